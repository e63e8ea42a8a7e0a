// jd_rules.h -- which of its built forms a sweep runs: host rules by dimension, precision,
// jump law and jump rate.  Plain C++ without CUDA, so that any host can check them.
#pragma once

#include "jd.h"

namespace jd {

// Mean number of jumps per step of a path.  A problem without a jump law has none, whatever
// its intensity says (a law may be set later, with the intensity already there).
inline double jump_rate(jd_jump_law law, double lambda, double T, int Nt) {
  return law == JD_JUMP_NONE ? 0.0 : lambda * T / (double)Nt;
}

// What the rules go by: the compiled dimension, the precision and the jumps.
struct FormKey {
  int D;
  bool f64;
  bool one_jump;   // steps with one jump take the short path (one_jump of the kernels): the
                   // slot's words lie as compiled for D, and the law is additive for d > 2
  double rate;     // jump_rate
};
inline FormKey form_key(int D, bool f64, const jd_problem_desc &q) {
  const bool packed = (q.d + 1) / 2 == (D + 1) / 2;
  return FormKey{D, f64, packed && (D <= 2 || q.jump_law != JD_JUMP_KS),
                 jump_rate(q.jump_law, q.lambda, q.T, q.Nt)};
}

// Chunk length: the records hold a lane's jumps of a chunk but in rare chunks, and a pass of
// slot draws serves many lanes.
inline int fwd_chunk_len(double rate, int most) {
  const int n = rate <= 0.015 ? 16 : rate <= 0.03 ? 8 : 4;
  return n < most ? n : most;
}

// Whether a sweep takes its steps in chunks, by the jump rate per step.  The store sweep and
// every FP64 sweep gain or tie at any rate; the other FP32 sweeps pay about 6% for the
// chunks' passes without jumps and gain from about lambda dt = 0.005 on.  One launch at M =
// 2^20, N_t = 160, d = 2 FP32, step by step -> in chunks, in ms:
//   lambda dt          0            0.002         0.01          0.05          0.2           0.4
//   cost          0.91 -> 0.97  1.01 -> 1.06  1.32 -> 1.23  2.33 -> 1.94  5.88 -> 3.27  9.96 -> 7.08
//   store         1.11 -> 1.04  1.21 -> 1.15  1.56 -> 1.38  2.66 -> 2.24  6.38 -> 3.83  10.5 -> 8.48
//   checkpoints   0.94 -> 0.99  1.02 -> 1.09  1.32 -> 1.25  2.30 -> 1.97  5.97 -> 3.34  10.1 -> 7.55
//   store, pair   1.25 -> 1.22  1.38 -> 1.39  1.82 -> 1.79  4.16 -> 3.03  12.9 -> 6.65  21.9 -> 15.7
//   ckpt., pair   1.11 -> 1.15  1.21 -> 1.27  1.59 -> 1.51  3.16 -> 2.44  10.1 -> 4.69  18.4 -> 11.9
//   recompute     1.26 -> 1.35  1.39 -> 1.47  1.80 -> 1.70  3.18 -> 2.75  12.1 -> 12.1  23.7 -> 22.1
//   adjoint (replay)
// (double precision, M = 2^15: store sweep 1.17 -> 1.17, 1.30 -> 1.28, 1.68 -> 1.49, 2.68 ->
// 2.17, 4.32 -> 4.14 ms up to 0.2.)  Between 0.004 and 0.007 the forms are within 3%.
constexpr double FWD_CHUNK_RATE = 0.006;
// What a launch runs: a sweep without stored states, the single store sweep, the replay of the
// recompute adjoint.
enum SweepKind { SWEEP_PLAIN, SWEEP_STORE, SWEEP_REPLAY };

// d > 2: whether a one-jump step's slot draws are the whole warp's (coop_slot0_draws).  A lane
// alone draws with its warp waiting; the warp-wide form costs the steps without jumps a
// ballot and registers, and takes the jump lanes one after another, so it pays between a
// lowest and a highest jump rate per step.  One launch, N_t = 160, one lane -> warp, in ms:
//   lambda dt                        0              0.002          0.01           0.05
//   FP32 d = 8  M = 200,003  cost    0.65 -> 0.67   0.75 -> 0.71   1.04 -> 0.87   2.45 -> 1.78
//                            store   0.71 -> 0.78   0.80 -> 0.83   1.13 -> 1.01   2.51 -> 2.22
//                            replay  1.04 -> 1.08   1.37 -> 1.20   2.81 -> 2.00   6.24 -> 5.08
//   FP32 d = 4               cost    0.34 -> 0.37   0.38 -> 0.40   0.50 -> 0.50   0.89 -> 0.94
//                            replay  0.57 -> 0.57   0.63 -> 0.61   0.81 -> 0.76   1.76 -> 1.57
//   FP64 d = 8  M = 16,000   store   1.86 -> 1.86   2.20 -> 2.00   3.08 -> 2.50   5.63 -> 4.20
//   FP64 d = 4               store   0.87 -> 0.88   1.02 -> 0.94   1.44 -> 1.20   2.53 -> 2.15
// (at 0.2 the warp-wide FP32 sweeps are slower again: d = 8 store 6.7 against 5.4.)  Where no
// step takes the one-jump path the form only costs: Keilson-Storer d = 8, FP32, M = 2^17, store
// sweep 1.17 -> 1.33 ms at 0.01, 1.52 -> 1.83 at 0.02, cost 1.07 -> 1.17 and 1.47 -> 1.63.
inline bool coop_slots(const FormKey &f, SweepKind kind) {
  if (!f.one_jump) return false;
  if (f.f64) return f.rate > 0.0005 && f.rate <= 0.1;
  if (f.D == 8) return f.rate > (kind == SWEEP_STORE ? 0.005 : 0.0015) && f.rate <= 0.08;
  return kind == SWEEP_REPLAY ? f.rate > 0.003 && f.rate <= 0.08 : f.rate > 0.01 && f.rate <= 0.03;
}

// The form of a forward sweep or replay: in chunks (d <= 2) or with warp-wide slot draws (d > 2).
inline bool fwd_chunks(const FormKey &f, SweepKind kind) {
  if (f.D > 2) return coop_slots(f, kind);
  return f.f64 || kind == SWEEP_STORE || f.rate > FWD_CHUNK_RATE;
}

// Parameter gradients: the jump draws are kept up to this jump rate per step; beyond it a
// segment's jumps outgrow the records and most steps have several (M = 2^19, N_t = 160, d = 2
// FP32, regenerated -> kept: 0.80 -> 0.86 ms without jumps, 1.36 -> 0.94 at 0.002, 3.29 ->
// 1.16 at 0.01, 7.82 -> 4.16 at 0.05, 10.9 -> 9.8 at 0.1, 16.0 -> 20.0 at 0.2).
constexpr double THETA_KEEP_RATE = 0.12;
inline bool theta_keeps(const FormKey &f) { return f.rate <= THETA_KEEP_RATE; }

}  // namespace jd
