// jd_rules.h -- which of its built forms a sweep runs: host rules by dimension, precision,
// jump law and jump rate.  Plain C++ without CUDA, so that any host can check them.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>

#include "jd.h"

namespace jd {

// Mean number of jumps per step of a path.  A problem without a jump law has none, whatever
// its intensity says (a law may be set later, with the intensity already there).
inline double jump_rate(jd_jump_law law, double lambda, double T, int Nt) {
  return law == JD_JUMP_NONE ? 0.0 : lambda * T / (double)Nt;
}

// Keilson-Storer, d <= 2: whether a step with one jump takes the short path.  Where a third of
// the jump steps and more have several jumps, a warp pays for both routines at nearly every step:
// all through build_jump_step the FP32 cost sweep took 3.10 against 3.46 ms at lambda dt = 0.55,
// the store sweep 3.24 against 3.59, at 1.2 4.46 against 4.87 (M = 2^18, N_t = 160).
inline bool ks_one_jump(double rate) { return rate <= 0.5; }

// What the rules go by: the compiled dimension, the precision and the jumps.
struct FormKey {
  int D;
  bool f64;
  bool one_jump;   // a step with one jump can take the short path: the slot's words lie as
                   // compiled for D, and the law is additive for d > 2
  bool ks;         // Keilson-Storer law
  double rate;     // jump_rate
  int64_t M;       // paths
};
inline FormKey form_key(int D, bool f64, const jd_problem_desc &q) {
  const bool packed = (q.d + 1) / 2 == (D + 1) / 2;
  const bool ks = q.jump_law == JD_JUMP_KS;
  return FormKey{D, f64, packed && (D <= 2 || !ks), ks, jump_rate(q.jump_law, q.lambda, q.T, q.Nt), q.M};
}

// Chunk length: the records hold a lane's jumps of a chunk but in rare chunks, and a pass of
// slot draws serves many lanes.
inline int fwd_chunk_len(double rate, int most) {
  const int n = rate <= 0.015 ? 16 : rate <= 0.03 ? 8 : 4;
  return n < most ? n : most;
}

// What a launch runs: a forward sweep (cost, checkpoints, stored states; the last two also for a
// pair of controls) or the replay of the recompute adjoint.
enum SweepKind { SWEEP_COST, SWEEP_CKPT, SWEEP_STORE, SWEEP_STORE_PAIR, SWEEP_CKPT_PAIR, SWEEP_REPLAY };

// Whether the steps with one jump take the short path.
inline bool one_jump_path(const FormKey &f) { return f.one_jump && (!f.ks || ks_one_jump(f.rate)); }

// d > 2: whether a one-jump step's slot draws are the whole warp's (coop_slot0_draws).  A lane
// alone draws with its warp waiting; the warp-wide form costs the steps without jumps a
// ballot and registers, and takes the jump lanes one after another, so it pays between a
// lowest and a highest jump rate per step.  One launch, N_t = 160, one lane -> warp, in ms:
//   lambda dt                        0              0.002          0.01           0.05
//   FP32 d = 8  M = 200,003  cost    0.65 -> 0.67   0.75 -> 0.71   1.04 -> 0.87   2.45 -> 1.78
//                            store   0.71 -> 0.78   0.80 -> 0.83   1.13 -> 1.01   2.51 -> 2.22
//                            replay  1.04 -> 1.08   1.37 -> 1.20   2.81 -> 2.00   6.24 -> 5.08
//   FP32 d = 4               cost    0.34 -> 0.37   0.38 -> 0.40   0.51 -> 0.50   0.89 -> 0.94
//                            replay  0.57 -> 0.57   0.63 -> 0.61   0.81 -> 0.76   1.76 -> 1.57
//   FP64 d = 8  M = 16,000   store   1.86 -> 1.86   2.20 -> 2.00   3.08 -> 2.50   5.63 -> 4.20
//   FP64 d = 4               store   0.87 -> 0.88   1.02 -> 0.94   1.44 -> 1.20   2.53 -> 2.15
// (at 0.2 the warp-wide FP32 sweeps are slower again: d = 8 store 6.7 against 5.4.)  FP32 d = 4
// gains only where the chip is full: replay at 0.02 0.173 -> 0.178 ms for M = 8000, 0.212 -> 0.207
// at 20,000, 0.283 -> 0.261 at 40,000 (at 0.05 0.256 -> 0.285, 0.330 -> 0.332, 0.434 -> 0.398);
// cost at 0.02 0.126 -> 0.135, 0.151 -> 0.157, 0.199 -> 0.197, 0.632 -> 0.609 at 200,003, and
// between 0.01 and 0.03 only; its store sweep not for every size even there (0.718 -> 0.700 at
// 200,003, but 0.271 -> 0.281 at 50,001 and 0.03).  Where no step takes the one-jump path the form
// only costs: Keilson-Storer d = 8, FP32, M = 2^17, store sweep 1.17 -> 1.33 ms at 0.01, 1.52 ->
// 1.83 at 0.02, cost 1.07 -> 1.17 and 1.47 -> 1.63.
inline bool coop_slots(const FormKey &f, SweepKind kind) {
  if (!f.one_jump) return false;
  if (f.f64) return f.rate > 0.0005 && f.rate <= 0.1;
  if (f.D == 8) return f.rate > (kind == SWEEP_STORE ? 0.005 : 0.0015) && f.rate <= 0.08;
  if (kind == SWEEP_REPLAY) return f.M >= 152 * 128 && f.rate > 0.003 && f.rate <= 0.08;
  return (kind == SWEEP_COST || kind == SWEEP_CKPT) && f.M >= 152 * 256 && f.rate > 0.01 && f.rate <= 0.025;
}

// d <= 2: whether a sweep takes its steps in chunks, by the jump rate per step.  The chunks'
// passes cost a little where almost nothing jumps, and at high rates most jump steps have three
// jumps or more and go to the general routine either way.  One launch at N_t = 160, step by
// step -> in chunks, in ms (pair: checkpoints; FP32 M = 2^18, but 2^20 up to 0.006, pairs up to
// 0.002; FP64 2^15):
//   lambda dt              0             0.002         0.006         0.1           0.3           0.5           0.6
//   FP32 d = 1  cost       0.85 -> 0.85  0.95 -> 0.98  1.12 -> 1.09  0.96 -> 0.62  2.32 -> 1.30  3.12 -> 2.52  3.37 -> 3.10
//               ckpt.      0.83 -> 0.88  0.93 -> 1.00  1.10 -> 1.11  0.95 -> 0.63  2.34 -> 1.31  3.16 -> 2.50  3.42 -> 3.09
//               store      1.07 -> 0.87  1.17 -> 1.03  1.36 -> 1.19  1.06 -> 0.70  2.46 -> 1.47  3.24 -> 2.66  3.50 -> 3.22
//               pair       0.94 -> 0.90  1.05 -> 1.06  0.35 -> 0.33  1.45 -> 0.77  4.35 -> 2.18  6.13 -> 4.26  6.66 -> 5.46
//               replay     1.08 -> 1.09  1.19 -> 1.19  1.40 -> 1.29  1.25 -> 1.19  4.14 -> 3.90  5.95 -> 5.82  6.57 -> 6.55
//   FP32 d = 2  cost       0.93 -> 0.89  1.02 -> 0.99  1.18 -> 1.08  0.94 -> 0.62  2.31 -> 1.35  3.11 -> 2.58  3.36 -> 3.21
//               store      1.12 -> 0.98  1.22 -> 1.10  1.40 -> 1.22  1.05 -> 0.73  2.44 -> 1.68  3.23 -> 3.06  3.47 -> 3.71
//               pair       1.08 -> 1.09  1.19 -> 1.21  0.38 -> 0.37  1.40 -> 0.85  4.11 -> 2.42  5.68 -> 4.89  6.19 -> 6.21
//               replay     1.27 -> 1.25  1.41 -> 1.36  1.64 -> 1.49  1.45 -> 1.54  4.98 -> 5.22  7.30 -> 7.27  8.12 -> 7.99
//   FP64 d = 1  store      0.61 -> 0.61  0.74 -> 0.70  0.93 -> 0.75  2.38 -> 1.61  4.12 -> 3.08  5.03 -> 4.82  5.36 -> 5.67
//   FP64 d = 2  store      0.81 -> 0.79  0.91 -> 0.89  1.09 -> 0.99  2.46 -> 2.02  4.04 -> 4.07  4.83 -> 5.35  5.13 -> 5.84
//               replay     1.05 -> 1.05  1.19 -> 1.18  1.41 -> 1.32  3.23 -> 2.87  6.76 -> 6.90  8.76 -> 9.30  9.49 -> 10.2
//   FP64 KS     store      0.71 -> 0.79  0.84 -> 0.89  1.04 -> 0.96  2.68 -> 1.94  4.73 -> 4.42  5.79 -> 5.92  6.19 -> 6.48
// (The FP32 replay of d = 2 also takes 0.73 -> 0.58 at 0.03, 3.95 -> 3.78 at 0.07 and 12.1 -> 13.4
// at 0.2, M = 2^20: 5 blocks of it fit an SM in chunks, 6 step by step.  While all its blocks are
// resident it is faster in chunks at every rate: at 0.2 0.744 -> 0.622 for M = 13,000, 1.37 -> 1.21
// at 80,000, but 1.55 -> 2.11 at 110,000.  At 1.2 the FP32 store sweep of d = 2 takes 4.6 -> 6.3.)
inline bool chunk_steps(const FormKey &f, SweepKind kind) {
  double lo = 0.0, hi = 0.5;
  if (f.f64) {
    if (f.D == 2) hi = f.ks ? 0.45 : 0.3;   // Keilson-Storer at 0.4 5.27 -> 5.12
    if (f.ks && kind != SWEEP_REPLAY) lo = 0.004;
  } else {
    if (f.D == 2 && kind == SWEEP_REPLAY && f.M > 152 * 5 * 128) hi = 0.08;
    if (f.D == 1 && (kind == SWEEP_COST || kind == SWEEP_CKPT)) lo = 0.005;
  }
  return f.rate >= lo && f.rate <= hi;
}

// The form of a forward sweep or replay: in chunks (d <= 2) or with warp-wide slot draws (d > 2).
inline bool fwd_chunks(const FormKey &f, SweepKind kind) {
  return f.D > 2 ? coop_slots(f, kind) : chunk_steps(f, kind);
}

// Draw pre-pass: a problem with d <= 2 of few paths (its sweeps are latency-bound: each
// thread's steps are a chain of dependent operations, and the Philox and Box-Muller of every
// step sit on that chain) takes its main-stream draws in one parallel kernel first, when
// their buffers stay small.  Its sweeps then run few lanes per warp (SPREAD_LANES), which costs
// them instruction issue as the paths grow (a pair's two controls are sweeps of their own), and
// save more where more steps jump.  The limits per kind of sweep and jump rate lie below the path
// count from which the other form is faster; that count, measured at N_t = 200 with the draws held
// (Keilson-Storer as d = 2 where it is not given):
//   lambda dt          0       0.002   0.007   0.015   0.03    0.07    0.2
//   FP32 cost   d = 1  7200    7800    7500    10800   11300   13000+  13000+
//               d = 2  3800    5000    7000    9100    10200   11000   11000
//        ckpt.  d = 1  7400    7800    6300    10200   10700   13000+  13000+
//               d = 2  none    none    2900    5500    7900    10200   10600
//        store  d = 1  none    none    3500    8100    9600    10700   12100
//               d = 2  none    none    4800    8900    8400    10500   13000+
//        store, d = 1  none    none    2600    5100    6900    8300    10400
//        pair   d = 2  none    1100    2500    5100    7000    8200    10400
//        ckpt., d = 1  none    3100    5000    7700    8500    9900    11200
//        pair   d = 2  1200    1800    3700    5600    7600    9000    10400
//   FP64 single d = 1  9300    10100   10600   10900   11300   11700   10200
//               d = 2  6100    6800    7200    7600    7900    8400    9700
//        pair   d = 1  6000    6500    6900    7200    7400    7400    7200
//               d = 2  4100    4600    5000    5300    5700    6000    6300
//               KS     5000    5900    6300    6300    6400    6400    6600
// ("none": the other form is faster at 1000 paths already: FP32 d = 1 store sweep of 3000 paths
// at 0.0005 45 against 58 us, its pair 48 against 74.)
inline int64_t pre_max_paths(const FormKey &f, SweepKind kind) {
  if (f.D > 2) return 0;
  // multiples of 152 paths (an SM's share) by rate: below 0.004, 0.01, 0.02, 0.05, 0.1, above
  static const unsigned char f32[5][2][6] = {
      {{40, 40, 64, 64, 64, 64}, {24, 40, 56, 64, 64, 64}},    // cost: d = 1, d = 2
      {{40, 40, 64, 64, 64, 64}, {0, 16, 32, 48, 64, 64}},     // checkpoints
      {{0, 20, 48, 56, 64, 64}, {0, 28, 52, 52, 64, 64}},      // store
      {{0, 16, 32, 44, 52, 64}, {0, 16, 32, 44, 52, 64}},      // store, pair
      {{16, 32, 48, 52, 64, 64}, {8, 24, 36, 48, 56, 64}}};    // checkpoints, pair
  const int c = f.rate < 0.004 ? 0 : f.rate < 0.01 ? 1 : f.rate < 0.02 ? 2 : f.rate < 0.05 ? 3 : f.rate < 0.1 ? 4 : 5;
  if (f.f64) {
    if (kind != SWEEP_STORE_PAIR && kind != SWEEP_CKPT_PAIR) return 152 * (f.D == 1 ? 56 : 40);
    static const unsigned char pair[3][6] = {
        {40, 44, 44, 48, 48, 46}, {28, 32, 32, 32, 36, 40}, {32, 40, 40, 40, 40, 40}};   // d = 1, d = 2, KS
    return 152 * (int64_t)pair[f.ks && f.D == 2 ? 2 : f.D - 1][c];
  }
  return 152 * (int64_t)f32[kind][f.D - 1][c];
}
// The largest of the limits.
inline int64_t pre_top_paths(int D, bool f64) { return D > 2 ? 0 : 152 * (!f64 ? 64 : D == 1 ? 56 : 40); }

// Parameter gradients: whether the recompute adjoint keeps its jump steps' draws (adj_theta_body;
// built for d <= 2 and FP32 d = 4).  Without jumps its passes cost a little; at high rates a
// segment's jumps outgrow the records and most jump steps have several.  One launch at N_t =
// 160, regenerated -> kept, in ms (FP32 d <= 2 M = 2^20, d = 4 2^17; FP64 2^15):
//   lambda dt    0             0.0002        0.0005*       0.02          0.1           0.12          0.14          0.17
//   FP32 d = 1   1.29 -> 1.33  1.39 -> 1.34  1.48 -> 1.36  7.63 -> 2.70  17.1 -> 15.1  18.7 -> 18.4  20.2 -> 21.7  22.4 -> 26.2
//        d = 2   1.55 -> 1.56  1.66 -> 1.58  1.75 -> 1.59  9.01 -> 2.93  20.0 -> 17.6  21.8 -> 21.7  23.7 -> 25.7  26.3 -> 31.2
//        KS      1.53 -> 1.55  1.66 -> 1.56  1.75 -> 1.58  9.72 -> 3.09  21.8 -> 20.4  24.0 -> 25.3  26.2 -> 30.0  29.2 -> 36.4
//        d = 4   0.57 -> 0.64  0.60 -> 0.64  0.64 -> 0.64  5.01 -> 1.98  11.3 -> 11.6  12.6 -> 13.9  13.8 -> 16.0  15.3 -> 18.7
//   FP64 d = 1   0.83 -> 0.83  0.93 -> 0.86  0.99 -> 0.87  3.57 -> 1.64  6.70 -> 4.85  7.22 -> 6.04  7.60 -> 6.82  8.17 -> 7.90
//        d = 2   1.22 -> 1.22  1.31 -> 1.25  1.36 -> 1.27  3.89 -> 2.43  6.86 -> 5.50  7.33 -> 6.57  7.68 -> 7.34  8.14 -> 8.34
// (* 0.0004; d = 4 at 0.07 9.16 -> 7.82.)
inline bool theta_keeps(const FormKey &f) {
  if (f.D > 2) return f.rate > 0.0004 && f.rate <= 0.09;
  return f.rate > 0.0 && f.rate <= (f.f64 ? 0.16 : f.ks ? 0.11 : 0.12);
}

// Feedback forward sweep: whether a step with one jump takes its slot's draws in straight code
// beside the plan's loops of the other jump steps.  At high rates a warp runs both at nearly every
// step, sooner where a ring's lanes wait for one another (ring_kind 2 and 3); in FP64 the loops
// cost no more than the straight code at any rate.  Forward without stored states, N_t = 60,
// loops -> straight, in us (FP32 M = 2^18, FP64 2^15):
//   lambda dt                   0.02          0.1           0.15          0.2           0.3           1
//   FP32 4 x 4                  396 -> 282    641 -> 487    704 -> 604    765 -> 720    880 -> 927    1439 -> 1578
//        10 x 10                522 -> 417    820 -> 675    897 -> 800    975 -> 934    1122 -> 1173  1832 -> 1970
//        16 x 16                813 -> 728    1205 -> 1094  1318 -> 1246  1428 -> 1396  1641 -> 1684  2677 -> 2785
//        4 x 4, rings of 200    491 -> 334    686 -> 648    762 -> 801    828 -> 890    939 -> 1034   1514 -> 1652
//        16 x 16, rings of 200  999 -> 826    1392 -> 1351  1537 -> 1565  1650 -> 1722  1855 -> 1951  2913 -> 3045
//   FP64 10 x 10                4517 -> 4506  6449 -> 6537  7090 -> 7238  7563 -> 7817  8769 -> 9144  14026 -> 14455
inline bool fb_one_slot(bool f64, int ring_kind, double rate) {
  return !f64 && rate <= (ring_kind <= 1 ? 0.25 : 0.13);
}

// Feedback jump log: records per path (at most 1024; 0: no jumps).  The expected records and a
// wide Poisson margin; in FP32 only of the steps that are logged: a path's log closes at its first
// step with three jumps (probability p3 per step) and a logged step has one or two records, so at
// lambda dt = 0.5 and N_t = 1000 the log holds 69 steps on average and 1000 steps' records would
// be mostly never written.  Four times the mean number of logged steps covers 98% of the paths.
inline int fb_log_capacity(const jd_problem_desc &q) {
  const double r = jump_rate(q.jump_law, q.lambda, q.T, q.Nt);
  if (!(r > 0.0)) return 0;
  double steps = q.Nt, most = 1024.0;
  if (q.prec == JD_FP32) {
    const double p3 = r < 0.05 ? r * r * r / 6.0 * (1.0 - 0.75 * r) : 1.0 - std::exp(-r) * (1.0 + r + 0.5 * r * r);
    if (p3 * q.Nt > 1e-3) steps = std::min(steps, std::ceil(4.0 * (1.0 - std::pow(1.0 - p3, q.Nt)) / p3));
    most = std::min(most, 2.0 * steps);
  }
  const double mean = r * steps;
  return (int)std::min(most, std::ceil(mean + 6.0 * std::sqrt(mean) + 8.0));
}

// Whether the device has room for a feedback jump log of that many bytes: another problem or
// another library on the device cannot ask for its memory back, so it takes a quarter of what is
// free at most.
inline bool fb_log_fits(size_t bytes, size_t free_bytes) { return bytes <= free_bytes / 4; }

}  // namespace jd
