// rkck45_relay.cu -- Keller-Miksis phase mode for ensembles of at most two warps
// of systems per SM: the trial of 32 systems runs in seven or eight warps.
//
// Such an ensemble takes as long as its longest system, one trial after the other,
// and a lone warp's FP64 operations, dependent or not, take 64 cycles each: 190 of
// them in the main warp of rkck45_teams.cu make its trial 15,500 cycles, while three
// of the SM's four FP64 pipes stand idle.  Here the chain that a trial cannot do
// without stays in the main warp, 15 operations a stage (the new y2, the reciprocal
// 1 / (y1 D), the terms of the acceleration that it multiplies), and the rest runs
// beside it in warps of other sub-partitions:
//   - sums: the sums over the slopes, in order, up to the newest slope, the next
//     stage's y1 and the error estimate;
//   - power: the polytropic power, for stage 2 also the numerator, and at the end the
//     error norm and the next step;
//   - numerator, factors: what the acceleration takes from y2, with and without the
//     power;
//   - drive (two, three of them with two frequencies): the stages' drives and what
//     the error norm needs besides the error.
// Every operation is that of ck_phased_kernel, so are the bits.  A trial takes 10,200
// cycles (two frequencies 11,000; Dormand-Prince, whose error waits for the last
// slope, 10,900).  Milliseconds in teams of three warps and here: 1,073 systems x 2
// periods 32.5 / 20.9, 4,608 frequencies x 3 48.8 / 31.3, two frequencies and
// Dormand-Prince (6,097 x 2) 48.3 / 34.5; two relays on every SM: 9,700 x 2 32.6 /
// 21.9.  Three would not fit the registers; from there on the teams keep more of
// the pipes busy.
//
// What bounds a trial now: stages 3 to 6 take 1,390 cycles each, 950 of them FP64
// issue of the chain, 30 the reciprocal's seed, the rest a wait and two posts; stage 2
// (2,300) waits for its power and drive, 900 cycles of dependent integer products
// that need the new step; the end (600 after the last slope) for error norm and step.
// What was tried: messages of value and trial number in one 128-bit word, polled (a
// round trip of 360 cycles against 260 through mbarriers); a barrier per kind of
// message (1,900 cycles a stage: each wait costs some 100 cycles, so everything that
// the main warp needs arrives on one); the main warp's stages unrolled (1,600:
// instruction fetch).
//
// Messages go through shared memory; a barrier of the mailbox has one phase per
// trial, which ends when all its senders have posted.  The main warp starts a trial
// only when it has received everything of the one before, so no barrier is ever more
// than one phase ahead of a receiver and no slot is written before it has been read.
// Waits are bounded; when one of the main warp's expires, its systems and all it
// still claims are retired with ENS_SYS_TIMEOUT, and a helper whose wait expires
// leaves.
#include "common.cuh"
#include "controller.cuh"
#include "mailbox.cuh"
#include "rhs.cuh"

namespace ens {

namespace {

// barriers of a relay; index s - 2 for stage s = 2..7
enum : int {
  kSlope = 0, kPow = 6, kAll = 12, kPower = 18, kStart = 24, kSecond = 25, kErr0 = 26, kErr = 27, kCtl = 28, kBars = 29
};

struct __align__(16) Relay {
  double x[6][32], v[6][32], k[6][32];   // a stage's state; the second slope component of the stage before
  double n[6][32];                       // the acceleration's numerator as far as it needs only the power
  double b[6][32], o[6][32], e[6][32], q[6][32];   // factors of its other terms
  double pv[6][32];                      // sum over the slopes known so far for the next stage
  double fs[5][32], fc[5][32];           // drives of stages 2..6
  double g[6][32];                       // the power of y1
  double t[32], h[32], y[2][32], a31k1x[32];
  double f2[2][32];                      // sine and cosine of stage 2's second frequency
  double err[2][32], r0[32], w1[32];     // error estimate; ratio of its first component, weight of the second
  double dt[32];                         // the next step, negative after a rejection
  long long sys[32];                     // the lane's system, -1 when none are left
  unsigned long long bar[kBars];
};

// weight of slope i in row r: rows 2..6 the stages, 7 the new state, 8 the error estimate
template <int PAIR>
__device__ constexpr double weight(int r, int i) {
  if (PAIR == kDormandPrince) {
    constexpr double A[7][7] = {{dp::a21, 0, 0, 0, 0, 0, 0},
                                {dp::a31, dp::a32, 0, 0, 0, 0, 0},
                                {dp::a41, dp::a42, dp::a43, 0, 0, 0, 0},
                                {dp::a51, dp::a52, dp::a53, dp::a54, 0, 0, 0},
                                {dp::a61, dp::a62, dp::a63, dp::a64, dp::a65, 0, 0},
                                {dp::b1, 0, dp::b3, dp::b4, dp::b5, dp::b6, 0},
                                {dp::e1, 0, dp::e3, dp::e4, dp::e5, dp::e6, dp::e7}};
    return A[r - 2][i - 1];
  }
  constexpr double A[7][7] = {{ck::a21, 0, 0, 0, 0, 0, 0},
                              {ck::a31, ck::a32, 0, 0, 0, 0, 0},
                              {ck::a41, ck::a42, ck::a43, 0, 0, 0, 0},
                              {ck::a51, ck::a52, ck::a53, ck::a54, 0, 0, 0},
                              {ck::a61, ck::a62, ck::a63, ck::a64, ck::a65, 0, 0},
                              {ck::b1, 0, ck::b3, ck::b4, 0, ck::b6, 0},
                              {ck::d1, 0, ck::d3, ck::d4, ck::d5, ck::d6, 0}};
  return A[r - 2][i - 1];
}
// by pair and stage - 2: weight of the newest slope in the stage after, time of the stage in steps
static __constant__ double kNewest[2][5] = {{ck::a32, ck::a43, ck::a54, ck::a65, ck::b6},
                                            {dp::a32, dp::a43, dp::a54, dp::a65, dp::b6}};
template <int PAIR>
__device__ __forceinline__ double stage_time(int stage) {
  if (PAIR == kDormandPrince)
    return stage == 2 ? dp::c2 : stage == 3 ? dp::c3 : stage == 4 ? dp::c4 : stage == 5 ? dp::c5 : 1.0;
  return stage == 2 ? ck::c2 : stage == 3 ? ck::c3 : stage == 4 ? ck::c4 : stage == 5 ? ck::c5 : ck::c6;
}

// FP64 operations that keep their place among the waits
__device__ __forceinline__ double vfma(double a, double b, double c) {
  double r;
  asm volatile("fma.rn.f64 %0, %1, %2, %3;" : "=d"(r) : "d"(a), "d"(b), "d"(c));
  return r;
}
__device__ __forceinline__ double vmul(double a, double b) {
  double r;
  asm volatile("mul.rn.f64 %0, %1, %2;" : "=d"(r) : "d"(a), "d"(b));
  return r;
}
__device__ __forceinline__ double vadd(double a, double b) {
  double r;
  asm volatile("add.rn.f64 %0, %1, %2;" : "=d"(r) : "d"(a), "d"(b));
  return r;
}

__device__ __forceinline__ bool all(bool ok) { return __all_sync(0xffffffffu, ok); }
// the next phase of a barrier that has one per trial
__device__ __forceinline__ bool await_trial(Relay& m, int bar, uint32_t trial) { return await(&m.bar[bar], trial); }
__device__ __forceinline__ bool all_await(Relay& m, int bar, uint32_t trial) {
  return all(await(&m.bar[bar], trial));
}

// the system of the lane, reloaded when it changes; false when none are left
template <class Sys>
__device__ __forceinline__ bool follow(const AdaptArgs& a, const Relay& m, int lane, Sys& s, long long& cur) {
  const long long sys = m.sys[lane];
  if (sys != cur) {
    if (sys < 0) return false;
    cur = sys;
    s.load(a.params, a.n, cur);
  }
  return true;
}

// powers of the stages' y1, then error norm and step factor
template <class Sys>
__device__ __forceinline__ void power_warp(const AdaptArgs& a, Relay& m) {
  const int lane = threadIdx.x & 31;
  Sys s;
  long long cur = -2;
  for (uint32_t trial = 0;; ++trial) {
    // stage 2 waits for its power, so its numerator is made here too
    double A = 0.0, o = 0.0;
#pragma unroll 1
    for (int k = 0; k < 6; ++k) {
      if (!all_await(m, k == 0 ? kSlope : kPow + k, trial)) return;
      const double x = m.x[k][lane];
      if (k == 0) {
        if (!all(follow(a, m, lane, s, cur))) return;
        const double v = m.v[0][lane];
        A = vfma(s.C1, v, s.C0);
        o = vfma(s.C9, v, 1.0);
      }
      const double g = s.early_power(x);
      if (k == 0) {
        m.n[0][lane] = vfma(-s.C2, o, vmul(A, g));
        post(&m.bar[kAll]);
      } else {
        m.g[k][lane] = g;
        post(&m.bar[kPower + k]);
      }
    }
    const double h = m.h[lane];
    if (!all_await(m, kErr, trial)) return;
    const double E = nnmax(m.r0[lane], err_ratio(m.err[1][lane], m.w1[lane]));
    const double hf = h * step_factor(E);
    m.dt[lane] = accept(E) ? nnmax(nnmin(hf, a.dt_max), a.dt_min) : -hf;
    post(&m.bar[kCtl]);
  }
}

// the numerator as far as it needs only the power
template <class Sys>
__device__ __forceinline__ void numerator_warp(const AdaptArgs& a, Relay& m) {
  const int lane = threadIdx.x & 31;
  Sys s;
  long long cur = -2;
  for (uint32_t trial = 0;; ++trial) {
    if (!all_await(m, kSlope, trial) || !all(follow(a, m, lane, s, cur))) return;
#pragma unroll 1
    for (int k = 1; k < 6; ++k) {
      if (!all_await(m, kSlope + k, trial)) return;
      const double v = m.v[k][lane];
      const double A = vfma(s.C1, v, s.C0), o = vfma(s.C9, v, 1.0);
      if (!all_await(m, kPower + k, trial)) return;
      m.n[k][lane] = vfma(-s.C2, o, vmul(A, m.g[k][lane]));
      post(&m.bar[kAll + k]);
    }
  }
}

// drives of the stages: warp 0 those of stages 2, 4 and 6, warp 1 of stages 3 and 5; of
// two frequencies warp 0 takes stages 2 and 4, warp 1 the second one of stage 2, then
// stages 5 and 6, warp 2 stage 3.  Warps 0 and 1 end with what the
// error norm takes from the first component and the weight of the second.
template <class Sys, int PAIR>
__device__ __forceinline__ void drive_warp(const AdaptArgs& a, Relay& m, int which) {
  const int lane = threadIdx.x & 31;
  Sys s;
  long long cur = -2;
  for (uint32_t trial = 0;; ++trial) {
    if (!all_await(m, kStart, trial) || !all(follow(a, m, lane, s, cur))) return;
    const double t = m.t[lane], h = m.h[lane];
    // one sine and cosine per iteration, so that its code is there once
    int stage = which == 0 || (Sys::kDual && which == 1) ? 2 : 3;
    if (!Sys::kDual) {
      // stage 2 waits for its drive: a polynomial in either warp
      const double ts = fma(stage_time<PAIR>(2), h, t);
      bool sine;
      const double z = which == 0 ? sincos2pi_half<true>(ts, &sine) : sincos2pi_half<false>(ts, &sine);
      (sine ? m.fs : m.fc)[0][lane] = (sine ? s.C5 : s.C7) * z;
      post(&m.bar[kAll]);
      stage = which == 0 ? 4 : 3;
    }
    bool second = Sys::kDual && which == 1;
    typename Sys::Drive d{};
#pragma unroll 1
    while (stage <= 6) {
      const double ts = fma(stage_time<PAIR>(stage), h, t);
      double sn, cs;
      sincos2pi_fx(second ? fma(s.C11, ts, s.C12f) : ts, &sn, &cs);
      if (!second) {
        d = {s.C5 * sn, s.C7 * cs};
        if (Sys::kDual) {
          if (stage > 2) {
            second = true;
            continue;
          }
          if (!all_await(m, kSecond, trial)) return;
          d = {fma(s.C6, m.f2[0][lane], d.fs), fma(s.C8, m.f2[1][lane], d.fc)};
        }
      } else if (stage == 2) {
        m.f2[0][lane] = sn;
        m.f2[1][lane] = cs;
        post(&m.bar[kSecond]);
        stage = 5;
        second = false;
        continue;
      } else {
        d = {fma(s.C6, sn, d.fs), fma(s.C8, cs, d.fc)};
        second = false;
      }
      m.fs[stage - 2][lane] = d.fs;
      m.fc[stage - 2][lane] = d.fc;
      post(&m.bar[kAll + stage - 2]);
      stage = Sys::kDual ? (stage == 2 ? 4 : stage == 5 ? 6 : 7) : stage + 2;
    }
    if (which == 0) {
      if (!all_await(m, kPow + 5, trial)) return;
      const double w = err_weight(m.y[0][lane], m.x[5][lane], a.rtol, a.atol);
      if (!all_await(m, kErr0, trial)) return;
      m.r0[lane] = nnmax(0.0, err_ratio(m.err[0][lane], w));
      post(&m.bar[kErr]);
    } else if (which == 1) {
      if (!all_await(m, kSlope + 5, trial)) return;
      m.w1[lane] = err_weight(m.y[1][lane], m.v[5][lane], a.rtol, a.atol);
      post(&m.bar[kErr]);
    }
  }
}

// factors of the numerator's other terms
template <class Sys>
__device__ __forceinline__ void factors_warp(const AdaptArgs& a, Relay& m) {
  const int lane = threadIdx.x & 31;
  Sys s;
  long long cur = -2;
  for (uint32_t trial = 0;; ++trial) {
#pragma unroll 1
    for (int k = 0; k < 6; ++k) {
      if (!all_await(m, kSlope + k, trial)) return;
      if (k == 0) {
        if (!all(follow(a, m, lane, s, cur))) return;
      }
      const double v = m.v[k][lane];
      const double b = vfma(s.C4, v, s.C3), e = vfma(s.C9h, v, 1.5), q = vmul(v, v), o = vfma(s.C9, v, 1.0);
      m.b[k][lane] = b;
      m.e[k][lane] = e;
      m.q[k][lane] = q;
      m.o[k][lane] = o;
      post(&m.bar[kAll + k]);
    }
  }
}

// sums over the slopes, in the order of the one-warp kernel
template <int PAIR>
__device__ __forceinline__ void sums_warp(const AdaptArgs& a, Relay& m) {
  const int lane = threadIdx.x & 31;
  for (uint32_t trial = 0;; ++trial) {
    double sv[9], sx[9], h = 0.0, y0 = 0.0;
#pragma unroll
    for (int s = 2; s <= 7; ++s) {
      if (!all_await(m, kSlope + s - 2, trial)) return;
      const double kv = m.k[s - 2][lane], kx = m.v[s - 2][lane];   // slopes s - 1 (second) and s (first component)
      if (s == 2) {
        if (!all(m.sys[lane] >= 0)) return;
        h = m.h[lane];
        y0 = m.y[0][lane];
        sx[3] = m.a31k1x[lane];
      }
      if (s <= 6) {
        // the next stage's y1, what is known of its y2, then the later rows
        m.x[s - 1][lane] = vfma(h, vfma(weight<PAIR>(s + 1, s), kx, sx[s + 1]), y0);
        post(&m.bar[kPow + s - 1]);
        if (s > 2) {
          sv[s + 1] = vfma(weight<PAIR>(s + 1, s - 1), kv, sv[s + 1]);
          m.pv[s - 2][lane] = sv[s + 1];
        }
        post(&m.bar[kAll + s - 2]);
        const double k1x = m.y[1][lane];
#pragma unroll
        for (int r = (s == 2 ? 4 : s + 2); r <= 8; ++r) {
          if (s == 2) {
            sv[r] = weight<PAIR>(r, 1) * kv;
            sx[r] = weight<PAIR>(r, 1) * k1x;
          } else if (weight<PAIR>(r, s - 1) != 0.0) {
            sv[r] = fma(weight<PAIR>(r, s - 1), kv, sv[r]);
          }
          if (weight<PAIR>(r, s) != 0.0) sx[r] = fma(weight<PAIR>(r, s), kx, sx[r]);
        }
      } else {
        sv[8] = vfma(weight<PAIR>(8, 6), kv, sv[8]);
        if (PAIR == kDormandPrince) {   // the main warp adds the last slope's term of the second component
          m.pv[5][lane] = sv[8];
          post(&m.bar[kAll + 5]);
          m.err[0][lane] = h * fma(weight<PAIR>(8, 7), kx, sx[8]);
          post(&m.bar[kErr0]);
        } else {
          m.err[1][lane] = vmul(h, sv[8]);
          post(&m.bar[kErr]);
        }
      }
      if (PAIR == kCashKarp && s == 6) {
        m.err[0][lane] = h * sx[8];
        post(&m.bar[kErr0]);
      }
    }
  }
}

template <class Sys, int PAIR>
__device__ __forceinline__ void main_warp(const AdaptArgs& a, Relay& m) {
  const int lane = threadIdx.x & 31;
  const double tau_end = a.t0 + a.phase_len;
  const uint64_t deadline = global_ns() + a.timeout_ns;
  uint32_t trial = 0;
  bool timed_out = false;
  Sys s;
  typename Sys::Drive d0, dn;  // drive at the phase start, at the end of the trial
  double y[2], k1v;            // state, first slope's second component (the first is y2)
  double tau = a.t0, rest = a.phase_len, dt = a.dt0, ymax = 0.0, ymin = 0.0;  // rest of the phase, > 0
  double a21k1x = 0.0, a21k1v = 0.0, a31k1x = 0.0, a31k1v = 0.0;
  int32_t ph = 0, st = 0;
  uint32_t trials = 0, nacc = 0, nrej = 0, nrhs = 0;
  bool fresh = true;           // the next trial's first stage counts as an evaluation

  auto start_system = [&](int64_t sys) {
    s.load(a.params, a.n, sys);
    y[0] = a.y0[sys];
    y[1] = a.y0[a.n + sys];
    tau = a.t0;
    rest = tau_end - tau;
    dt = a.dt0;
    ph = 0;
    st = timed_out ? kStTimeout : 0;
    trials = nacc = nrej = nrhs = 0;
    fresh = true;
    ymax = ymin = y[0];
    d0 = s.drive(a.t0);
    k1v = s.accel_at(y[0], y[1], s.early_power(y[0]), d0);
    a21k1x = weight<PAIR>(2, 1) * y[1];
    a21k1v = weight<PAIR>(2, 1) * k1v;
    a31k1x = weight<PAIR>(3, 1) * y[1];
    a31k1v = weight<PAIR>(3, 1) * k1v;
  };
  auto record = [&](int64_t sys) {
    ymax = omax(ymax, y[0]);
    ymin = omin(ymin, y[0]);
    if (ph >= a.n_transient) {
      a.acc[(int64_t)(2 * (ph - a.n_transient)) * a.n + sys] = ymax;
      a.acc[(int64_t)(2 * (ph - a.n_transient) + 1) * a.n + sys] = ymin;
    }
  };
  auto finish_system = [&](int64_t sys) {
    // recorded phases that were not completed are marked NaN
    for (int p = max(ph, a.n_transient); p < a.n_phases; ++p) {
      a.acc[(int64_t)(2 * (p - a.n_transient)) * a.n + sys] = __longlong_as_double(0x7ff8000000000000LL);
      a.acc[(int64_t)(2 * (p - a.n_transient) + 1) * a.n + sys] = __longlong_as_double(0x7ff8000000000000LL);
    }
    a.y[sys] = y[0];
    a.y[a.n + sys] = y[1];
    a.t_out[sys] = tau;
    a.dt_out[sys] = dt;
    a.status[sys] = st;
    a.nacc[sys] = nacc;
    a.nrej[sys] = nrej;
    a.nrhs[sys] = nrhs;
    if (st) atomicOr(&a.scratch->any_status, (unsigned)st);
  };
  auto next_system = [&]() -> int64_t {
    return a.first_by_subpartition ? claim_next_after_ranked(a, 32) : claim(a, false, 0, 0);
  };

  int64_t i;
  if (a.first_by_subpartition) {
    const int64_t rank = blockIdx.x * (int64_t)32 + lane;
    i = rank < a.n ? (int64_t)a.order[rank] : -1;
  } else {
    i = claim(a, true, 32, lane);
  }
  long long shown = i >= 0 ? i : 0;   // a lane without a system computes on system 0 and stores nothing

  bool taken = false;
  auto count = [&]() {   // of the trial that ended
    nrhs += pair_rhs(PAIR) + (fresh ? 1u : 0u);
    fresh = PAIR == kCashKarp && taken;  // Dormand-Prince counts k7 among the trial's evaluations
    nacc += taken ? 1u : 0u;
    nrej += taken ? 0u : 1u;
  };
  // step and second stage of the next trial
  bool next_clamped = false;
  double next_h = 0.0, next_x = 0.0, next_v = 0.0;
  auto begin = [&]() {
    next_clamped = nnbits(dt) >= nnbits(rest);
    next_h = next_clamped ? rest : dt;
    next_x = vfma(next_h, a21k1x, y[0]);
    next_v = vfma(next_h, a21k1v, y[1]);
  };
  bool special = true, need = true, under = false, was_clamped = false, ends = false, counted = true, ok = true;
  for (;;) {
    if (__builtin_expect(special, 0)) {
      if (__any_sync(0xffffffffu, !ok)) timed_out = true;   // a helper is lost: retire all there is to claim
      if (!need) {
        count();
        counted = true;
        if (under && i >= 0) st |= kStDtUnderflow;
        if (taken && ends) {
          record(i);
          ++ph;
          if (ph >= a.n_phases) {
            finish_system(i);
            i = next_system();
            need = i >= 0;
          } else {
            // the first stage takes the drive of the phase start
            if ((PAIR == kDormandPrince || !was_clamped) &&
                (nnbits(dn.fs) != nnbits(d0.fs) || nnbits(dn.fc) != nnbits(d0.fc))) {
              k1v = s.accel_at(y[0], y[1], m.g[5][lane], d0);
              a21k1v = weight<PAIR>(2, 1) * k1v;
              a31k1v = weight<PAIR>(3, 1) * k1v;
            }
            tau = a.t0;
            rest = tau_end - tau;
            fresh = true;
            ymax = ymin = y[0];
          }
        }
      }
      do {
        if (need) {
          if (i >= 0) shown = i;
          start_system(shown);
          need = false;
        }
        // systems that ran out of a budget or failed close their phase with what it has
        if (i >= 0 && st == 0) {
          if (timed_out) st |= kStTimeout;
          else if (trials >= (uint64_t)a.max_steps) st |= kStMaxSteps;
        }
        if (i >= 0 && st != 0) {
          if (ph < a.n_phases) {
            record(i);
            ++ph;
          }
          finish_system(i);
          i = next_system();
          need = i >= 0;
        }
      } while (__any_sync(0xffffffffu, need));
      if (!__any_sync(0xffffffffu, i >= 0)) break;
      begin();
    }
    const bool clamped = next_clamped;
    const double h = next_h;
    double x = next_x, v = next_v, kv = k1v, pv = a31k1v;
    was_clamped = clamped;
    m.t[lane] = tau;
    m.h[lane] = h;
    m.sys[lane] = shown;
    post(&m.bar[kStart]);
    m.y[0][lane] = y[0];
    m.y[1][lane] = y[1];
    m.a31k1x[lane] = a31k1x;
    m.k[0][lane] = kv;
    m.pv[0][lane] = pv;
    m.x[0][lane] = x;
    m.v[0][lane] = v;
    post(&m.bar[kSlope]);
    if (!counted) count();
    ymax = omax(ymax, y[0]);  // the end of the last accepted trial
    ymin = omin(ymin, y[0]);
    ++trials;
    // 1 / (y1 D), D = y1 (1 - C9 y2) + C4 C9, as rcp_nr refines it
    double D, w;
    auto reciprocal = [&]() {
      D = vfma(x, vfma(-s.C9, v, 1.0), s.C4C9);
      const double xD = vmul(x, D);
      asm volatile("rcp.approx.ftz.f64 %0, %1;" : "=d"(w) : "d"(xD));
      const double e = vfma(-xD, w, 1.0);
      w = vfma(vfma(e, e, e), w, w);
    };
    typename Sys::Drive d;
#pragma unroll 1
    for (int c = 0; c < 5; ++c) {   // stages 2..6
      reciprocal();
      const double rx = vmul(D, w), yw = vmul(x, w);
      ok &= await_trial(m, kAll + c, trial);
      double N = vfma(-m.b[c][lane], rx, m.n[c][lane]);
      N = vfma(-m.e[c][lane], m.q[c][lane], N);
      d = {m.fs[c][lane], m.fc[c][lane]};
      if (PAIR == kCashKarp && c == 3) dn = d;   // c5 = 1
      N = vfma(-d.fs, m.o[c][lane], N);
      N = vfma(-x, d.fc, N);
      pv = m.pv[c][lane];
      const double newest = kNewest[PAIR == kDormandPrince][c];
      x = m.x[c + 1][lane];
      kv = vmul(N, yw);
      v = vfma(h, vfma(newest, kv, pv), y[1]);
      m.k[c + 1][lane] = kv;
      m.v[c + 1][lane] = v;
      post(&m.bar[kSlope + c + 1]);
    }
    if (PAIR == kDormandPrince) dn = d;
    reciprocal();
    const double tau_sum = vadd(tau, h), tau_new = clamped ? tau_end : tau_sum, rest_new = vadd(tau_end, -tau_new);
    const double a21k1x_new = vmul(weight<PAIR>(2, 1), v), a31k1x_new = vmul(weight<PAIR>(3, 1), v);
    const double rx = vmul(D, w), yw = vmul(x, w);
    if (PAIR == kDormandPrince || !clamped) d = dn;
    else d = d0;
    ok &= await_trial(m, kAll + 5, trial);
    {
      double N = vfma(-m.b[5][lane], rx, m.n[5][lane]);
      N = vfma(-m.e[5][lane], m.q[5][lane], N);
      N = vfma(-d.fs, m.o[5][lane], N);
      N = vfma(-x, d.fc, N);
      if (PAIR == kDormandPrince) pv = m.pv[5][lane];
      kv = vmul(N, yw);
    }
    // x, v are the trial's end state and kv the next trial's first slope, if this
    // one is accepted; a Cash-Karp trial that was shortened to the end of the phase
    // is followed by a phase start
    if (PAIR == kDormandPrince) {
      m.err[1][lane] = vmul(h, vfma(weight<PAIR>(8, 7), kv, pv));
      post(&m.bar[kErr]);
    }
    const double a21k1v_new = vmul(weight<PAIR>(2, 1), kv), a31k1v_new = vmul(weight<PAIR>(3, 1), kv);
    if ((trial & 127u) == 127u && global_ns() > deadline) timed_out = true;
    const bool spent = timed_out || trials >= (uint64_t)a.max_steps;
    ends = okey(tau_new) >= okey(tau_end);   // !(tau < tau_end): tau + h may round onto the end
    ok &= await_trial(m, kCtl, trial);
    ++trial;
    const double step = m.dt[lane], next = absd(step);
    const bool accepted = !(__double2hiint(step) < 0);
    // the outcome without branches, so that lanes that reject cost the others nothing
    taken = accepted && ok && i >= 0;
    dt = accepted && clamped ? dt : next;
    tau = taken ? tau_new : tau;
    rest = taken ? rest_new : rest;
    y[0] = taken ? x : y[0];
    y[1] = taken ? v : y[1];
    k1v = taken ? kv : k1v;
    a21k1x = taken ? a21k1x_new : a21k1x;
    a21k1v = taken ? a21k1v_new : a21k1v;
    a31k1x = taken ? a31k1x_new : a31k1x;
    a31k1v = taken ? a31k1v_new : a31k1v;
    begin();
    under = !taken && nnbits(dt) < nnbits(a.dt_min);
    counted = false;
    special = __any_sync(0xffffffffu, !ok || (i >= 0 && (spent || (taken ? ends : under))));
  }
  m.sys[lane] = -1;
  post(&m.bar[kSlope]);
  post(&m.bar[kStart]);
}

// Block = 8 warps, one relay.  Warp w of a block runs on sub-partition w mod 4: the
// main warp has the FP64 pipe of one to itself; numerator and first drive warp share
// one, sums and second drive warp another, power and factors the last.  A block that
// starts at an odd multiple of 8 warps, the second of its SM, takes them in reverse,
// so that the two main warps do not meet (which only the speed depends on).
template <class Sys, int PAIR>
__global__ void __launch_bounds__(256, 2) ck_phased_relay_kernel(AdaptArgs a) {
  __shared__ Relay m;
  __shared__ unsigned flip;
  const int w = (int)(threadIdx.x >> 5);
  if (threadIdx.x == 0) {
    for (int k = 0; k < kBars; ++k) {
      // the main warp waits for numerator, factors, sums and drive (stage 2's in two halves),
      // the power warp for the error estimate, a ratio and a weight
      int senders = 1;
      if (k >= kAll && k < kAll + 5) senders = k == kAll && !Sys::kDual ? 5 : 4;
      if (k == kAll + 5) senders = PAIR == kDormandPrince ? 3 : 2;   // no drive, Cash-Karp no sums
      if (k == kErr) senders = 3;
      init_bar(m.bar + k, senders);
    }
    unsigned id;
    asm volatile("mov.u32 %0, %warpid;" : "=r"(id));
    flip = (id >> 3) & 1u;
  }
  __syncthreads();
  const int role = (w & 4) | (flip ? 3 - (w & 3) : (w & 3));
  if (role == 0) main_warp<Sys, PAIR>(a, m);
  else if (role == 1) numerator_warp<Sys>(a, m);
  else if (role == 2) sums_warp<PAIR>(a, m);
  else if (role == 3) power_warp<Sys>(a, m);
  else if (role == 7) factors_warp<Sys>(a, m);
  else if (Sys::kDual || role != 4) drive_warp<Sys, PAIR>(a, m, role == 4 ? 2 : role - 5);
}

}  // namespace

// An adaptive launch of blocks of 32 systems, with 8 warps for each: Keller-Miksis
// phase mode with the exponent 21/5.
cudaError_t launch_ck45_relay(unsigned flags, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s) {
  if (a.n == 0) return cudaSuccess;
  if (a.n_phases <= 0 || (flags & kKmGeneralExponent)) return cudaErrorNotSupported;
  if (L.grid <= 0 || L.grid > 0x7fffffffLL || L.block != 32) return cudaErrorInvalidConfiguration;
  const dim3 g((unsigned)L.grid), b(256);
  const bool dual = flags & kKmDual;
  if (a.pair == kDormandPrince) {
    if (dual) ck_phased_relay_kernel<KellerMiksis<true, true>, kDormandPrince><<<g, b, 0, s>>>(a);
    else ck_phased_relay_kernel<KellerMiksis<false, true>, kDormandPrince><<<g, b, 0, s>>>(a);
  } else if (a.pair == kCashKarp) {
    if (dual) ck_phased_relay_kernel<KellerMiksis<true, true>, kCashKarp><<<g, b, 0, s>>>(a);
    else ck_phased_relay_kernel<KellerMiksis<false, true>, kCashKarp><<<g, b, 0, s>>>(a);
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace ens
