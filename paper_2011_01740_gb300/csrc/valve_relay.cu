// valve_relay.cu -- event mode of the relief valve for ensembles of at most four warps
// of systems per SM: the trial of 32 systems runs in four warps.
//
// Such an ensemble takes as long as its longest system, and in ck_events_kernel
// (rkck45.cu) its warp issues 140 FP64 instructions of 64 cycles a trial one after the
// other, beside the integer chains of the square root and the controller: 12,800
// cycles.  Only the third component, y3' = beta (q - y1 sqrt(y3)), depends on the root,
// so the main warp keeps that component's chain (root, slope, newest term of the
// stage, 1,280 cycles a stage) and the event rules, and other warps, on other
// sub-partitions, do the rest for the same 32 lanes:
//   - motion: stage sums and slopes of the first two components, which need y3 of the
//     stage alone;
//   - sums: the sums over the third component's older slopes and its error estimate;
//   - control: error norm and next step, while the main warp takes the next trial's
//     first slope and the event tests for the case that this one is accepted.
// Every operation is that of ck_events_kernel, so are the bits.  Milliseconds there and
// here for 16 time units: 1,000 valves 21.4 / 16.8, 9,700 21.4 / 17.6, 19,456 (four
// relays on every SM) 21.6 / 20.1.  A trial ends with event roots (2,700 cycles where
// a lane of the warp has one) or the error norm, whichever is later.
// What was tried: helper warps for the root and the controller alone (21.7: each
// stage's root then makes a round trip of 260 cycles); the event tests in the sums
// warp (17.3); the error weights there (17.1).
//
// Messages, bounded waits and what follows when one expires are those of
// rkck45_relay.cu.
#include "common.cuh"
#include "controller.cuh"
#include "events.cuh"
#include "mailbox.cuh"
#include "rhs.cuh"

namespace ens {

namespace {

// barriers, one phase per trial; index s - 2 for stage s = 2..7
enum : int { kStart = 0, kP = 1, kX = 7, kK = 13, kS = 18, kV = 22, kErrV = 23, kErrP = 24, kEnd = 25, kCtl = 26, kBars = 27 };

struct __align__(16) ValveRelay {
  double p[6][32], x[6][32];         // y3 and y1 of a stage
  double k[6][32];                   // third slope component of stages 1..6
  double pp[4][32];                  // its sums known so far for stages 4..7
  double h[32], y[3][32], k1v[32];   // the trial: length, state, second component of the first slope
  double v7[32], kv7[32];            // y2 and its slope at the trial's end
  double err[3][32];
  double dt[32];                     // the next step, negative after a rejection
  long long sys[32];                 // the lane's system, -1 when none are left
  unsigned long long bar[kBars];
};

// weight of slope i in row r: rows 2..6 the stages, 7 the new state, 8 the error estimate
__device__ constexpr double weight(int r, int i) {
  constexpr double A[7][6] = {{ck::a21, 0, 0, 0, 0, 0},
                              {ck::a31, ck::a32, 0, 0, 0, 0},
                              {ck::a41, ck::a42, ck::a43, 0, 0, 0},
                              {ck::a51, ck::a52, ck::a53, ck::a54, 0, 0},
                              {ck::a61, ck::a62, ck::a63, ck::a64, ck::a65, 0},
                              {ck::b1, 0, ck::b3, ck::b4, 0, ck::b6},
                              {ck::d1, 0, ck::d3, ck::d4, ck::d5, ck::d6}};
  return A[r - 2][i - 1];
}
// weight of the newest slope in the stage after, by stage - 2
static __constant__ double kNewest[5] = {ck::a32, ck::a43, ck::a54, ck::a65, ck::b6};

__device__ __forceinline__ bool all(bool ok) { return __all_sync(0xffffffffu, ok); }
__device__ __forceinline__ bool all_await(ValveRelay& m, int bar, uint32_t trial) { return all(await(&m.bar[bar], trial)); }

// first and second component, both sums and slopes
__device__ __forceinline__ void motion_warp(const AdaptArgs& a, ValveRelay& m) {
  const int lane = threadIdx.x & 31;
  ReliefValve s;
  long long cur = -2;
  for (uint32_t trial = 0;; ++trial) {
    if (!all_await(m, kStart, trial)) return;
    const long long sys = m.sys[lane];
    if (!all(sys >= 0)) return;
    if (sys != cur) {
      cur = sys;
      s.load(a.params, a.n, cur);
    }
    const double h = m.h[lane], x0 = m.y[0][lane], v0 = m.y[1][lane];
    double kx[8], kv[8], x, v;   // slopes 1..7
    kx[1] = v0;
    kv[1] = m.k1v[lane];
    x = fma(h, smul(weight(2, 1), kx[1]), x0);
    m.x[0][lane] = x;
    post(&m.bar[kX]);
    v = fma(h, smul(weight(2, 1), kv[1]), v0);
#pragma unroll
    for (int g = 2; g <= 7; ++g) {
      // x, v: stage g; the next stage's first component needs no more than v
      kx[g] = v;
      double xn = 0.0;
      if (g < 7) {
        double z = smul(weight(g + 1, 1), kx[1]);
#pragma unroll
        for (int j = 2; j <= g; ++j)
          if (weight(g + 1, j) != 0.0) z = fma(weight(g + 1, j), kx[j], z);
        xn = fma(h, z, x0);
        m.x[g - 1][lane] = xn;
        post(&m.bar[kX + g - 1]);
      }
      const double xd = sadd(x, s.delta);
      double z = 0.0;
      if (g < 7) {
        z = smul(weight(g + 1, 1), kv[1]);
#pragma unroll
        for (int j = 2; j < g; ++j)
          if (weight(g + 1, j) != 0.0) z = fma(weight(g + 1, j), kv[j], z);
      }
      double ex = 0.0, ev = 0.0;
      if (g == 6) {   // the error estimate up to the slope that is still to come
        ex = smul(weight(8, 1), kx[1]);
        ev = smul(weight(8, 1), kv[1]);
#pragma unroll
        for (int j = 3; j <= 6; ++j) {
          ex = fma(weight(8, j), kx[j], ex);
          if (j < 6) ev = fma(weight(8, j), kv[j], ev);
        }
        m.err[0][lane] = smul(h, ex);
      }
      if (!all_await(m, kP + g - 2, trial)) return;
      kv[g] = fma(-s.kappa, v, ssub(m.p[g - 2][lane], xd));
      if (g == 7) {
        m.kv7[lane] = kv[7];
        post(&m.bar[kEnd]);
        break;
      }
      v = fma(h, fma(weight(g + 1, g), kv[g], z), v0);
      if (g == 6) {
        m.v7[lane] = v;
        post(&m.bar[kV]);
        m.err[1][lane] = smul(h, fma(weight(8, 6), kv[6], ev));
        post(&m.bar[kErrV]);
      }
      x = xn;
    }
  }
}

// sums over the third component's slopes
__device__ __forceinline__ void sums_warp(ValveRelay& m) {
  const int lane = threadIdx.x & 31;
  for (uint32_t trial = 0;; ++trial) {
    if (!all_await(m, kStart, trial) || !all(m.sys[lane] >= 0)) return;
    const double h = m.h[lane], k1 = m.k[0][lane];
    double z[9];
#pragma unroll
    for (int r = 4; r <= 8; ++r) z[r] = smul(weight(r, 1), k1);
#pragma unroll
    for (int g = 2; g <= 6; ++g) {
      if (!all_await(m, kK + g - 2, trial)) return;
      const double k = m.k[g - 1][lane];
#pragma unroll
      for (int r = g + 2; r <= 8; ++r) {
        if (weight(r, g) != 0.0) z[r] = fma(weight(r, g), k, z[r]);
        if (r == g + 2 && r <= 7) {
          m.pp[r - 4][lane] = z[r];
          post(&m.bar[kS + r - 4]);
        }
      }
    }
    m.err[2][lane] = smul(h, z[8]);
    post(&m.bar[kErrP]);
  }
}

// error norm and next step
__device__ __forceinline__ void control_warp(const AdaptArgs& a, ValveRelay& m) {
  const int lane = threadIdx.x & 31;
  for (uint32_t trial = 0;; ++trial) {
    if (!all_await(m, kStart, trial) || !all(m.sys[lane] >= 0)) return;
    const double h = m.h[lane], y0 = m.y[0][lane], y1 = m.y[1][lane], y2 = m.y[2][lane];
    if (!all_await(m, kX + 5, trial)) return;
    const double w0 = err_weight(y0, m.x[5][lane], a.rtol, a.atol);
    if (!all_await(m, kV, trial)) return;
    const double w1 = err_weight(y1, m.v7[lane], a.rtol, a.atol);
    if (!all_await(m, kP + 5, trial)) return;
    const double w2 = err_weight(y2, m.p[5][lane], a.rtol, a.atol);
    if (!all_await(m, kErrV, trial) || !all_await(m, kErrP, trial)) return;
    double E = nnmax(0.0, err_ratio(m.err[0][lane], w0));
    E = nnmax(E, err_ratio(m.err[1][lane], w1));
    E = nnmax(E, err_ratio(m.err[2][lane], w2));
    const double hf = smul(h, step_factor(E));
    m.dt[lane] = accept(E) ? nnmax(nnmin(hf, a.dt_max), a.dt_min) : -hf;
    post(&m.bar[kCtl]);
  }
}

__device__ __forceinline__ void main_warp(const AdaptArgs& a, ValveRelay& m) {
  constexpr int D = 3;
  const int lane = threadIdx.x & 31;
  const uint64_t deadline = global_ns() + a.timeout_ns;
  const double etol = a.event_tol;
  const long long kt = okey(etol), knt = okey(-etol);
  uint32_t trial = 0;
  bool timed_out = false, ok = true;
  ReliefValve s;
  double y[D], k1[D], y5[D], kn[D];
  double t = a.t0, dt = a.dt0, h_ev = 0.0, ymin = 0.0;
  int32_t st = 0, ev_retries = 0;
  uint32_t trials = 0, nacc = 0, nrej = 0, nrhs = 0, nmax = 0, nimp = 0;
  bool k1v = false, fresh = true, stuck = false;   // first slope there; counts as an evaluation

  auto start_system = [&](int64_t sys) {
    s.load(a.params, a.n, sys);
#pragma unroll
    for (int c = 0; c < D; ++c) y[c] = a.y0[c * a.n + sys];
    t = a.t0;
    dt = a.dt0;
    h_ev = 0.0;
    st = timed_out ? kStTimeout : 0;
    ev_retries = 0;
    trials = nacc = nrej = nrhs = nmax = nimp = 0;
    k1v = false;
    stuck = false;
    ymin = (t >= a.acc_t_start) ? y[0] : __longlong_as_double(0x7ff0000000000000LL);
  };
  auto clear_ring = [&](int64_t sys) {
    for (int r = 0; r < kRing; ++r) a.acc[(int64_t)r * a.n + sys] = __longlong_as_double(0x7ff8000000000000LL);
  };
  auto finish_system = [&](int64_t sys) {
#pragma unroll
    for (int c = 0; c < D; ++c) a.y[c * a.n + sys] = y[c];
    a.acc[(int64_t)kRing * a.n + sys] = ymin;
    a.acc[(int64_t)(kRing + 1) * a.n + sys] = (double)nmax;
    a.acc[(int64_t)(kRing + 2) * a.n + sys] = (double)nimp;
    a.t_out[sys] = t;
    a.dt_out[sys] = dt;
    a.status[sys] = st;
    a.nacc[sys] = nacc;
    a.nrej[sys] = nrej;
    a.nrhs[sys] = nrhs;
    if (st) atomicOr(&a.scratch->any_status, (unsigned)st);
  };

  int64_t i = claim(a, true, 32, lane);
  long long shown = i >= 0 ? i : 0;
  start_system(shown);   // a lane without a system computes on system 0 and stores nothing
  if (i >= 0) clear_ring(i);
  auto next_system = [&]() {
    finish_system(i);
    i = claim(a, false, 0, 0);
    if (i >= 0) {
      shown = i;
      start_system(i);
      clear_ring(i);
    }
  };

  for (;;) {
    // everything but trials: retired systems, intervals on the seat
    while (i >= 0) {
      if (st == 0) {
        if (timed_out) st |= kStTimeout;
        else if (!stuck && trials >= (uint64_t)a.max_steps) st |= kStMaxSteps;
      }
      if (st != 0) {
        next_system();
      } else if (stuck) {
        // closed-form interval on the seat: y1 = y2 = 0, y3' = beta q
        const double t_lift = t + (s.delta - y[2]) / (s.beta * s.q);
        if (t_lift >= a.t1) {
          y[2] = y[2] + s.beta * s.q * (a.t1 - t);
          t = a.t1;
        } else {
          y[2] = s.delta;
          t = t_lift;
          stuck = false;
        }
        k1v = false;
        if (okey(t) >= okey(a.acc_t_start) && okey(y[0]) < okey(ymin)) ymin = y[0];
        if (okey(t) >= okey(a.t1)) next_system();
      } else {
        break;
      }
    }
    if (!__any_sync(0xffffffffu, i >= 0)) break;
    double h = dt;
    int limited = 0;
    const double rest = ssub(a.t1, t);  // > 0 before the end
    if (nnbits(h) >= nnbits(rest)) {
      h = rest;
      limited = 1;
    }
    if (nnbits(h_ev) > 0 && nnbits(h_ev) < nnbits(h)) {  // h_ev >= 0
      h = h_ev;
      limited = 2;
    }
    if (!k1v) {
      s.f(t, y, k1);
      k1v = true;
      fresh = true;
    }
    m.h[lane] = h;
#pragma unroll
    for (int c = 0; c < D; ++c) m.y[c][lane] = y[c];
    m.k1v[lane] = k1[1];
    m.k[0][lane] = k1[2];
    m.sys[lane] = shown;
    double p = fma(h, smul(ck::a21, k1[2]), y[2]);
    post(&m.bar[kStart]);
    double sum = smul(ck::a31, k1[2]);
    // the third slope component at y3 = p: its root here, y1 from the motion warp
    auto slope = [&](int c) {
      m.p[c][lane] = p;
      post(&m.bar[kP + c]);
      const double r = sqrt_fx(__double2hiint(p) < 0 ? 0.0 : p);
      uint32_t phase = trial;
      ok &= await(&m.bar[kX + c], phase);
      return smul(s.beta, fma(-m.x[c][lane], r, s.q));
    };
#pragma unroll 1
    for (int c = 0; c < 5; ++c) {
      const double k = slope(c);
      m.k[c + 1][lane] = k;
      post(&m.bar[kK + c]);
      if (c > 0) {
        uint32_t phase = trial;
        ok &= await(&m.bar[kS + c - 1], phase);
        sum = m.pp[c - 1][lane];
      }
      p = fma(h, fma(kNewest[c], k, sum), y[2]);
    }
    // the next trial's first slope, if this one is accepted without an event
    kn[2] = slope(5);
    y5[0] = m.x[5][lane];
    y5[2] = p;
    {
      uint32_t phase = trial;
      ok &= await(&m.bar[kEnd], phase);
    }
    y5[1] = kn[0] = m.v7[lane];
    kn[1] = m.kv7[lane];
    // the event tests, for a trial that is accepted, while its error norm is on the way
    double best = 2.0;
    bool overshoot = false;
    if (okey(y5[0]) < knt) {  // impact beyond the band
      const double frac = (okey(y[0]) > kt) ? event_frac(y[0], k1[0], y5[0], h) : 0.5;
      best = nnmin(frac, best);
      overshoot = true;
    }
    if (okey(y[1]) > kt && okey(y5[1]) < knt) {  // maximum beyond the band
      const double frac = event_frac(y[1], k1[1], y5[1], h);
      best = nnmin(frac, best);
      overshoot = true;
    }
    nrhs += 5u + (fresh ? 1u : 0u);
    fresh = false;
    ++trials;
    if ((trial & 127u) == 127u && global_ns() > deadline) timed_out = true;
    uint32_t phase = trial++;
    ok &= await(&m.bar[kCtl], phase);
    const double step = m.dt[lane], next = absd(step);
    const bool lost = !__all_sync(0xffffffffu, ok);
    if (lost) timed_out = true;   // a helper is gone: retire all there is to claim
    if (i < 0 || lost) continue;
    if (__double2hiint(step) < 0) {
      ++nrej;
      dt = next;
      h_ev = 0.0;
      if (nnbits(dt) < nnbits(a.dt_min)) st |= kStDtUnderflow;
    } else {
      if (overshoot) {
        if (++ev_retries > kEventRetries) st |= kStEventNoConverge;
        else h_ev = smul(h, best);
      } else {
        const double y1_old = y[1];
#pragma unroll
        for (int c = 0; c < D; ++c) {
          y[c] = y5[c];
          k1[c] = kn[c];
        }
        t = (limited == 1) ? a.t1 : sadd(t, h);
        fresh = true;   // the impact law below takes the slope back
        ++nacc;
        ev_retries = 0;
        h_ev = 0.0;
        if (!limited) dt = next;
        if (okey(y1_old) > kt && nnbits(absd(y[1])) <= nnbits(etol)) {  // Poincare point
          a.acc[(int64_t)(nmax % kRing) * a.n + i] = y[0];
          ++nmax;
        }
        // impact law when |y1| <= tol and y2 < 0 (okey(-0.0) = -1: -0 is not below zero)
        if (nnbits(absd(y[0])) <= nnbits(etol) && okey(y[1]) < -1LL) {
          y[0] = 0.0;
          y[1] = -s.r * y[1];
          k1v = false;
          ++nimp;
          const double push = s.delta - y[2];
          if (push > 0.0 && y[1] * y[1] <= 2.0 * push * etol) {
            y[1] = 0.0;
            stuck = true;
          }
        }
        if (okey(t) >= okey(a.acc_t_start) && okey(y[0]) < okey(ymin)) ymin = y[0];
        if (okey(t) >= okey(a.t1)) next_system();
      }
    }
  }
  m.sys[lane] = -1;
  post(&m.bar[kStart]);
}

// block = 4 warps, one relay
__global__ void __launch_bounds__(128, 4) ck_events_relay_kernel(AdaptArgs a) {
  __shared__ ValveRelay m;
  __shared__ unsigned turn;
  if (threadIdx.x == 0) {
    init_bars(m.bar, kBars);
    unsigned id;
    asm volatile("mov.u32 %0, %warpid;" : "=r"(id));
    turn = id >> 2;
  }
  __syncthreads();
  const int role = (int)((threadIdx.x >> 5) + turn) & 3;
  if (role == 0) main_warp(a, m);
  else if (role == 1) motion_warp(a, m);
  else if (role == 2) sums_warp(m);
  else control_warp(a, m);
}

}  // namespace

cudaError_t launch_ck45_events_relay(const AdaptArgs& a, AdaptLaunch L, cudaStream_t s) {
  if (a.n == 0) return cudaSuccess;
  if (a.pair != kCashKarp) return cudaErrorNotSupported;
  if (L.grid <= 0 || L.grid > 0x7fffffffLL || L.block != 32) return cudaErrorInvalidConfiguration;
  ck_events_relay_kernel<<<dim3((unsigned)L.grid), 128, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace ens
