// rkck45_teams.cu -- Keller-Miksis phase mode with a team of three warps per 32
// systems.
//
// In ck_phased_kernel (rkck45.cu) one warp carries a system's whole trial: about
// 200 FP64 instructions, each 64 cycles of its sub-partition's FP64 pipe (a
// dependent one costs no more: 65), and some 3,500 integer instructions (the
// polytropic power, the forcing's sine and cosine, the controller's roots and
// reciprocals in fixed point).  A warp issues in order, and the integer chains
// come out as long runs in which the FP64 pipe idles: a lone warp's trial takes
// 21,500 cycles, 13,100 of them FP64 issue.
//
// Here the two kinds of work run in different warps, which the hardware
// interleaves cycle by cycle.  The main warp of a team holds 32 systems and does
// the FP64 work; for the same 32 lanes
//   - the power warp computes the polytropic power at each stage's y1.  As
//     y1' = y2, a stage's y1 needs only the y2 of earlier stages: the main warp
//     sends it before it completes the acceleration of the stage before, and has
//     the power when it needs it.  At the trial's end it computes the error norm
//     and the step factor while the main warp already evaluates the next trial's
//     first stage on the trial's end state (discarded after a rejection);
//   - the drive warp computes the drives of the trial's stages, which depend on
//     the time alone.
// Every operation is that of ck_phased_kernel, so are the bits.  Milliseconds
// there and here: 1,073 systems x 2 periods 45.1 / 32.9, 4,608 frequencies x 3
// 68.2 / 48.9, two frequencies and Dormand-Prince (6,097 x 2) 69.4 / 48.5; with
// longest-first claiming 65,536 x 2 47.6 / 36.7, 131,044 x 6 189.4 (6 warps per
// SM) / 166.4 (5 teams).  Registers allow 5 teams per SM, which keep the FP64 pipe
// 82 % busy (131,044 x 64); enough systems let more plain warps do better (262,144 x 2:
// 105.1 here, 97.0 with 12 plain warps), see teams_fit in abi.cu; up to two warps of
// systems per SM the relay (rkck45_relay.cu) does.
// What was tried: one helper warp for both kinds (37.4 ms on 1,073 systems; its
// power then waits for a drive); the helpers' stages unrolled (fast while all teams
// of an SM run in step, 151 ms on 131,044 x 4 when they do not: instruction cache);
// the power spelled out a stage earlier in the one-warp kernel (45.3 -> 50.6 ms).
//
// Messages go through a mailbox in shared memory, on mbarriers with one phase per
// trial: the sender's lanes write, one lane arrives; the receiver waits for the
// phase.  A stage's power and drive arrive on one barrier (a wait costs some 60 cycles:
// 131,044 x 3 periods 81.8 -> 81.1 ms).  The main warp has received everything of a
// trial before it starts the next, so no barrier is ever more than one phase ahead of
// its receiver.  Waits are bounded; when one of the
// main warp's expires, its systems and all it still claims are retired with
// ENS_SYS_TIMEOUT, and a helper whose wait expires leaves.
#include "common.cuh"
#include "controller.cuh"
#include "mailbox.cuh"
#include "rhs.cuh"

namespace ens {

namespace {

constexpr int kMaxTeams = 5;             // teams of three warps per block

// barriers of a team's mailbox
enum : int { kReq = 0, kAll = 6, kCtlReq = 12, kCtlRsp = 13, kStart = 14, kBars = 15 };

struct __align__(16) Mailbox {
  double x[6][32];             // power request: y1 of a stage
  double g[6][32];             // its reply
  double t[32], h[32];         // trial start: its time and length,
  long long sys[32];           //              the lane's system
  double fs[5][32], fc[5][32]; // drives of stages 2..6
  double v[6][32];             // controller request: y, y5, error estimate
  double e[32], fac[32];       // its reply: error norm, step factor
  int run;                     // 0: no systems left
  unsigned long long bar[kBars];
};

// stage times of stages 2..6 in steps (a stage at t + h is fma(1, h, t), the same bits)
template <int PAIR>
__device__ __forceinline__ double stage_c(int stage) {
  if (PAIR == kDormandPrince)
    return stage == 2 ? dp::c2 : stage == 3 ? dp::c3 : stage == 4 ? dp::c4 : stage == 5 ? dp::c5 : 1.0;
  return stage == 2 ? ck::c2 : stage == 3 ? ck::c3 : stage == 4 ? ck::c4 : stage == 5 ? ck::c5 : ck::c6;
}

// the next phase of a barrier that has one per trial
__device__ __forceinline__ bool all_await(Mailbox& m, int bar, uint32_t trial) {
  return __all_sync(0xffffffffu, await(&m.bar[bar], trial));
}

// Both helpers' loops over the stages stay rolled: unrolled (50 KB) they thrash the
// instruction cache as soon as the teams of an SM run out of step.

// powers of the stages' y1 and, at the trial's end, error norm and step factor
template <class Sys>
__device__ __forceinline__ void power_warp(const AdaptArgs& a, Mailbox& m) {
  const int lane = threadIdx.x & 31;
  const Sys s{};
  for (uint32_t trial = 0;; ++trial) {
#pragma unroll 1
    for (int k = 0; k < 6; ++k) {
      if (!all_await(m, kReq + k, trial)) return;
      if (k == 0 && !m.run) return;
      m.g[k][lane] = s.early_power(m.x[k][lane]);
      post(&m.bar[kAll + k]);
    }
    if (!all_await(m, kCtlReq, trial)) return;
    const double y[2] = {m.v[0][lane], m.v[1][lane]}, y5[2] = {m.v[2][lane], m.v[3][lane]},
                 err[2] = {m.v[4][lane], m.v[5][lane]};
    const double E = err_norm<2>(y, y5, err, a.rtol, a.atol);
    m.e[lane] = E;
    m.fac[lane] = step_factor(E);
    post(&m.bar[kCtlRsp]);
  }
}

// drives of the stages
template <class Sys, int PAIR>
__device__ __forceinline__ void drive_warp(const AdaptArgs& a, Mailbox& m) {
  const int lane = threadIdx.x & 31;
  Sys s;
  long long cur = -1;
  for (uint32_t trial = 0;; ++trial) {
    if (!all_await(m, kStart, trial) || !m.run) return;
    if (m.sys[lane] != cur) {
      cur = m.sys[lane];
      s.load(a.params, a.n, cur);
    }
    const double t = m.t[lane], h = m.h[lane];
#pragma unroll 1
    for (int stage = 2; stage <= 6; ++stage) {
      const typename Sys::Drive d = s.drive(fma(stage_c<PAIR>(stage), h, t));
      m.fs[stage - 2][lane] = d.fs;
      m.fc[stage - 2][lane] = d.fc;
      post(&m.bar[kAll + stage - 2]);
    }
  }
}

template <class Sys, int PAIR>
__device__ __forceinline__ void main_warp(const AdaptArgs& a, Mailbox& m, int W, int w) {
  const int lane = threadIdx.x & 31, lanes = 32 * W;
  const double tau_end = a.t0 + a.phase_len;
  const uint64_t deadline = global_ns() + a.timeout_ns;
  uint32_t trial = 0, iter = 0;
  bool timed_out = false, dead = false;
  Sys s;
  typename Sys::Drive d0, dn;  // drive at the phase start, at the end of the trial
  double y[2], k1v;            // state, first slope's second component (the first is y2)
  double tau = a.t0, rest = a.phase_len, dt = a.dt0, ymax = 0.0, ymin = 0.0;  // rest of the phase, > 0
  constexpr double a21 = PAIR == kDormandPrince ? dp::a21 : ck::a21;
  double a21k1x = 0.0, a21k1v = 0.0;   // a21 times the first slope
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
    a21k1x = a21 * y[1];
    a21k1v = a21 * k1v;
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
    return a.first_by_subpartition ? claim_next_after_ranked(a, lanes) : claim(a, false, 0, 0);
  };

  int64_t i = a.first_by_subpartition ? claim_first_by_subpartition(a, W, w)
                                      : claim(a, true, lanes, 32 * w + lane);
  long long shown = i >= 0 ? i : 0;   // a lane without a system computes on system 0 and stores nothing
  start_system(shown);

  while (__any_sync(0xffffffffu, i >= 0)) {
    if ((++iter & 127u) == 0 && global_ns() > deadline) timed_out = true;
    // budgets; retired systems close their phase with what it has
    if (i >= 0 && st == 0) {
      if (timed_out) st |= kStTimeout;
      else if (trials >= (uint64_t)a.max_steps) st |= kStMaxSteps;
    }
    while (i >= 0 && st != 0) {
      if (ph < a.n_phases) {
        record(i);
        ++ph;
      }
      finish_system(i);
      i = next_system();
      if (i >= 0) {
        shown = i;
        start_system(i);
      }
    }
    __syncwarp();
    if (dead) continue;
    double h = dt;
    bool clamped = false;
    if (nnbits(h) >= nnbits(rest)) {
      h = rest;
      clamped = true;
    }
    double y5[2], E, fac;
    [[maybe_unused]] double k1n;
    bool ok = true;
    // the rest of a stage's acceleration with its power, requested earlier, and drive
    auto finish_stage = [&](int stage, const typename Sys::Half& p, typename Sys::Drive& d) {
      uint32_t phase = trial;   // one phase per trial
      ok &= await(&m.bar[kAll + stage - 2], phase);
      const typename Sys::Half2 q = s.accel_more(p);   // the pipe works while they arrive
      d = {m.fs[stage - 2][lane], m.fc[stage - 2][lane]};
      return s.accel_last(p, q, s.accel_mid(p, q, m.g[stage - 2][lane]), d.fs, d.fc);
    };
    auto request = [&](int stage, double x) {
      m.x[stage - 2][lane] = x;
      post(&m.bar[kReq + stage - 2]);
    };
    if constexpr (PAIR == kCashKarp) {
      typename Sys::Drive d;
      const double k1x = y[1];
      const double x2 = fma(h, a21k1x, y[0]);
      m.t[lane] = tau;
      m.h[lane] = h;
      m.sys[lane] = shown;
      m.run = 1;
      request(2, x2);
      post(&m.bar[kStart]);
      ymax = omax(ymax, y[0]);  // the end of the last accepted trial
      ymin = omin(ymin, y[0]);
      const double k2x = fma(h, a21k1v, y[1]);
      const double x3 = fma(h, fma(ck::a32, k2x, ck::a31 * k1x), y[0]);
      const typename Sys::Half q2 = s.accel_begin(x2, k2x);
      request(3, x3);
      const double k2v = finish_stage(2, q2, d);
      const double k3x = fma(h, fma(ck::a32, k2v, ck::a31 * k1v), y[1]);
      const double x4 = fma(h, fma(ck::a43, k3x, fma(ck::a42, k2x, ck::a41 * k1x)), y[0]);
      const typename Sys::Half q3 = s.accel_begin(x3, k3x);
      request(4, x4);
      const double k3v = finish_stage(3, q3, d);
      const double k4x = fma(h, fma(ck::a43, k3v, fma(ck::a42, k2v, ck::a41 * k1v)), y[1]);
      const double x5 = fma(h, fma(ck::a54, k4x, fma(ck::a53, k3x, fma(ck::a52, k2x, ck::a51 * k1x))), y[0]);
      const typename Sys::Half q4 = s.accel_begin(x4, k4x);
      request(5, x5);
      const double k4v = finish_stage(4, q4, d);
      const double k5x = fma(h, fma(ck::a54, k4v, fma(ck::a53, k3v, fma(ck::a52, k2v, ck::a51 * k1v))), y[1]);
      const double x6 =
          fma(h, fma(ck::a65, k5x, fma(ck::a64, k4x, fma(ck::a63, k3x, fma(ck::a62, k2x, ck::a61 * k1x)))), y[0]);
      const typename Sys::Half q5 = s.accel_begin(x5, k5x);
      request(6, x6);
      const double k5v = finish_stage(5, q5, dn);  // c5 = 1: the drive at the trial's end
      const double k6x =
          fma(h, fma(ck::a65, k5v, fma(ck::a64, k4v, fma(ck::a63, k3v, fma(ck::a62, k2v, ck::a61 * k1v)))), y[1]);
      y5[0] = fma(h, fma(ck::b6, k6x, fma(ck::b4, k4x, fma(ck::b3, k3x, ck::b1 * k1x))), y[0]);
      const typename Sys::Half q6 = s.accel_begin(x6, k6x);
      request(7, y5[0]);
      m.v[0][lane] = y[0];
      m.v[1][lane] = y[1];
      m.v[2][lane] = y5[0];
      m.v[4][lane] =
          h * fma(ck::d6, k6x, fma(ck::d5, k5x, fma(ck::d4, k4x, fma(ck::d3, k3x, ck::d1 * k1x))));
      const double k6v = finish_stage(6, q6, d);
      y5[1] = fma(h, fma(ck::b6, k6v, fma(ck::b4, k4v, fma(ck::b3, k3v, ck::b1 * k1v))), y[1]);
      m.v[3][lane] = y5[1];
      m.v[5][lane] =
          h * fma(ck::d6, k6v, fma(ck::d5, k5v, fma(ck::d4, k4v, fma(ck::d3, k3v, ck::d1 * k1v))));
      post(&m.bar[kCtlReq]);
      // the next trial's first stage, if this one is accepted; a trial that was
      // shortened to the end of the phase is followed by a phase start
      const typename Sys::Half qn = s.accel_begin(y5[0], y5[1]);
      uint32_t phase = trial;
      ok &= await(&m.bar[kAll + 5], phase);
      {
        const typename Sys::Half2 q = s.accel_more(qn);
        k1n = s.accel_last(qn, q, s.accel_mid(qn, q, m.g[5][lane]), clamped ? d0.fs : dn.fs, clamped ? d0.fc : dn.fc);
      }
    } else {
      typename Sys::Drive d;
      const double k1x = y[1];
      const double x2 = fma(h, a21k1x, y[0]);
      m.t[lane] = tau;
      m.h[lane] = h;
      m.sys[lane] = shown;
      m.run = 1;
      request(2, x2);
      post(&m.bar[kStart]);
      ymax = omax(ymax, y[0]);  // the end of the last accepted trial
      ymin = omin(ymin, y[0]);
      const double k2x = fma(h, a21k1v, y[1]);
      const double x3 = fma(h, fma(dp::a32, k2x, dp::a31 * k1x), y[0]);
      const typename Sys::Half q2 = s.accel_begin(x2, k2x);
      request(3, x3);
      const double k2v = finish_stage(2, q2, d);
      const double k3x = fma(h, fma(dp::a32, k2v, dp::a31 * k1v), y[1]);
      const double x4 = fma(h, fma(dp::a43, k3x, fma(dp::a42, k2x, dp::a41 * k1x)), y[0]);
      const typename Sys::Half q3 = s.accel_begin(x3, k3x);
      request(4, x4);
      const double k3v = finish_stage(3, q3, d);
      const double k4x = fma(h, fma(dp::a43, k3v, fma(dp::a42, k2v, dp::a41 * k1v)), y[1]);
      const double x5 = fma(h, fma(dp::a54, k4x, fma(dp::a53, k3x, fma(dp::a52, k2x, dp::a51 * k1x))), y[0]);
      const typename Sys::Half q4 = s.accel_begin(x4, k4x);
      request(5, x5);
      const double k4v = finish_stage(4, q4, d);
      const double k5x = fma(h, fma(dp::a54, k4v, fma(dp::a53, k3v, fma(dp::a52, k2v, dp::a51 * k1v))), y[1]);
      const double x6 =
          fma(h, fma(dp::a65, k5x, fma(dp::a64, k4x, fma(dp::a63, k3x, fma(dp::a62, k2x, dp::a61 * k1x)))), y[0]);
      const typename Sys::Half q5 = s.accel_begin(x5, k5x);
      request(6, x6);
      const double k5v = finish_stage(5, q5, d);
      const double k6x =
          fma(h, fma(dp::a65, k5v, fma(dp::a64, k4v, fma(dp::a63, k3v, fma(dp::a62, k2v, dp::a61 * k1v)))), y[1]);
      y5[0] = fma(h, fma(dp::b6, k6x, fma(dp::b5, k5x, fma(dp::b4, k4x, fma(dp::b3, k3x, dp::b1 * k1x)))), y[0]);
      const typename Sys::Half q6 = s.accel_begin(x6, k6x);
      request(7, y5[0]);
      const double k6v = finish_stage(6, q6, dn);  // c6 = c7 = 1
      y5[1] = fma(h, fma(dp::b6, k6v, fma(dp::b5, k5v, fma(dp::b4, k4v, fma(dp::b3, k3v, dp::b1 * k1v)))), y[1]);
      // stage 7 = the next trial's first stage
      const typename Sys::Half qn = s.accel_begin(y5[0], y5[1]);
      uint32_t phase = trial;
      ok &= await(&m.bar[kAll + 5], phase);
      {
        const typename Sys::Half2 q = s.accel_more(qn);
        k1n = s.accel_last(qn, q, s.accel_mid(qn, q, m.g[5][lane]), dn.fs, dn.fc);
      }
      m.v[0][lane] = y[0];
      m.v[1][lane] = y[1];
      m.v[2][lane] = y5[0];
      m.v[3][lane] = y5[1];
      m.v[4][lane] = h * fma(dp::e7, y5[1],
                             fma(dp::e6, k6x, fma(dp::e5, k5x, fma(dp::e4, k4x, fma(dp::e3, k3x, dp::e1 * k1x)))));
      m.v[5][lane] = h * fma(dp::e7, k1n,
                             fma(dp::e6, k6v, fma(dp::e5, k5v, fma(dp::e4, k4v, fma(dp::e3, k3v, dp::e1 * k1v)))));
      post(&m.bar[kCtlReq]);
    }
    uint32_t phase = trial++;
    ok &= await(&m.bar[kCtlRsp], phase);
    E = m.e[lane];
    fac = m.fac[lane];
    const double hf = h * fac;
    // what the next trial starts with if this one is accepted
    const double tau_new = clamped ? tau_end : tau + h, rest_new = tau_end - tau_new;
    const double a21k1x_new = a21 * y5[1], a21k1v_new = a21 * k1n;
    if (!__all_sync(0xffffffffu, ok)) {
      dead = timed_out = true;
      continue;
    }
    // the outcome without branches, so that lanes that reject cost the others nothing
    const bool live = i >= 0, taken = accept(E) && live;
    nrhs += pair_rhs(PAIR) + (fresh ? 1u : 0u);
    fresh = PAIR == kCashKarp && taken;  // Dormand-Prince counts k7 among the trial's evaluations
    ++trials;
    nacc += taken ? 1u : 0u;
    nrej += taken ? 0u : 1u;
    const double bounded = nnmax(nnmin(hf, a.dt_max), a.dt_min);
    dt = taken ? (clamped ? dt : bounded) : hf;
    tau = taken ? tau_new : tau;
    rest = taken ? rest_new : rest;
    y[0] = taken ? y5[0] : y[0];
    y[1] = taken ? y5[1] : y[1];
    k1v = taken ? k1n : k1v;
    a21k1x = taken ? a21k1x_new : a21k1x;
    a21k1v = taken ? a21k1v_new : a21k1v;
    if (!taken && nnbits(dt) < nnbits(a.dt_min)) st |= kStDtUnderflow;  // retired before the next trial
    if (taken && okey(tau) >= okey(tau_end)) {  // !(tau < tau_end): tau + h may round onto the end
      record(i);
      ++ph;
      if (ph >= a.n_phases) {
        finish_system(i);
        i = next_system();
        if (i >= 0) {
          shown = i;
          start_system(i);
        }
      } else {
        // the first stage takes the drive of the phase start
        if ((PAIR == kDormandPrince || !clamped) &&
            (nnbits(dn.fs) != nnbits(d0.fs) || nnbits(dn.fc) != nnbits(d0.fc))) {
          k1v = s.accel_at(y[0], y[1], m.g[5][lane], d0);
          a21k1v = a21 * k1v;
        }
        tau = a.t0;
        rest = tau_end - tau;
        fresh = true;
        ymax = ymin = y[0];
      }
    }
  }
  m.run = 0;
  post(&m.bar[kReq]);
  post(&m.bar[kStart]);
}

// block = W main warps, W power warps, W drive warps
template <class Sys, int PAIR>
__global__ void __launch_bounds__(96 * kMaxTeams) ck_phased_teams_kernel(AdaptArgs a) {
  __shared__ Mailbox boxes[kMaxTeams];
  const int W = (int)blockDim.x / 96, w = (int)(threadIdx.x >> 5);
  if (threadIdx.x < (unsigned)W) {
    // the main warp waits for a stage's power and drive together
    for (int k = 0; k < kBars; ++k) init_bar(boxes[threadIdx.x].bar + k, k >= kAll && k < kAll + 5 ? 2 : 1);
  }
  __syncthreads();
  // Warps of a block go to the sub-partitions in turn.  Of five teams two main warps
  // share one: that with three warps, beside a single helper (131,044 systems x 3
  // periods 81.1 -> 80.5 ms)
  constexpr int kFive[15] = {1, 2, 3, 0, 5, 6, 7, 4, 8, 9, 10, 11, 12, 13, 14};
  const int r = W == 5 ? kFive[w] : w;
  if (r < W) main_warp<Sys, PAIR>(a, boxes[r], W, r);
  else if (r < 2 * W) power_warp<Sys>(a, boxes[r - W]);
  else drive_warp<Sys, PAIR>(a, boxes[r - 2 * W]);
}

}  // namespace

// An adaptive launch of L.block systems per block, with three threads for each:
// Keller-Miksis phase mode with the exponent 21/5, at most 160 systems a block.
cudaError_t launch_ck45_teams(unsigned flags, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s) {
  if (a.n == 0) return cudaSuccess;
  if (a.n_phases <= 0 || (flags & kKmGeneralExponent)) return cudaErrorNotSupported;
  if (L.grid <= 0 || L.grid > 0x7fffffffLL || L.block < 32 || L.block % 32 || L.block > 32 * kMaxTeams)
    return cudaErrorInvalidConfiguration;
  const dim3 g((unsigned)L.grid), b(3 * (unsigned)L.block);
  const bool dual = flags & kKmDual;
  if (a.pair == kDormandPrince) {
    if (dual) ck_phased_teams_kernel<KellerMiksis<true, true>, kDormandPrince><<<g, b, 0, s>>>(a);
    else ck_phased_teams_kernel<KellerMiksis<false, true>, kDormandPrince><<<g, b, 0, s>>>(a);
  } else if (a.pair == kCashKarp) {
    if (dual) ck_phased_teams_kernel<KellerMiksis<true, true>, kCashKarp><<<g, b, 0, s>>>(a);
    else ck_phased_teams_kernel<KellerMiksis<false, true>, kCashKarp><<<g, b, 0, s>>>(a);
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace ens
