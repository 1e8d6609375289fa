// abi.cu -- the C ABI of include/ens.h: contexts, host planner, launch
// selection, CUDA-graph replay and the autotuner.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <tuple>
#include <vector>

#include "common.cuh"

namespace ens {
cudaError_t launch_rk4(int sys, bool strict, const Rk4Args& a, int block, int spt, cudaStream_t s);
cudaError_t launch_ck45(int sys, unsigned flags, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_ck45_fp32c(unsigned flags, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_ck45_df(unsigned flags, bool unrolled, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_ck45_df_teams(unsigned flags, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_ck45_df_events(const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_ck45_teams(unsigned flags, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_ck45_relay(unsigned flags, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_ck45_events_relay(const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_ck45_spt2(int sys, unsigned flags, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s);
cudaError_t launch_order(const int64_t* steps, int64_t n, int32_t* order, unsigned* hist,
                         cudaStream_t s);
cudaError_t launch_rhs_eval(int sys, unsigned flags, int64_t n, const double* P, const double* t,
                            const double* y, double* dy, cudaStream_t s);
}  // namespace ens

using namespace ens;

struct ens_ctx {
  int device = 0;
  int sm_count = 0;
  ens_system sys = ENS_SYS_TOY_X2P;
  ens_solver solver = ENS_RK4;
  ens_tol tol{};
  int64_t n = 0;
  int dim = 0, npar = 0;
  int64_t acc_rows = 0;
  double t0 = 0.0, t1 = 0.0;
  unsigned km_flags = 0;  // Keller-Miksis kernel selection (kKmDual, kKmGeneralExponent)
  // device buffers
  double* params = nullptr;
  double* y0 = nullptr;
  double* y = nullptr;
  double* t_out = nullptr;
  double* dt_out = nullptr;
  double* acc = nullptr;
  int32_t* status = nullptr;
  int64_t* nacc = nullptr;
  int64_t* nrej = nullptr;
  int64_t* nrhs = nullptr;
  int32_t* order = nullptr;     // claim order (cost_order)
  unsigned* hist = nullptr;     // histogram scratch of the claim-order sort
  Scratch* scratch = nullptr;
  ens_launch launch{};
  // who chose it: what the caller set stays, the default and the tuner's choice follow the parameters
  enum { kDefault, kTuned, kCaller } launch_by = kDefault;
  // CUDA graph of one solve
  cudaGraphExec_t gexec = nullptr;
  cudaStream_t graph_stream = nullptr;
  bool graph_valid = false;
  cudaStream_t last_stream = nullptr;
  // events around the main solve kernel of the last solve (ens_kernel_ms)
  cudaEvent_t kev[2] = {nullptr, nullptr};
  bool kev_recorded = false;
  // claim order already in c->order for the tuner's shortened solves
  bool order_ready = false;
  // candidates and main-kernel times of the last ens_autotune
  std::vector<ens_tune_row> tune_rows;
  char err[512] = {0};
};

namespace {

thread_local char g_create_err[512] = {0};

void set_err(ens_ctx* c, const char* fmt, ...) {
  char* buf = c ? c->err : g_create_err;
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, 512, fmt, ap);
  va_end(ap);
}

ens_status cuda_fail(ens_ctx* c, cudaError_t e, const char* what) {
  set_err(c, "%s: %s", what, cudaGetErrorString(e));
  return ENS_ECUDA;
}

#define ENS_CUDA(ctx, call)                                          \
  do {                                                               \
    cudaError_t e_ = (call);                                         \
    if (e_ != cudaSuccess) return cuda_fail((ctx), e_, #call);       \
  } while (0)

// The launch of a context whose caller sets none.  Every line lies between
// measured shapes (GB300, 152 SMs; milliseconds of a whole pass, horizons of 2
// to 6 periods or 16 time units); all shapes give the same results.
//   Up to one warp per SM sub-partition (128 systems per SM) every system
//   starts at once, so an order only costs its pilot, and blocks of one warp
//   put each warp on a sub-partition of its own: FP64 without a team kernel,
//   split precision 16,384 14.4 against 17.4 (160 x 1, longest first).
//   FP64 Keller-Miksis phases with teams: a relay holds a warp of systems and two
//   fit on an SM, so up to there (64 systems per SM) all start at once (5,120: 21.3,
//   with an order 22.7); above, one relay per SM that claims the longest first
//   (19,200: 22.8, all at once in teams 35.0), then two (25,600: 25.1, one 27.6;
//   51,200: 31.5, 3 teams 38.1), then 3 teams (65,536: 38.7, two relays 39.7), 4
//   (90,000, kernel alone: 40.7, 3 teams 49.6), 5 (kernels alone, 560 systems per SM 41.9, 4
//   teams 39.8; 640: 43.1 / 44.8; 131,044 x 2: 52.4 / 59.0; x 4: 110.6, 6 plain warps
//   126.3), then 8 plain
//   warps (200,000 x 2: 78.5, 5 teams 80.3), then 12 (262,144 x 2: 97.0, 5 teams
//   105.1; 524,288: 199 / 209); other FP64 phases 5 warps (65,536: 57.6, 6 warps
//   58.9), then 6 (131,044: 207 / 221 at 5), then 12.  Split precision, kernels
//   alone: 4 (65,536 x 4: 14.2, 8 warps 16.0), then 8 (131,044: 16.2, 4 warps 20.5), 12
//   (262,144: 19.5 / 23.1 at 8), 16 (524,288: 37.9 / 74.9 at 5), 24 from there.
//   Double-float phases, kernels alone: teams on 2 of the sub-partitions (32,768 x 4:
//   54.0, 3 teams 61.0), 3 (65,536: 61.9, 2 teams 80.6), 4 (431 systems per SM x 4 64.7, 3
//   teams 64.4; 439: 64.9 / 65.5; 90,000: 65.8 / 84.1), 6 (650 per SM x 2 38.0, 4 teams 36.0;
//   710: 38.5 / 39.4; 131,044: 81.8 / 95.2), then 12 plain warps (262,144 x 2: 60.8, 8 warps
//   71.1), then 16 (524,288 x 2: 111.6, 12 120.9).  Two frequencies leave the plain
//   launch earlier, as four teams of three warps do not fit (19,200 x 2: 40.8 / 29.2).
//   Valves take about the same number of steps each, and neighbours take them
//   alike, which claiming by cost breaks up: plain launches of 1 warp a block
//   (1,000: 17.0, in one warp a trial 21.5 / 25.4; 32,768: 25.8 / 37.2; 65,536: 46.4 / 60.7; 262,144: 168 /
//   211; 2 warps a block 21.4, 28.2, 46.7 and 170); double-float ones of 8, whose
//   warps share the fetch of a long trial (65,536: 20.8, 1 warp a block 21.8; 524,288:
//   132 / 136; persistent 5 warps per SM 282).
bool has_teams(const ens_ctx* c);

ens_launch default_launch(const ens_ctx* c) {
  ens_launch L{};
  L.mode = ENS_LAUNCH_PLAIN;
  L.block = 32;
  const int64_t per_sm = c->n / std::max(1, c->sm_count);  // systems per SM
  if (c->solver == ENS_RK4) return L;
  if (c->sys == ENS_SYS_RELIEF_VALVE && c->tol.n_phases == 0) {
    if (c->tol.prec == ENS_FP32X2) L.block = 256;
    return L;
  }
  const bool teams = has_teams(c), dual_df = c->tol.prec == ENS_FP32X2 && (c->km_flags & kKmDual);
  if (c->n <= (int64_t)c->sm_count * (teams || dual_df ? 64 : 128)) {
    if (c->tol.prec == ENS_FP32X2) L.block = 64;  // 16,384 x 2: 33.0, one warp a block 35.7
    if (c->tol.prec == ENS_FP64 && !teams) L.block = 128;  // exponent 3.99, 16,384 x 1: 49.6, one warp a block 52.0
    return L;
  }
  L.mode = ENS_LAUNCH_PERSISTENT;
  L.blocks_per_sm = 1;
  L.cost_order = 1;
  if (c->tol.prec == ENS_FP32_COMP) {
    L.block = per_sm < 700 || (per_sm >= 1300 && per_sm < 2600) ? 128 : 256;
    L.blocks_per_sm = per_sm < 1300 ? 1 : per_sm < 2600 ? 3 : per_sm < 5200 ? 2 : 3;
  } else if (c->tol.prec == ENS_FP32X2) {
    L.block = per_sm < 320 ? 64 : per_sm < 440 ? 96 : per_sm < 710 ? 128 : per_sm < 1300 ? 192 : per_sm < 2600 ? 128 : 256;
    L.blocks_per_sm = per_sm < 1300 ? 1 : per_sm < 2600 ? 3 : 2;
  } else if (teams && per_sm < 410) {
    L.block = 32;
    L.blocks_per_sm = per_sm < 145 ? 1 : 2;
  } else if (teams && per_sm < 1300) {
    L.block = per_sm < 480 ? 96 : per_sm < 600 ? 128 : 160;
  } else if (per_sm < 1300) {
    L.block = per_sm < 640 ? 160 : 192;
  } else if (per_sm < 1700 && teams) {
    L.block = 256;
  } else {
    L.block = 128;
    L.blocks_per_sm = 3;
  }
  return L;
}

int spt_of(const ens_launch& L) { return L.systems_per_thread <= 0 ? 1 : L.systems_per_thread; }

bool valid_launch(const ens_launch& L) {
  if (L.mode != ENS_LAUNCH_PLAIN && L.mode != ENS_LAUNCH_PERSISTENT) return false;
  if (L.block < 32 || L.block > 256 || (L.block % 32) != 0) return false;
  if (L.mode == ENS_LAUNCH_PERSISTENT && (L.blocks_per_sm < 1 || L.blocks_per_sm > 32)) return false;
  const int spt = spt_of(L);
  if (spt != 1 && spt != 2 && spt != 4) return false;
  return true;
}

template <class T>
cudaError_t dalloc(T** p, size_t count) {
  *p = nullptr;
  if (count == 0) count = 1;
  return cudaMalloc((void**)p, count * sizeof(T));
}

void free_buffers(ens_ctx* c) {
  cudaFree(c->params);
  cudaFree(c->y0);
  cudaFree(c->y);
  cudaFree(c->t_out);
  cudaFree(c->dt_out);
  cudaFree(c->acc);
  cudaFree(c->status);
  cudaFree(c->nacc);
  cudaFree(c->nrej);
  cudaFree(c->nrhs);
  cudaFree(c->order);
  cudaFree(c->hist);
  cudaFree(c->scratch);
  if (c->gexec) cudaGraphExecDestroy(c->gexec);
  c->gexec = nullptr;
  for (cudaEvent_t& e : c->kev) {
    if (e) cudaEventDestroy(e);
    e = nullptr;
  }
}

// Record one of the main-kernel timing events on s.  Inside a stream capture
// the record becomes an event node of the graph (external record), so every
// replay of the graph records it again.
cudaError_t record_kernel_event(ens_ctx* c, int which, cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &cs);
  if (e != cudaSuccess) return e;
  return cs == cudaStreamCaptureStatusActive ? cudaEventRecordWithFlags(c->kev[which], s, cudaEventRecordExternal)
                                             : cudaEventRecord(c->kev[which], s);
}

ens_status detect_flags(ens_ctx* c) {
  c->km_flags = 0;
  if (!is_km(c->sys) || c->n == 0) return ENS_OK;
  ENS_CUDA(c, cudaMemset(&c->scratch->any_status, 0, sizeof(unsigned)));
  ENS_CUDA(c, launch_km_flags(c->params, c->n, &c->scratch->any_status, 0));
  unsigned flag = 0;
  ENS_CUDA(c, cudaMemcpy(&flag, &c->scratch->any_status, sizeof(unsigned), cudaMemcpyDeviceToHost));
  c->km_flags = flag;
  return ENS_OK;
}

uint64_t timeout_ns(const ens_tol& t) {
  const double s = t.timeout_s > 0.0 ? t.timeout_s : 600.0;
  return (uint64_t)(s * 1e9);
}

// Whether the Keller-Miksis phases of an FP64 launch run in teams of three warps
// per 32 systems (rkck45_teams.cu): up to 5 teams per SM, which is what the
// registers hold and where the FP64 pipe still has room (1,073 to 131,044 systems:
// a seventh to a third faster).  Launches of more warps per SM, chosen where
// systems abound, keep the one-warp kernel: 524,288 systems 199 ms at 12 warps
// per SM against 209 ms in 5 teams.
bool has_teams(const ens_ctx* c) {
  return c->sys == ENS_SYS_KELLER_MIKSIS && c->tol.n_phases > 0 && c->tol.prec == ENS_FP64 &&
         c->solver != ENS_RK4 && !(c->km_flags & kKmGeneralExponent);
}
bool teams_fit(const ens_ctx* c, AdaptLaunch L) {
  return has_teams(c) && L.spt == 1 && L.block <= 160 && L.grid * (L.block / 32) <= 5 * (int64_t)c->sm_count;
}

// Of those, up to two warps of systems per SM run in relays (rkck45_relay.cu), which
// is what the registers hold: the longest system bounds the run, and its trial takes
// two thirds of the teams' time (1 system 30.3 / 19.5 ms, 9,700 x 2 periods 32.6 / 21.9).
bool relay_fits(const ens_ctx* c, AdaptLaunch L) {
  return teams_fit(c, L) && L.grid * (L.block / 32) <= 2 * (int64_t)c->sm_count;
}

// Whether the valves of an FP64 Cash-Karp launch run in relays (valve_relay.cu): blocks
// of one warp of systems, up to the four per SM that fit (1,000 valves x 16 time units
// 21.4 -> 16.8 ms, 19,456 21.6 -> 20.1).
bool valve_relay_fits(const ens_ctx* c, const AdaptArgs& a, AdaptLaunch L) {
  return c->sys == ENS_SYS_RELIEF_VALVE && a.n_phases == 0 && a.pair == kCashKarp && L.spt == 1 && L.block == 32 &&
         L.grid <= 4 * (int64_t)c->sm_count;
}

// The same for double-float phases, in teams of two or three (df64.cu): up to 6 per SM,
// and 8 in persistent blocks of 7 or 8 (131,044 x 2, longest first: 6 teams 40.5 ms, 8 44.5;
// the one-warp kernel in 8 warps 44.9, in 12 60.2; 262,144 x 2: 6 teams 80.1, 12 warps
// 63.6).
bool df_teams_fit(const ens_ctx* c, const AdaptArgs& a, AdaptLaunch L) {
  return L.grid * (L.block / 32) <= (a.persistent && L.block > 192 ? 8 : 6) * (int64_t)c->sm_count;
}

// Whether the other double-float phases take the kernel with unrolled stages: where the
// longest trials bound them, that is for up to 10 warps of systems per SM (37,000 x 2 in
// blocks of 64: 25.4 ms, rolled 31.1; 45,000: 27.2 / 33.1; 65,536, 13 to 14 warps, random
// order: 49.2 / 45.2) and, with one frequency, in up to 8 warps per SM that claim up to four
// systems a lane (65,536 x 2 in 8 warps 30.5 / 33.9; 131,044, longest first, 30.8 / 33.4;
// 262,144 57.1 / 51.1; two frequencies, 131,044: 83.3 / 74.3).
bool df_unrolled(const ens_ctx* c, AdaptLaunch L) {
  const int64_t lanes = L.grid * L.block, warp = 32 * (int64_t)c->sm_count;
  return c->n <= 10 * warp || (!(c->km_flags & kKmDual) && lanes <= 8 * warp && c->n <= 4 * lanes);
}

// the adaptive kernel of the context's precision
cudaError_t launch_adaptive(const ens_ctx* c, const AdaptArgs& a, AdaptLaunch L, cudaStream_t s) {
  if (c->tol.prec == ENS_FP32_COMP) return launch_ck45_fp32c(c->km_flags, a, L, s);
  if (c->tol.prec == ENS_FP32X2) {
    if (c->sys == ENS_SYS_RELIEF_VALVE) return launch_ck45_df_events(a, L, s);
    // a plain launch of up to 8 warps per SM in blocks of two, whatever its own, so that each SM
    // gets its share (16,384 x 2 in 8 warps a block 40.1 -> 26.7 ms; above 6 warps, where as
    // many teams fit, 37,000 x 2 in the one-warp kernel 25.4, in 8 teams a block 41.1)
    if (!a.persistent && L.block > 64 && c->n <= 256 * (int64_t)c->sm_count) L = AdaptLaunch{(c->n + 63) / 64, 64};
    if (!df_teams_fit(c, a, L)) return launch_ck45_df(c->km_flags, df_unrolled(c, L), a, L, s);
    return launch_ck45_df_teams(c->km_flags, a, L, s);
  }
  if (L.spt == 2) return launch_ck45_spt2(c->sys, c->km_flags, a, L, s);
  if (valve_relay_fits(c, a, L)) return launch_ck45_events_relay(a, L, s);
  if (relay_fits(c, L)) return launch_ck45_relay(c->km_flags, a, AdaptLaunch{L.grid * (L.block / 32), 32}, s);
  if (teams_fit(c, L)) {
    // a plain launch in blocks of one team, whatever its own: five of those fit on an SM, but
    // two of two teams and one of three or four, whose rest would wait for the first ones
    // (24,320 x 2 in blocks of two and four teams 44.3 and 47.1 ms, of one 27.4; 20,000 x 2 in
    // blocks of three 43.5, of one 26.3).  Persistent launches keep theirs: resident blocks claim
    // for those that wait (20,000 x 2 in 128 x 2 25.6)
    if (!a.persistent) L = AdaptLaunch{(c->n + 31) / 32, 32};
    return launch_ck45_teams(c->km_flags, a, L, s);
  }
  return launch_ck45(c->sys, c->km_flags, a, L, s);
}

// Two systems per thread: the FP64 Cash-Karp phase mode of the Keller-Miksis
// model with one driving frequency and the exponent 21/5, persistent launch
// of at most 128 threads per block.  The static part is checked when the
// launch is set, the parameter-dependent part (km_flags) when it runs.
bool spt2_static_ok(const ens_ctx* c, const ens_launch& L) {
  return c->solver == ENS_RKCK45 && c->sys == ENS_SYS_KELLER_MIKSIS && c->tol.n_phases > 0 &&
         (c->tol.prec == ENS_FP64 || c->tol.prec == ENS_FP64_STRICT) && L.mode == ENS_LAUNCH_PERSISTENT &&
         L.block <= 128;
}
const char* kSpt2Msg =
    "systems_per_thread 2 runs the FP64 Cash-Karp phase mode of the Keller-Miksis model (one driving frequency, "
    "C10 = 21/5) in a persistent launch of at most 128 threads per block; the other adaptive solves take 1";

AdaptArgs adapt_args(ens_ctx* c) {
  AdaptArgs a{};
  a.n = c->n;
  a.params = c->params;
  a.y0 = c->y0;
  a.y = c->y;
  a.t_out = c->t_out;
  a.dt_out = c->dt_out;
  a.acc = c->acc;
  a.status = c->status;
  a.nacc = c->nacc;
  a.nrej = c->nrej;
  a.nrhs = c->nrhs;
  a.order = nullptr;
  a.scratch = c->scratch;
  a.rtol = c->tol.rtol;
  a.atol = c->tol.atol;
  a.dt0 = c->tol.dt0;
  a.dt_min = c->tol.dt_min;
  a.dt_max = c->tol.dt_max;
  a.event_tol = c->tol.event_tol;
  a.t0 = c->t0;
  a.t1 = c->t1;
  a.phase_len = c->tol.phase_len;
  a.acc_t_start = c->tol.acc_t_start;
  a.max_steps = c->tol.max_steps;
  a.n_phases = c->tol.n_phases;
  a.n_transient = c->tol.n_transient;
  a.acc_phases = c->tol.n_phases - c->tol.n_transient;
  a.persistent = 0;
  a.pair = c->solver == ENS_DOPRI5 ? kDormandPrince : kCashKarp;
  a.timeout_ns = timeout_ns(c->tol);
  return a;
}

AdaptLaunch adapt_launch(const ens_ctx* c, const ens_launch& L) {
  AdaptLaunch out;
  out.block = L.block;
  out.spt = spt_of(L);
  if (L.mode == ENS_LAUNCH_PERSISTENT) {
    out.grid = (int64_t)c->sm_count * L.blocks_per_sm;
    const int64_t slots = (int64_t)L.block * out.spt;
    const int64_t need = (c->n + slots - 1) / slots;  // never more lanes than systems
    if (out.grid > need) out.grid = need;
    if (out.grid < 1) out.grid = 1;
  } else {
    out.grid = (c->n + L.block - 1) / L.block;
  }
  return out;
}

// The claim order for longest-first scheduling: a pilot of one phase (or 1/16
// of the horizon) of every system in plain mode, then the systems sorted by
// decreasing pilot step count into c->order.  The pilot only ranks the
// systems (the claim order never changes what a system computes), so it runs at
// a tolerance of at least kPilotTol, and Keller-Miksis phases are ranked at
// kPhasePilotTol in split precision: a trial of the
// longest system, which bounds the pilot, takes 2.9 us there against 10.4 us
// in FP64 (131,044 systems: pilot and sort 1.6 ms, at 1e-7 in FP64 14).
// The tangent system keeps a pilot of its own: its steps follow the tangent vector too
// (131,044 x 2 periods 173 ms, ranked by the plain system 240).
// kPilotTrials bounds a system whose float pilot would be held up by rounding; it
// ranks with the longest.
ens_status enqueue_order(ens_ctx* c, const AdaptArgs& a, cudaStream_t s) {
  AdaptArgs p = a;
  p.persistent = 0;
  p.order = nullptr;
  if (p.n_phases > 0) {
    p.n_phases = 1;
    p.n_transient = 0;
    p.acc_phases = 1;
  } else {
    p.t1 = p.t0 + (p.t1 - p.t0) / 16.0;
  }
  const bool split = c->sys == ENS_SYS_KELLER_MIKSIS && p.n_phases > 0;
  const double loosest = split ? kPhasePilotTol : kPilotTol;
  p.rtol = std::max(p.rtol, loosest);
  p.atol = std::max(p.atol, loosest);
  AdaptLaunch PL{(c->n + 127) / 128, 128};
  cudaError_t e;
  if (split) {
    p.max_steps = std::min<int64_t>(p.max_steps, kPilotTrials);
    e = launch_ck45_fp32c(c->km_flags, p, PL, s);
  } else {
    e = launch_adaptive(c, p, PL, s);
  }
  if (e != cudaSuccess) return cuda_fail(c, e, "pilot launch");
  e = launch_order(c->nacc, c->n, c->order, c->hist, s);
  if (e != cudaSuccess) return cuda_fail(c, e, "order launch");
  ENS_CUDA(c, cudaMemsetAsync(c->scratch, 0, sizeof(Scratch), s));
  return ENS_OK;
}

// Enqueue one solve (no graph) with launch L.  frac < 1 runs the same systems
// over a fraction of the horizon, for the tuner: phase mode keeps
// max(1, round(frac n_phases)) phases (transient phases scaled alike),
// event and plain mode integrate frac of [t0, t1], RK4 takes
// max(1, round(frac n_steps)) steps.  A shortened solve reuses the claim
// order the tuner computed (order_ready) instead of running its own pilot.
ens_status enqueue_solve(ens_ctx* c, const ens_launch& L, cudaStream_t s, double frac = 1.0) {
  const bool full = !(frac < 1.0);
  ENS_CUDA(c, cudaMemsetAsync(c->scratch, 0, sizeof(Scratch), s));
  if (c->solver == ENS_RK4) {
    Rk4Args a{};
    a.n = c->n;
    a.params = c->params;
    a.y0 = c->y0;
    a.y = c->y;
    a.t_out = c->t_out;
    a.dt_out = c->dt_out;
    a.status = c->status;
    a.nacc = c->nacc;
    a.nrej = c->nrej;
    a.nrhs = c->nrhs;
    a.scratch = c->scratch;
    a.t0 = c->t0;
    a.dt = c->tol.dt0;
    a.nsteps = full ? c->tol.n_steps
                    : std::min<int64_t>(c->tol.n_steps, std::max<int64_t>(1, std::llround(frac * c->tol.n_steps)));
    ENS_CUDA(c, record_kernel_event(c, 0, s));
    cudaError_t e = launch_rk4(c->sys, c->tol.prec == ENS_FP64_STRICT, a, L.block, spt_of(L), s);
    if (e != cudaSuccess) return cuda_fail(c, e, "rk4 launch");
    ENS_CUDA(c, record_kernel_event(c, 1, s));
    c->kev_recorded = true;
    return ENS_OK;
  }
  if (c->tol.prec == ENS_FP32X2 && (c->km_flags & kKmGeneralExponent)) {
    set_err(c, "ENS_FP32X2 needs C10 = 21/5 (polytropic exponent 1.4) in every system");
    return ENS_ENOTSUP;
  }
  if (spt_of(L) != 1 &&
      (spt_of(L) != 2 || !spt2_static_ok(c, L) || (c->km_flags & (kKmDual | kKmGeneralExponent)))) {
    set_err(c, "%s", kSpt2Msg);
    return ENS_ENOTSUP;
  }
  AdaptArgs a = adapt_args(c);
  if (!full) {
    if (a.n_phases > 0) {
      const int32_t np = (int32_t)std::max<long long>(1, std::llround(frac * a.n_phases));
      const int32_t nt = std::min<int32_t>((int32_t)(frac * a.n_transient), np - 1);
      a.n_phases = std::min(a.n_phases, np);
      a.n_transient = std::max<int32_t>(0, std::min(a.n_transient, nt));
      a.acc_phases = a.n_phases - a.n_transient;
    } else {
      a.t1 = a.t0 + (a.t1 - a.t0) * frac;
    }
  }
  a.persistent = L.mode == ENS_LAUNCH_PERSISTENT;
  if (a.persistent && L.cost_order) {
    if (full || !c->order_ready) {
      ens_status st = enqueue_order(c, adapt_args(c), s);
      if (st != ENS_OK) return st;
    }
    a.order = c->order;
  }
  AdaptLaunch AL = adapt_launch(c, L);
  // the phase-mode FP64 and tangent kernels rank the first claims by
  // sub-partition when one block runs per SM
  a.first_by_subpartition = a.persistent && a.order && a.n_phases > 0 && L.blocks_per_sm == 1 &&
                            spt_of(L) == 1 && (c->tol.prec == ENS_FP64 || c->tol.prec == ENS_FP64_STRICT);
  ENS_CUDA(c, record_kernel_event(c, 0, s));
  cudaError_t e = launch_adaptive(c, a, AL, s);
  if (e != cudaSuccess) return cuda_fail(c, e, "adaptive launch");
  ENS_CUDA(c, record_kernel_event(c, 1, s));
  c->kev_recorded = true;
  return ENS_OK;
}

std::mutex g_tune_mu;

}  // namespace

namespace ens {
// Message of a failed call that has no context, returned by ens_last_error(NULL).
void set_call_error(const char* msg) { set_err(nullptr, "%s", msg); }

// Keller-Miksis kernel selection: bit kKmDual if any system drives with a
// second frequency (C6 or C8 != 0), bit kKmGeneralExponent if any C10 is not
// within 4 ulp of 21/5 (then pow() is used instead of the fifth-root form).
__global__ void km_flags_kernel(const double* C, int64_t n, unsigned* flags) {
  const double lo = 4.2 - 4 * 8.881784197001252e-16, hi = 4.2 + 4 * 8.881784197001252e-16;
  unsigned f = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (C[6 * n + i] != 0.0 || C[8 * n + i] != 0.0) f |= kKmDual;
    const double e = C[10 * n + i];
    if (!(e >= lo && e <= hi)) f |= kKmGeneralExponent;
  }
  if (f) atomicOr(flags, f);
}

cudaError_t launch_km_flags(const double* C, int64_t n, unsigned* flags, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4096);
  km_flags_kernel<<<(unsigned)blocks, 256, 0, s>>>(C, n, flags);
  return cudaGetLastError();
}

ens_status check_tol(ens_ctx* c, ens_solver solver, ens_system sys, const ens_tol& t) {
  if (solver == ENS_RK4) {
    if (!(t.dt0 > 0.0) || t.n_steps < 0) {
      set_err(c, "RK4 needs dt0 > 0 and n_steps >= 0");
      return ENS_EINVAL;
    }
    if (sys != ENS_SYS_TOY_X2P && sys != ENS_SYS_LORENZ) {
      set_err(c, "RK4 runs the smooth systems (x2p, Lorenz); the relief valve needs event "
                 "handling and Keller-Miksis needs step control");
      return ENS_ENOTSUP;
    }
    if (t.prec != ENS_FP64 && t.prec != ENS_FP64_STRICT) {
      set_err(c, "RK4 supports ENS_FP64 and ENS_FP64_STRICT");
      return ENS_ENOTSUP;
    }
    return ENS_OK;
  }
  if (!(t.rtol >= 0.0) || !(t.atol >= 0.0) || !(t.rtol > 0.0 || t.atol > 0.0) || !(t.dt0 > 0.0) ||
      !(t.dt_min > 0.0) || !(t.dt_max >= t.dt_min) || t.max_steps <= 0 || t.n_phases < 0) {
    set_err(c, "adaptive solve needs rtol, atol >= 0 (not both 0), 0 < dt_min <= dt_max, dt0 > 0, "
               "max_steps > 0, n_phases >= 0");
    return ENS_EINVAL;
  }
  if (t.n_phases > 0 && !(t.phase_len > 0.0)) {
    set_err(c, "phase mode needs phase_len > 0");
    return ENS_EINVAL;
  }
  if (t.n_transient < 0 || (t.n_phases > 0 ? t.n_transient >= t.n_phases : t.n_transient != 0)) {
    set_err(c, "n_transient must satisfy 0 <= n_transient < n_phases (0 outside phase mode)");
    return ENS_EINVAL;
  }
  if (sys == ENS_SYS_RELIEF_VALVE && !(t.event_tol > 0.0)) {
    set_err(c, "the relief valve needs event_tol > 0");
    return ENS_EINVAL;
  }
  if (sys == ENS_SYS_KELLER_MIKSIS_TANGENT && !(t.n_phases > 0 && t.prec == ENS_FP64)) {
    set_err(c, "the tangent system runs in phase mode (n_phases > 0) in FP64");
    return ENS_ENOTSUP;
  }
  if (sys == ENS_SYS_RELIEF_VALVE && t.n_phases > 0) {
    set_err(c, "the relief valve runs in event mode (n_phases must be 0)");
    return ENS_ENOTSUP;
  }
  if (t.prec == ENS_FP32_COMP && !(sys == ENS_SYS_KELLER_MIKSIS && t.n_phases > 0 && solver == ENS_RKCK45)) {
    set_err(c, "ENS_FP32_COMP is implemented for the Keller-Miksis phase mode with Cash-Karp");
    return ENS_ENOTSUP;
  }
  if (t.prec == ENS_FP32X2 && !(solver == ENS_RKCK45 && ((sys == ENS_SYS_KELLER_MIKSIS && t.n_phases > 0) ||
                                                          (sys == ENS_SYS_RELIEF_VALVE && t.n_phases == 0)))) {
    set_err(c, "ENS_FP32X2 is implemented with Cash-Karp for the Keller-Miksis phase mode and the relief "
               "valve's event mode");
    return ENS_ENOTSUP;
  }
  if (t.prec != ENS_FP64 && t.prec != ENS_FP32_COMP && t.prec != ENS_FP32X2) {
    set_err(c, "adaptive solves support ENS_FP64, ENS_FP32_COMP and ENS_FP32X2");
    return ENS_ENOTSUP;
  }
  return ENS_OK;
}

}  // namespace ens

namespace {

// tuned launch and its candidate table per (system, solver, precision, n,
// phases, transient phases, horizon, device, tolerances, kind of parameters: the
// kernels and the candidates depend on km_flags)
std::map<std::tuple<int, int, int, int64_t, int, int, double, int, double, double, unsigned>,
         std::pair<ens_launch, std::vector<ens_tune_row>>>
    g_tune_cache;

}  // namespace

extern "C" {

const char* ens_version(void) { return "ens 0.1 (sm_103a)"; }

ens_status ens_create(ens_ctx** out, ens_system sys, int64_t n, const double* params,
                      const double* y0, const double t_span[2], ens_solver solver,
                      const ens_tol* tol) {
  if (!out) {
    set_err(nullptr, "out is NULL");
    return ENS_EINVAL;
  }
  *out = nullptr;
  if (n < 0 || !tol || !t_span || (n > 0 && (!params || !y0))) {
    set_err(nullptr, "bad arguments: n < 0 or a NULL tol / t_span / params / y0");
    return ENS_EINVAL;
  }
  if (sys_dim(sys) == 0) {
    set_err(nullptr, "unknown system %d", (int)sys);
    return ENS_EINVAL;
  }
  if (solver != ENS_RK4 && solver != ENS_RKCK45 && solver != ENS_DOPRI5) {
    set_err(nullptr, "unknown solver %d", (int)solver);
    return ENS_EINVAL;
  }
  ens_status st = check_tol(nullptr, solver, sys, *tol);
  if (st != ENS_OK) return st;
  if (solver != ENS_RK4 && tol->n_phases == 0 && !(t_span[1] > t_span[0])) {
    set_err(nullptr, "t_span[1] must exceed t_span[0]");
    return ENS_EINVAL;
  }
  ens_ctx* c = new (std::nothrow) ens_ctx();
  if (!c) {
    set_err(nullptr, "host allocation failed");
    return ENS_ENOMEM;
  }
  c->sys = sys;
  c->solver = solver;
  c->tol = *tol;
  c->n = n;
  c->dim = sys_dim(sys);
  c->npar = sys_npar(sys);
  c->t0 = t_span[0];
  c->t1 = t_span[1];
  if (solver != ENS_RK4) {
    if (tol->n_phases > 0)
      c->acc_rows = (sys == ENS_SYS_KELLER_MIKSIS_TANGENT ? 3 : 2) * (int64_t)(tol->n_phases - tol->n_transient);
    else if (sys == ENS_SYS_RELIEF_VALVE) c->acc_rows = kPrvAccRows;
  }
  cudaError_t e = cudaGetDevice(&c->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device);
  const size_t nn = (size_t)n;
  if (e == cudaSuccess) e = dalloc(&c->params, nn * c->npar);
  if (e == cudaSuccess) e = dalloc(&c->y0, nn * c->dim);
  if (e == cudaSuccess) e = dalloc(&c->y, nn * c->dim);
  if (e == cudaSuccess) e = dalloc(&c->t_out, nn);
  if (e == cudaSuccess) e = dalloc(&c->dt_out, nn);
  if (e == cudaSuccess) e = dalloc(&c->acc, nn * (size_t)std::max<int64_t>(c->acc_rows, 1));
  if (e == cudaSuccess) e = dalloc(&c->status, nn);
  if (e == cudaSuccess) e = dalloc(&c->nacc, nn);
  if (e == cudaSuccess) e = dalloc(&c->nrej, nn);
  if (e == cudaSuccess) e = dalloc(&c->nrhs, nn);
  if (e == cudaSuccess) e = dalloc(&c->order, nn);
  if (e == cudaSuccess) e = dalloc(&c->hist, 512);
  if (e == cudaSuccess) e = dalloc(&c->scratch, 1);
  if (e == cudaSuccess) e = cudaEventCreate(&c->kev[0]);
  if (e == cudaSuccess) e = cudaEventCreate(&c->kev[1]);
  if (e != cudaSuccess) {
    set_err(nullptr, "device allocation: %s", cudaGetErrorString(e));
    free_buffers(c);
    delete c;
    return e == cudaErrorMemoryAllocation ? ENS_ENOMEM : ENS_ECUDA;
  }
  // zero the outputs so that reads before a solve are defined
  const size_t zero_sizes[] = {nn * c->dim * sizeof(double), nn * sizeof(double), nn * sizeof(double),
                               nn * (size_t)std::max<int64_t>(c->acc_rows, 1) * sizeof(double),
                               nn * sizeof(int32_t), nn * sizeof(int64_t), nn * sizeof(int64_t),
                               nn * sizeof(int64_t)};
  void* zero_ptrs[] = {c->y, c->t_out, c->dt_out, c->acc, c->status, c->nacc, c->nrej, c->nrhs};
  for (int k = 0; k < 8 && e == cudaSuccess; ++k)
    if (zero_sizes[k]) e = cudaMemset(zero_ptrs[k], 0, zero_sizes[k]);
  if (e == cudaSuccess && n > 0)
    e = cudaMemcpy(c->params, params, nn * c->npar * sizeof(double), cudaMemcpyDefault);
  if (e == cudaSuccess && n > 0) e = cudaMemcpy(c->y0, y0, nn * c->dim * sizeof(double), cudaMemcpyDefault);
  if (e == cudaSuccess) e = cudaMemset(c->scratch, 0, sizeof(Scratch));
  if (e != cudaSuccess) {
    set_err(nullptr, "input copy: %s", cudaGetErrorString(e));
    free_buffers(c);
    delete c;
    return ENS_ECUDA;
  }
  st = detect_flags(c);
  if (st != ENS_OK) {
    set_err(nullptr, "%s", c->err);
    free_buffers(c);
    delete c;
    return st;
  }
  c->launch = default_launch(c);
  *out = c;
  return ENS_OK;
}

ens_status ens_set_inputs(ens_ctx* c, const double* params, const double* y0, void* stream) {
  if (!c) return ENS_EINVAL;
  if (c->n == 0) return ENS_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t nn = (size_t)c->n;
  if (params)
    ENS_CUDA(c, cudaMemcpyAsync(c->params, params, nn * c->npar * sizeof(double), cudaMemcpyDefault, s));
  if (y0) ENS_CUDA(c, cudaMemcpyAsync(c->y0, y0, nn * c->dim * sizeof(double), cudaMemcpyDefault, s));
  c->last_stream = s;
  if (params && is_km(c->sys)) {
    ENS_CUDA(c, cudaStreamSynchronize(s));
    const unsigned was = c->km_flags;
    ens_status st = detect_flags(c);
    if (st != ENS_OK) return st;
    if (was != c->km_flags) {
      c->graph_valid = false;
      if (c->launch_by != ens_ctx::kCaller) {
        const int graph = c->launch.use_graph;
        c->launch = default_launch(c);
        c->launch.use_graph = graph;
        c->launch_by = ens_ctx::kDefault;
      }
    }
  }
  return ENS_OK;
}

ens_status ens_set_launch(ens_ctx* c, const ens_launch* cfg) {
  if (!c) return ENS_EINVAL;
  ens_launch L = cfg ? *cfg : default_launch(c);
  if (!valid_launch(L)) {
    set_err(c, "invalid launch: mode %d block %d blocks_per_sm %d", L.mode, L.block, L.blocks_per_sm);
    return ENS_EINVAL;
  }
  if (c->solver == ENS_RK4 && L.mode != ENS_LAUNCH_PLAIN) {
    set_err(c, "RK4 runs a plain launch (systems_per_thread systems per thread)");
    return ENS_ENOTSUP;
  }
  if (c->solver != ENS_RK4 && spt_of(L) != 1 && (spt_of(L) != 2 || !spt2_static_ok(c, L))) {
    set_err(c, "%s", kSpt2Msg);
    return ENS_ENOTSUP;
  }
  c->launch = L;
  c->launch_by = cfg ? ens_ctx::kCaller : ens_ctx::kDefault;
  c->graph_valid = false;
  return ENS_OK;
}

ens_status ens_get_launch(const ens_ctx* c, ens_launch* cfg) {
  if (!c || !cfg) return ENS_EINVAL;
  *cfg = c->launch;
  return ENS_OK;
}

ens_status ens_solve(ens_ctx* c, void* stream) {
  if (!c) return ENS_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  c->last_stream = s;
  if (c->n == 0) return ENS_OK;
  if (!c->launch.use_graph) return enqueue_solve(c, c->launch, s);
  if (!c->graph_valid || c->graph_stream != s) {
    if (c->gexec) cudaGraphExecDestroy(c->gexec);
    c->gexec = nullptr;
    cudaGraph_t g = nullptr;
    // a private capture stream keeps the caller's stream free of capture state
    cudaStream_t cap = nullptr;
    ENS_CUDA(c, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
      cudaStreamDestroy(cap);
      return cuda_fail(c, e, "cudaStreamBeginCapture");
    }
    ens_status st = enqueue_solve(c, c->launch, cap);
    e = cudaStreamEndCapture(cap, &g);
    cudaStreamDestroy(cap);
    if (st != ENS_OK) {
      if (g) cudaGraphDestroy(g);
      return st;
    }
    if (e != cudaSuccess) return cuda_fail(c, e, "cudaStreamEndCapture");
    e = cudaGraphInstantiate(&c->gexec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(c, e, "cudaGraphInstantiate");
    c->graph_valid = true;
    c->graph_stream = s;
  }
  ENS_CUDA(c, cudaGraphLaunch(c->gexec, s));
  return ENS_OK;
}

ens_status ens_sync(ens_ctx* c) {
  if (!c) return ENS_EINVAL;
  ENS_CUDA(c, cudaStreamSynchronize(c->last_stream));
  if (c->n == 0) return ENS_OK;
  unsigned any = 0;
  ENS_CUDA(c, cudaMemcpy(&any, &c->scratch->any_status, sizeof(unsigned), cudaMemcpyDeviceToHost));
  if (any & kStTimeout) {
    set_err(c, "solve stopped at its wall-clock budget (%.1f s)", c->tol.timeout_s);
    return ENS_ETIMEOUT;
  }
  if (any) {
    set_err(c, "some systems finished with status bits 0x%x", any);
    return ENS_ESYSTEM;
  }
  return ENS_OK;
}

ens_status ens_kernel_ms(ens_ctx* c, double* ms) {
  if (!c || !ms) return ENS_EINVAL;
  *ms = 0.0;
  if (!c->kev_recorded) {
    set_err(c, "no solve kernel has been enqueued on this context");
    return ENS_EINVAL;
  }
  float f = 0.0f;
  ENS_CUDA(c, cudaEventElapsedTime(&f, c->kev[0], c->kev[1]));
  *ms = (double)f;
  return ENS_OK;
}

ens_status ens_read(ens_ctx* c, int which, void* dst, size_t dst_bytes) {
  if (!c) return ENS_EINVAL;
  const size_t nn = (size_t)c->n;
  const void* src = nullptr;
  size_t bytes = 0;
  switch (which) {
    case ENS_STATE: src = c->y; bytes = nn * c->dim * sizeof(double); break;
    case ENS_ACC: src = c->acc; bytes = nn * (size_t)c->acc_rows * sizeof(double); break;
    case ENS_STATUS: src = c->status; bytes = nn * sizeof(int32_t); break;
    case ENS_NSTEPS: src = c->nacc; bytes = nn * sizeof(int64_t); break;
    case ENS_NREJ: src = c->nrej; bytes = nn * sizeof(int64_t); break;
    case ENS_NRHS: src = c->nrhs; bytes = nn * sizeof(int64_t); break;
    case ENS_TIME: src = c->t_out; bytes = nn * sizeof(double); break;
    case ENS_DT: src = c->dt_out; bytes = nn * sizeof(double); break;
    default: set_err(c, "unknown selector %d", which); return ENS_EINVAL;
  }
  if (bytes == 0) return ENS_OK;
  if (!dst || dst_bytes < bytes) {
    set_err(c, "destination holds %zu bytes, selector %d needs %zu", dst_bytes, which, bytes);
    return ENS_EINVAL;
  }
  ENS_CUDA(c, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, c->last_stream));
  ENS_CUDA(c, cudaStreamSynchronize(c->last_stream));
  return ENS_OK;
}

int64_t ens_acc_rows(const ens_ctx* c) { return c ? c->acc_rows : 0; }
int64_t ens_size(const ens_ctx* c) { return c ? c->n : 0; }
int32_t ens_dim(const ens_ctx* c) { return c ? c->dim : 0; }
int32_t ens_npar(const ens_ctx* c) { return c ? c->npar : 0; }

ens_status ens_autotune(ens_ctx* c, void* stream, ens_launch* best) {
  if (!c) return ENS_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  c->last_stream = s;
  if (c->n == 0) {
    if (best) *best = c->launch;
    return ENS_OK;
  }
  const double horizon = c->solver == ENS_RK4 ? (double)c->tol.n_steps : c->t1 - c->t0;
  const auto key = std::make_tuple((int)c->sys, (int)c->solver, (int)c->tol.prec, c->n,
                                   (int)c->tol.n_phases, (int)c->tol.n_transient, horizon, c->device, c->tol.rtol,
                                   c->tol.atol, c->km_flags);
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) {
      const bool graph = c->launch.use_graph;
      c->launch = it->second.first;
      c->launch_by = ens_ctx::kTuned;
      c->launch.use_graph = graph;
      c->tune_rows = it->second.second;
      c->graph_valid = false;
      if (best) *best = c->launch;
      return ENS_OK;
    }
  }
  c->tune_rows.clear();
  auto mk = [](int mode, int block, int bps, int co, int spt) {
    ens_launch L{};
    L.mode = mode;
    L.block = block;
    L.blocks_per_sm = bps;
    L.cost_order = co;
    L.systems_per_thread = spt;
    return L;
  };
  // Time one candidate: the main kernel of a shortened solve (CUDA events
  // recorded by enqueue_solve around that launch).
  double frac = 1.0;
  auto time_one = [&](const ens_launch& L, float* ms) -> ens_status {
    ens_status st = enqueue_solve(c, L, s, frac);
    if (st != ENS_OK) return st;
    ENS_CUDA(c, cudaStreamSynchronize(s));
    ENS_CUDA(c, cudaEventElapsedTime(ms, c->kev[0], c->kev[1]));
    c->tune_rows.push_back(ens_tune_row{L, (double)*ms, frac});
    return ENS_OK;
  };
  ens_launch best_L = c->launch;
  float best_ms = 1e30f;
  auto consider = [&](const ens_launch& L) -> ens_status {
    float ms = 0.f;
    ens_status st = time_one(L, &ms);
    if (st != ENS_OK) return st;
    if (ms < best_ms) {
      best_ms = ms;
      best_L = L;
    }
    return ENS_OK;
  };
  ens_status st = ENS_OK;
  if (c->solver == ENS_RK4) {
    // fixed step: every system takes the same steps, so the shape only
    // decides occupancy and ILP (systems per thread).  Whole solves up to
    // 1e9 system-steps (Lorenz at N = 768,000 takes about 40 ms), else an
    // eighth of the steps; each candidate runs twice (the first launch of a
    // kernel variant includes its loading) and keeps the faster time.
    frac = (double)c->n * (double)c->tol.n_steps <= 1e9 ? 1.0 : 0.125;
    for (int spt : {1, 2, 4})
      for (int b : {32, 64, 128, 256}) {
        if (st != ENS_OK) break;
        const ens_launch L = mk(ENS_LAUNCH_PLAIN, b, 0, 0, spt);
        float ms0 = 0.f, ms1 = 0.f;
        st = time_one(L, &ms0);
        if (st == ENS_OK) st = time_one(L, &ms1);
        if (st != ENS_OK) break;
        // one row per candidate, holding the timing the choice uses (the faster)
        c->tune_rows.erase(c->tune_rows.end() - 2);
        c->tune_rows.back().ms = (double)std::min(ms0, ms1);
        if (std::min(ms0, ms1) < best_ms) {
          best_ms = std::min(ms0, ms1);
          best_L = L;
        }
      }
  } else {
    // Adaptive: the run time is the larger of the throughput bound (more
    // warps per SM feed the FP64 pipe better) and the longest system's chain
    // (every warp that shares an SM slows it).  Both scale with the horizon,
    // so an eighth of the phases (or of the time span) of every system keeps
    // the balance of the full solve.  The claim order comes from the same
    // one-phase pilot as the full solve's and is computed once here.
    frac = 0.125;
    if (c->tol.n_phases > 0 && c->tol.n_phases < 8) frac = 1.0;
    AdaptArgs a = adapt_args(c);
    st = enqueue_order(c, a, s);
    if (st == ENS_OK) c->order_ready = true;
    // warm-up at the default shape; shrink the horizon while one shortened
    // solve takes more than 0.6 s (down to one phase or 1/128 of the span)
    float ms = 0.f;
    const ens_launch L0 = mk(ENS_LAUNCH_PERSISTENT, 160, 1, 1, 1);
    if (st == ENS_OK) st = enqueue_solve(c, L0, s, frac);
    if (st == ENS_OK) {
      cudaError_t e = cudaStreamSynchronize(s);
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, c->kev[0], c->kev[1]);
      if (e != cudaSuccess) st = cuda_fail(c, e, "autotune warm-up");
    }
    // at least two phases: the first one holds the transient from the initial state
    const double min_frac = c->tol.n_phases > 0 ? 2.0 / c->tol.n_phases : 1.0 / 128;
    while (st == ENS_OK && ms > 600.f) {
      if (frac * 0.5 < min_frac) break;
      frac *= 0.5;
      ms *= 0.5f;
    }
    // warps per SM, block, blocks per SM
    const int shapes[][3] = {{3, 96, 1},  {4, 128, 1},  {5, 160, 1},  {6, 192, 1},  {7, 224, 1},
                             {8, 256, 1}, {12, 192, 2}, {16, 256, 2}, {24, 256, 3}};
    // the launch of an untuned context, where the lists below lack it
    const ens_launch untuned = default_launch(c);
    const bool plain = untuned.mode == ENS_LAUNCH_PLAIN;
    bool listed = plain;
    for (const auto& sh : shapes) listed |= sh[1] == untuned.block && sh[2] == untuned.blocks_per_sm;
    const bool relays = has_teams(c) && c->n > 64 * (int64_t)c->sm_count;   // not every system starts at once
    listed |= relays && untuned.block == 32;
    if (st == ENS_OK && !listed) st = consider(mk(untuned.mode, untuned.block, untuned.blocks_per_sm, untuned.cost_order, 1));
    if (relays)
      for (const int bps : {1, 2})
        if (st == ENS_OK) st = consider(mk(ENS_LAUNCH_PERSISTENT, 32, bps, 1, 1));
    for (const auto& sh : shapes)
      if (st == ENS_OK) st = consider(mk(ENS_LAUNCH_PERSISTENT, sh[1], sh[2], 1, 1));
    // the best of these without longest-first claiming, and a plain launch
    if (st == ENS_OK) st = consider(mk(ENS_LAUNCH_PERSISTENT, best_L.block, best_L.blocks_per_sm, 0, 1));
    if (st == ENS_OK) st = consider(mk(ENS_LAUNCH_PLAIN, plain ? untuned.block : 128, 0, 0, 1));
    // two systems per thread where the kernel exists: 6 and 8 warps per SM
    // (236 registers a thread leave room for 8), longest first
    for (const int b : {96, 128}) {
      const ens_launch L2 = mk(ENS_LAUNCH_PERSISTENT, b, 2, 1, 2);
      if (st == ENS_OK && spt2_static_ok(c, L2) && !(c->km_flags & (kKmDual | kKmGeneralExponent)))
        st = consider(L2);
    }
    // The two fastest candidates again on twice the horizon, and the faster
    // of those is the choice: shapes whose tails differ (a plain launch waits
    // for the longest system of every block, a persistent one refills its
    // lanes) can trade places as the horizon grows, and on the 1024 x 1024
    // double-float grid a plain launch that led on 1/32 of the horizon took
    // 12.8 s against 10.0 s for the persistent shape on the whole solve.
    if (st == ENS_OK && frac < 1.0 && c->tune_rows.size() >= 2) {
      std::vector<ens_tune_row> ranked(c->tune_rows.begin(), c->tune_rows.end());
      std::stable_sort(ranked.begin(), ranked.end(),
                       [](const ens_tune_row& x, const ens_tune_row& y) { return x.ms < y.ms; });
      frac = std::min(1.0, 2.0 * frac);
      best_ms = 1e30f;
      for (int r = 0; r < 2 && st == ENS_OK; ++r) st = consider(ranked[r].launch);
    }
    c->order_ready = false;
  }
  if (st != ENS_OK) return st;
  best_L.use_graph = c->launch.use_graph;
  c->launch = best_L;
  c->launch_by = ens_ctx::kTuned;
  c->graph_valid = false;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache[key] = std::make_pair(best_L, c->tune_rows);
  }
  if (best) *best = best_L;
  return ENS_OK;
}

int32_t ens_autotune_table(const ens_ctx* c, ens_tune_row* rows, int32_t cap) {
  if (!c) return 0;
  const int32_t n = (int32_t)c->tune_rows.size();
  for (int32_t k = 0; k < n && k < cap && rows; ++k) rows[k] = c->tune_rows[k];
  return n;
}

ens_status ens_eval_rhs(ens_system sys, int64_t n, const double* params, const double* t, const double* y,
                        double* dy, void* stream) {
  if (n < 0 || sys_dim(sys) == 0) return ENS_EINVAL;
  if (n == 0) return ENS_OK;
  if (!params || !t || !y || !dy) return ENS_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned flags = 0;
  if (is_km(sys)) {
    unsigned* f = nullptr;
    if (cudaMalloc(&f, sizeof(unsigned)) != cudaSuccess) return ENS_ENOMEM;
    cudaMemsetAsync(f, 0, sizeof(unsigned), s);
    cudaError_t e = launch_km_flags(params, n, f, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&flags, f, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(f);
    if (e != cudaSuccess) return ENS_ECUDA;
  }
  return launch_rhs_eval(sys, flags, n, params, t, y, dy, s) == cudaSuccess ? ENS_OK : ENS_ECUDA;
}

const char* ens_last_error(const ens_ctx* c) { return c ? c->err : g_create_err; }

void ens_destroy(ens_ctx* c) {
  if (!c) return;
  free_buffers(c);
  delete c;
}

}  // extern "C"
