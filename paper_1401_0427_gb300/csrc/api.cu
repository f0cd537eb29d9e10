// C ABI of the library (declarations and contracts in include/lbm_sw.h).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>

#include "internal.h"
#include "launch_plan.h"

namespace {

// Smallest 2D FP32 grid (cells) that AUTO steps with temporal blocking: 640^2 ran 10 .. 37 %
// faster fused (K = 4) than one step per launch, 512^2 with a wall and an inflow side 19 %
// slower.
constexpr long long kAutoTemporalCells = 3LL << 17;

// 2D FP32 grids below this size (cells) take several steps per launch on register tiles under
// AUTO where the wavefront does not apply or two waves of tiles cover the grid.  us per step, tiles
// against the wavefront, BGK and MRT: two waves 740^2 3.9 / 4.1 and 5.4 / 5.7, with walls 4.6 / 4.9
// and 6.1 / 6.2; three waves 768^2 4.2 / 4.1 and 5.9 / 5.7, 900 x 600 with walls 5.5 / 4.6 and 7.3 / 5.8.
constexpr long long kTileCells = 5LL << 17;

int fail(lbm_sw* h, int code, const char* fmt, ...) {
  if (h) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    std::vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    h->err = buf;
  }
  return code;
}

int cuda_fail(lbm_sw* h, cudaError_t e, const char* what) {
  return fail(h, e == cudaErrorMemoryAllocation ? LBM_SW_E_NOMEM : LBM_SW_E_CUDA, "%s: %s (%s)", what,
              cudaGetErrorString(e), cudaGetErrorName(e));
}

#define LBM_CUDA(h, call, what)                       \
  do {                                                \
    cudaError_t e_ = (call);                          \
    if (e_ != cudaSuccess) return cuda_fail(h, e_, what); \
  } while (0)

long long round_up(long long v, long long m) { return (v + m - 1) / m * m; }

size_t state_bytes(const lbm_sw* h) { return static_cast<size_t>(h->q) * h->plane * h->elem; }

template <class T>
lbm::StepArgs<T> args(const lbm_sw* h, int src_buf) {
  return lbm::handle_args<T>(h, src_buf);
}

lbm::ConstsD consts(const lbm_sw* h) { return lbm::handle_consts(h); }

// Whether lbm_sw_step fuses temporal_k steps per launch: FP32 2D TEMPORAL handles without
// obstacles, with the BGK collision or with MRT where the two-column kernel applies.
bool temporal_active(const lbm_sw* h) {
  if (h->p.dim != 2 || h->kernel != LBM_SW_KERNEL_TEMPORAL || h->p.precision != LBM_SW_FP32 || h->has_obstacles)
    return false;
  if (!h->mrt) return true;
  // MRT: the two-column kernel's K; under AUTO from 2^19 cells (868^2 with walls and inflow:
  // +14 % fused at K = 4; 724^2 even, 628^2 -12 %)
  const bool large = static_cast<long long>(h->p.nx) * h->p.ny >= (1LL << 19);
  return lbm::temporal_mrt_supported(h->p.bc, h->p.nx, h->temporal_k) && (large || !h->auto_kernel);
}

// Steps per fused launch with obstacles (FP32 BGK TEMPORAL handles with an even temporal_steps; 8
// runs as 6), 0: one step per launch.
int obstacle_k(const lbm_sw* h) {
  if (!h->has_obstacles || h->p.dim != 2 || h->kernel != LBM_SW_KERNEL_TEMPORAL || h->p.precision != LBM_SW_FP32 ||
      h->mrt || h->temporal_k % 2)
    return 0;
  return std::min(h->temporal_k, 6);
}

// What takes a launch of two steps where register tiles run: tiles reload their halo for little then.
// The wavefront where it applies, for even widths without solid cells (us, tiles / wavefront: 700 x 600 9.7 / 9.3
// periodic and 11.3 / 9.3 with sides, 200 x 2000 10.1 / 9.8 and 11.8 / 9.9, 1024 x 512 12.1 / 11.1 and 13.1 /
// 11.3; 801 x 601 11.4 / 13.1); two single steps for MRT with sides from 5 * 2^14 cells on (450 x 200 7.6 / 6.7,
// 640^2 12.8 / 12.3, 1024 x 512 15.2 / 13.8; 256^2 4.6 / 5.1).
// Four steps (four at a time): BGK on even widths by the estimates of both (us, tiles / wavefront: 700 x 600 periodic 14.4 /
// 13.4, 900 x 500 15.8 / 14.1, 1024 x 512 16.7 / 15.3 and with sides 20.7 / 18.3; 640^2 13.7 / 15.2 and 16.1 / 17.9).  Launches of
// other sizes run on tiles: six steps 18 to 21 against 23 to 31.
enum class TwoSteps { tile, wave, singles };
TwoSteps two_steps(const lbm_sw* h) {
  const bool per = h->p.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC && h->p.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC;
  if (h->has_obstacles) return TwoSteps::tile;
  if (h->mrt) return !per && static_cast<long long>(h->p.nx) * h->p.ny >= (5LL << 14) ? TwoSteps::singles : TwoSteps::tile;
  return temporal_active(h) && h->p.nx % 2 == 0 ? TwoSteps::wave : TwoSteps::tile;
}

// The launches of n > 0 steps where register tiles run, as even as they come: launch(steps) for each.
template <class F>
int for_tile_launches(const lbm_sw* h, int n, F&& launch) {
  const int k = h->tile_k;
  const int count = (n + k - 1) / k, base = n / count, extra = n % count;
  for (int i = 0; i < count; ++i) {
    const int steps = i < extra ? base + 1 : base;
    const bool singles = steps == 2 && two_steps(h) == TwoSteps::singles;
    int rc = launch(singles ? 1 : steps);
    if (rc == LBM_SW_OK && singles) rc = launch(1);
    if (rc != LBM_SW_OK) return rc;
  }
  return LBM_SW_OK;
}

// Launch plan of a fused handle (launch_plan.h): K, and whether odd sizes above one may run
// (BGK with every side periodic: the paired kernel with an even left halo at K = 3 and 5 on
// large grids, else the one-column kernel).
int plan_fused_launches(const lbm_sw* h, int n, int* plan, int max_plan) {
  const bool odd_ok = !h->mrt && h->p.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC &&
                      h->p.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC;
  return lbm::plan_launches(h->temporal_k, odd_ok, n, plan, max_plan);
}
static_assert(64 > lbm::kMaxTail, "plan buffers of lbm_sw_step and lbm_sw_step_plan hold a whole tail");

// One step from buffer `from` into the other buffer, on stream st (the TEMPORAL choice
// takes single steps with the VEC kernel).
cudaError_t launch_one_step(lbm_sw* h, int from, cudaStream_t st) {
  const int variant = h->kernel == LBM_SW_KERNEL_TEMPORAL ? LBM_SW_KERNEL_VEC : h->kernel;
  if (h->has_obstacles) {
    const unsigned char* mask = variant == LBM_SW_KERNEL_SIMPLE ? h->solid : h->solid_flags;
    return h->p.precision == LBM_SW_FP64
               ? lbm::launch_step2d_obstacle<double>(args<double>(h, from), consts(h), mask, variant, st)
               : lbm::launch_step2d_obstacle<float>(args<float>(h, from), consts(h), mask, variant, st);
  }
  if (h->p.precision == LBM_SW_FP64) {
    auto a = args<double>(h, from);
    return h->p.dim == 1 ? lbm::launch_step1d<double>(a, consts(h), st)
                         : lbm::launch_step2d<double>(a, consts(h), variant, st);
  }
  auto a = args<float>(h, from);
  return h->p.dim == 1 ? lbm::launch_step1d<float>(a, consts(h), st)
                       : lbm::launch_step2d<float>(a, consts(h), variant, st);
}

// Rows of every plane between the state (src, dst: its first row) and a dense array: a kernel on the
// device, a 2D copy per plane from or to the host.
cudaError_t planes_out(lbm_sw* h, const char* src, void* dst, size_t row, size_t dplane, int rows, int on_device) {
  const long long pitch = h->pitch * static_cast<long long>(h->elem), plane = h->plane * static_cast<long long>(h->elem);
  if (on_device) {
    h->launches += 1;
    return lbm::copy_planes({src, pitch, plane, dst, static_cast<long long>(row), static_cast<long long>(dplane),
                             static_cast<long long>(row), rows, h->q, dst}, h->elem, h->stream);
  }
  for (int p = 0; p < h->q; ++p) {
    const cudaError_t e = cudaMemcpy2DAsync(static_cast<char*>(dst) + p * dplane, row, src + p * plane, pitch, row, rows,
                                            cudaMemcpyDeviceToHost, h->stream);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
cudaError_t planes_in(lbm_sw* h, char* dst, const void* src, size_t row, size_t dplane, int rows, int on_device) {
  const long long pitch = h->pitch * static_cast<long long>(h->elem), plane = h->plane * static_cast<long long>(h->elem);
  if (on_device) {
    h->launches += 1;
    return lbm::copy_planes({src, static_cast<long long>(row), static_cast<long long>(dplane), dst, pitch, plane,
                             static_cast<long long>(row), rows, h->q, src}, h->elem, h->stream);
  }
  for (int p = 0; p < h->q; ++p) {
    const cudaError_t e = cudaMemcpy2DAsync(dst + p * plane, pitch, static_cast<const char*>(src) + p * dplane, row, row,
                                            rows, cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Capture graph_chunk steps starting from buffer `from` (graph_chunk is even, so the
// chunk ends in the buffer it started from).
int build_graph(lbm_sw* h, int from) {
  if (!h->capture_stream)
    LBM_CUDA(h, cudaStreamCreateWithFlags(&h->capture_stream, cudaStreamNonBlocking), "cudaStreamCreate");
  LBM_CUDA(h, cudaStreamBeginCapture(h->capture_stream, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture");
  cudaError_t le = cudaSuccess;
  int b = from;
  for (int i = 0; i < h->graph_chunk && le == cudaSuccess; ++i, b ^= 1) le = launch_one_step(h, b, h->capture_stream);
  cudaGraph_t g = nullptr;
  cudaError_t ce = cudaStreamEndCapture(h->capture_stream, &g);
  if (le != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    return cuda_fail(h, le, "step launch during graph capture");
  }
  if (ce != cudaSuccess) return cuda_fail(h, ce, "cudaStreamEndCapture");
  cudaError_t ie = cudaGraphInstantiate(&h->graph[from], g, 0);
  cudaGraphDestroy(g);
  if (ie != cudaSuccess) return cuda_fail(h, ie, "cudaGraphInstantiate");
  return LBM_SW_OK;
}

int validate(const lbm_sw_params* p, lbm_sw* h) {
  if (p->dim != 1 && p->dim != 2) return fail(h, LBM_SW_E_ARG, "dim must be 1 or 2 (got %d)", p->dim);
  if (p->nx < 1 || p->ny < 1) return fail(h, LBM_SW_E_ARG, "nx and ny must be >= 1 (got %d, %d)", p->nx, p->ny);
  if (p->dim == 1 && p->ny != 1) return fail(h, LBM_SW_E_ARG, "ny must be 1 when dim == 1");
  if (p->nx > (1 << 30) || p->ny > (1 << 30)) return fail(h, LBM_SW_E_ARG, "nx, ny must be <= 2^30");
  if (p->precision != LBM_SW_FP32 && p->precision != LBM_SW_FP64)
    return fail(h, LBM_SW_E_ARG, "precision must be LBM_SW_FP32 or LBM_SW_FP64");
  if (!(p->g > 0) || !std::isfinite(p->g)) return fail(h, LBM_SW_E_ARG, "g must be finite and > 0");
  if (!(p->lambda > 0) || !std::isfinite(p->lambda)) return fail(h, LBM_SW_E_ARG, "lambda must be finite and > 0");
  if (!(p->s >= 0 && p->s < 2)) return fail(h, LBM_SW_E_ARG, "s must be in [0, 2)");
  if (!(p->a >= 0) || !std::isfinite(p->a)) return fail(h, LBM_SW_E_ARG, "a must be finite and >= 0");
  const int nsides = p->dim == 1 ? 2 : 4;
  for (int s = 0; s < nsides; ++s) {
    if (p->bc[s] < LBM_SW_BC_PERIODIC || p->bc[s] > LBM_SW_BC_INFLOW)
      return fail(h, LBM_SW_E_ARG, "bc[%d] = %d is not a LBM_SW_BC_* value", s, p->bc[s]);
    if (p->bc[s] == LBM_SW_BC_INFLOW) {
      if (!(p->inflow[s][0] > 0) || !std::isfinite(p->inflow[s][0]) || !std::isfinite(p->inflow[s][1]) ||
          !std::isfinite(p->inflow[s][2]))
        return fail(h, LBM_SW_E_ARG, "inflow[%d] must be finite with depth > 0", s);
    }
  }
  for (int pair = 0; pair < nsides; pair += 2)
    if ((p->bc[pair] == LBM_SW_BC_PERIODIC) != (p->bc[pair + 1] == LBM_SW_BC_PERIODIC))
      return fail(h, LBM_SW_E_ARG, "periodic sides come in pairs (bc[%d], bc[%d])", pair, pair + 1);
  if (p->kernel < LBM_SW_KERNEL_AUTO || p->kernel > LBM_SW_KERNEL_TEMPORAL)
    return fail(h, LBM_SW_E_ARG, "kernel must be a LBM_SW_KERNEL_* value");
  if ((p->dim == 2 && p->kernel == LBM_SW_KERNEL_CLUSTER) ||
      (p->dim == 1 && (p->kernel == LBM_SW_KERNEL_VEC || p->kernel == LBM_SW_KERNEL_TEMPORAL)))
    return fail(h, LBM_SW_E_ARG, "kernel: CLUSTER is for 1D handles, VEC and TEMPORAL for 2D handles");
  if (p->temporal_steps != 0 && !lbm::temporal_steps_supported(p->temporal_steps))
    return fail(h, LBM_SW_E_ARG, "temporal_steps must be 0 or 2 .. 8");
  for (int r = 0; r < 5; ++r)
    if (p->reserved[r] != 0) return fail(h, LBM_SW_E_ARG, "reserved fields must be zero");
  return LBM_SW_OK;
}

thread_local std::string g_create_error;

}  // namespace

namespace lbm {
// AUTO without a wish for temporal_steps.
bool tile_active(const lbm_sw* h) {
  return h->tile_k > 0 && ((!temporal_active(h) && obstacle_k(h) == 0) || h->tile_waves <= 2);
}

void set_create_error(const char* msg) { g_create_error = msg ? msg : ""; }
}  // namespace lbm

extern "C" {

int lbm_sw_abi_version(void) { return LBM_SW_ABI_VERSION; }

const char* lbm_sw_status_string(int status) {
  switch (status) {
    case LBM_SW_OK: return "ok";
    case LBM_SW_E_ARG: return "invalid argument";
    case LBM_SW_E_CUDA: return "CUDA error";
    case LBM_SW_E_UNSTABLE: return "unstable state (NaN/Inf or depth <= 0)";
    case LBM_SW_E_STATE: return "call not valid in the current state";
    case LBM_SW_E_NOMEM: return "out of device memory";
    default: return "unknown status";
  }
}

int lbm_sw_params_init(lbm_sw_params* p) {
  if (!p) return LBM_SW_E_ARG;
  std::memset(p, 0, sizeof(*p));
  p->dim = 2;
  p->precision = LBM_SW_FP32;
  p->g = 1.0;
  p->lambda = 8.0;
  p->s = 1.8;
  p->a = 0.05;
  for (int s = 0; s < 4; ++s) {
    p->bc[s] = LBM_SW_BC_PERIODIC;
    p->inflow[s][0] = 1.0;
  }
  p->kernel = LBM_SW_KERNEL_AUTO;
  return LBM_SW_OK;
}

const char* lbm_sw_last_error(const lbm_sw* h) { return h ? h->err.c_str() : "null handle"; }

const char* lbm_sw_create_error(void) { return g_create_error.c_str(); }

void lbm_sw_destroy(lbm_sw* h) {
  if (!h) return;
  cudaStreamSynchronize(h->stream);
  for (int i = 0; i < 2; ++i) {
    if (h->graph[i]) cudaGraphExecDestroy(h->graph[i]);
    if (h->buf[i]) cudaFree(h->buf[i]);
  }
  h->tape_memory->close();
  if (h->capture_stream) cudaStreamDestroy(h->capture_stream);
  if (h->inflow_feq) cudaFree(h->inflow_feq);
  if (h->moments_staging) cudaFree(h->moments_staging);
  if (h->mail1d) cudaFree(h->mail1d);
  if (h->pop_staging) cudaFree(h->pop_staging);
  if (h->diag_partials) cudaFree(h->diag_partials);
  if (h->diag_done) cudaFree(h->diag_done);
  if (h->diag_host) cudaFreeHost(h->diag_host);
  if (h->solid) cudaFree(h->solid);
  delete h;
}

int lbm_sw_create(const lbm_sw_params* p, lbm_sw** out) {
  if (!out) return LBM_SW_E_ARG;
  *out = nullptr;
  if (!p) return LBM_SW_E_ARG;
  g_create_error.clear();
  lbm_sw* h = nullptr;
  try {
    h = new lbm_sw;  // allocates for its members too
  } catch (const std::bad_alloc&) {
    return LBM_SW_E_NOMEM;
  }
  int rc = validate(p, h);
  if (rc != LBM_SW_OK) {
    g_create_error = h->err;  // the handle is not returned: keep the message per thread
    delete h;
    return rc;
  }
  h->p = *p;
  h->stream = static_cast<cudaStream_t>(p->stream);
  h->q = p->dim == 1 ? 5 : 13;
  h->elem = p->precision == LBM_SW_FP64 ? 8 : 4;
  h->pitch = round_up(p->nx, 32);
  h->plane = round_up(h->pitch * p->ny, 64);  // 256-byte aligned planes in FP32 and FP64
  const bool all_periodic = p->bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC && p->bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC;
  // default steps per fused launch: 4 below 2^20 cells (shorter wavefront fill), else 6
  const long long cells = static_cast<long long>(p->nx) * p->ny;
  h->temporal_k = p->temporal_steps ? p->temporal_steps : (cells < (1LL << 20) ? 4 : 6);
  h->auto_kernel = p->kernel == LBM_SW_KERNEL_AUTO;
  if (p->dim == 2) {
    // AUTO: temporal blocking where it was measured faster (FP32, at least 3 * 2^17 cells,
    // all sides periodic or the two-column kernel: even K), otherwise one vectorised step
    // per launch
    const int k = h->temporal_k;
    const bool temporal = p->precision == LBM_SW_FP32 && (all_periodic || k % 2 == 0) && cells >= kAutoTemporalCells;
    h->kernel = p->kernel == LBM_SW_KERNEL_AUTO ? (temporal ? LBM_SW_KERNEL_TEMPORAL : LBM_SW_KERNEL_VEC) : p->kernel;
  } else {
    h->kernel = p->kernel == LBM_SW_KERNEL_AUTO ? LBM_SW_KERNEL_CLUSTER : p->kernel;
  }
  h->graph_chunk = p->graph_chunk == 0 ? 64 : (p->graph_chunk < 0 ? 0 : p->graph_chunk + (p->graph_chunk & 1));

  auto bail = [&](int code) {
    const cudaError_t last = cudaGetLastError();  // device_alloc leaves none
    g_create_error = std::string("create: ") + lbm_sw_status_string(code) + ": " +
                     cudaGetErrorString(last == cudaSuccess && code == LBM_SW_E_NOMEM ? cudaErrorMemoryAllocation : last);
    lbm_sw_destroy(h);
    return code;
  };
  if (cudaGetDevice(&h->device) != cudaSuccess) return bail(LBM_SW_E_CUDA);
  if (cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess)
    return bail(LBM_SW_E_CUDA);
  if (h->auto_kernel && p->temporal_steps == 0 && p->dim == 2 && p->precision == LBM_SW_FP32 &&
      static_cast<long long>(p->nx) * p->ny < kTileCells)
    h->tile_k = lbm::tile_steps(p->nx, p->ny, std::max(h->sm_count, 1), &h->tile_waves);
  // (not where launches are of five steps at most, so that longer runs take fours too: 760 x 740 3.9 us per step on tiles
  // against 4.05, with sides 4.3 and 4.9)
  h->wave4 = h->tile_k > 5 && p->nx % 2 == 0 && lbm::temporal4_us(p->nx, p->ny, all_periodic, h->sm_count) <
                                                    lbm::tile4_us(p->nx, p->ny, all_periodic, h->sm_count);
  const size_t bytes = state_bytes(h);
  for (int i = 0; i < 2; ++i) {
    if (lbm::device_alloc(&h->buf[i], bytes) != cudaSuccess) return bail(LBM_SW_E_NOMEM);
    if (cudaMemsetAsync(h->buf[i], 0, bytes, h->stream) != cudaSuccess) return bail(LBM_SW_E_CUDA);
  }
  if (lbm::device_alloc(&h->inflow_feq, 4 * h->q * h->elem) != cudaSuccess) return bail(LBM_SW_E_NOMEM);
  if (h->kernel == LBM_SW_KERNEL_CLUSTER && p->nx <= lbm::kWindows1dMaxCells &&
      lbm::device_alloc(&h->mail1d, p->precision == LBM_SW_FP64 ? lbm::mail1d_bytes<double>(p->nx)
                                                         : lbm::mail1d_bytes<float>(p->nx)) != cudaSuccess)
    return bail(LBM_SW_E_NOMEM);
  if (lbm::device_alloc(&h->diag_partials, 5 * sizeof(double) * lbm::diag_max_blocks()) != cudaSuccess)
    return bail(LBM_SW_E_NOMEM);
  if (lbm::device_alloc(&h->diag_done, sizeof(unsigned)) != cudaSuccess) return bail(LBM_SW_E_NOMEM);
  if (cudaMemsetAsync(h->diag_done, 0, sizeof(unsigned), h->stream) != cudaSuccess) return bail(LBM_SW_E_CUDA);
  if (cudaMallocHost(&h->diag_host, 8 * sizeof(double)) != cudaSuccess) return bail(LBM_SW_E_NOMEM);
  cudaError_t e;
  if (p->precision == LBM_SW_FP64)
    e = p->dim == 1 ? lbm::launch_inflow_feq1d<double>(static_cast<double*>(h->inflow_feq), p->bc, p->inflow, consts(h), h->stream)
                    : lbm::launch_inflow_feq2d<double>(static_cast<double*>(h->inflow_feq), p->bc, p->inflow, consts(h), h->stream);
  else
    e = p->dim == 1 ? lbm::launch_inflow_feq1d<float>(static_cast<float*>(h->inflow_feq), p->bc, p->inflow, consts(h), h->stream)
                    : lbm::launch_inflow_feq2d<float>(static_cast<float*>(h->inflow_feq), p->bc, p->inflow, consts(h), h->stream);
  if (e != cudaSuccess) return bail(LBM_SW_E_CUDA);
  h->launches += 1;
  if (cudaStreamSynchronize(h->stream) != cudaSuccess) return bail(LBM_SW_E_CUDA);
  *out = h;
  return LBM_SW_OK;
}

int lbm_sw_set_state(lbm_sw* h, const double* depth, const double* hu, const double* hv, int on_device) {
  if (!h) return LBM_SW_E_ARG;
  if (!depth || !hu || (h->p.dim == 2 && !hv && on_device))
    return fail(h, LBM_SW_E_ARG, "set_state: depth and hu are required (and hv for device input in 2D)");
  const size_t n = static_cast<size_t>(h->p.nx) * h->p.ny;
  const double *d = depth, *u = hu, *v = (h->p.dim == 2) ? hv : nullptr;
  if (!on_device) {
    if (!h->moments_staging)
      LBM_CUDA(h, lbm::device_alloc(&h->moments_staging, 3 * n * sizeof(double)), "cudaMalloc(moments staging)");
    double* s = h->moments_staging;
    LBM_CUDA(h, cudaMemcpyAsync(s, depth, n * sizeof(double), cudaMemcpyHostToDevice, h->stream), "copy h");
    LBM_CUDA(h, cudaMemcpyAsync(s + n, hu, n * sizeof(double), cudaMemcpyHostToDevice, h->stream), "copy hu");
    if (h->p.dim == 2) {
      if (hv)
        LBM_CUDA(h, cudaMemcpyAsync(s + 2 * n, hv, n * sizeof(double), cudaMemcpyHostToDevice, h->stream), "copy hv");
      else
        LBM_CUDA(h, cudaMemsetAsync(s + 2 * n, 0, n * sizeof(double), h->stream), "zero hv");
    }
    d = s;
    u = s + n;
    v = h->p.dim == 2 ? s + 2 * n : nullptr;
  }
  cudaError_t e;
  // the equilibrium is written into the current buffer (as the destination of "args")
  const int from = 1 - h->cur;
  if (h->p.precision == LBM_SW_FP64)
    e = h->p.dim == 1 ? lbm::launch_init1d<double>(args<double>(h, from), consts(h), d, u, h->stream)
                      : lbm::launch_init2d<double>(args<double>(h, from), consts(h), d, u, v, h->stream);
  else
    e = h->p.dim == 1 ? lbm::launch_init1d<float>(args<float>(h, from), consts(h), d, u, h->stream)
                      : lbm::launch_init2d<float>(args<float>(h, from), consts(h), d, u, v, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "set_state kernel launch");
  h->launches += 1;
  if (!on_device) LBM_CUDA(h, cudaStreamSynchronize(h->stream), "set_state synchronize");
  h->has_state = true;
  h->steps_done = 0;
  return LBM_SW_OK;
}

int lbm_sw_step(lbm_sw* h, int n) {
  if (!h) return LBM_SW_E_ARG;
  if (n < 0) return fail(h, LBM_SW_E_ARG, "step: n must be >= 0 (got %d)", n);
  if (!h->has_state) return fail(h, LBM_SW_E_STATE, "step: no state set (call set_state or set_populations)");
  if (h->p.dim == 1 && h->kernel == LBM_SW_KERNEL_CLUSTER && n > 0) {
    if (h->p.nx <= lbm::kWindows1dMaxCells) {
      const bool fp64 = h->p.precision == LBM_SW_FP64;
      cudaError_t e = fp64 ? lbm::launch_step1d_windows<double>(args<double>(h, h->cur), consts(h), n, h->mail1d,
                                                                h->sm_count, h->stream)
                           : lbm::launch_step1d_windows<float>(args<float>(h, h->cur), consts(h), n, h->mail1d,
                                                               h->sm_count, h->stream);
      if (e != cudaSuccess) return cuda_fail(h, e, "line step launch");
      h->cur ^= 1;
      h->steps_done += n;
      h->launches += 1;
      return LBM_SW_OK;
    }
  }
  if (n > 0 && lbm::tile_active(h))
    return for_tile_launches(h, n, [&](int k) {
      const auto a = args<float>(h, h->cur);
      const unsigned char* flags = h->has_obstacles ? h->solid_flags : nullptr;
      const cudaError_t e =
          k == 1 ? launch_one_step(h, h->cur, h->stream)
          : (k == 2 && two_steps(h) == TwoSteps::wave) || (k == 4 && h->wave4 && !h->mrt && temporal_active(h))
              ? lbm::launch_step2d_temporal(a, consts(h), k, h->stream, h->sm_count)
              : lbm::launch_step2d_tile(a, consts(h), k, flags, h->stream, h->sm_count);
      if (e != cudaSuccess) return cuda_fail(h, e, "tile step launch");
      h->cur ^= 1;
      h->steps_done += k;
      h->launches += 1;
      return static_cast<int>(LBM_SW_OK);
    });
  if (const int ko = obstacle_k(h)) {
    int plan[64];
    while (n > 0) {
      const int count = lbm::plan_launches(ko, false, n, plan, 64);
      for (int i = 0; i < count; ++i) {
        const int k = plan[i];
        const cudaError_t e = k == 1 ? launch_one_step(h, h->cur, h->stream)
                                     : lbm::launch_step2d_temporal_obstacle(args<float>(h, h->cur), consts(h),
                                                                            h->solid_flags, k, h->stream, h->sm_count);
        if (e != cudaSuccess) return cuda_fail(h, e, "obstacle step launch");
        h->cur ^= 1;
        n -= k;
        h->steps_done += k;
        h->launches += 1;
      }
    }
    return LBM_SW_OK;
  }
  if (temporal_active(h)) {
    int plan[64];
    while (n > 0) {
      const int count = plan_fused_launches(h, n, plan, 64);
      for (int i = 0; i < count; ++i) {
        const int k = plan[i];
        cudaError_t e;
        if (k == 1) {  // one step per launch (the vectorised kernel; FP32 here)
          e = lbm::launch_step2d<float>(args<float>(h, h->cur), consts(h), LBM_SW_KERNEL_VEC, h->stream);
        } else {
          e = h->mrt ? lbm::launch_step2d_temporal_mrt(args<float>(h, h->cur), consts(h), k, h->stream, h->sm_count)
                     : lbm::launch_step2d_temporal(args<float>(h, h->cur), consts(h), k, h->stream, h->sm_count);
        }
        if (e != cudaSuccess) return cuda_fail(h, e, k == 1 ? "step kernel launch" : "temporal step launch");
        h->cur ^= 1;
        n -= k;
        h->steps_done += k;
        h->launches += 1;
      }
    }
    return LBM_SW_OK;
  }
  while (n > 0) {
    if (h->graph_chunk > 0 && n >= h->graph_chunk) {
      if (!h->graph[h->cur]) {
        int rc = build_graph(h, h->cur);
        if (rc != LBM_SW_OK) return rc;
      }
      LBM_CUDA(h, cudaGraphLaunch(h->graph[h->cur], h->stream), "cudaGraphLaunch");
      n -= h->graph_chunk;
      h->steps_done += h->graph_chunk;
      h->launches += h->graph_chunk;
    } else {
      cudaError_t e = launch_one_step(h, h->cur, h->stream);
      if (e != cudaSuccess) return cuda_fail(h, e, "step kernel launch");
      h->cur ^= 1;
      n -= 1;
      h->steps_done += 1;
      h->launches += 1;
    }
  }
  return LBM_SW_OK;
}

int lbm_sw_step_plan(const lbm_sw* h, int n, int* sizes, int max_sizes) {
  if (!h || n < 0 || max_sizes < 0 || (max_sizes > 0 && !sizes)) return LBM_SW_E_ARG;
  int count = 0;
  auto put = [&](int k) {
    if (count < max_sizes) sizes[count] = k;
    ++count;
  };
  if (n == 0) return 0;
  if (h->p.dim == 1 && h->kernel == LBM_SW_KERNEL_CLUSTER) {
    if (h->p.nx <= lbm::kWindows1dMaxCells) {
      put(n);
      return count;
    }
  }
  if (lbm::tile_active(h)) {
    for_tile_launches(h, n, [&](int k) {
      put(k);
      return static_cast<int>(LBM_SW_OK);
    });
    return count;
  }
  const int ko = obstacle_k(h);
  if (ko || temporal_active(h)) {
    int plan[64];
    while (n > 0) {
      const int c = ko ? lbm::plan_launches(ko, false, n, plan, 64) : plan_fused_launches(h, n, plan, 64);
      for (int i = 0; i < c; ++i) {
        put(plan[i]);
        n -= plan[i];
      }
    }
    return count;
  }
  for (int i = 0; i < n; ++i) put(1);
  return count;
}

int lbm_sw_get_moments(lbm_sw* h, double* depth, double* hu, double* hv, int on_device) {
  if (!h) return LBM_SW_E_ARG;
  if (!depth || !hu) return fail(h, LBM_SW_E_ARG, "get_moments: depth and hu are required");
  if (!h->has_state) return fail(h, LBM_SW_E_STATE, "get_moments: no state set");
  const size_t n = static_cast<size_t>(h->p.nx) * h->p.ny;
  double *d = depth, *u = hu, *v = (h->p.dim == 2) ? hv : nullptr;
  if (!on_device) {
    if (!h->moments_staging)
      LBM_CUDA(h, lbm::device_alloc(&h->moments_staging, 3 * n * sizeof(double)), "cudaMalloc(moments staging)");
    d = h->moments_staging;
    u = d + n;
    v = (h->p.dim == 2 && hv) ? d + 2 * n : nullptr;
  }
  cudaError_t e;
  const int from = h->cur;
  if (h->p.precision == LBM_SW_FP64)
    e = h->p.dim == 1 ? lbm::launch_moments1d<double>(args<double>(h, from), d, u, h->stream)
                      : lbm::launch_moments2d<double>(args<double>(h, from), d, u, v, h->stream);
  else
    e = h->p.dim == 1 ? lbm::launch_moments1d<float>(args<float>(h, from), d, u, h->stream)
                      : lbm::launch_moments2d<float>(args<float>(h, from), d, u, v, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "moments kernel launch");
  h->launches += 1;
  if (!on_device) {
    LBM_CUDA(h, cudaMemcpyAsync(depth, d, n * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "copy h");
    LBM_CUDA(h, cudaMemcpyAsync(hu, u, n * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "copy hu");
    if (v) LBM_CUDA(h, cudaMemcpyAsync(hv, v, n * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "copy hv");
    LBM_CUDA(h, cudaStreamSynchronize(h->stream), "get_moments synchronize");
  }
  return LBM_SW_OK;
}

int lbm_sw_diagnostics(lbm_sw* h, double out[4]) {
  if (!h || !out) return h ? fail(h, LBM_SW_E_ARG, "diagnostics: out is NULL") : LBM_SW_E_ARG;
  if (!h->has_state) return fail(h, LBM_SW_E_STATE, "diagnostics: no state set");
  cudaError_t e = h->p.precision == LBM_SW_FP64
                      ? lbm::launch_diagnostics<double>(args<double>(h, h->cur), h->q, h->diag_partials, h->diag_done, h->diag_host, h->sm_count, h->stream)
                      : lbm::launch_diagnostics<float>(args<float>(h, h->cur), h->q, h->diag_partials, h->diag_done, h->diag_host, h->sm_count, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "diagnostics kernel launch");
  h->launches += 1;
  LBM_CUDA(h, cudaStreamSynchronize(h->stream), "diagnostics synchronize");
  for (int k = 0; k < 4; ++k) out[k] = h->diag_host[k];
  if (h->diag_host[4] > 0)
    return fail(h, LBM_SW_E_UNSTABLE, "diagnostics: %.0f cells with NaN/Inf or depth <= 0", h->diag_host[4]);
  return LBM_SW_OK;
}

int lbm_sw_get_populations(lbm_sw* h, void* dst, int on_device) {
  if (!h) return LBM_SW_E_ARG;
  if (!dst) return fail(h, LBM_SW_E_ARG, "get_populations: dst is NULL");
  if (!h->has_state) return fail(h, LBM_SW_E_STATE, "get_populations: no state set");
  const size_t row = static_cast<size_t>(h->p.nx) * h->elem;
  const size_t dplane = row * h->p.ny;
  const char* src = static_cast<const char*>(h->buf[h->cur]);
  LBM_CUDA(h, planes_out(h, src, dst, row, dplane, h->p.ny, on_device), "copy populations out");
  if (!on_device) LBM_CUDA(h, cudaStreamSynchronize(h->stream), "get_populations synchronize");
  return LBM_SW_OK;
}

int lbm_sw_set_populations(lbm_sw* h, const void* src, int on_device, int form) {
  if (!h) return LBM_SW_E_ARG;
  if (!src) return fail(h, LBM_SW_E_ARG, "set_populations: src is NULL");
  if (form != LBM_SW_POST_COLLISION && form != LBM_SW_PRE_COLLISION)
    return fail(h, LBM_SW_E_ARG, "set_populations: form must be LBM_SW_POST_COLLISION or LBM_SW_PRE_COLLISION");
  const size_t row = static_cast<size_t>(h->p.nx) * h->elem;
  const size_t dplane = row * h->p.ny;
  if (form == LBM_SW_POST_COLLISION) {
    char* dst = static_cast<char*>(h->buf[h->cur]);
    LBM_CUDA(h, planes_in(h, dst, src, row, dplane, h->p.ny, on_device), "copy populations in");
  } else {
    const void* dense = src;
    if (!on_device) {
      if (!h->pop_staging)
        LBM_CUDA(h, lbm::device_alloc(&h->pop_staging, h->q * dplane), "cudaMalloc(population staging)");
      LBM_CUDA(h, cudaMemcpyAsync(h->pop_staging, src, h->q * dplane, cudaMemcpyHostToDevice, h->stream),
               "copy populations in");
      dense = h->pop_staging;
    }
    const int from = 1 - h->cur;  // write into the current buffer
    cudaError_t e;
    if (h->p.precision == LBM_SW_FP64)
      e = h->p.dim == 1 ? lbm::launch_collide1d_dense<double>(args<double>(h, from), consts(h), static_cast<const double*>(dense), h->stream)
                        : lbm::launch_collide2d_dense<double>(args<double>(h, from), consts(h), static_cast<const double*>(dense),
                                                              h->has_obstacles ? h->solid : nullptr, h->stream);
    else
      e = h->p.dim == 1 ? lbm::launch_collide1d_dense<float>(args<float>(h, from), consts(h), static_cast<const float*>(dense), h->stream)
                        : lbm::launch_collide2d_dense<float>(args<float>(h, from), consts(h), static_cast<const float*>(dense),
                                                             h->has_obstacles ? h->solid : nullptr, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "collide kernel launch");
    h->launches += 1;
  }
  if (!on_device) LBM_CUDA(h, cudaStreamSynchronize(h->stream), "set_populations synchronize");
  h->has_state = true;
  h->steps_done = 0;
  return LBM_SW_OK;
}

int lbm_sw_get_rows(lbm_sw* h, int y0, int nrows, void* dst, int on_device) {
  if (!h) return LBM_SW_E_ARG;
  if (!dst) return fail(h, LBM_SW_E_ARG, "get_rows: dst is NULL");
  if (h->p.dim != 2) return fail(h, LBM_SW_E_ARG, "get_rows: rows are for 2D handles");
  if (y0 < 0 || nrows < 0 || y0 > h->p.ny - nrows)
    return fail(h, LBM_SW_E_ARG, "get_rows: rows [%d, %d) outside [0, %d)", y0, y0 + nrows, h->p.ny);
  if (!h->has_state) return fail(h, LBM_SW_E_STATE, "get_rows: no state set");
  if (nrows == 0) return LBM_SW_OK;
  const size_t row = static_cast<size_t>(h->p.nx) * h->elem;
  const size_t dplane = row * nrows;
  const char* src = static_cast<const char*>(h->buf[h->cur]) + static_cast<size_t>(y0) * h->pitch * h->elem;
  LBM_CUDA(h, planes_out(h, src, dst, row, dplane, nrows, on_device), "copy rows out");
  if (!on_device) LBM_CUDA(h, cudaStreamSynchronize(h->stream), "get_rows synchronize");
  return LBM_SW_OK;
}

int lbm_sw_set_rows(lbm_sw* h, int y0, int nrows, const void* src, int on_device) {
  if (!h) return LBM_SW_E_ARG;
  if (!src) return fail(h, LBM_SW_E_ARG, "set_rows: src is NULL");
  if (h->p.dim != 2) return fail(h, LBM_SW_E_ARG, "set_rows: rows are for 2D handles");
  if (y0 < 0 || nrows < 0 || y0 > h->p.ny - nrows)
    return fail(h, LBM_SW_E_ARG, "set_rows: rows [%d, %d) outside [0, %d)", y0, y0 + nrows, h->p.ny);
  if (!h->has_state) return fail(h, LBM_SW_E_STATE, "set_rows: no state set");
  if (nrows == 0) return LBM_SW_OK;
  const size_t row = static_cast<size_t>(h->p.nx) * h->elem;
  const size_t dplane = row * nrows;
  char* dst = static_cast<char*>(h->buf[h->cur]) + static_cast<size_t>(y0) * h->pitch * h->elem;
  LBM_CUDA(h, planes_in(h, dst, src, row, dplane, nrows, on_device), "copy rows in");
  if (!on_device) LBM_CUDA(h, cudaStreamSynchronize(h->stream), "set_rows synchronize");
  return LBM_SW_OK;
}

int lbm_sw_diagnostics_rows(lbm_sw* h, int y0, int nrows, double out[4]) {
  if (!h || !out) return h ? fail(h, LBM_SW_E_ARG, "diagnostics_rows: out is NULL") : LBM_SW_E_ARG;
  if (y0 < 0 || nrows < 1 || y0 > h->p.ny - nrows)
    return fail(h, LBM_SW_E_ARG, "diagnostics_rows: rows [%d, %d) outside [0, %d)", y0, y0 + nrows, h->p.ny);
  if (!h->has_state) return fail(h, LBM_SW_E_STATE, "diagnostics_rows: no state set");
  cudaError_t e;
  if (h->p.precision == LBM_SW_FP64) {
    auto a = args<double>(h, h->cur);
    a.src += static_cast<long long>(y0) * h->pitch;
    a.ny = nrows;
    e = lbm::launch_diagnostics<double>(a, h->q, h->diag_partials, h->diag_done, h->diag_host, h->sm_count, h->stream);
  } else {
    auto a = args<float>(h, h->cur);
    a.src += static_cast<long long>(y0) * h->pitch;
    a.ny = nrows;
    e = lbm::launch_diagnostics<float>(a, h->q, h->diag_partials, h->diag_done, h->diag_host, h->sm_count, h->stream);
  }
  if (e != cudaSuccess) return cuda_fail(h, e, "diagnostics kernel launch");
  h->launches += 1;
  LBM_CUDA(h, cudaStreamSynchronize(h->stream), "diagnostics synchronize");
  for (int k = 0; k < 4; ++k) out[k] = h->diag_host[k];
  if (h->diag_host[4] > 0)
    return fail(h, LBM_SW_E_UNSTABLE, "diagnostics: %.0f cells with NaN/Inf or depth <= 0", h->diag_host[4]);
  return LBM_SW_OK;
}

int lbm_sw_set_relaxation(lbm_sw* h, const double* rates, int count) {
  if (!h) return LBM_SW_E_ARG;
  if (!rates) {
    h->mrt = false;
  } else {
    const int want = h->p.dim == 1 ? 5 : 13;
    if (count != want) return fail(h, LBM_SW_E_ARG, "set_relaxation: %d rates expected (got %d)", want, count);
    static const int map2[10] = {1, 2, 3, 4, 6, 7, 8, 10, 11, 12};
    static const int map1[3] = {1, 2, 4};
    const int n = h->p.dim == 1 ? 3 : 10;
    const int* map = h->p.dim == 1 ? map1 : map2;
    for (int i = 0; i < n; ++i) {
      const double r = rates[map[i]];
      if (!(r >= 0.0 && r < 2.0)) return fail(h, LBM_SW_E_ARG, "set_relaxation: rate %d = %g is not in [0, 2)", map[i], r);
    }
    for (int i = 0; i < 10; ++i) h->mrt_rates[i] = i < n ? rates[map[i]] : 0.0;
    h->mrt = true;
  }
  // the captured graphs hold the old constants
  for (int i = 0; i < 2; ++i)
    if (h->graph[i]) {
      cudaGraphExecDestroy(h->graph[i]);
      h->graph[i] = nullptr;
    }
  return LBM_SW_OK;
}

int lbm_sw_set_obstacle(lbm_sw* h, const unsigned char* solid, int on_device) {
  if (!h) return LBM_SW_E_ARG;
  if (h->p.dim != 2) return fail(h, LBM_SW_E_ARG, "set_obstacle: obstacles are for 2D handles");
  if (!solid) {
    h->has_obstacles = false;
  } else {
    const size_t n = static_cast<size_t>(h->p.nx) * h->p.ny, at = static_cast<size_t>(round_up(n, 256));
    const bool flags = h->kernel != LBM_SW_KERNEL_SIMPLE;
    if (!h->solid) {
      LBM_CUDA(h, lbm::device_alloc(&h->solid, at + (flags ? static_cast<size_t>(h->plane) : 0)), "cudaMalloc (obstacle mask)");
      if (flags) h->solid_flags = h->solid + at;
    }
    const bool direct = on_device && flags && lbm::kernel_reaches(solid);  // the flags' kernel copies the mask too
    if (!direct) {
      LBM_CUDA(h, cudaMemcpyAsync(h->solid, solid, n, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                  h->stream), "obstacle mask copy");
      // the caller may reuse its buffer when this returns
      LBM_CUDA(h, cudaStreamSynchronize(h->stream), "set_obstacle synchronize");
    }
    if (flags) {
      LBM_CUDA(h, lbm::launch_obstacle_flags(direct ? solid : h->solid, direct ? h->solid : nullptr, h->solid_flags,
                                             h->p.nx, h->p.ny, h->pitch, h->p.bc, h->stream),
               "obstacle flags launch");
      h->launches += 1;
    }
    if (direct) LBM_CUDA(h, cudaStreamSynchronize(h->stream), "set_obstacle synchronize");
    h->has_obstacles = true;
  }
  // the captured graphs hold the previous step kernel
  for (int i = 0; i < 2; ++i)
    if (h->graph[i]) {
      cudaGraphExecDestroy(h->graph[i]);
      h->graph[i] = nullptr;
    }
  return LBM_SW_OK;
}

int lbm_sw_synchronize(lbm_sw* h) {
  if (!h) return LBM_SW_E_ARG;
  LBM_CUDA(h, cudaStreamSynchronize(h->stream), "synchronize");
  return LBM_SW_OK;
}

int lbm_sw_get_info(const lbm_sw* h, lbm_sw_info* out) {
  if (!h || !out) return LBM_SW_E_ARG;
  out->q = h->q;
  out->kernel = h->kernel;
  if (h->p.dim == 1 && h->kernel == LBM_SW_KERNEL_CLUSTER && h->p.nx > lbm::kWindows1dMaxCells)
    out->kernel = LBM_SW_KERNEL_SIMPLE;
  out->pitch = static_cast<size_t>(h->pitch);
  out->population_bytes = static_cast<size_t>(h->q) * h->p.nx * h->p.ny * h->elem;
  out->bytes_per_update = 2.0 * h->q * static_cast<double>(h->elem);
  out->steps_done = h->steps_done;
  out->kernel_launches = h->launches;
  out->steps_per_launch = 1;
  if (out->kernel == LBM_SW_KERNEL_CLUSTER) out->steps_per_launch = 0;
  if (temporal_active(h)) out->steps_per_launch = h->temporal_k;
  return LBM_SW_OK;
}

}  // extern "C"
