// Pressure solve that allocates nothing.
//
// Some callers cannot call cudaMalloc: a host framework that owns all device memory
// through its own pool and forbids other allocations, a process running under a hard
// device-memory cap, or latency-sensitive code that must not trigger the device-wide
// synchronisation that cudaMalloc and cudaFree imply.  ccm_solve_pressure_noalloc serves
// them: it solves the same system as ccm_solve_pressure in FP64 with the Jacobi
// preconditioner, whatever the case's precision and preconditioner settings, but its scratch
// lives in one file-scope __device__ array of fixed size instead of memory the library
// allocates.  The kernel is the resident one-barrier solve (pcg_fused.cu) in its built-in plan:
// a tile's vectors stay in shared memory, so the array holds the right-hand side, the first
// residual and the mailboxes of the tiles.  Every grid within the limit has such a plan
// (tests/test_fused_plan.py goes through them all); where the smallest tiles are wide and flat
// their rings would not fit the mailboxes, and the plan takes narrower or taller ones (500x150:
// 150 tiles of 256x2 instead of 512x1).  A singular case (no outflow side) projects onto zero mean at the start and the end.
// The caller passes the right-hand side and the solution in device memory of its own.
//
// The array (about 6.4 MB) stays resident on every GPU that loads the library until the
// process exits.  Every call uses the same array, so calls that overlap on the GPU (from
// two streams or two threads) race; the array keeps the previous call's contents, so this
// file clears what must start at zero.  The first call on a device looks up the device
// address of the array once (cudaGetSymbolAddress with that device current); make that
// first call before any stream capture.
#include <math.h>
#include <stddef.h>

#include <mutex>
#include <string>

#include "ccm_host.h"

namespace {

using namespace ccm;

constexpr size_t kMaxElems = CCM_NOALLOC_MAX_ELEMS;
constexpr size_t kMaxPartials = 8192;
constexpr int kMaxDevices = 64;

struct Scratch {
  double b[kMaxElems];           // right-hand side restricted to active cells
  double r[kMaxElems];           // the tiles' first residual
  ulonglong2 mail[2 * kMaxElems];  // the tiles' mailboxes
  double partials[kMaxPartials];
  unsigned long long fxacc[kFxAccWords];
  double rr, bb;
  int iters, converged;
  int bar_err, pad;
  unsigned int bar_count[kBarWords];
};

static __device__ __align__(256) Scratch g_scratch;

std::mutex g_mu;
void* g_addr[kMaxDevices] = {};

__global__ void k_masked_copy(Geom g, const int8_t* act, const double* src, double* dst) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) - 1;
  const int j = (int)(blockIdx.y * blockDim.y + threadIdx.y) - 1;
  if (i > g.nx + 1 || j > g.ny + 1) return;
  const size_t k = g.idx(i, j);
  dst[k] = act[k] ? src[k] : 0.0;
}

__global__ void k_mask(Geom g, const int8_t* act, double* x) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) - 1;
  const int j = (int)(blockIdx.y * blockDim.y + threadIdx.y) - 1;
  if (i > g.nx + 1 || j > g.ny + 1) return;
  const size_t k = g.idx(i, j);
  if (!act[k]) x[k] = 0.0;
}

ccm_status fail(ccm_status s, const std::string& m) {
  set_last_error(m);
  return s;
}

// Device address of the scratch array on the current device (looked up once per device).
cudaError_t scratch_address(Scratch** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_addr[dev]) {
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_scratch);
    if (e != cudaSuccess) return e;
    g_addr[dev] = ptr;
  }
  *out = (Scratch*)g_addr[dev];
  return cudaSuccess;
}

}  // namespace

extern "C" ccm_status ccm_solve_pressure_noalloc(ccm_case c, const double* rhs_dev, double* phi_dev,
                                                 ccm_solve_stats* stats) {
  set_last_error("");
  if (!c || !rhs_dev || !phi_dev) return fail(CCM_E_INVALID, "null argument");
  CaseSolveView v;
  if (!case_solve_view(c, &v)) return fail(CCM_E_STATE, "set_geometry must come first");
  if (v.g.px || v.g.py) return fail(CCM_E_INVALID, "periodic cases are not supported by this solve");
  const size_t n = v.g.count();
  if (n > kMaxElems)
    return fail(CCM_E_INVALID, "grid too large for the fixed scratch: (ny+3)*pitch = " + std::to_string(n) +
                                   " elements, the maximum is " + std::to_string(kMaxElems));
  if ((size_t)pcg_partials_needed() > kMaxPartials) return fail(CCM_E_INVALID, "too many multiprocessors");
  Scratch* S = nullptr;
  cudaError_t e = scratch_address(&S);
  if (e != cudaSuccess) return fail(CCM_E_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
  cudaStream_t st = v.st;
  // the barrier counter and its error flag hold the previous call's (the kernel clears or writes
  // the rest of the scratch before it reads it)
  if ((e = cudaMemsetAsync(&S->bar_err, 0, 2 * sizeof(int) + sizeof(unsigned int) * kBarWords, st)) != cudaSuccess)
    return fail(CCM_E_CUDA, std::string("cudaMemsetAsync: ") + cudaGetErrorString(e));
  const dim3 blk(64, 4), grd((v.g.nx + 3 + 63) / 64, (v.g.ny + 3 + 3) / 4);
  k_masked_copy<<<grd, blk, 0, st>>>(v.g, v.act, rhs_dev, S->b);
  k_mask<<<grd, blk, 0, st>>>(v.g, v.act, phi_dev);
  FusedSolve f{};
  f.a = scaled_solve_of(v, phi_dev, S->b, nullptr, nullptr, nullptr, nullptr, nullptr);
  f.a.partials = S->partials;
  f.a.bar = Barrier{S->bar_count, &S->bar_err, 2000000000LL};
  f.a.out = PcgOut{&S->iters, &S->rr, &S->bb, &S->converged, nullptr, nullptr};
  f.fxacc = S->fxacc;
  f.R[0] = S->r;
  f.mail = S->mail;
  f.mail_slots = 2 * kMaxElems;
  f.resident = 1;
  f.zero_mean = v.zero_mean;
  e = cudaSuccess;
  if (v.zero_mean) {
    e = project_zero_mean(v.g, v.act, phi_dev, S->partials, v.n_act, st);
    if (e == cudaSuccess) e = project_zero_mean(v.g, v.act, S->b, S->partials, v.n_act, st);
  }
  if (e == cudaSuccess) e = run_poisson_fused(f, st);
  if (e == cudaSuccess && v.zero_mean) e = project_zero_mean(v.g, v.act, phi_dev, S->partials, v.n_act, st);
  if (e != cudaSuccess)
    return fail(CCM_E_CUDA, std::string("Poisson PCG launch: ") + cudaGetErrorString(e));
  struct { double rr, bb; int iters, converged; int err, pad; } h{};
  static_assert(sizeof(h) == offsetof(Scratch, bar_count) - offsetof(Scratch, rr), "layout");
  if ((e = cudaMemcpyAsync(&h, &S->rr, sizeof(h), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(st)) != cudaSuccess)
    return fail(CCM_E_CUDA, std::string("reading the solve statistics: ") + cudaGetErrorString(e));
  if (h.err) return fail(CCM_E_TIMEOUT, "a device-wide barrier gave up waiting");
  if (stats) {
    stats->iters = h.iters;
    stats->outer = 1;
    stats->rel_res = h.bb > 0 ? sqrt(h.rr / h.bb) : 0.0;
    stats->converged = h.converged;
  }
  if (!h.converged) return fail(CCM_E_NOT_CONVERGED, "Poisson PCG reached its iteration limit");
  return CCM_OK;
}
