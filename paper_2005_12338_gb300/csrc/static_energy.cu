// rssri_energy_static: the Eq. 26 energy of a caller-held self-energy, for
// callers that may not allocate device memory.
//
// Some callers cannot call cudaMalloc: code running while a stream is being
// captured into a CUDA graph (an allocation there breaks the capture), hosts
// that hand every byte of device memory to their own pool allocator and forbid
// libraries from allocating behind their back, and real-time loops that must
// not hit the allocator's synchronisation.  This entry point creates no handle
// and allocates nothing: its only scratch (partial traces and counters of
// finished blocks) is file-scope __device__ memory of fixed size, loaded with
// the library and held by every GPU that loads it until the process exits.
//
// One launch: the block that finishes last adds the partial traces (a second
// launch for that cost as much as the traces of small problems).  The blocks of
// a launch count modulo their number, on a counter that only launches of as many
// blocks use: whatever calls overlap, each leaves the counter where it was, so that
// an overlap, which the interface forbids, spoils the overlapping calls alone.
#include <mutex>

#include "trace.cuh"

namespace {

// RSSRI_STATIC_MAX_TAU partial traces (32 KiB), then a counter for every number of
// blocks up to that (16 KiB), zero between calls.
static __device__ __align__(256) double
    g_energy_scratch[RSSRI_STATIC_MAX_TAU + RSSRI_STATIC_MAX_TAU / 2];
static_assert(RSSRI_STATIC_MAX_TAU >= rssri::TRACE_SLOTS, "slots of trace_parts");

constexpr int kMaxDevices = 64;
std::mutex g_mutex;
double *g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device.  The symbol's
// host-side name is only a stand-in: the address must come from
// cudaGetSymbolAddress with that device current.  Looked up once per device.
cudaError_t scratch_on_current_device(double **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_scratch_ptr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_energy_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = static_cast<double *>(p);
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

// Partial traces by block (p, t); the last block to finish forms
// e_corr = -(sum_t w_t tr[t]) / ne, summed in tau order (the same order as
// the energy of rssri_sigma).
__global__ void __launch_bounds__(256) static_energy_kernel(const double *__restrict__ sigma,
                                                            const double *__restrict__ gb,
                                                            const double *__restrict__ tau_w, int n,
                                                            double ne, double *scratch,
                                                            double *__restrict__ e_corr) {
  __shared__ bool last;
  const long long nn = (long long)n * n;
  const int t = blockIdx.y, parts = gridDim.x, nt = gridDim.y;
  const unsigned blocks = parts * nt;  // <= RSSRI_STATIC_MAX_TAU
  unsigned *count = reinterpret_cast<unsigned *>(scratch + RSSRI_STATIC_MAX_TAU) + blocks - 1;
  const double s = rssri::trace_part(sigma + t * nn, gb + t * nn, n, blockIdx.x, parts);
  if (threadIdx.x == 0) {
    scratch[(long long)t * parts + blockIdx.x] = s;
    __threadfence();
    last = atomicInc(count, blocks - 1) == blocks - 1;  // the last one wraps it to 0
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const double b = rssri::trace_weighted(tau_w, scratch, parts, nt);
  if (threadIdx.x == 0) e_corr[0] = -b / ne;
}

}  // namespace

extern "C" int rssri_energy_static(const double *sigma, const double *gb, const double *tau_w,
                                   int n, int n_tau, int n_occ, double *e_corr, void *stream) {
  if (!sigma || !gb || !tau_w || !e_corr) return RSSRI_ERR_INVALID_ARG;
  if (n < 1 || n > 4096 || n_occ < 1 || n_tau < 1) return RSSRI_ERR_INVALID_ARG;
  if (n_tau > RSSRI_STATIC_MAX_TAU) return RSSRI_ERR_INVALID_ARG;  // beyond the static scratch
  double *scratch = nullptr;
  cudaError_t e = scratch_on_current_device(&scratch);
  if (e != cudaSuccess) return RSSRI_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  static_energy_kernel<<<dim3(rssri::trace_parts(n, n_tau), n_tau), 256, 0, s>>>(
      sigma, gb, tau_w, n, 2.0 * n_occ, scratch, e_corr);
  e = cudaGetLastError();
  return e == cudaSuccess ? RSSRI_OK : RSSRI_ERR_CUDA;
}
