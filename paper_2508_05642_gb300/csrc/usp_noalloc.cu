// usp_noalloc.cu -- per-cell moments of a caller-owned particle state with no
// device allocation at all.
//
// Some callers cannot let a library allocate device memory: frameworks that
// carve all device memory out of their own pool at start-up and forbid any
// later cudaMalloc, code that must not trigger the implicit device
// synchronisation cudaMalloc/cudaFree can cause in the middle of a time step,
// or hosts running under a hard device-memory budget.  usp_moments_noalloc
// serves them: it computes the same per-cell moments as usp_moments, but its
// working space (the FP64 per-cell accumulators) lives in the file-scope
// device array below, of fixed size, kept on each device until the process
// exits.  With CUDA's lazy module loading (the default), the array is
// reserved on a device when the library's module is first loaded there,
// which is at the first call on that device at the latest (that call also
// looks up the array's address): a caller that must not see any reservation
// inside its time loop makes one warm-up call at start-up, or sets
// CUDA_MODULE_LOADING=EAGER.  The address looked up at a device's first call
// is kept, so a cudaDeviceReset between calls is not supported.  The caller
// passes the inputs and the output buffer.
//
// Every call shares that one array and leaves its last contents there: each
// call clears it first on the caller's stream.  Two calls whose work overlaps
// on the GPU (for instance on two streams at once) race on it.
#include <cuda_runtime.h>

#include <mutex>

#include "../../include/usp.h"
#include "usp_sums.cuh"

// Scratch: 20 FP64 sums for each of up to USP_NOALLOC_MAX_CELLS cells
// (20 x 8192 x 8 B = 1.25 MiB on every device that loads the library).
static __device__ __align__(256) double g_na_scratch[20 * USP_NOALLOC_MAX_CELLS];

namespace {

constexpr int kNaAcc = usp::kRawN;   // accumulators per cell
constexpr double kNaKB = 1.380649e-23;  // Boltzmann constant [J/K]

// what the moments need of the species: R = k_B / m and Theta_vib
struct NaGas {
  double R, theta_v;
};

// temperature whose e_vib = R Theta / (exp(Theta/T) - 1) equals R Theta ebar
__device__ __forceinline__ double na_T_vib(const NaGas& g, double ebar) {
  if (ebar <= 0.0) return 0.0;
  return g.theta_v / log1p(1.0 / ebar);
}

// Device address of g_na_scratch, looked up once per device (host code may
// not use the symbol itself as a device pointer).
constexpr int kMaxDevices = 64;
double* g_na_ptr[kMaxDevices] = {nullptr};
std::mutex g_na_mutex;

// Per cell (G threads each) its sums cleared and its reference velocity (usp_sums.cuh)
// into the rows of U.
template <int G>
__global__ void __launch_bounds__(usp::kRawBlock)
na_references(int ncell, const int64_t* __restrict__ off, const double* __restrict__ cx,
              const double* __restrict__ cy, const double* __restrict__ cz,
              double* __restrict__ acc, double* __restrict__ out) {
  const int c = blockIdx.x * (usp::kRawBlock / G) + threadIdx.x / G;
  if (c >= ncell) return;   // uniform over the G threads
  if (threadIdx.x % G < kNaAcc) acc[(size_t)c * kNaAcc + threadIdx.x % G] = 0.0;
  usp::raw_reference<G>(off[c], off[c + 1] - off[c], cx, cy, cz, out + ncell + c, ncell);
}

// Raw sums of every cell about its reference velocity, one
// pass; blockIdx.y walks the cells.  Bound by the FP64 pipe (22 to 26
// operations per particle, 2 lanes per clock and SM).
__global__ void __launch_bounds__(usp::kRawBlock)
na_sums(int ncell, int chunk_min, const int64_t* __restrict__ off, const double* __restrict__ cx,
        const double* __restrict__ cy, const double* __restrict__ cz,
        const double* __restrict__ er, const int32_t* __restrict__ lev, double* __restrict__ acc,
        const double* __restrict__ out) {
  for (int c = blockIdx.y; c < ncell; c += gridDim.y) {
    const double* w = out + ncell + c;
    usp::raw_cell(off[c], off[c + 1] - off[c], chunk_min,
                  [&] { return usp::RawRef{{w[0], w[ncell], w[2 * (size_t)ncell]}}; }, cx, cy, cz,
                  er, lev, acc + (size_t)c * kNaAcc);
  }
}

// one thread per cell; the reference velocities are in the rows of U
__global__ void na_assemble(NaGas gas, int ncell, const int64_t* __restrict__ off,
                            const double* __restrict__ acc, double* __restrict__ out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const double R = gas.R;
  const long long n = off[c + 1] - off[c];
  if (n <= 0) {
    for (int f = 0; f < USP_NMOM; ++f) out[(size_t)f * ncell + c] = 0.0;
    return;
  }
  const double w[3] = {out[ncell + c], out[2 * (size_t)ncell + c], out[3 * (size_t)ncell + c]};
  const usp::RawMoments m = usp::raw_moments(acc + (size_t)c * kNaAcc, (double)n, w);
  out[c] = (double)n;
  for (int i = 0; i < 3; ++i) out[(size_t)(1 + i) * ncell + c] = m.U[i];
  out[(size_t)4 * ncell + c] = (m.P[0] + m.P[1] + m.P[2]) / (3.0 * R);
  out[(size_t)5 * ncell + c] = m.eps / R;
  out[(size_t)6 * ncell + c] = na_T_vib(gas, m.lev);
  for (int i = 0; i < 6; ++i) out[(size_t)(7 + i) * ncell + c] = m.P[i];
  for (int i = 0; i < 3; ++i) {
    out[(size_t)(13 + i) * ncell + c] = m.qt[i];
    out[(size_t)(16 + i) * ncell + c] = m.qr[i];
    out[(size_t)(19 + i) * ncell + c] = m.ql[i] * R * gas.theta_v;
  }
}

// Look up the device address of the scratch array for the current device,
// once per device.
int na_scratch_for_current_device(double** ptr) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return USP_ECUDA;
  if (dev < 0 || dev >= kMaxDevices) return USP_ENOTSUP;
  std::lock_guard<std::mutex> lock(g_na_mutex);
  if (!g_na_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_na_scratch) != cudaSuccess || !p) return USP_ECUDA;
    g_na_ptr[dev] = (double*)p;
  }
  *ptr = g_na_ptr[dev];
  return USP_OK;
}

}  // namespace

extern "C" int usp_moments_noalloc(const usp_species* sp, int n_cells, const int64_t* d_offsets,
                                   const double* d_cx, const double* d_cy, const double* d_cz,
                                   const double* d_erot, const int32_t* d_lev, double* d_out,
                                   void* stream) {
  if (!sp || !d_offsets || !d_out || n_cells <= 0) return USP_EINVAL;
  if (n_cells > USP_NOALLOC_MAX_CELLS) return USP_EINVAL;
  if (!d_cx || !d_cy || !d_cz || !d_erot || !d_lev) return USP_EINVAL;
  if (!(sp->m > 0.0) || !(sp->theta_v > 0.0)) return USP_EINVAL;
  double* acc = nullptr;
  const int rc = na_scratch_for_current_device(&acc);
  if (rc != USP_OK) return rc;
  NaGas gas;
  gas.R = kNaKB / sp->m;
  gas.theta_v = sp->theta_v;
  cudaStream_t st = (cudaStream_t)stream;
  // an error left by the caller's earlier work is not this call's: report it
  // without launching (and without clearing it)
  if (cudaPeekAtLastError() != cudaSuccess) return USP_ECUDA;
  if (usp::ref_by_warp(n_cells))
    na_references<32><<<(n_cells + 7) / 8, usp::kRawBlock, 0, st>>>(n_cells, d_offsets, d_cx, d_cy,
                                                                    d_cz, acc, d_out);
  else
    na_references<usp::kRawBlock><<<n_cells, usp::kRawBlock, 0, st>>>(n_cells, d_offsets, d_cx, d_cy,
                                                                      d_cz, acc, d_out);
  if (cudaGetLastError() != cudaSuccess) return USP_ECUDA;
  na_sums<<<dim3(usp::raw_blocks(n_cells), n_cells), usp::kRawBlock, 0, st>>>(
      n_cells, usp::raw_chunk(n_cells), d_offsets, d_cx, d_cy, d_cz, d_erot, d_lev, acc, d_out);
  if (cudaGetLastError() != cudaSuccess) return USP_ECUDA;
  na_assemble<<<(n_cells + 63) / 64, 64, 0, st>>>(gas, n_cells, d_offsets, acc, d_out);
  if (cudaGetLastError() != cudaSuccess) return USP_ECUDA;
  return USP_OK;
}
