// hca_o2_residual_noalloc: the oxygen solve's true-residual check on
// caller-owned device arrays, without any device allocation.
//
// Who needs this: code that may not call cudaMalloc on the path where it
// checks a field -- for example a caller running inside another framework's
// memory pool that must not be bypassed, a real-time loop where an
// allocation's latency or its implicit device synchronisation is not
// allowed, or an embedding that only hands the library raw pointers.  Such a
// caller cannot create a handle (which owns its device buffers) just to ask
// "how well does this K solve the oxygen system linearised about K_prev?".
//
// This entry point answers that with the same arithmetic as the handle's
// true-residual kernel: per site r = b - A(K_prev) K with the 7-point
// Neumann operator, summed per chunk of rows (1 to 32, by the lattice's size)
// and then over chunks in a fixed order.  The per-chunk partial sums, the arrival count and the result
// live in the file-scope device array `g_noalloc` below instead of memory
// the caller or the library would allocate.  Its size is fixed at compile
// time (kNoAllocMaxChunks chunks: ny * nz <= 65536 rows, e.g. 256 x 256 in
// y, z with any nx), it occupies about 33 KB on every GPU that loads the library
// until the process exits, and every call shares it.  Calls that overlap on
// the GPU (two streams, or two host threads) race on it and must be
// serialised by the caller.
//
// The array's device address is looked up on every call, with the caller's
// device current (cudaGetSymbolAddress is a host-side lookup and allocates
// nothing).  A cached address could outlive the context it belongs to: after
// a device reset the module is loaded again and the array may move.
//
// A small lattice's call is latency: the FP64 arithmetic (one warp
// instruction occupies a quarter of a multiprocessor for 76 cycles) is spread
// over all multiprocessors by short chunks and trimmed to ~25 operations a
// site (|b|^2 counts vessels, c n comes from a table), and where the GPU can
// write pageable host memory (Grace) the result goes straight to the caller's
// stack instead of through a copy.  48^3: 42 -> 28 us a call.
#include <cuda_runtime.h>

#include <atomic>

#include "hca_internal.cuh"

namespace {

constexpr int kNoAllocMaxChunks = 2048;
constexpr int kNoAllocRows = 32;       // most rows per chunk
constexpr int kNoAllocThreads = 256;   // fixed: the reduction order depends on it

struct NoAllocScratch {
  double partial[kNoAllocMaxChunks][2];  // per chunk: |r|^2, |b|^2
  double result[2];                      // |r| / |b|, the number of the call it belongs to
  // the call's number (upper bits) and the chunks it has finished (lower 16):
  // every block raises the number to its own call's before it counts itself,
  // so what an earlier call left (one that overlapped another, or was cut
  // short) drops out, and no memset has to come before the kernel
  unsigned long long ticket;
  unsigned long long pad;
};
constexpr int kArrivalBits = 16;
static_assert(kNoAllocMaxChunks < 1 << kArrivalBits, "a call's arrivals fit their bits");

static __device__ __align__(256) NoAllocScratch g_noalloc;

// out: where the result goes besides the scratch array (host memory the GPU
// can write, or null).
__global__ void __launch_bounds__(kNoAllocThreads) k_o2_residual_noalloc(
    NoAllocScratch* __restrict__ sc, unsigned long long call, int nx, int ny, int nz, int chunk_rows, double c, double phi_K, double K1, double b0,
    double r_K, const uint8_t* __restrict__ state, const double* __restrict__ K_prev,
    const double* __restrict__ K, double* out) {
  __shared__ double s_cn[7];   // c times a neighbour count
  if (threadIdx.x < 7) s_cn[threadIdx.x] = c * (double)threadIdx.x;
  __syncthreads();
  const int rows = ny * nz;
  const int row0 = blockIdx.x * chunk_rows;
  const int nrow = min(chunk_rows, rows - row0);
  const int nsite = nrow * nx;   // at most the lattice's sites: below 2^31
  const long long plane = (long long)nx * ny;
  double rr = 0.0;
  int vessels = 0;
  for (long long t0 = threadIdx.x; t0 < nsite; t0 += kNoAllocThreads) {
    const int t = (int)t0, jr = t / nx;
    const int j = row0 + jr;
    const int x = t - jr * nx;
    const int z = j / ny, y = j - z * ny;
    const long long i = (long long)j * nx + x;
    const uint8_t s = state[i];
    const bool xm = x > 0, xp = x < nx - 1, ym = y > 0, yp = y < ny - 1, zm = z > 0, zp = z < nz - 1;
    const double Ki = K[i];
    const double kxm = xm ? K[i - 1] : 0.0, kxp = xp ? K[i + 1] : 0.0;
    const double kym = ym ? K[i - nx] : 0.0, kyp = yp ? K[i + nx] : 0.0;
    const double kzm = zm ? K[i - plane] : 0.0, kzp = zp ? K[i + plane] : 0.0;
    double d = s_cn[xm + xp + ym + yp + zm + zp];
    if (s == HCA_PROLIF || s == HCA_QUIESC || s == HCA_STROMA) d += phi_K / (K1 + K_prev[i]);
    const bool vessel = s == HCA_VESSEL;
    if (vessel) d += r_K;
    vessels += vessel;
    const double nb = ((kxm + kxp) + (kym + kyp)) + (kzm + kzp);
    const double r = (vessel ? b0 : 0.0) - (d * Ki - c * nb);
    rr += r * r;
  }
  double bb = (double)vessels * (b0 * b0);
  // fixed-order block reduction: warp xor trees, then warp sums in order
  __shared__ double s_w[kNoAllocThreads / 32][2];
  for (int o = 16; o > 0; o >>= 1) {
    rr += __shfl_xor_sync(0xffffffffu, rr, o);
    bb += __shfl_xor_sync(0xffffffffu, bb, o);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    s_w[warp][0] = rr;
    s_w[warp][1] = bb;
  }
  __syncthreads();
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    double a0 = 0.0, a1 = 0.0;
    for (int w = 0; w < kNoAllocThreads / 32; ++w) {
      a0 += s_w[w][0];
      a1 += s_w[w][1];
    }
    sc->partial[blockIdx.x][0] = a0;
    sc->partial[blockIdx.x][1] = a1;
    __threadfence();
    atomicMax(&sc->ticket, call << kArrivalBits);
    s_last = atomicAdd(&sc->ticket, 1ull) == (call << kArrivalBits) + gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  // last block: chunk partials in a fixed order (thread t takes t, t + 256, ...)
  __threadfence();
  double p0 = 0.0, p1 = 0.0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += kNoAllocThreads) {
    p0 += __ldcg(&sc->partial[k][0]);
    p1 += __ldcg(&sc->partial[k][1]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    p0 += __shfl_xor_sync(0xffffffffu, p0, o);
    p1 += __shfl_xor_sync(0xffffffffu, p1, o);
  }
  __syncthreads();
  if (lane == 0) {
    s_w[warp][0] = p0;
    s_w[warp][1] = p1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a0 = 0.0, a1 = 0.0;
    for (int w = 0; w < kNoAllocThreads / 32; ++w) {
      a0 += s_w[w][0];
      a1 += s_w[w][1];
    }
    const double rel = a1 > 0.0 ? sqrt(a0 / a1) : 0.0;
    sc->result[0] = rel;
    sc->result[1] = (double)call;
    if (out) *out = rel;
  }
}

}  // namespace

extern "C" int hca_o2_residual_noalloc(const hca_config* cfg, const uint8_t* state, const double* K_prev,
                                       const double* K, double* rel_out, void* stream) {
  if (!cfg || !state || !K_prev || !K || !rel_out) return HCA_ERR_ARG;
  if (cfg->struct_size != sizeof(hca_config)) return HCA_ERR_ARG;
  if (cfg->nx < 1 || cfg->ny < 1 || cfg->nz < 1 || !(cfg->dx > 0)) return HCA_ERR_ARG;
  // the same parameter checks as handle creation, for the fields read here
  if (!(cfg->D_K > 0) || !(cfg->phi_K >= 0) || !(cfg->K1 > 0) || !(cfg->r_K >= 0) || !(cfg->K0 >= 0))
    return HCA_ERR_ARG;
  // only the quasi-steady operator: with a time-dependent oxygen scheme the
  // handle's right-hand side also depends on the previous field
  if (cfg->o2_scheme != 0) return HCA_ERR_ARG;
  const long long rows = (long long)cfg->ny * cfg->nz;
  if ((rows + kNoAllocRows - 1) / kNoAllocRows > kNoAllocMaxChunks) return HCA_ERR_ARG;   // beyond the fixed scratch size
  if ((long long)cfg->nx * rows > 2147483647LL) return HCA_ERR_ARG;
  // about four blocks a multiprocessor where the lattice has the rows
  const long long want = (rows + 607) / 608, least = (rows + kNoAllocMaxChunks - 1) / kNoAllocMaxChunks;
  const int chunk_rows = (int)(want > kNoAllocRows ? kNoAllocRows : want > least ? want : least);
  const long long chunks = (rows + chunk_rows - 1) / chunk_rows;
  // device address of the scratch array in the current device's context (the
  // host-side symbol is only a stand-in, not a device address)
  void* addr = nullptr;
  if (cudaGetSymbolAddress(&addr, g_noalloc) != cudaSuccess || !addr) {
    (void)cudaGetLastError();
    return HCA_ERR_CUDA;
  }
  NoAllocScratch* sc = (NoAllocScratch*)addr;
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0, ats = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&ats, cudaDevAttrPageableMemoryAccess, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return HCA_ERR_CUDA;
  }
  const double c = cfg->D_K / (cfg->dx * cfg->dx), b0 = cfg->r_K * cfg->K0;
  // A call that overlaps another may find no last block, as the two count in
  // one place: then the result still reads as the mark (or belongs to another
  // call) and the check runs once more.
  static std::atomic<unsigned long long> calls{0};
  const double mark = -1.0;
  volatile double res = mark;
  for (int attempt = 0; attempt < 2 && res == mark; ++attempt) {
    const unsigned long long call = ++calls;   // (2^48 of them)
    k_o2_residual_noalloc<<<(unsigned)chunks, kNoAllocThreads, 0, s>>>(
        sc, call, cfg->nx, cfg->ny, cfg->nz, chunk_rows, c, cfg->phi_K, cfg->K1, b0, cfg->r_K, state, K_prev, K,
        ats ? const_cast<double*>(&res) : nullptr);
    double got[2] = {mark, 0.0};
    if (cudaGetLastError() != cudaSuccess ||
        (!ats && cudaMemcpyAsync(got, sc->result, sizeof(got), cudaMemcpyDeviceToHost, s) != cudaSuccess) ||
        cudaStreamSynchronize(s) != cudaSuccess) {
      (void)cudaGetLastError();
      return HCA_ERR_CUDA;
    }
    if (!ats && got[1] == (double)call) res = got[0];
  }
  if (!isfinite(res)) return HCA_ERR_NONFINITE;
  if (res == mark) return HCA_ERR_CUDA;
  *rel_out = res;
  return HCA_OK;
}
