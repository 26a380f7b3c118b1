// iccg_spmv_dot_noalloc: q = A p and <p, q> without any device allocation.
//
// Some callers cannot allocate device memory at the point where they need a
// sparse product: latency-critical loops that must not pay for the
// allocator's implicit device synchronisation, and host frameworks that own
// all device memory through their own pool and forbid raw cudaMalloc (an
// allocation behind their back would break their accounting or fail under
// their memory cap).  This entry point serves them: the caller passes every
// input and output as device pointers, and the only scratch the kernel needs
// (one partial sum per CTA plus the arrival counters of the deterministic
// two-level reduction) lives in a fixed file-scope __device__ array.
//
// That array is part of the module: every GPU that loads the library holds
// it until the process exits.  All calls share it, and it keeps the contents
// of the last call, so the counters that must start at zero are cleared at
// the start of every call (a memset on the caller's stream, not an
// allocation).  Two calls whose kernels overlap on the GPU (different streams,
// or different host threads) race on the array and give wrong results.
//
// The first call on each device looks up the array's device address with
// cudaGetSymbolAddress (with that device current) and caches it.  The stream
// must belong to the current device (the cached address is that device's
// copy of the array).
#include <algorithm>
#include <cstddef>
#include <mutex>

#include "iccg_internal.h"

namespace {

constexpr int kNaWarps = 8;                       // warps per CTA
constexpr int kNaRowsPerCta = kNaWarps * 32;      // one row per lane
constexpr int kNaGrid = 4 * 152;                  // CTAs of a launch at most: those a GB300 holds at once
constexpr int kNaGroup = 32;                      // CTAs per first-level group
constexpr int kNaGroups = kNaGrid / kNaGroup;

struct NaScratch {
  double part[kNaGrid];           // per-CTA partial of <p, q>
  double gsum[kNaGroups];         // per-group sums
  unsigned int gticket[kNaGroups];
  unsigned int ticket;            // groups finished
};

static_assert(kNaGroups * kNaGroup == kNaGrid, "the CTAs must split into whole groups");
static_assert(int64_t(ICCG_NOALLOC_MAX_ROWS) + int64_t(kNaGrid) * kNaRowsPerCta <= INT32_MAX, "a row index past the last");
static_assert(offsetof(NaScratch, ticket) == offsetof(NaScratch, gticket) + sizeof(NaScratch::gticket), "cleared together");

static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NaScratch)];

__device__ __forceinline__ double na_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// one value per thread -> thread 0, fixed order
__device__ __forceinline__ double na_cta_sum(double v, double *red) {
  v = na_warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < int(blockDim.x >> 5); ++k) s += red[k];
  return s;
}

__device__ __forceinline__ bool na_last(unsigned int *ticket, unsigned int expected, int *flag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    *flag = atomicAdd(ticket, 1u) == expected - 1 ? 1 : 0;
    if (*flag) __threadfence();
  }
  __syncthreads();
  return *flag != 0;
}

// Two forms, by the number of rows.
//
// More rows than kNaGrid CTAs hold: a persistent grid.  A warp takes slices of 32
// rows, whose CSR entries are one range.  A slice of at most kNaChunk entries (8 a
// row: 5- and 7-point) is copied into shared memory coalesced, and a lane then
// sums its own row from there, the gathers of kNaBatch entries in flight
// (consecutive rows gather neighbouring elements of p); the next slice's row
// pointers and entries are loaded while the current one is summed.  A slice with
// more entries is read a lane per row from global memory (na_row): staged in
// chunks, only the few lanes whose rows lie in the chunk would work at a time,
// and an FP64 instruction costs a warp the same for 1 lane as for 32.  Bound by
// memory traffic and, equally, by the FP64 rate, which is why the <p, q> sum
// runs once per CTA over all its slices, not once per 256 rows.  7-point 160^3
// 130 us with a CTA per 256 rows, 87 so; 27-point 155^3 377 and 352 (in chunks
// 877).
//
// Fewer rows: a CTA per 256 rows, a lane per row, with the registers and the L1
// that 64 warps an SM leave (latency bound; there is no next slice to load
// meanwhile: 27-point 50^3 24 us, graph of degree 16, 100,000 rows 23 us, both
// forms at 7-point 50^3 15 us).
constexpr int kNaChunk = 256;
constexpr int kNaBatch = 8;

struct NaChunk {
  int32_t c[kNaChunk / 32];
  double v[kNaChunk / 32];
};

__device__ __forceinline__ void na_load(NaChunk &k, const int32_t *colind, const double *val, int64_t b, int cnt,
                                        int lane) {
#pragma unroll
  for (int u = 0; u < kNaChunk / 32; ++u) {
    const int e = u * 32 + lane;
    k.c[u] = e < cnt ? __ldg(colind + b + e) : 0;
    k.v[u] = e < cnt ? __ldg(val + b + e) : 0.0;
  }
}

// <p, q> from the lanes' shares: over the CTA, groups of CTAs, the groups
__device__ __forceinline__ void na_finish(double acc, double *red, int *flag, NaScratch *s, double *pq) {
  const double cta = na_cta_sum(acc, red);
  const int g = blockIdx.x / kNaGroup;
  const int g0 = g * kNaGroup;
  const int gs = min(kNaGroup, int(gridDim.x) - g0);
  if (threadIdx.x == 0) s->part[blockIdx.x] = cta;
  if (!na_last(&s->gticket[g], unsigned(gs), flag)) return;
  const double gv = na_cta_sum(threadIdx.x < gs ? __ldcg(&s->part[g0 + threadIdx.x]) : 0.0, red);
  if (threadIdx.x == 0) s->gsum[g] = gv;
  const unsigned ng = (gridDim.x + kNaGroup - 1) / kNaGroup;
  if (!na_last(&s->ticket, ng, flag)) return;
  double t = 0.0;
  for (unsigned k = threadIdx.x; k < ng; k += blockDim.x) t += __ldcg(&s->gsum[k]);
  const double total = na_cta_sum(t, red);
  if (threadIdx.x == 0) *pq = total;
}

// A lane's row [b, e): the gathers of kNaWalk entries in flight while the next
// ones' columns and values are loaded
constexpr int kNaWalk = 4;
__device__ __forceinline__ double na_row(const int32_t *colind, const double *val, const double *p, int64_t b,
                                         int64_t e) {
  colind += b;
  val += b;
  const int len = int(e - b);
  double sum = 0.0;
  int32_t c[kNaWalk];
  double v[kNaWalk];
#pragma unroll
  for (int u = 0; u < kNaWalk; ++u) {
    c[u] = u < len ? __ldg(colind + u) : 0;
    v[u] = u < len ? __ldg(val + u) : 0.0;
  }
  for (int k0 = 0; k0 < len; k0 += kNaWalk) {
    double x[kNaWalk], w[kNaWalk];
#pragma unroll
    for (int u = 0; u < kNaWalk; ++u) {
      x[u] = k0 + u < len ? __ldg(p + c[u]) : 0.0;
      w[u] = v[u];
    }
    const int n0 = k0 + kNaWalk;
#pragma unroll
    for (int u = 0; u < kNaWalk; ++u) {
      c[u] = n0 + u < len ? __ldg(colind + n0 + u) : 0;
      v[u] = n0 + u < len ? __ldg(val + n0 + u) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kNaWalk; ++u)
      if (k0 + u < len) sum += w[u] * x[u];
  }
  return sum;
}

__global__ void __launch_bounds__(kNaRowsPerCta, 4)
spmv_dot_noalloc_kernel(int n, const int64_t *__restrict__ rowptr, const int32_t *__restrict__ colind,
                        const double *__restrict__ val, const double *__restrict__ p, double *__restrict__ q,
                        double *__restrict__ pq, NaScratch *s) {
  __shared__ double red[kNaWarps];
  __shared__ int flag;
  __shared__ double sval[kNaWarps][kNaChunk];
  __shared__ int32_t scol[kNaWarps][kNaChunk];
  const int lane = threadIdx.x & 31;
  double *sv = sval[threadIdx.x >> 5];
  int32_t *sc = scol[threadIdx.x >> 5];
  double acc = 0.0;
  const int stride = int(gridDim.x) * kNaRowsPerCta;
  int i = blockIdx.x * kNaRowsPerCta + threadIdx.x;
  int64_t rs = 0, re = 0;
  if (i - lane < n) {
    rs = rowptr[min(i, n)];
    re = rowptr[min(i + 1, n)];
  }
  NaChunk nx;
  {
    const int64_t e0 = __shfl_sync(0xffffffffu, rs, 0), e1 = __shfl_sync(0xffffffffu, re, 31);
    na_load(nx, colind, val, e0, e1 - e0 <= kNaChunk ? int(e1 - e0) : 0, lane);
  }
  while (i - lane < n) {
    const int in = i + stride;   // below ICCG_NOALLOC_MAX_ROWS + kNaGrid * kNaRowsPerCta
    const bool more = in - lane < n;
    const int64_t rsn = more ? rowptr[min(in, n)] : 0, ren = more ? rowptr[min(in + 1, n)] : 0;
    const int64_t e0 = __shfl_sync(0xffffffffu, rs, 0), e1 = __shfl_sync(0xffffffffu, re, 31);
    const bool staged = e1 - e0 <= kNaChunk;
    const double pi = i < n ? p[i] : 0.0;
    double sum = 0.0;
    if (staged) {
      __syncwarp();   // every lane is done with the previous slice
#pragma unroll
      for (int u = 0; u < kNaChunk / 32; ++u) {
        sc[u * 32 + lane] = nx.c[u];
        sv[u * 32 + lane] = nx.v[u];
      }
      __syncwarp();
    }
    // (the walk before the next slice's loads: their registers in turn)
    if (!staged) sum = na_row(colind, val, p, rs, re);
    const int64_t f0 = __shfl_sync(0xffffffffu, rsn, 0), f1 = __shfl_sync(0xffffffffu, ren, 31);
    na_load(nx, colind, val, f0, f1 - f0 <= kNaChunk ? int(f1 - f0) : 0, lane);
    if (staged) {
      const int hi = int(re - e0);
      for (int k0 = int(rs - e0); k0 < hi; k0 += kNaBatch) {
        double x[kNaBatch];
#pragma unroll
        for (int u = 0; u < kNaBatch; ++u) x[u] = k0 + u < hi ? p[sc[k0 + u]] : 0.0;
#pragma unroll
        for (int u = 0; u < kNaBatch; ++u)
          if (k0 + u < hi) sum += sv[k0 + u] * x[u];
      }
    }
    if (i < n) {
      q[i] = sum;
      acc += pi * sum;
    }
    rs = rsn;
    re = ren;
    i = in;
  }
  na_finish(acc, red, &flag, s, pq);
}

// a CTA per 256 rows
__global__ void __launch_bounds__(kNaRowsPerCta)
spmv_dot_noalloc_small(int n, const int64_t *__restrict__ rowptr, const int32_t *__restrict__ colind,
                       const double *__restrict__ val, const double *__restrict__ p, double *__restrict__ q,
                       double *__restrict__ pq, NaScratch *s) {
  __shared__ double red[kNaWarps];
  __shared__ int flag;
  const int i = blockIdx.x * kNaRowsPerCta + threadIdx.x;
  double acc = 0.0;
  if (i < n) {
    double sum = 0.0;
    for (int64_t e = rowptr[i]; e < rowptr[i + 1]; ++e) sum += val[e] * p[colind[e]];
    q[i] = sum;
    acc = p[i] * sum;
  }
  na_finish(acc, red, &flag, s, pq);
}

std::mutex g_na_mutex;
NaScratch *g_na_ptr[64] = {nullptr};

}  // namespace

extern "C" iccg_status iccg_spmv_dot_noalloc(int32_t n, const int64_t *rowptr, const int32_t *colind,
                                             const double *val, const double *p, double *q, double *pq,
                                             iccg_stream_t stream) {
  if (n < 0 || n > ICCG_NOALLOC_MAX_ROWS) return ICCG_ERR_ARG;
  if (!pq || (n > 0 && (!rowptr || !colind || !val || !p || !q))) return ICCG_ERR_ARG;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ICCG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the scratch address below is the current device's copy: a stream of
  // another device would run the kernel against the wrong GPU's memory
  int sdev = -1;
  if (cudaStreamGetDevice(st, &sdev) != cudaSuccess) return ICCG_ERR_ARG;
  if (sdev != dev) return ICCG_ERR_ARG;
  NaScratch *s = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_na_mutex);
    if (!g_na_ptr[dev]) {
      void *addr = nullptr;
      if (cudaGetSymbolAddress(&addr, g_noalloc_scratch) != cudaSuccess || !addr) return ICCG_ERR_CUDA;
      g_na_ptr[dev] = static_cast<NaScratch *>(addr);
    }
    s = g_na_ptr[dev];
  }
  if (n == 0) return cudaMemsetAsync(pq, 0, sizeof(double), st) == cudaSuccess ? ICCG_OK : ICCG_ERR_CUDA;
  const int ctas = (n + kNaRowsPerCta - 1) / kNaRowsPerCta;
  // the arrival counters must start at zero; the previous call left them at
  // their final counts
  // (one memset over both, adjacent: a second one cost 2 us per call)
  if (cudaMemsetAsync(s->gticket, 0, sizeof(s->gticket) + sizeof(s->ticket), st) != cudaSuccess) return ICCG_ERR_CUDA;
  // the launch's own status (cudaGetLastError would also report, and clear,
  // an error that earlier unrelated work of the caller left pending)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(std::min(ctas, kNaGrid)));
  cfg.blockDim = dim3(unsigned(kNaRowsPerCta));
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, ctas <= kNaGrid ? spmv_dot_noalloc_small : spmv_dot_noalloc_kernel, n, rowptr, colind,
                            val, p, q, pq, s) == cudaSuccess
             ? ICCG_OK
             : ICCG_ERR_CUDA;
}
