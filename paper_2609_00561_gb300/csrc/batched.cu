// Batched ICCG: many systems of uneven size, several right-hand sides each,
// in one cooperative launch (the PCG loop lives inside the kernel; the launch
// is replayed as a CUDA graph).  Each system is the block-multicolor ICCG of
// the single-system path (Alg. 1 for the substitutions, standard PCG around
// it) applied to all of its right-hand sides at once.
//
// Layout.  Per system, every n-vector is stored row-major over the
// right-hand sides: v[i * kp + j] (kp = nrhs rounded up to a power of two
// <= 32), so the values of one row for all right-hand sides are one
// contiguous line.  A "chain" of kp lanes (lane j = right-hand side j) walks
// rows; a matrix or factor entry is loaded once per chain and broadcast to
// its lanes, and every vector access of the chain is one coalesced line.
//
// Schedule.  The grid is split into per-system CTA ranges (assign_ctas, at
// least one CTA each); a system's CTAs synchronise only among themselves (a
// bounded-wait barrier per system), so systems progress independently.  Per
// iteration and system: p update | SpMV and <p,q> | x / r update | forward colors
// (the last color's backward sweep fused) | backward colors and the sums, with a
// barrier after each phase (2 n_c + 2 for two colors or more).  A warp owns a
// whole block at a time (batch_precond): everything but the in-block recurrence
// is done for all rows at once, the recurrence itself (rows in order, Alg. 1) on
// shared memory only.  For small blocks, and for wide rows with many right-hand
// sides, a chain owns a block instead and walks its rows, the x / r update of a
// color in front of them (batch_precond_walk; batch_walks says when).  Reductions
// are per right-hand side, per CTA, summed in a fixed order by every CTA of the
// system after a barrier.
// A right-hand side that converged (or met a non-finite value) is frozen.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "iccg_internal.h"

namespace iccg {
namespace {

constexpr int kBatchMaxBlock = 64;   // rows of a block (its row values in shared memory)
constexpr int kBatchCap = 512;       // most entries a warp stages (6 KB)
constexpr long long kBatchSpinLimit = 1ll << 27;

struct BatchSys {
  int32_t n, nc, cta0, cta1;
  const int32_t *arp, *acol;
  const double *aval;
  const int32_t *lrp, *lcol, *urp, *ucol;
  const double *lv64, *uv64, *dv64;
  const float *lv32, *uv32, *dv32;
  const int32_t *cblk;     // [nc + 1] first block of each color
  const int32_t *bptr;     // [nb + 1] first row of each block
  const int32_t *perm;     // row -> original row
  double *x, *r, *p, *q;   // [n][kp]
  void *y, *z;             // [n][kp], precision of the preconditioner
  const double *bin;       // [k][n], original numbering (staging)
  double *xio;             // [k][n], original numbering: x0 in, x out (staging)
  double *part;            // [CTAs of the system][4][kp] partial sums
  double *hist;            // [maxit + 1][kp]
  int32_t *iters;          // [kp]
  int32_t *status;         // [kp] per right-hand side
  GridBar *bar;
  unsigned long long wait_ns;   // bounded barrier wait (ns)
};

template <typename PT> __device__ __forceinline__ const PT *b_lv(const BatchSys &S);
template <> __device__ __forceinline__ const double *b_lv<double>(const BatchSys &S) { return S.lv64; }
template <> __device__ __forceinline__ const float *b_lv<float>(const BatchSys &S) { return S.lv32; }
template <typename PT> __device__ __forceinline__ const PT *b_uv(const BatchSys &S);
template <> __device__ __forceinline__ const double *b_uv<double>(const BatchSys &S) { return S.uv64; }
template <> __device__ __forceinline__ const float *b_uv<float>(const BatchSys &S) { return S.uv32; }
template <typename PT> __device__ __forceinline__ const PT *b_dv(const BatchSys &S);
template <> __device__ __forceinline__ const double *b_dv<double>(const BatchSys &S) { return S.dv64; }
template <> __device__ __forceinline__ const float *b_dv<float>(const BatchSys &S) { return S.dv32; }

__device__ __forceinline__ unsigned b_ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long b_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier over the nct CTAs of one system, with a bounded wait (false for
// the whole CTA when this or another CTA of the system gave up).
__device__ __forceinline__ bool sys_sync(GridBar *bar, unsigned nct, unsigned &gen, int *flag,
                                         unsigned long long wait_ns) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();
    const unsigned arrived = atomicAdd(&bar->count, 1u);
    if (arrived == nct - 1) {
      atomicExch(&bar->count, 0u);
      __threadfence();
      atomicExch(&bar->gen, gen + 1);
    } else {
      const unsigned long long t0 = b_ns();
      // the clock is read on every poll (a short limit must take effect at
      // the first poll); the error word of other CTAs every 64 polls
      for (long long k = 1; b_ld_acquire(&bar->gen) == gen; ++k) {
        if (b_ns() - t0 > wait_ns || k > kBatchSpinLimit ||
            ((k & 63) == 0 && b_ld_acquire(&bar->err) != 0u)) {
          atomicExch(&bar->err, 1u);
          ok = 0;
          break;
        }
        __nanosleep(32);
      }
    }
    __threadfence();
    gen = gen + 1;
    *flag = ok && b_ld_acquire(&bar->err) == 0u;
  }
  __syncthreads();
  return *flag != 0;
}

// Exact float -> double by bit arithmetic (about 8 integer instructions, 3
// cycles of an SM per warp against 16 for the conversion instruction, which
// shares this GPU's scarce FP64 rate); subnormals, infinities and NaN take the
// instruction.
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0u) return double(f);
  return __hiloint2double(int((b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), int(b << 29));
}
__device__ __forceinline__ double widen(double d) { return d; }

// Per-right-hand-side CTA sum: every lane holds v for its (chain, j); the
// sums over the CTA's chains (fixed order) go to part_slot[j]: over a warp's
// chains by shuffles, then over the warps.
__device__ __forceinline__ void cta_rhs_sum(double v, double *red, int kp, double *part_slot) {
  for (int o = 16; o >= kp; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  __syncthreads();
  if (lane < kp) red[w * kp + lane] = v;
  __syncthreads();
  if (threadIdx.x < kp) {
    double s = 0.0;
    for (int c = 0; c < W; ++c) s += red[c * kp + threadIdx.x];
    part_slot[threadIdx.x] = s;
  }
}

// Sum over the system's CTAs of part[.][slot][j] (fixed order) into out[j],
// j < kp; every CTA computes the same values.  The CTA's chains take the CTAs
// in turn (their loads in flight together: one thread per j walking them took
// 10 us for 100 CTAs), then one thread per j adds the chains' sums.
// (The walk's kernel without unrolling: the registers of eight loads cost it 8%
// with 32 right-hand sides in FP64.)
template <bool WALK>
__device__ __forceinline__ void sys_rhs_sum(const double *part, int nct, int kp, int slot, double *out, double *red) {
  const int ch = threadIdx.x / kp, j = threadIdx.x % kp, nchain = blockDim.x / kp;
  const int used = min(nchain, 16);
  __syncthreads();
  if (ch < used) {
    double s = 0.0;
#pragma unroll (WALK ? 1 : 8)
    for (int c = ch; c < nct; c += used) s += __ldcg(part + (size_t(c) * 4 + slot) * kp + j);
    red[ch * kp + j] = s;
  }
  __syncthreads();
  if (threadIdx.x < kp) {
    double s = 0.0;
    for (int c = 0; c < used; ++c) s += red[c * kp + threadIdx.x];
    out[threadIdx.x] = s;
  }
  __syncthreads();
}

// A warp's shared memory: w (row values of the current block, one per
// right-hand side), the block's 1/L_ii, row pointers and the in-block / other-
// color boundary of every row, and its entries (col, val; val holds PT in the
// substitutions, double in the SpMV), cap of them; a range with more entries
// is read from global memory.
constexpr int kSpmvRows = 16;   // rows of a warp's SpMV tile
struct BatchSmem {
  int o_dv, o_val, o_col, o_rp, o_sp, bytes;
  int chain;   // the walk: values of a chain's row scratch
};
__host__ __device__ inline BatchSmem batch_smem_plan(int smax, int kp, int cap, int elem) {
  const int rows = smax > kSpmvRows ? smax : kSpmvRows;
  BatchSmem m{};
  int o = r16b(smax * kp * elem);
  m.o_dv = o; o += r16b(smax * elem);
  m.o_val = o; o += r16b(cap * 8);
  m.o_col = o; o += r16b(cap * 4);
  m.o_rp = o; o += r16b((rows + 1) * 4);
  m.o_sp = o; o += r16b(rows * 4);
  m.bytes = o;
  return m;
}

// The block (or SpMV tile) a warp works on: rows [r0, r0 + nr), entries from
// e0; in shared memory when staged (index entry - e0).
template <typename VT>
struct BatchRows {
  int r0, nr, e0;
  bool staged;
  const int32_t *gcol;
  const VT *gval;
  const int32_t *scol;
  const VT *sval;
  const int32_t *rp;   // rp[k]: first entry of row r0 + k, from e0
  __device__ __forceinline__ int col(int e) const { return staged ? scol[e] : __ldg(gcol + e0 + e); }
  __device__ __forceinline__ VT val(int e) const { return staged ? sval[e] : __ldg(gval + e0 + e); }
};

template <typename VT>
__device__ __forceinline__ BatchRows<VT> stage_rows(const int32_t *rp, const int32_t *col, const VT *val, int r0,
                                                    int r1, unsigned char *sm, const BatchSmem &m, int cap, int lane) {
  BatchRows<VT> b;
  b.r0 = r0;
  b.nr = r1 - r0;
  b.e0 = __ldg(rp + r0);
  const int ne = __ldg(rp + r1) - b.e0;
  b.staged = ne <= cap;
  b.gcol = col;
  b.gval = val;
  int32_t *sc = reinterpret_cast<int32_t *>(sm + m.o_col), *srp = reinterpret_cast<int32_t *>(sm + m.o_rp);
  VT *sv = reinterpret_cast<VT *>(sm + m.o_val);
  for (int k = lane; k <= b.nr; k += kWarp) srp[k] = __ldg(rp + r0 + k) - b.e0;
  if (b.staged) {
#pragma unroll 4
    for (int e = lane; e < ne; e += kWarp) {
      sc[e] = __ldg(col + b.e0 + e);
      sv[e] = __ldg(val + b.e0 + e);
    }
  }
  b.scol = sc;
  b.sval = sv;
  b.rp = srp;
  return b;
}

// block blk of a substitution: its rows staged with 1/L_ii and, per row, the
// first entry past the other colors (L) or past the block (U)
template <typename PT, bool UPPER>
__device__ __forceinline__ BatchRows<PT> stage_block(const BatchSys &S, int blk, unsigned char *sm,
                                                     const BatchSmem &m, int cap, int lane) {
  __syncwarp();   // the previous block's readers are done
  const int r0 = __ldg(S.bptr + blk), r1 = __ldg(S.bptr + blk + 1);
  const BatchRows<PT> b = UPPER ? stage_rows<PT>(S.urp, S.ucol, b_uv<PT>(S), r0, r1, sm, m, cap, lane)
                                : stage_rows<PT>(S.lrp, S.lcol, b_lv<PT>(S), r0, r1, sm, m, cap, lane);
  PT *sdv = reinterpret_cast<PT *>(sm + m.o_dv);
  int32_t *ssp = reinterpret_cast<int32_t *>(sm + m.o_sp);
  for (int k = lane; k < b.nr; k += kWarp) sdv[k] = __ldg(b_dv<PT>(S) + r0 + k);
  __syncwarp();
  for (int k = lane; k < b.nr; k += kWarp) {
    int e = b.rp[k];
    const int e1 = b.rp[k + 1], bound = UPPER ? r1 : r0;
    while (e < e1 && b.col(e) < bound) ++e;
    ssp[k] = e;
  }
  __syncwarp();
  return b;
}

constexpr int kBatchRowsU = 4;   // rows a chain has in flight

// The rows' sources (r forward, y backward) minus their entries to other colors
// into w.  A chain takes every NC-th row, kBatchRowsU of them in flight.
template <typename PT, bool UPPER>
__device__ __forceinline__ void block_other(const BatchSys &S, const BatchRows<PT> &b, PT *w, const int32_t *ssp, int kp,
                                            int j, int ch, int NC) {
  const PT *y = reinterpret_cast<const PT *>(S.y);
  const PT *g = UPPER ? reinterpret_cast<const PT *>(S.z) : y;
  for (int k0 = ch; k0 < b.nr; k0 += NC * kBatchRowsU) {
    int e[kBatchRowsU], len[kBatchRowsU], most = 0;
    PT acc[kBatchRowsU], x[kBatchRowsU][3];
    double ri[kBatchRowsU];
#pragma unroll
    for (int u = 0; u < kBatchRowsU; ++u) {
      const int k = k0 + u * NC;
      const size_t at = size_t(b.r0 + k) * kp + j;
      const bool ok = k < b.nr;
      if (UPPER) acc[u] = ok ? __ldcg(y + at) : PT(0);
      else ri[u] = ok ? __ldcg(S.r + at) : 0.0;
      e[u] = ok ? (UPPER ? ssp[k] : b.rp[k]) : 0;
      len[u] = ok ? (UPPER ? b.rp[k + 1] : ssp[k]) - e[u] : 0;
      most = max(most, len[u]);
    }
#pragma unroll
    for (int u = 0; u < kBatchRowsU; ++u)
#pragma unroll
      for (int i = 0; i < 3; ++i)
        x[u][i] = i < len[u] ? __ldcg(g + size_t(b.col(e[u] + i)) * kp + j) : PT(0);
#pragma unroll
    for (int u = 0; u < kBatchRowsU; ++u) {
      if (!UPPER) acc[u] = PT(ri[u]);
#pragma unroll
      for (int i = 0; i < 3; ++i)
        if (i < len[u]) acc[u] -= b.val(e[u] + i) * x[u][i];
    }
    for (int t = 3; t < most; t += 3) {
#pragma unroll
      for (int u = 0; u < kBatchRowsU; ++u)
#pragma unroll
        for (int i = 0; i < 3; ++i)
          x[u][i] = t + i < len[u] ? __ldcg(g + size_t(b.col(e[u] + t + i)) * kp + j) : PT(0);
#pragma unroll
      for (int u = 0; u < kBatchRowsU; ++u)
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (t + i < len[u]) acc[u] -= b.val(e[u] + t + i) * x[u][i];
    }
#pragma unroll
    for (int u = 0; u < kBatchRowsU; ++u)
      if (k0 + u * NC < b.nr) w[(k0 + u * NC) * kp + j] = acc[u];
  }
}

// The in-block recurrence, rows in order (forward) or in reverse (backward),
// by one chain on shared memory; a lane reads only its own right-hand side.
template <typename PT, bool UPPER>
__device__ __forceinline__ void block_chain(const BatchRows<PT> &b, PT *w, const PT *sdv, const int32_t *ssp, int kp,
                                            int j) {
  for (int q = 0; q < b.nr; ++q) {
    const int k = UPPER ? b.nr - 1 - q : q;
    PT acc = w[k * kp + j];
    const int e1 = UPPER ? ssp[k] : b.rp[k + 1];
    for (int e = UPPER ? b.rp[k] : ssp[k]; e < e1; ++e) acc -= b.val(e) * w[(b.col(e) - b.r0) * kp + j];
    w[k * kp + j] = acc * sdv[k];
  }
}

// r of kBatchRowsU rows of a chain, from row k0 (0 past the block)
template <typename PT>
__device__ __forceinline__ void block_r(const BatchSys &S, const BatchRows<PT> &b, int kp, int j, int k0, int NC,
                                        double (&r)[kBatchRowsU]) {
#pragma unroll
  for (int u = 0; u < kBatchRowsU; ++u) {
    const int k = k0 + u * NC;
    r[u] = k < b.nr ? __ldcg(S.r + size_t(b.r0 + k) * kp + j) : 0.0;
  }
}

// the block's y from w
template <typename PT>
__device__ __forceinline__ void block_store_y(const BatchSys &S, const BatchRows<PT> &b, const PT *w, int kp, int j,
                                              int ch, int NC) {
  PT *y = reinterpret_cast<PT *>(S.y);
  for (int k = ch; k < b.nr; k += NC) y[size_t(b.r0 + k) * kp + j] = w[k * kp + j];
}

// the block's z from w and its share of <r, z>; r: that of the chain's first
// rows, the following ones loaded a step ahead
template <typename PT>
__device__ __forceinline__ void block_store_z(const BatchSys &S, const BatchRows<PT> &b, const PT *w, int kp, int j,
                                              int ch, int NC, double (&r)[kBatchRowsU], double &rz) {
  PT *z = reinterpret_cast<PT *>(S.z);
  for (int k0 = ch; k0 < b.nr; k0 += NC * kBatchRowsU) {
    double next[kBatchRowsU];
    block_r<PT>(S, b, kp, j, k0 + NC * kBatchRowsU, NC, next);
#pragma unroll
    for (int u = 0; u < kBatchRowsU; ++u) {
      const int k = k0 + u * NC;
      if (k < b.nr) {
        const PT v = w[k * kp + j];
        z[size_t(b.r0 + k) * kp + j] = v;
        rz += r[u] * widen(v);
      }
      r[u] = next[u];
    }
  }
}

// One substitution pass of a system; rz receives the lane's share of <r, z>, r
// in 64 bits times the z that is stored (with an FP32 preconditioner <y, y>,
// y = L^-1 r, differs from it by 1e-8, and an overflow of z would not show).
// A warp owns a block at a time and works in three parts: every row minus its
// entries to other colors (block_other: all chains of the warp, several rows
// each in flight), the in-block recurrence (block_chain: shared memory only;
// the rows' r is loaded meanwhile), the results (block_store_y / _z).  The
// block's static data is staged ahead; the first block of the next color before
// the barrier that ends the current one.
//
// Bound by latency: a chain that walks its block row by row pays two to three
// dependent L2 loads for each of 32 rows, 60-120 us for a color phase; split
// so, a phase costs a few such trips (8 systems of sides 16..64, 16 right-hand
// sides, FP32, blocks of 32 rows: 143 ms with the walk, 82 ms so; 4 systems of
// sides 16..48, 4 right-hand sides, FP64, ten iterations: 20.1 and 4.8 ms).  What remains is still latency: a
// color of one system has fewer blocks than its CTAs have warps.
template <typename PT>
__device__ __forceinline__ bool batch_precond(const BatchSys &S, unsigned char *sm, const BatchSmem &m, int cap, int kp,
                                              int gw, int total, double &rz, unsigned nct, unsigned &gen, int *flag) {
  const int lane = threadIdx.x & 31, j = lane % kp, ch = lane / kp, NC = kWarp / kp;
  PT *w = reinterpret_cast<PT *>(sm);
  const PT *sdv = reinterpret_cast<const PT *>(sm + m.o_dv);
  const int32_t *ssp = reinterpret_cast<const int32_t *>(sm + m.o_sp);
  const int nc = S.nc;
  BatchRows<PT> b;
  int blk = __ldg(S.cblk) + gw;
  bool have = blk < __ldg(S.cblk + 1);
  if (have) b = stage_block<PT, false>(S, blk, sm, m, cap, lane);
  for (int c = 0; c < nc; ++c) {
    const bool last = c == nc - 1;
    const int b1 = __ldg(S.cblk + c + 1);
    while (have) {
      block_other<PT, false>(S, b, w, ssp, kp, j, ch, NC);
      __syncwarp();
      if (ch == 0) block_chain<PT, false>(b, w, sdv, ssp, kp, j);
      __syncwarp();
      if (!last) {
        block_store_y<PT>(S, b, w, kp, j, ch, NC);
      } else {
        // the last color: backward sweep of the same block at once (no
        // later colors), y in w
        b = stage_block<PT, true>(S, blk, sm, m, cap, lane);
        double r[kBatchRowsU];
        block_r<PT>(S, b, kp, j, ch, NC, r);
        if (ch == 0) block_chain<PT, true>(b, w, sdv, ssp, kp, j);
        __syncwarp();
        block_store_z<PT>(S, b, w, kp, j, ch, NC, r, rz);
      }
      blk += total;
      have = blk < b1;
      if (have) b = stage_block<PT, false>(S, blk, sm, m, cap, lane);
    }
    const int cn = last ? nc - 2 : c + 1;
    if (cn >= 0) {
      blk = __ldg(S.cblk + cn) + gw;
      have = blk < __ldg(S.cblk + cn + 1);
      if (have) b = last ? stage_block<PT, true>(S, blk, sm, m, cap, lane) : stage_block<PT, false>(S, blk, sm, m, cap, lane);
    }
    // every color's results (for the last color: its z) complete before the
    // next color reads them
    if (!sys_sync(S.bar, nct, gen, flag, S.wait_ns)) return false;
  }
  for (int c = nc - 2; c >= 0; --c) {
    const int b1 = __ldg(S.cblk + c + 1);
    while (have) {
      block_other<PT, true>(S, b, w, ssp, kp, j, ch, NC);
      double r[kBatchRowsU];
      block_r<PT>(S, b, kp, j, ch, NC, r);
      __syncwarp();
      if (ch == 0) block_chain<PT, true>(b, w, sdv, ssp, kp, j);
      __syncwarp();
      block_store_z<PT>(S, b, w, kp, j, ch, NC, r, rz);
      blk += total;
      have = blk < b1;
      if (have) b = stage_block<PT, true>(S, blk, sm, m, cap, lane);
    }
    if (c > 0) {
      blk = __ldg(S.cblk + c - 1) + gw;
      have = blk < __ldg(S.cblk + c);
      if (have) b = stage_block<PT, true>(S, blk, sm, m, cap, lane);
      if (!sys_sync(S.bar, nct, gen, flag, S.wait_ns)) return false;
    }
  }
  return true;
}

// A times a [n][kp] vector, a warp per tile of kSpmvRows rows whose entries are
// staged coalesced, a chain per row, R rows of a chain in flight (8 entries each
// at R = 1 or 2, 4 at R = 4).  INIT: r = r - A x (r holds b), returns the share of <r, r>;
// else q = A p, the share of <p, q>.
template <int R, bool INIT>
__device__ __forceinline__ double batch_spmv(const BatchSys &S, unsigned char *sm, const BatchSmem &m, int cap, int kp,
                                             int gw, int total, bool act) {
  constexpr int E = R < 4 ? 8 : 4;
  const int lane = threadIdx.x & 31, j = lane % kp, ch = lane / kp, NC = kWarp / kp;
  const double *v = INIT ? S.x : S.p;
  const int ntile = (S.n + kSpmvRows - 1) / kSpmvRows;
  double acc = 0.0;
  for (int t = gw; t < ntile; t += total) {
    __syncwarp();
    const int r0 = t * kSpmvRows, r1 = min(S.n, r0 + kSpmvRows);
    const BatchRows<double> b = stage_rows<double>(S.arp, S.acol, S.aval, r0, r1, sm, m, cap, lane);
    __syncwarp();
    if (!act) continue;
    for (int k0 = ch; k0 < b.nr; k0 += NC * R) {
      int e[R], len[R], most = 0;
      double s[R], own[R], rb[R];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const int k = k0 + u * NC;
        const bool ok = k < b.nr;
        e[u] = ok ? b.rp[k] : 0;
        len[u] = ok ? b.rp[k + 1] - e[u] : 0;
        most = max(most, len[u]);
        s[u] = 0.0;
        const size_t at = size_t(b.r0 + k) * kp + j;
        own[u] = ok && !INIT ? __ldcg(v + at) : 0.0;
        rb[u] = ok && INIT ? __ldcg(S.r + at) : 0.0;
      }
      for (int t0 = 0; t0 < most; t0 += E) {
        double x[R][E];
#pragma unroll
        for (int u = 0; u < R; ++u)
#pragma unroll
          for (int i = 0; i < E; ++i)
            x[u][i] = t0 + i < len[u] ? __ldcg(v + size_t(b.col(e[u] + t0 + i)) * kp + j) : 0.0;
#pragma unroll
        for (int u = 0; u < R; ++u)
#pragma unroll
          for (int i = 0; i < E; ++i)
            if (t0 + i < len[u]) s[u] += b.val(e[u] + t0 + i) * x[u][i];
      }
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const int k = k0 + u * NC;
        if (k >= b.nr) continue;
        const size_t at = size_t(b.r0 + k) * kp + j;
        if (INIT) {
          const double ri = rb[u] - s[u];
          S.r[at] = ri;
          acc += ri * ri;
        } else {
          S.q[at] = s[u];
          acc += own[u] * s[u];
        }
      }
    }
  }
  return acc;
}

// The same by walking (UPDATE: with the x / r update in front of the forward
// sweep): a chain owns a block at a time and resolves it row by row; w is the
// chain's scratch (block rows x kp).  A warp serves 32 / kp blocks at once, so
// that it has more blocks in flight than batch_precond and, one latency after
// another, needs longer for each (batch_walks: which is the better one when).
template <typename PT, bool UPDATE>
__device__ __forceinline__ bool batch_precond_walk(const BatchSys &S, PT *w, int kp, int j, int gc, int total,
                                              double alpha, bool act, double &rr, double &rz, unsigned nct,
                                              unsigned &gen, int *flag) {
  const PT *lv = b_lv<PT>(S), *uv = b_uv<PT>(S), *dv = b_dv<PT>(S);
  PT *y = reinterpret_cast<PT *>(S.y);
  PT *z = reinterpret_cast<PT *>(S.z);
  const int nc = S.nc;
  for (int c = 0; c < nc; ++c) {
    const bool last = c == nc - 1;
    const int b1 = __ldg(S.cblk + c + 1);
    for (int blk = __ldg(S.cblk + c) + gc; blk < b1; blk += total) {
      const int r0 = __ldg(S.bptr + blk), r1 = __ldg(S.bptr + blk + 1);
      for (int i = r0; i < r1; ++i) {
        double ri = __ldcg(S.r + size_t(i) * kp + j);
        if (UPDATE && act) {
          ri -= alpha * __ldcg(S.q + size_t(i) * kp + j);
          S.r[size_t(i) * kp + j] = ri;
          S.x[size_t(i) * kp + j] = __ldcg(S.x + size_t(i) * kp + j) + alpha * __ldcg(S.p + size_t(i) * kp + j);
          rr += ri * ri;
        }
        PT acc = PT(ri);
        const int e1 = __ldg(S.lrp + i + 1);
        for (int e = __ldg(S.lrp + i); e < e1; ++e) {
          const int col = __ldg(S.lcol + e);
          const PT v = __ldg(lv + e);
          const PT yc = col >= r0 ? w[(col - r0) * kp + j] : __ldcg(y + size_t(col) * kp + j);
          acc -= v * yc;
        }
        const PT yi = acc * __ldg(dv + i);
        w[(i - r0) * kp + j] = yi;
        if (!last) y[size_t(i) * kp + j] = yi;
      }
      if (last) {
        // the last color: backward sweep of the same block at once (no
        // later colors), y in the scratch
        for (int i = r1 - 1; i >= r0; --i) {
          PT acc = w[(i - r0) * kp + j];
          const int e1 = __ldg(S.urp + i + 1);
          for (int e = __ldg(S.urp + i); e < e1; ++e) acc -= __ldg(uv + e) * w[(__ldg(S.ucol + e) - r0) * kp + j];
          const PT zi = acc * __ldg(dv + i);
          w[(i - r0) * kp + j] = zi;
          z[size_t(i) * kp + j] = zi;
          rz += __ldcg(S.r + size_t(i) * kp + j) * widen(zi);
        }
      }
    }
    // every color's results (for the last color: its z) complete before the
    // next color reads them
    if (!sys_sync(S.bar, nct, gen, flag, S.wait_ns)) return false;
  }
  for (int c = nc - 2; c >= 0; --c) {
    const int b1 = __ldg(S.cblk + c + 1);
    for (int blk = __ldg(S.cblk + c) + gc; blk < b1; blk += total) {
      const int r0 = __ldg(S.bptr + blk), r1 = __ldg(S.bptr + blk + 1);
      for (int i = r1 - 1; i >= r0; --i) {
        PT acc = __ldcg(y + size_t(i) * kp + j);
        const int e1 = __ldg(S.urp + i + 1);
        for (int e = __ldg(S.urp + i); e < e1; ++e) {
          const int col = __ldg(S.ucol + e);
          const PT zc = col < r1 ? w[(col - r0) * kp + j] : __ldcg(z + size_t(col) * kp + j);
          acc -= __ldg(uv + e) * zc;
        }
        const PT zi = acc * __ldg(dv + i);
        w[(i - r0) * kp + j] = zi;
        z[size_t(i) * kp + j] = zi;
        rz += __ldcg(S.r + size_t(i) * kp + j) * widen(zi);
      }
    }
    if (c > 0 && !sys_sync(S.bar, nct, gen, flag, S.wait_ns)) return false;
  }
  return true;
}

// A times a [n][kp] vector by walking: a chain per row (INIT or R = 1) or R
// consecutive rows of a chain together.  INIT and results as in batch_spmv.
template <int R, bool INIT>
__device__ __forceinline__ double batch_spmv_walk(const BatchSys &S, int kp, int j, int gc, int total, bool act) {
  const double *v = INIT ? S.x : S.p;
  const int n = S.n;
  double acc = 0.0;
  if (!act) return acc;
  if constexpr (INIT || R == 1) {
    for (int i = gc; i < n; i += total) {
      const size_t at = size_t(i) * kp + j;
      double s = 0.0;
      const int e1 = __ldg(S.arp + i + 1);
      for (int e = __ldg(S.arp + i); e < e1; ++e)
        s += __ldg(S.aval + e) * __ldcg(v + size_t(__ldg(S.acol + e)) * kp + j);
      if (INIT) {
        const double ri = __ldcg(S.r + at) - s;
        S.r[at] = ri;
        acc += ri * ri;
      } else {
        S.q[at] = s;
        acc += __ldcg(v + at) * s;
      }
    }
  } else {
    for (int i0 = gc * R; i0 < n; i0 += total * R) {
      int e0[R], e1[R];
      double s[R];
      int len = 0;
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const bool in = i0 + u < n;
        e0[u] = in ? __ldg(S.arp + i0 + u) : 0;
        e1[u] = in ? __ldg(S.arp + i0 + u + 1) : 0;
        s[u] = 0.0;
        len = max(len, e1[u] - e0[u]);
      }
      // the rows' t-th entries together (each row's sum in entry order)
      for (int t = 0; t < len; ++t) {
#pragma unroll
        for (int u = 0; u < R; ++u)
          if (e0[u] + t < e1[u])
            s[u] += __ldg(S.aval + e0[u] + t) * __ldcg(v + size_t(__ldg(S.acol + e0[u] + t)) * kp + j);
      }
#pragma unroll
      for (int u = 0; u < R; ++u)
        if (i0 + u < n) {
          S.q[size_t(i0 + u) * kp + j] = s[u];
          acc += __ldcg(v + size_t(i0 + u) * kp + j) * s[u];
        }
    }
  }
  return acc;
}

// R: rows of a chain in flight in the SpMV (1, 2 or 4); WALK: the walking
// forms, with a chain's row scratch as its only shared memory
template <typename PT, int R, bool WALK>
__global__ void __launch_bounds__(kMaxWarpsPerCta * kWarp, 1)
batch_kernel(const BatchSys *sys, const int32_t *cta_sys, int k, int kp, BatchSmem plan, int cap, int maxit,
             double tol) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ BatchSys S;
  __shared__ int flag;
  __shared__ double sv[4][32];    // per right-hand side: bb / rr / pq / rz sums
  __shared__ double st_rz[32], st_beta[32], st_bn[32];
  __shared__ int st_act[32];
  __shared__ int any_act;
  if (threadIdx.x == 0) S = sys[cta_sys[blockIdx.x]];
  __syncthreads();
  const int nchain = blockDim.x / kp;
  const int ch = threadIdx.x / kp, j = threadIdx.x % kp;
  const int lc = blockIdx.x - S.cta0;
  const unsigned nct = unsigned(S.cta1 - S.cta0);
  const int gc = lc * nchain + ch, total = int(nct) * nchain;
  const int W = blockDim.x / kWarp, warp = threadIdx.x / kWarp;
  const int gw = lc * W + warp, totalw = int(nct) * W;
  unsigned char *wsm = smem + size_t(warp) * plan.bytes;
  PT *wch = reinterpret_cast<PT *>(smem) + size_t(ch) * plan.chain;
  double *red = reinterpret_cast<double *>(smem + size_t(W) * plan.bytes);
  double *mypart = S.part + size_t(lc) * 4 * kp;
  const int n = S.n;
  unsigned gen = 0;
  bool ok = true;
  const bool real = j < k;

  // solve start: x, b (in r) in the internal numbering; p = 0; <b,b>
  double acc = 0.0;
  for (int i = gc; i < n; i += total) {
    const int o = __ldg(S.perm + i);
    const double bi = real ? __ldcg(S.bin + size_t(j) * n + o) : 0.0;
    S.x[size_t(i) * kp + j] = real ? __ldcg(S.xio + size_t(j) * n + o) : 0.0;
    S.r[size_t(i) * kp + j] = bi;
    S.p[size_t(i) * kp + j] = 0.0;
    acc += bi * bi;
  }
  cta_rhs_sum(acc, red, kp, mypart + 0 * kp);
  ok = sys_sync(S.bar, nct, gen, &flag, S.wait_ns);
  // r0 = b - A x0, <r0, r0> (a row's b is read and r written by its own lane)
  if (ok) {
    if constexpr (WALK) acc = batch_spmv_walk<R, true>(S, kp, j, gc, total, true);
    else acc = batch_spmv<R, true>(S, wsm, plan, cap, kp, gw, totalw, true);
    cta_rhs_sum(acc, red, kp, mypart + 1 * kp);
    ok = sys_sync(S.bar, nct, gen, &flag, S.wait_ns);
  }
  // z0 = M^-1 r0, <r0, z0>
  double rr = 0.0, rz = 0.0;
  if (ok) {
    if constexpr (WALK) ok = batch_precond_walk<PT, false>(S, wch, kp, j, gc, total, 0.0, false, rr, rz, nct, gen, &flag);
    else ok = batch_precond<PT>(S, wsm, plan, cap, kp, gw, totalw, rz, nct, gen, &flag);
  }
  if (ok) {
    cta_rhs_sum(rz, red, kp, mypart + 3 * kp);
    ok = sys_sync(S.bar, nct, gen, &flag, S.wait_ns);
  }
  int it = 0;
  if (ok) {
    sys_rhs_sum<WALK>(S.part, int(nct), kp, 0, sv[0], red);
    sys_rhs_sum<WALK>(S.part, int(nct), kp, 1, sv[1], red);
    sys_rhs_sum<WALK>(S.part, int(nct), kp, 3, sv[3], red);
    if (threadIdx.x < kp) {
      const int t = threadIdx.x;
      const double bn = sqrt(sv[0][t]);
      st_bn[t] = bn;
      st_rz[t] = sv[3][t];
      st_beta[t] = 0.0;
      int a = 0, status = ICCG_OK;
      double rn = 0.0;
      if (t < k && bn > 0.0) {
        rn = sqrt(sv[1][t]) / bn;
        if (!isfinite(rn) || !isfinite(sv[3][t])) status = ICCG_ERR_NONFINITE;
        else if (rn <= tol) status = ICCG_OK;
        else if (maxit <= 0) status = ICCG_NOT_CONVERGED;
        else a = 1;
      }
      st_act[t] = a;
      if (lc == 0) {
        S.hist[t] = rn;
        S.iters[t] = 0;
        S.status[t] = a ? ICCG_NOT_CONVERGED : status;
      }
    }
    if (threadIdx.x == 0) {
      int a = 0;
      for (int t = 0; t < kp; ++t) a |= st_act[t];
      any_act = a;
    }
    __syncthreads();
  }
  while (ok && any_act) {
    const bool act = st_act[j] != 0;
    const double beta = st_beta[j];
    // p = z + beta p (U rows of a chain in flight)
    const PT *z = reinterpret_cast<const PT *>(S.z);
    constexpr int U = WALK ? R : kBatchRowsU;
    if (act) {
      for (int i0 = gc; i0 < n; i0 += total * U) {
        double zz[U], pp[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u * total;
          zz[u] = i < n ? widen(__ldcg(z + size_t(i) * kp + j)) : 0.0;
          pp[u] = i < n ? __ldcg(S.p + size_t(i) * kp + j) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i0 + u * total < n) S.p[size_t(i0 + u * total) * kp + j] = zz[u] + beta * pp[u];
      }
    }
    if (!(ok = sys_sync(S.bar, nct, gen, &flag, S.wait_ns))) break;
    // q = A p, <p, q>
    if constexpr (WALK) acc = batch_spmv_walk<R, false>(S, kp, j, gc, total, act);
    else acc = batch_spmv<R, false>(S, wsm, plan, cap, kp, gw, totalw, act);
    cta_rhs_sum(acc, red, kp, mypart + 2 * kp);
    if (!(ok = sys_sync(S.bar, nct, gen, &flag, S.wait_ns))) break;
    sys_rhs_sum<WALK>(S.part, int(nct), kp, 2, sv[2], red);
    const double alpha = act ? st_rz[j] / sv[2][j] : 0.0;
    rr = 0.0;
    rz = 0.0;
    if constexpr (WALK) {
      // x / r update, z = M^-1 r, <r,r>, <r,z>
      if (!(ok = batch_precond_walk<PT, true>(S, wch, kp, j, gc, total, alpha, act, rr, rz, nct, gen, &flag))) break;
    } else {
      // x / r update and <r,r> over all rows at once (in front of each color's
      // forward sweep, where only that color's blocks are at work, it took twice
      // as long), then z = M^-1 r and <r,z>
      if (act) {
        for (int i0 = gc; i0 < n; i0 += total * kBatchRowsU) {
          double ri[kBatchRowsU], qi[kBatchRowsU], xi[kBatchRowsU], pi[kBatchRowsU];
#pragma unroll
          for (int u = 0; u < kBatchRowsU; ++u) {
            const int i = i0 + u * total;
            const size_t at = size_t(i) * kp + j;
            ri[u] = i < n ? __ldcg(S.r + at) : 0.0;
            qi[u] = i < n ? __ldcg(S.q + at) : 0.0;
            xi[u] = i < n ? __ldcg(S.x + at) : 0.0;
            pi[u] = i < n ? __ldcg(S.p + at) : 0.0;
          }
#pragma unroll
          for (int u = 0; u < kBatchRowsU; ++u) {
            const int i = i0 + u * total;
            if (i < n) {
              const size_t at = size_t(i) * kp + j;
              ri[u] -= alpha * qi[u];
              S.r[at] = ri[u];
              S.x[at] = xi[u] + alpha * pi[u];
              rr += ri[u] * ri[u];
            }
          }
        }
      }
      if (!(ok = sys_sync(S.bar, nct, gen, &flag, S.wait_ns))) break;
      if (!(ok = batch_precond<PT>(S, wsm, plan, cap, kp, gw, totalw, rz, nct, gen, &flag))) break;
    }
    cta_rhs_sum(rr, red, kp, mypart + 1 * kp);
    cta_rhs_sum(rz, red, kp, mypart + 3 * kp);
    if (!(ok = sys_sync(S.bar, nct, gen, &flag, S.wait_ns))) break;
    sys_rhs_sum<WALK>(S.part, int(nct), kp, 1, sv[1], red);
    sys_rhs_sum<WALK>(S.part, int(nct), kp, 3, sv[3], red);
    ++it;
    if (threadIdx.x < kp) {
      const int t = threadIdx.x;
      if (st_act[t]) {
        const double rn = sqrt(sv[1][t]) / st_bn[t];
        int a = 1, status = ICCG_NOT_CONVERGED;
        if (!isfinite(rn) || !isfinite(sv[3][t])) { a = 0; status = ICCG_ERR_NONFINITE; }
        else if (rn <= tol) { a = 0; status = ICCG_OK; }
        else if (it >= maxit) { a = 0; status = ICCG_NOT_CONVERGED; }
        else {
          st_beta[t] = sv[3][t] / st_rz[t];
          st_rz[t] = sv[3][t];
        }
        if (lc == 0) {
          S.hist[size_t(it) * kp + t] = rn;
          S.iters[t] = it;
          S.status[t] = status;
        }
        st_act[t] = a;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int a = 0;
      for (int t = 0; t < kp; ++t) a |= st_act[t];
      any_act = a;
    }
    __syncthreads();
  }
  if (ok) {
    for (int i = gc; i < n; i += total)
      if (real) S.xio[size_t(j) * n + __ldg(S.perm + i)] = st_bn[j] > 0.0 ? __ldcg(S.x + size_t(i) * kp + j) : 0.0;
  } else if (lc == 0 && threadIdx.x < kp) {
    S.status[threadIdx.x] = ICCG_ERR_TIMEOUT;
  }
}

int pow2_at_least(int k) {
  int p = 1;
  while (p < k) p <<= 1;
  return p;
}

// allow dynamic shared memory up to the opt-in limit minus the kernel's
// static shared memory
template <typename K>
cudaError_t allow_smem_b(K kernel) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              optin - int(fa.sharedSizeBytes) - 256);
}

using BatchKernel = void (*)(const BatchSys *, const int32_t *, int, int, BatchSmem, int, int, double);

template <typename PT>
BatchKernel batch_kernel_of(int R, bool walk) {
  if (walk) return R == 4 ? batch_kernel<PT, 4, true> : (R == 2 ? batch_kernel<PT, 2, true> : batch_kernel<PT, 1, true>);
  return R == 4 ? batch_kernel<PT, 4, false> : (R == 2 ? batch_kernel<PT, 2, false> : batch_kernel<PT, 1, false>);
}

BatchKernel batch_kernel_of(bool fp32, int R, bool walk) {
  return fp32 ? batch_kernel_of<float>(R, walk) : batch_kernel_of<double>(R, walk);
}

}  // namespace
}  // namespace iccg

using namespace iccg;

struct iccg_batch {
  int device = 0;
  cudaStream_t stream = nullptr;
  int nsys = 0, k = 0, kp = 0, smax = 1;
  int cap = 0;           // entries of a block or SpMV tile staged per warp
  bool walk_better = false;   // the walk is the better form for these systems
  bool walk = false;          // the launch shape's form
  bool fp32 = false;
  std::vector<iccg_ctx *> ctxs;
  std::vector<int32_t> n;
  std::vector<void *> allocs;
  // per system device buffers
  std::vector<double *> x, r, p, q, bin, xio, part, hist;
  std::vector<void *> y, z;
  std::vector<int32_t *> iters, status, cblk, bptr;
  GridBar *bars = nullptr;
  BatchSys *d_sys = nullptr;
  int32_t *d_cta_sys = nullptr;
  int hist_cap = 0;
  // launch shape
  int W = 8, cps = 1, grid = 0, smem = 0, max_part_ctas = 0;
  int R = 1;             // rows per chain and pass (SpMV, p update)
  bool by_work = true;         // CTAs per system by rows x estimated iterations, else by rows
  std::vector<double> work;    // rows x estimated iterations of each system
  std::vector<int32_t> cta0;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  int graph_maxit = -1;
  double graph_tol = -1.0;
  bool direct = false;   // the runtime refused to capture the cooperative launch: launch it directly
  unsigned long long wait_ns = kDefaultWaitNs;   // barrier wait limit of the batched kernel
  std::string err_msg;
};

namespace {

cudaError_t b_alloc(iccg_batch *b, void **p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes + 64);
  if (e != cudaSuccess) return e;
  b->allocs.push_back(*p);
  return cudaMemsetAsync(*p, 0, bytes + 64, b->stream);
}

// a warp's shared memory: the block buffers, or (walk) the rows of its chains' blocks
BatchSmem batch_plan(const iccg_batch *b, bool walk) {
  const int elem = b->fp32 ? 4 : 8;
  if (!walk) return batch_smem_plan(b->smax, b->kp, b->cap, elem);
  BatchSmem m{};
  m.bytes = kWarp * b->smax * elem;
  m.chain = b->smax * b->kp;
  return m;
}

int batch_smem(const iccg_batch *b, int W, bool walk) { return W * batch_plan(b, walk).bytes + W * kWarp * 8; }

int batch_occupancy(const iccg_batch *b, int W, bool walk) {
  int nb = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_kernel_of(b->fp32, b->R, walk),
                                                                      W * kWarp, size_t(batch_smem(b, W, walk)));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}

void destroy_batch_graph(iccg_batch *b) {
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->gexec = nullptr;
  b->graph = nullptr;
}

// Rows times an estimate of the iterations: CG takes O(sqrt(kappa)) of them,
// and for a discretised elliptic operator lambda_min / lambda_max is about
// n^(-2/3) (times a constant all systems share) plus the diagonal dominance
// delta = min_i (a_ii - sum_j |a_ij|) / a_ii that a shift adds (0.2 delta in the
// same unit: 7-point rows give 2.5 / side^2 + delta / 2).  Only the ratio
// between systems matters: a system's CTAs work on it alone, so the batch ends
// when the slowest system does.
double system_work(const HostLayout &H) {
  double delta = 1.0;
  for (int32_t i = 0; i < H.n; ++i) {
    double off = 0.0, d = 0.0;
    for (int32_t e = H.arp[i]; e < H.arp[i + 1]; ++e) {
      if (H.acol[e] == i) d = H.aval[e];
      else off += std::fabs(H.aval[e]);
    }
    delta = std::min(delta, d > 0.0 ? (d - off) / d : 0.0);
  }
  const double n = double(H.n);
  return n / std::sqrt(std::pow(n, -2.0 / 3.0) + 0.2 * std::max(delta, 0.0));
}

// CTA ranges per system (>= 1 each) for a grid of G CTAs, in proportion to the
// systems' rows or (by_work) to rows x estimated iterations; returns false when
// G < nsys.  8 systems of sides 16..64 with shifts in [1e-4, 1e-1] need 24 to 79
// iterations.
bool assign_ctas(iccg_batch *b, int G) {
  if (G < b->nsys) return false;
  double tot = 0.0;
  std::vector<double> wt(b->nsys);
  for (int s = 0; s < b->nsys; ++s) {
    wt[s] = b->by_work ? b->work[s] : double(b->n[s]);
    tot += wt[s];
  }
  std::vector<int32_t> c(b->nsys, 1);
  int used = b->nsys;
  // largest remainder over the CTAs beyond one per system
  std::vector<double> want(b->nsys);
  for (int s = 0; s < b->nsys; ++s) want[s] = double(G) * wt[s] / tot;
  for (int s = 0; s < b->nsys; ++s) {
    const int extra = std::max(0, int(want[s]) - 1);
    c[s] += extra;
    used += extra;
  }
  while (used > G) {
    int best = -1;
    for (int s = 0; s < b->nsys; ++s)
      if (c[s] > 1 && (best < 0 || double(c[s]) - want[s] > double(c[best]) - want[best])) best = s;
    if (best < 0) break;
    c[best]--;
    used--;
  }
  while (used < G) {
    int best = 0;
    for (int s = 1; s < b->nsys; ++s)
      if (want[s] - double(c[s]) > want[best] - double(c[best])) best = s;
    c[best]++;
    used++;
  }
  b->cta0.assign(b->nsys + 1, 0);
  for (int s = 0; s < b->nsys; ++s) b->cta0[s + 1] = b->cta0[s] + c[s];
  b->grid = b->cta0[b->nsys];
  return true;
}

iccg_status upload_plan(iccg_batch *b, int maxit) {
  // per-system descriptors for the current CTA assignment and history size
  std::vector<BatchSys> hs(b->nsys);
  std::vector<int32_t> cs(b->grid);
  for (int s = 0; s < b->nsys; ++s) {
    const iccg_ctx *c = b->ctxs[s];
    const Params &P = c->P;
    BatchSys &S = hs[s];
    std::memset(&S, 0, sizeof(S));
    S.n = b->n[s];
    S.nc = c->H.n_c;
    S.cta0 = b->cta0[s];
    S.cta1 = b->cta0[s + 1];
    S.arp = P.arp; S.acol = P.acol; S.aval = P.aval;
    S.lrp = P.lrp; S.lcol = P.lcol; S.urp = P.urp; S.ucol = P.ucol;
    S.lv64 = P.lval; S.uv64 = P.uval; S.dv64 = P.invd;
    S.lv32 = P.lval32; S.uv32 = P.uval32; S.dv32 = P.invd32;
    S.cblk = b->cblk[s];
    S.bptr = b->bptr[s];
    S.perm = P.perm;
    S.x = b->x[s]; S.r = b->r[s]; S.p = b->p[s]; S.q = b->q[s];
    S.y = b->y[s]; S.z = b->z[s];
    S.bin = b->bin[s];
    S.xio = b->xio[s];
    S.part = b->part[s];
    S.hist = b->hist[s];
    S.iters = b->iters[s];
    S.status = b->status[s];
    S.bar = b->bars + s;
    S.wait_ns = b->wait_ns;
    for (int g = S.cta0; g < S.cta1; ++g) cs[g] = s;
  }
  if (cudaMemcpyAsync(b->d_sys, hs.data(), sizeof(BatchSys) * hs.size(), cudaMemcpyHostToDevice, b->stream) !=
          cudaSuccess ||
      cudaMemcpyAsync(b->d_cta_sys, cs.data(), sizeof(int32_t) * cs.size(), cudaMemcpyHostToDevice, b->stream) !=
          cudaSuccess) {
    b->err_msg = std::string("batch plan upload: ") + cudaGetErrorString(cudaGetLastError());
    return ICCG_ERR_CUDA;
  }
  (void)maxit;
  return ICCG_OK;
}

cudaError_t batch_launch(iccg_batch *b, cudaStream_t s, int maxit, double tol) {
  cudaError_t e = cudaMemsetAsync(b->bars, 0, sizeof(GridBar) * size_t(b->nsys), s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(b->grid));
  cfg.blockDim = dim3(unsigned(b->W * kWarp));
  cfg.dynamicSmemBytes = size_t(b->smem);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const BatchSys *sys = b->d_sys;
  const int32_t *cts = b->d_cta_sys;
  return cudaLaunchKernelEx(&cfg, batch_kernel_of(b->fp32, b->R, b->walk), sys, cts, b->k, b->kp,
                            batch_plan(b, b->walk), b->cap, maxit, tol);
}

// Where the walk is the better form (400 combinations of 8 batches, blocks of 1
// to 64 rows, 1 to 32 right-hand sides and both precisions, ten iterations;
// taking the better one everywhere would gain 0.4% more on average).  A warp per
// block pays where a block fills its chains and the blocks of a color do not
// outnumber the warps; the walk is better
//  - for blocks of one and two rows (4 systems of sides 16..48, one-row blocks:
//    0.65 against 8.1 ms with one right-hand side, 4.7 against 10.7 with 16; at
//    worst 1.2 times the warp form's time: 20,000-row graph, two rows, one
//    right-hand side);
//  - for blocks of three to five rows with 16 or 32 right-hand sides (two chains
//    or one to a warp: 27-point, 4-row blocks, 32: 0.74 of the time) or with
//    more blocks a color than `warps` (sides 16..48, 4-row blocks, 4 right-hand
//    sides: 0.70; with half as many blocks, one side of 40: 1.15);
//  - for a single chain to a warp on wide rows (32 right-hand sides; 17 entries a
//    row 0.72 to 1.15, 27-point 0.67 to 1.0, spring network 0.43 to 0.8; at 9
//    entries and below the warp form is better from 8-row blocks on);
//  - in FP32 for two chains on rows above 32 entries whose blocks are not staged
//    (spring network, 16 right-hand sides, blocks of 32 rows: 0.87; FP64 1.07).
bool batch_walks(const iccg_batch *b, int warps) {
  double rows = 0.0, blocks = 0.0, entries = 0.0, per_color = 0.0;
  for (const iccg_ctx *c : b->ctxs) {
    rows += c->H.n;
    blocks += c->H.n_b;
    entries += double(c->H.acol.size());
    per_color += double(c->H.n_b) / c->H.n_c;
  }
  const double mean = rows / blocks, wide = entries / rows;
  if (mean < 3.0) return true;
  if (mean < 6.0 && (b->kp >= 16 || per_color > warps)) return true;
  if (b->kp >= 32 && wide > 12.0) return true;
  return b->fp32 && b->kp >= 16 && wide > 32.0 && mean * wide > 2.0 * kBatchCap;
}

// The form a shape runs: the better one, or the walk where the block buffers do
// not fit beside one another (64-row blocks, 32 right-hand sides, FP64: above 9
// warps a CTA).
bool shape_walks(const iccg_batch *b, int W) { return b->walk_better || batch_occupancy(b, W, false) <= 0; }

iccg_status set_shape(iccg_batch *b, int W, int cps, int sms) {
  const bool walk = shape_walks(b, W);
  const int occ = batch_occupancy(b, W, walk);
  if (occ <= 0) {
    b->err_msg = "batched kernel does not fit an SM with this shape";
    return ICCG_ERR_ARG;
  }
  const int c = cps <= 0 ? occ : std::min(cps, occ);
  if (!assign_ctas(b, sms * c)) {
    b->err_msg = "more systems than resident CTAs";
    return ICCG_ERR_ARG;
  }
  if (b->grid > b->max_part_ctas) {
    b->err_msg = "CTA count above the partial-sum capacity";
    return ICCG_ERR_ARG;
  }
  b->W = W;
  b->cps = c;
  b->walk = walk;
  b->smem = batch_smem(b, W, walk);
  destroy_batch_graph(b);
  return ICCG_OK;
}

iccg_status ensure_hist(iccg_batch *b, int maxit) {
  if (maxit + 1 <= b->hist_cap) return ICCG_OK;
  const int cap = std::max(maxit + 1, 1024);
  for (int s = 0; s < b->nsys; ++s) {
    void *h = nullptr;
    if (b_alloc(b, &h, sizeof(double) * size_t(cap) * size_t(b->kp)) != cudaSuccess) {
      b->err_msg = "history allocation failed";
      return ICCG_ERR_CUDA;
    }
    b->hist[s] = static_cast<double *>(h);
  }
  b->hist_cap = cap;
  destroy_batch_graph(b);
  return ICCG_OK;
}

iccg_status run(iccg_batch *b, int maxit, double tol) {
  if (b->direct) {
    iccg_status st = upload_plan(b, maxit);
    if (st != ICCG_OK) return st;
    const cudaError_t e = batch_launch(b, b->stream, maxit, tol);
    if (e != cudaSuccess) {
      b->err_msg = std::string("batched launch: ") + cudaGetErrorString(e);
      return ICCG_ERR_CUDA;
    }
    return ICCG_OK;
  }
  if (!b->gexec || b->graph_maxit != maxit || b->graph_tol != tol) {
    destroy_batch_graph(b);
    iccg_status st = upload_plan(b, maxit);
    if (st != ICCG_OK) return st;
    cudaStream_t cs = nullptr;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
      b->err_msg = "capture stream";
      return ICCG_ERR_CUDA;
    }
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    cudaError_t el = e == cudaSuccess ? batch_launch(b, cs, maxit, tol) : e;
    cudaGraph_t g = nullptr;
    cudaError_t ee = e == cudaSuccess ? cudaStreamEndCapture(cs, &g) : e;
    cudaStreamDestroy(cs);
    if (el != cudaSuccess || ee != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      cudaGetLastError();
      b->direct = true;
      return run(b, maxit, tol);
    }
    b->graph = g;
    if (cudaGraphInstantiate(&b->gexec, g, 0) != cudaSuccess) {
      b->err_msg = "batched graph instantiate";
      destroy_batch_graph(b);
      return ICCG_ERR_CUDA;
    }
    b->graph_maxit = maxit;
    b->graph_tol = tol;
  }
  if (cudaGraphLaunch(b->gexec, b->stream) != cudaSuccess) {
    b->err_msg = std::string("batched graph launch: ") + cudaGetErrorString(cudaGetLastError());
    return ICCG_ERR_CUDA;
  }
  return ICCG_OK;
}

}  // namespace

extern "C" {

iccg_status iccg_batch_create(iccg_batch **out, iccg_ctx *const *ctxs, int32_t nsys, int32_t nrhs,
                              const iccg_batch_opts *opts) {
  if (!out) return ICCG_ERR_ARG;
  *out = nullptr;
  if (!ctxs || nsys < 1 || nrhs < 1 || nrhs > 32) return ICCG_ERR_ARG;
  iccg_batch_opts o{};
  if (opts) o = *opts;
  for (int k = 0; k < 4; ++k)
    if (o.reserved[k] != 0) return ICCG_ERR_ARG;
  if (o.warps_per_cta < 0 || o.warps_per_cta > kMaxWarpsPerCta || o.ctas_per_sm < 0) return ICCG_ERR_ARG;
  if (o.rows_per_thread != 0 && o.rows_per_thread != 1 && o.rows_per_thread != 2 && o.rows_per_thread != 4)
    return ICCG_ERR_ARG;
  for (int s = 0; s < nsys; ++s) {
    const iccg_ctx *c = ctxs[s];
    if (!c || !c->factored || c->H.n < 1) return ICCG_ERR_STATE;
    if (c->H.tile_colors != 0 || c->H.unit_colors != 0) return ICCG_ERR_ARG;   // set up with lane_block_max = -1
    if (c->device != ctxs[0]->device || c->fp32 != ctxs[0]->fp32) return ICCG_ERR_ARG;
    for (int j = 0; j < c->H.n_b; ++j)
      if (c->H.block_ptr[j + 1] - c->H.block_ptr[j] > kBatchMaxBlock) return ICCG_ERR_ARG;
  }
  iccg_batch *b = new iccg_batch();
  *out = b;
  b->device = ctxs[0]->device;
  b->stream = ctxs[0]->stream;
  b->nsys = nsys;
  b->k = nrhs;
  b->kp = pow2_at_least(nrhs);
  b->fp32 = ctxs[0]->fp32;
  b->ctxs.assign(ctxs, ctxs + nsys);
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != b->device) cudaSetDevice(b->device);
  cudaError_t e = cudaSuccess;
  for (int R : {1, 2, 4})
    for (bool walk : {false, true})
      if (e == cudaSuccess) e = allow_smem_b(batch_kernel_of(b->fp32, R, walk));
  const size_t pe = b->fp32 ? 4 : 8;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
  b->max_part_ctas = sms * 32;
  b->x.resize(nsys); b->r.resize(nsys); b->p.resize(nsys); b->q.resize(nsys);
  b->bin.resize(nsys); b->xio.resize(nsys); b->part.resize(nsys); b->hist.resize(nsys);
  b->y.resize(nsys); b->z.resize(nsys);
  b->iters.resize(nsys); b->status.resize(nsys); b->cblk.resize(nsys); b->bptr.resize(nsys);
  for (int s = 0; s < nsys && e == cudaSuccess; ++s) {
    const iccg_ctx *c = ctxs[s];
    const size_t n = size_t(c->H.n), kp = size_t(b->kp);
    b->n.push_back(c->H.n);
    const HostLayout &H = c->H;
    b->work.push_back(system_work(H));
    for (int j = 0; j < H.n_b; ++j) {
      const int r0 = H.block_ptr[j], r1 = H.block_ptr[j + 1];
      b->smax = std::max(b->smax, r1 - r0);
      b->cap = std::max(b->cap, std::max(H.lrp[r1] - H.lrp[r0], H.urp[r1] - H.urp[r0]));
    }
    for (int r0 = 0; r0 < H.n; r0 += kSpmvRows)
      b->cap = std::max(b->cap, H.arp[std::min(H.n, r0 + kSpmvRows)] - H.arp[r0]);
    b->cap = std::min(b->cap, kBatchCap);
    void *v = nullptr;
    if (e == cudaSuccess && (e = b_alloc(b, &v, 8 * n * kp)) == cudaSuccess) b->x[s] = static_cast<double *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, 8 * n * kp)) == cudaSuccess) b->r[s] = static_cast<double *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, 8 * n * kp)) == cudaSuccess) b->p[s] = static_cast<double *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, 8 * n * kp)) == cudaSuccess) b->q[s] = static_cast<double *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, pe * n * kp)) == cudaSuccess) b->y[s] = v;
    if (e == cudaSuccess && (e = b_alloc(b, &v, pe * n * kp)) == cudaSuccess) b->z[s] = v;
    if (e == cudaSuccess && (e = b_alloc(b, &v, 8 * n * size_t(b->k))) == cudaSuccess) b->bin[s] = static_cast<double *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, 8 * n * size_t(b->k))) == cudaSuccess) b->xio[s] = static_cast<double *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, 8 * size_t(b->max_part_ctas) * 4 * kp)) == cudaSuccess)
      b->part[s] = static_cast<double *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, 4 * kp)) == cudaSuccess) b->iters[s] = static_cast<int32_t *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, 4 * kp)) == cudaSuccess) b->status[s] = static_cast<int32_t *>(v);
    if (e == cudaSuccess && (e = b_alloc(b, &v, 4 * c->H.color_ptr.size())) == cudaSuccess) {
      b->cblk[s] = static_cast<int32_t *>(v);
      e = cudaMemcpyAsync(v, c->H.color_ptr.data(), 4 * c->H.color_ptr.size(), cudaMemcpyHostToDevice, b->stream);
    }
    if (e == cudaSuccess && (e = b_alloc(b, &v, 4 * c->H.block_ptr.size())) == cudaSuccess) {
      b->bptr[s] = static_cast<int32_t *>(v);
      e = cudaMemcpyAsync(v, c->H.block_ptr.data(), 4 * c->H.block_ptr.size(), cudaMemcpyHostToDevice, b->stream);
    }
  }
  void *v = nullptr;
  if (e == cudaSuccess && (e = b_alloc(b, &v, sizeof(GridBar) * size_t(nsys))) == cudaSuccess)
    b->bars = static_cast<GridBar *>(v);
  if (e == cudaSuccess && (e = b_alloc(b, &v, sizeof(BatchSys) * size_t(nsys))) == cudaSuccess)
    b->d_sys = static_cast<BatchSys *>(v);
  if (e == cudaSuccess && (e = b_alloc(b, &v, sizeof(int32_t) * size_t(b->max_part_ctas))) == cudaSuccess)
    b->d_cta_sys = static_cast<int32_t *>(v);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (prev >= 0 && prev != b->device) cudaSetDevice(prev);
  if (e != cudaSuccess) {
    b->err_msg = std::string("batch allocation: ") + cudaGetErrorString(e);
    return ICCG_ERR_CUDA;
  }
  int coop = 0;
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, b->device);
  if (!coop) {
    b->err_msg = "cooperative launch not supported";
    return ICCG_ERR_CUDA;
  }
  b->R = o.rows_per_thread > 0 ? o.rows_per_thread : 1;
  b->walk_better = batch_walks(b, 16 * sms);   // 2 CTAs of 8 warps an SM: the usual shape
  iccg_status st = set_shape(b, o.warps_per_cta > 0 ? o.warps_per_cta : 8, o.ctas_per_sm, sms);
  if (st != ICCG_OK) return st;
  if (o.autotune) {
    st = iccg_batch_tune(b, nullptr, 0.0, 0, nullptr);
    if (st != ICCG_OK) return st;
  }
  return ICCG_OK;
}

iccg_status iccg_batch_solve(iccg_batch *b, const double *const *B, double *const *X, double tol, int32_t maxit,
                             int32_t *iters, int32_t *status, double *const *res_hist) {
  if (!b || !B || !X || tol < 0 || !(tol == tol) || maxit < 0) return ICCG_ERR_ARG;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != b->device) cudaSetDevice(b->device);
  struct Restore {
    int p, d;
    ~Restore() { if (p >= 0 && p != d) cudaSetDevice(p); }
  } rs{prev, b->device};
  iccg_status st = ensure_hist(b, maxit);
  if (st != ICCG_OK) return st;
  cudaStream_t s = b->stream;
  for (int i = 0; i < b->nsys; ++i) {
    const size_t bytes = sizeof(double) * size_t(b->n[i]) * size_t(b->k);
    if (!B[i] || !X[i]) return ICCG_ERR_ARG;
    if (cudaMemcpyAsync(b->bin[i], B[i], bytes, cudaMemcpyDefault, s) != cudaSuccess ||
        cudaMemcpyAsync(b->xio[i], X[i], bytes, cudaMemcpyDefault, s) != cudaSuccess) {
      b->err_msg = "copy of B / X0";
      return ICCG_ERR_CUDA;
    }
  }
  st = run(b, maxit, tol);
  if (st != ICCG_OK) return st;
  std::vector<int32_t> it(size_t(b->kp)), stv(size_t(b->kp));
  std::vector<double> h;
  iccg_status worst = ICCG_OK;
  for (int i = 0; i < b->nsys; ++i) {
    const size_t bytes = sizeof(double) * size_t(b->n[i]) * size_t(b->k);
    if (cudaMemcpyAsync(X[i], b->xio[i], bytes, cudaMemcpyDefault, s) != cudaSuccess ||
        cudaMemcpyAsync(it.data(), b->iters[i], 4 * size_t(b->kp), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(stv.data(), b->status[i], 4 * size_t(b->kp), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
      b->err_msg = std::string("batched solve: ") + cudaGetErrorString(cudaGetLastError());
      return ICCG_ERR_CUDA;
    }
    for (int j = 0; j < b->k; ++j) {
      if (iters) iters[size_t(i) * b->k + j] = it[j];
      if (status) status[size_t(i) * b->k + j] = stv[j];
      const iccg_status sj = static_cast<iccg_status>(stv[j]);
      if (sj != ICCG_OK && (worst == ICCG_OK || sj != ICCG_NOT_CONVERGED)) worst = sj;
    }
    if (res_hist && res_hist[i]) {
      int mx = 0;
      for (int j = 0; j < b->k; ++j) mx = std::max(mx, it[j]);
      h.assign(size_t(mx + 1) * b->kp, 0.0);
      if (cudaMemcpy(h.data(), b->hist[i], sizeof(double) * h.size(), cudaMemcpyDeviceToHost) != cudaSuccess) {
        b->err_msg = "history copy";
        return ICCG_ERR_CUDA;
      }
      // res_hist[i]: [maxit + 1][nrhs]; entries past a right-hand side's
      // iteration count are 0
      for (int t = 0; t <= maxit; ++t)
        for (int j = 0; j < b->k; ++j)
          res_hist[i][size_t(t) * b->k + j] = (t <= it[j] && t <= mx) ? h[size_t(t) * b->kp + j] : 0.0;
    }
  }
  if (worst == ICCG_ERR_TIMEOUT) b->err_msg = "a barrier wait of the batched solve gave up";
  return worst;
}

iccg_status iccg_batch_tune(iccg_batch *b, const double *const *B, double tol, int32_t maxit, double *best_ms) {
  if (!b || (B && (tol < 0 || !(tol == tol) || maxit < 0))) return ICCG_ERR_ARG;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
  // every candidate shape solves the given right-hand sides from x0 = 0 to
  // (tol, maxit), or, without B, random right-hand sides for a fixed 20
  // iterations (tol 0); the fastest shape is kept
  std::vector<std::vector<double>> hb(b->nsys), hx(b->nsys);
  std::vector<const double *> Bp(b->nsys);
  std::vector<double *> X(b->nsys);
  uint64_t st = 0x9e3779b97f4a7c15ull;
  for (int s = 0; s < b->nsys; ++s) {
    hx[s].assign(size_t(b->n[s]) * b->k, 0.0);
    X[s] = hx[s].data();
    if (B) {
      Bp[s] = B[s];
      if (!B[s]) return ICCG_ERR_ARG;
      continue;
    }
    hb[s].resize(size_t(b->n[s]) * b->k);
    for (double &v : hb[s]) {
      st ^= st << 13; st ^= st >> 7; st ^= st << 17;
      v = double(st >> 11) * (1.0 / 9007199254740992.0) - 0.5;
    }
    Bp[s] = hb[s].data();
  }
  const double ttol = B ? tol : 0.0;
  const int tmax = B ? maxit : 20;
  const int Ws[3] = {4, 8, 16};
  double best = 1e300;
  bool bE = b->by_work;
  int bW = b->W, bC = b->cps;
  for (bool E : {false, true})
  for (int W : Ws) {
    const int occ = batch_occupancy(b, W, shape_walks(b, W));
    for (int cps = 1; cps <= std::min(occ, 4); cps *= 2) {
      b->by_work = E;
      if (set_shape(b, W, cps, sms) != ICCG_OK) continue;
      for (auto &x : hx) std::fill(x.begin(), x.end(), 0.0);
      // the first call captures the graph; the second is timed
      if (iccg_batch_solve(b, Bp.data(), X.data(), ttol, tmax, nullptr, nullptr, nullptr) == ICCG_ERR_CUDA) continue;
      for (auto &x : hx) std::fill(x.begin(), x.end(), 0.0);
      const auto t0 = std::chrono::steady_clock::now();
      const iccg_status r = iccg_batch_solve(b, Bp.data(), X.data(), ttol, tmax, nullptr, nullptr, nullptr);
      const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
      if (r == ICCG_ERR_CUDA || r == ICCG_ERR_TIMEOUT) continue;
      if (ms < best) { best = ms; bW = W; bC = cps; bE = E; }
    }
  }
  // rows per thread at the best shape
  b->by_work = bE;
  int bR = b->R;
  const int R0 = b->R;
  for (int R : {1, 2, 4}) {
    if (R == R0) continue;
    b->R = R;   // the shape's occupancy is that of this R's kernel
    if (set_shape(b, bW, bC, sms) != ICCG_OK) continue;
    for (auto &x : hx) std::fill(x.begin(), x.end(), 0.0);
    if (iccg_batch_solve(b, Bp.data(), X.data(), ttol, tmax, nullptr, nullptr, nullptr) == ICCG_ERR_CUDA) continue;
    for (auto &x : hx) std::fill(x.begin(), x.end(), 0.0);
    const auto t0 = std::chrono::steady_clock::now();
    const iccg_status r = iccg_batch_solve(b, Bp.data(), X.data(), ttol, tmax, nullptr, nullptr, nullptr);
    const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    if (r == ICCG_ERR_CUDA || r == ICCG_ERR_TIMEOUT) continue;
    if (ms < best) { best = ms; bR = R; }
  }
  b->R = bR;
  if (best_ms) *best_ms = best;
  return set_shape(b, bW, bC, sms);
}

iccg_status iccg_batch_set_wait_limit(iccg_batch *b, uint64_t wait_ns) {
  if (!b) return ICCG_ERR_ARG;
  b->wait_ns = wait_ns ? wait_ns : kDefaultWaitNs;
  destroy_batch_graph(b);   // the next solve uploads the descriptors again
  return ICCG_OK;
}

iccg_status iccg_batch_info(const iccg_batch *b, int32_t out[7]) {
  if (!b || !out) return ICCG_ERR_ARG;
  out[0] = b->W;
  out[1] = b->cps;
  out[2] = b->grid;
  out[3] = b->kp;
  out[4] = b->smax;
  out[5] = b->by_work ? 4 : 3;   // the CTA split: 4 by rows x estimated iterations, 3 by rows
  out[6] = b->R;
  return ICCG_OK;
}

iccg_status iccg_batch_last_error(const iccg_batch *b, const char **msg) {
  if (!b) return ICCG_ERR_ARG;
  if (msg) *msg = b->err_msg.c_str();
  return ICCG_OK;
}

void iccg_batch_destroy(iccg_batch *b) {
  if (!b) return;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != b->device) cudaSetDevice(b->device);
  if (b->stream) cudaStreamSynchronize(b->stream);
  destroy_batch_graph(b);
  for (void *p : b->allocs) cudaFree(p);
  if (prev >= 0 && prev != b->device) cudaSetDevice(prev);
  delete b;
}

}  // extern "C"
