// Device kernels of block-multicolor ICCG for sm_103a.
//
// One PCG iteration is 2*n_c + 1 launches (n_c = number of block colors):
//   p update             p = z + beta p
//   spmv                 q = A p, <p,q>; its last group sets alpha = (r,z)/(p,q)
//   fwd color 0..n_c-2   x += alpha p, r -= alpha q, <r,r>, then the forward
//                        substitution L y = r for the rows of that color
//                        (Alg. 1: colors in sequence, blocks of a color in
//                        parallel, rows of a block in order)
//   fused color n_c-1    the same, followed at once by the backward sweep of
//                        the last color (its rows have no later-color
//                        dependencies), <r,z> and <r,r>
//   bwd color n_c-2..0   backward substitution L^T z = y (the reverse sweep
//                        described after Alg. 1), <r,z> and <r,r>; the last
//                        group of the color-0 launch sums them, records the
//                        residual history, tests ||r||/||b|| <= tol and sets
//                        the CUDA-graph WHILE condition.
// Both sums are formed where the backward sweep reads r anyway, in one
// reduction per launch, and the forward launches reduce nothing.  (<r,z> is not
// taken as <y,y>, y = L^-1 r, although that needs no r: on ill-conditioned
// systems the two differ by more than a sum's rounding.)
//
// Substitution work mapping.  One warp owns a group: consecutive whole blocks
// of one color (at most 32R rows), or one block larger than that.  Blocks of
// one color share no edge, so the group's rows depend on earlier colors and
// on earlier rows of their own block only.  The warp works in two phases:
//   A  every row at once, one row per lane: the entries that point to earlier
//      colors (y or z gathers) and the fused x / r update;
//   B  the in-block dependencies, level by level: the rows of all the group's
//      blocks are listed by their depth in their block's dependency DAG, and
//      each level is processed with the rows packed across lanes, so every row
//      is computed exactly once and the FP64 lanes are mostly busy.  The
//      per-row arithmetic is the row of Alg. 1 (earlier-color terms first).
// GB300's FP64 FMA rate is 2 lanes/cycle/SM, so a DFMA issued with idle lanes
// costs as much as a full one; this packing is what keeps the FP64 pipe from
// becoming the bound.
//
// Memory: a fitting group's CSR segment of L or U, its row pointers, 1/L_ii,
// schedule and level pointers are copied into the warp's shared memory with
// cp.async (16-byte, L2 only, all in flight at once) before the kernel waits
// on its predecessor (programmatic dependent launch: griddepcontrol.wait), so
// this static traffic overlaps the previous launch.  A group too large for the
// shared-memory plan reads the same data from global memory.
//
// Vectors that other CTAs write during a solve (r, q, x, p, y, z) are read
// with L2 loads (ld.global.cg), so no SM ever sees a stale L1 line of them.
//
// Reductions are deterministic and two-level: every CTA writes its partial;
// the last CTA of each group of kGroup CTAs (arrival ticket) sums the group's
// partials in index order; the last group of the launch runs the epilogue.
#include <algorithm>
#include <cstdio>
#include <type_traits>

#include "iccg_internal.h"

namespace iccg {

namespace {

constexpr int kVecThreads = 256;
constexpr int kChunk = 4;    // row entries processed per predicated batch
constexpr int kRedWarp = 6;                        // reduction scratch of a warp (doubles)
constexpr int kRed = kRedWarp * kMaxWarpsPerCta;   // and of a CTA
enum StepMode { M_FWD = 0, M_BWD = 1, M_FUSED = 2 };

// Programmatic dependent launch: everything before this call runs while the
// previous launch finishes.  The next launch may start once every CTA of this
// one is past it, i.e. at most one launch waits beside the working one.  (Let
// off at the kernels' first instruction, five to ten launches piled up waiting
// and held the slots that the working launch's grid counts on.)
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
// 4- and 8-byte copies (.ca: cached in L1 as well)
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(gmem) : "memory");
}
template <typename PT>
__device__ __forceinline__ void cp_async_elem(PT *smem, const PT *gmem);
template <> __device__ __forceinline__ void cp_async_elem<double>(double *smem, const double *gmem) {
  cp_async8(smem, gmem);
}
template <> __device__ __forceinline__ void cp_async_elem<float>(float *smem, const float *gmem) {
  cp_async4(smem, gmem);
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
// all but the most recently committed group
__device__ __forceinline__ void cp_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Sums of a and b over the warp together: a's in lane 0, b's in lane 16.  An
// FP64 instruction costs a warp 64 cycles however many of its lanes it serves,
// so after one exchange the half warps carry one sum each: 5 additions for both.
__device__ __forceinline__ double warp_sum2(double a, double b) {
  const bool hi = (threadIdx.x & 16) != 0;
  const double u = __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
  double v = (hi ? b : a) + u;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, 16);
  return v;
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

// Sums of a and b over the CTA in a fixed order (red: 2 doubles a warp): the warps' sums one after another.  In warp 0, lane 0 returns a's
// and lane 16 b's (both in the same instructions).
__device__ __forceinline__ double cta_sum2(double a, double b, double *red) {
  double v = warp_sum2(a, b);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (nw == 1) return v;
  __syncthreads();
  if ((l & 15) == 0) red[(l >> 4) * nw + w] = v;
  __syncthreads();
  if (w == 0) {
    const double *p = red + (l >> 4) * nw;
    v = p[0];
    for (int k = 1; k < nw; ++k) v += p[k];
  }
  return v;
}

// Sum of one value per thread; result valid in thread 0.  Fixed order.
__device__ __forceinline__ double cta_sum(double v, double *red) { return cta_sum2(v, 0.0, red); }

// Deterministic sum of p[0..count) by the whole CTA (result in thread 0);
// optionally clears the entries.
__device__ __forceinline__ double cta_sum_array(double *p, int count, double *red, bool clear) {
  double s = 0.0;
#pragma unroll 4
  for (int k = threadIdx.x; k < count; k += blockDim.x) {
    s += __ldcg(p + k);
    if (clear) p[k] = 0.0;
  }
  return cta_sum(s, red);
}

// Arrival on a counter by thread 0 after a fence; true (for the whole CTA)
// for the last of `expected` arrivals, with which the counter wraps to 0.
__device__ __forceinline__ bool arrive_last(uint32_t *ticket, uint32_t expected, int *flag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const int last = atomicInc(ticket, expected - 1) == expected - 1 ? 1 : 0;
    if (last) __threadfence();
    *flag = last;
  }
  __syncthreads();
  return *flag != 0;
}

// First level: each CTA publishes its two sums (v of lanes 0 and 16 of its first
// warp); the last CTA of the group returns true with the group's in gv there.
__device__ __forceinline__ bool group_reduce(const Params &P, double v, double *red, int *flag, double &gv) {
  const int g = blockIdx.x / kGroup;
  const int g0 = g * kGroup;
  const int gs = min(kGroup, int(gridDim.x) - g0);
  if (threadIdx.x == 0) P.part0[blockIdx.x] = v;
  if (threadIdx.x == 16) {
    P.part1[blockIdx.x] = v;
    __threadfence();
  }
  if (!arrive_last(P.gticket + g, uint32_t(gs), flag)) return false;
  const bool in = threadIdx.x < unsigned(gs);
  gv = cta_sum2(in ? __ldcg(P.part0 + g0 + threadIdx.x) : 0.0, in ? __ldcg(P.part1 + g0 + threadIdx.x) : 0.0, red);
  return true;
}

// Second level: the last group of the launch.
__device__ __forceinline__ bool launch_last(const Params &P, int *flag) {
  const uint32_t ng = (gridDim.x + kGroup - 1) / kGroup;
  return arrive_last(&P.sc->ticket, ng, flag);
}

// A CSR segment: staged in shared memory (entry e at sv[e - bv], sc[e - bc])
// or read from global memory.
template <typename VT>
struct Seg {
  const VT *sv;
  const int32_t *sc;
  const VT *gv;
  const int32_t *gc;
  int bv, bc;
  bool staged;
  __device__ __forceinline__ VT v(int e) const { return staged ? sv[e - bv] : __ldg(gv + e); }
  __device__ __forceinline__ int32_t c(int e) const { return staged ? sc[e - bc] : __ldg(gc + e); }
};

// Issue the cp.async copies of the 16-byte-aligned cover of g[a, b) into s;
// returns the index of s[0] in g.  Device arrays carry 64 bytes of padding,
// so the cover stays inside the allocation; s needs (b - a) + 2 * (16 /
// sizeof(T)) elements.
template <typename T>
__device__ __forceinline__ int stage_cover(const T *g, int a, int b, T *s, int tid, int nthr) {
  constexpr int EV = 16 / sizeof(T);
  const int a0 = a & ~(EV - 1), a1 = (b + EV - 1) & ~(EV - 1);
  const int nv = (a1 - a0) / EV;
  for (int k = tid; k < nv; k += nthr) cp_async16(s + k * EV, g + a0 + k * EV);
  return a0;
}

// count of entries of [rb, re) whose column is below `bound` (columns sorted)
template <typename VT>
__device__ __forceinline__ int count_below(const Seg<VT> &S, int rb, int re, int bound) {
  int n = 0;
  for (int e = rb; e < re; ++e) n += S.c(e) < bound ? 1 : 0;
  return n;
}

// acc -= sum of v_e * x(c_e) over the entries e in [rb, re), ascending;
// loads in predicated batches of kChunk, then the FMAs of the batch.
template <typename VT, typename AT, typename Load>
__device__ __forceinline__ AT row_sub(const Seg<VT> &S, int rb, int re, AT acc, Load x) {
  for (int e0 = rb; e0 < re; e0 += kChunk) {
    int cc[kChunk];
    VT vv[kChunk];
#pragma unroll
    for (int j = 0; j < kChunk; ++j) {
      const bool ok = e0 + j < re;
      cc[j] = ok ? S.c(e0 + j) : -1;
      vv[j] = ok ? S.v(e0 + j) : VT(0);
    }
    AT xx[kChunk];
#pragma unroll
    for (int j = 0; j < kChunk; ++j) xx[j] = cc[j] >= 0 ? AT(x(cc[j])) : AT(0);
#pragma unroll
    for (int j = 0; j < kChunk; ++j)
      if (cc[j] >= 0) acc -= AT(vv[j]) * xx[j];
  }
  return acc;
}

template <typename PT> __device__ __forceinline__ const PT *lvals(const Params &P);
template <> __device__ __forceinline__ const double *lvals<double>(const Params &P) { return P.lval; }
template <> __device__ __forceinline__ const float *lvals<float>(const Params &P) { return P.lval32; }
template <typename PT> __device__ __forceinline__ const PT *uvals(const Params &P);
template <> __device__ __forceinline__ const double *uvals<double>(const Params &P) { return P.uval; }
template <> __device__ __forceinline__ const float *uvals<float>(const Params &P) { return P.uval32; }
template <typename PT> __device__ __forceinline__ const PT *invds(const Params &P);
template <> __device__ __forceinline__ const double *invds<double>(const Params &P) { return P.invd; }
template <> __device__ __forceinline__ const float *invds<float>(const Params &P) { return P.invd32; }

// alpha of this iteration, with the flag that the solve has ended: the graph
// loop runs several iterations per pass, and the launches of the iterations
// after the last one change nothing (false).
__device__ __forceinline__ bool load_alpha(const Params &P, double &alpha) {
  const double2 v = __ldcg(reinterpret_cast<const double2 *>(&P.sc->alpha));
  alpha = v.x;
  return v.y == 0.0;
}

// ---------------------------------------------------------------------------
// per-CTA shared memory of the substitution kernels (one CTA per group)
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ int r16(int bytes) { return (bytes + 15) & ~15; }

struct GroupSmemPlan {
  int o_sv, o_sc, o_rp, o_dv, o_sch, o_lp, o_w, o_spl, total;
};

__host__ __device__ __forceinline__ GroupSmemPlan group_smem_plan(int cap, int rows, int levs, int elem) {
  GroupSmemPlan p;
  int o = 0;
  p.o_sv = o; o += r16((cap + 8) * elem);
  p.o_sc = o; o += r16((cap + 8) * 4);
  p.o_rp = o; o += r16((rows + 9) * 4);
  p.o_dv = o; o += r16((rows + 8) * elem);
  p.o_sch = o; o += r16((rows + 8) * 4);
  p.o_lp = o; o += r16((levs + 9) * 4);
  p.o_w = o; o += r16(rows * elem);
  p.o_spl = o; o += r16(rows * 4);
  p.total = o;
  return p;
}

template <typename PT>
struct GroupSmem {
  PT *sv;
  int32_t *sc, *rp, *sch, *lp, *spl;
  PT *dv, *w;
};

template <typename PT>
__device__ __forceinline__ GroupSmem<PT> group_smem(unsigned char *base, const GroupSmemPlan &p) {
  unsigned char *m = base;
  GroupSmem<PT> s;
  s.sv = reinterpret_cast<PT *>(m + p.o_sv);
  s.sc = reinterpret_cast<int32_t *>(m + p.o_sc);
  s.rp = reinterpret_cast<int32_t *>(m + p.o_rp);
  s.dv = reinterpret_cast<PT *>(m + p.o_dv);
  s.sch = reinterpret_cast<int32_t *>(m + p.o_sch);
  s.lp = reinterpret_cast<int32_t *>(m + p.o_lp);
  s.w = reinterpret_cast<PT *>(m + p.o_w);
  s.spl = reinterpret_cast<int32_t *>(m + p.o_spl);
  return s;
}

__device__ __forceinline__ GroupDesc load_group(const GroupDesc *g) {
  const int4 *p = reinterpret_cast<const int4 *>(g);
  const int4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
  GroupDesc d;
  d.r0 = a.x; d.r1 = a.y; d.l0 = a.z; d.l1 = a.w;
  d.u0 = b.x; d.u1 = b.y; d.lf = b.z; d.lb = b.w;
  d.nlf = c.x; d.nlb = c.y; d.fit = c.z;
  return d;
}

// Where the static data of one sweep over a group lives (shared memory for a
// fitting group, global memory otherwise).
template <typename PT>
struct Sweep {
  Seg<PT> S;
  bool fit;
  int rpb, dvb, schb, lpb;       // index of the first staged element
  const int32_t *grp, *gsch;     // global row pointers / schedule
  const PT *gdv;
  int lev0, nlev;                // level pointers at levp[lev0 ..]
  __device__ __forceinline__ int rp(const GroupSmem<PT> &m, int i) const { return fit ? m.rp[i - rpb] : __ldg(grp + i); }
  __device__ __forceinline__ PT dv(const GroupSmem<PT> &m, int i) const { return fit ? m.dv[i - dvb] : __ldg(gdv + i); }
};

// index of the first element of the 16-byte-aligned cover that stage_cover copies
template <typename T>
__device__ __forceinline__ int cover_base(int a) { return a & ~(int(16 / sizeof(T)) - 1); }

// Describe where the static data of a forward (upper = false) or backward
// (upper = true) sweep over group d lives once sweep_issue's copies landed.
template <typename PT>
__device__ __forceinline__ Sweep<PT> sweep_desc(const Params &P, const GroupDesc &d, bool upper,
                                                const GroupSmem<PT> &m) {
  Sweep<PT> sw;
  sw.fit = d.fit != 0;
  sw.grp = upper ? P.urp : P.lrp;
  sw.gsch = upper ? P.sched_b : P.sched_f;
  sw.gdv = invds<PT>(P);
  sw.lev0 = upper ? d.lb : d.lf;
  sw.nlev = upper ? d.nlb : d.nlf;
  sw.S.gv = upper ? uvals<PT>(P) : lvals<PT>(P);
  sw.S.gc = upper ? P.ucol : P.lcol;
  sw.S.sv = m.sv;
  sw.S.sc = m.sc;
  sw.S.staged = sw.fit;
  sw.S.bv = sw.S.bc = 0;
  sw.rpb = sw.dvb = sw.schb = sw.lpb = 0;
  if (sw.fit) {
    const int e0 = upper ? d.u0 : d.l0;
    sw.S.bv = cover_base<PT>(e0);
    sw.S.bc = cover_base<int32_t>(e0);
    sw.rpb = cover_base<int32_t>(d.r0);
    sw.dvb = cover_base<PT>(d.r0);
    sw.schb = cover_base<int32_t>(d.r0);
    sw.lpb = cover_base<int32_t>(sw.lev0);
  }
  return sw;
}

// Issue (without committing) the cp.async copies of a fitting group's static
// sweep data into m; nothing for a group that reads global memory.
template <typename PT>
__device__ __forceinline__ void sweep_issue(const Params &P, const GroupDesc &d, bool upper, const GroupSmem<PT> &m,
                                            int tid, int nthr) {
  if (!d.fit) return;
  const int e0 = upper ? d.u0 : d.l0, e1 = upper ? d.u1 : d.l1;
  const int lev0 = upper ? d.lb : d.lf, nlev = upper ? d.nlb : d.nlf;
  stage_cover<PT>(upper ? uvals<PT>(P) : lvals<PT>(P), e0, e1, m.sv, tid, nthr);
  stage_cover<int32_t>(upper ? P.ucol : P.lcol, e0, e1, m.sc, tid, nthr);
  stage_cover<int32_t>(upper ? P.urp : P.lrp, d.r0, d.r1 + 1, m.rp, tid, nthr);
  stage_cover<PT>(invds<PT>(P), d.r0, d.r1, m.dv, tid, nthr);
  stage_cover<int32_t>(upper ? P.sched_b : P.sched_f, d.r0, d.r1, m.sch, tid, nthr);
  stage_cover<int32_t>(P.levp, lev0, lev0 + nlev + 1, m.lp, tid, nthr);
}

// Stage and describe the static data of one sweep; commits the copies, the
// caller waits.
template <typename PT>
__device__ __forceinline__ Sweep<PT> sweep_static(const Params &P, const GroupDesc &d, bool upper,
                                                  const GroupSmem<PT> &m, int tid, int nthr) {
  sweep_issue<PT>(P, d, upper, m, tid, nthr);
  cp_commit();
  return sweep_desc<PT>(P, d, upper, m);
}

// a row's shares of <r,r> and <r,z> (FP32 z widened exactly)
__device__ __forceinline__ void rz_add(double r, double z, double &rr, double &rz) {
  rr += r * r;
  rz += r * z;
}
__device__ __forceinline__ void rz_add(double r, float z, double &rr, double &rz) { rz_add(r, widen(z), rr, rz); }

// One sweep over a group.  UPPER = false: forward, L rows (entries to earlier
// colors are a prefix of each row, in-block entries the rest); the source is
// r (with the x / r update when UPDATE) and the result y.  UPPER = true:
// backward, U rows (in-block entries a prefix, later colors the rest); the
// source is y (shared memory when the fused kernel keeps y of a fitting group
// there) and the result z, with <r, z> and <r, r>.
// Fitting groups keep t / y / z in m.w; other groups work in place in the
// global result vector.
template <typename PT, bool UPPER, bool UPDATE>
__device__ __forceinline__ void group_sweep(const Params &P, const GroupDesc &d, const Sweep<PT> &sw,
                                            const GroupSmem<PT> &m, int tid, int nthr, double alpha,
                                            const double *pn, bool y_in_smem, bool store_result, double &rr_acc,
                                            double &rz_acc) {
  PT *yv = reinterpret_cast<PT *>(P.y);
  PT *zv = reinterpret_cast<PT *>(P.z);
  PT *res = UPPER ? zv : yv;        // global result vector
  const PT *ext = UPPER ? zv : yv;  // gathered for out-of-group columns
  const int r0 = d.r0, r1 = d.r1, nrows = r1 - r0;
  const bool fit = sw.fit;
  // phase A: out-of-group entries, all rows at once (one row per thread)
  for (int l = tid; l < nrows; l += nthr) {
    const int i = r0 + l;
    const int rb = sw.rp(m, i), re = sw.rp(m, i + 1);
    PT src;
    if (UPPER) {
      src = y_in_smem ? m.w[l] : __ldcg(yv + i);
    } else {
      double ri = __ldcg(P.r + i);
      if (UPDATE) {
        ri -= alpha * __ldcg(P.q + i);
        P.r[i] = ri;
        P.xh[i] = __ldcg(P.xh + i) + alpha * __ldcg(pn + i);
      }
      src = PT(ri);
    }
    const int split = rb + count_below(sw.S, rb, re, UPPER ? r1 : r0);
    const int xb = UPPER ? split : rb, xe = UPPER ? re : split;
    const PT t = row_sub<PT, PT>(sw.S, xb, xe, src, [&](int c) { return __ldcg(ext + c); });
    if (fit) {
      m.w[l] = t;
      m.spl[l] = split;
    } else {
      res[i] = t;
    }
  }
  __syncthreads();
  // phase B: in-block entries, level by level; a level's rows go to the
  // first threads, so only as many warps as the level needs issue FP64 work
  for (int lv = 0; lv < sw.nlev; ++lv) {
    const int p0 = fit ? m.lp[sw.lev0 + lv - sw.lpb] : __ldg(P.levp + sw.lev0 + lv);
    const int p1 = fit ? m.lp[sw.lev0 + lv + 1 - sw.lpb] : __ldg(P.levp + sw.lev0 + lv + 1);
    for (int p = p0 + tid; p < p1; p += nthr) {
      const int l = fit ? m.sch[r0 + p - sw.schb] : __ldg(sw.gsch + r0 + p);
      const int i = r0 + l;
      const int rb = sw.rp(m, i), re = sw.rp(m, i + 1);
      int ib, ie;
      PT acc;
      if (fit) {
        acc = m.w[l];
        ib = UPPER ? rb : m.spl[l];
        ie = UPPER ? m.spl[l] : re;
        acc = row_sub<PT, PT>(sw.S, ib, ie, acc, [&](int c) { return m.w[c - r0]; });
        m.w[l] = acc * sw.dv(m, i);
      } else {
        acc = __ldcg(res + i);
        const int split = rb + count_below(sw.S, rb, re, UPPER ? r1 : r0);
        ib = UPPER ? rb : split;
        ie = UPPER ? split : re;
        acc = row_sub<PT, PT>(sw.S, ib, ie, acc, [&](int c) { return __ldcg(res + c); });
        res[i] = acc * sw.dv(m, i);
      }
    }
    __syncthreads();
  }
  // results: fitting groups store from shared memory (coalesced)
  for (int l = tid; l < nrows; l += nthr) {
    const int i = r0 + l;
    const PT v = fit ? m.w[l] : __ldcg(res + i);
    if (fit && store_result) res[i] = v;
    if (UPPER) rz_add(__ldcg(P.r + i), v, rr_acc, rz_acc);
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// epilogues run by the last group of a launch
// ---------------------------------------------------------------------------
__device__ void set_condition(const Scalars *s, bool go, int iter) {
  if (!s->use_cond) return;
  cudaGraphSetConditional((cudaGraphConditionalHandle)s->cond_handle,
                          go && (s->cond_rest == 0 || iter < kFirstIterations) ? 1u : 0u);
  if (s->cond_rest) cudaGraphSetConditional((cudaGraphConditionalHandle)s->cond_rest, go ? 1u : 0u);
}

// What finish_iteration reads, loaded while the sums are still being formed.
struct IterScalars {
  double bnorm, tol, rz;
  int iter, maxit, status;
};
__device__ __forceinline__ IterScalars load_iter(const Scalars *s) {
  IterScalars v;
  v.bnorm = __ldcg(&s->bnorm);
  v.tol = __ldcg(&s->tol);
  v.rz = __ldcg(&s->rz);
  v.iter = __ldcg(&s->iter);
  v.maxit = __ldcg(&s->maxit);
  v.status = __ldcg(&s->status);
  return v;
}

// After the backward sweep of iteration k: residual history, stop test, beta;
// by warp 0, sum = rr in lane 0, rz in lane 16.  The two quotients (a division
// is a sequence of FP64 instructions) run side by side in the two lanes.
__device__ void finish_iteration(const Params &P, double sum, const IterScalars &v) {
  if (threadIdx.x >= kWarp) return;
  const bool l0 = threadIdx.x == 0;
  const double quot = (l0 ? sqrt(sum) : sum) / (l0 ? v.bnorm : v.rz);
  const double rz = __shfl_sync(0xffffffffu, sum, 16), beta = __shfl_sync(0xffffffffu, quot, 16);
  if (l0) {
    Scalars *s = P.sc;
    const int k = v.iter;
    const double rn = quot;
    int done = 0;
    // a bounded wait of this iteration gave up (a cooperative launch of the
    // sweep): the solve stops with that status
    if (v.status == ICCG_ERR_TIMEOUT) done = 1;
    else if (!isfinite(rn) || !isfinite(rz)) { s->status = ICCG_ERR_NONFINITE; done = 1; }
    else if (rn <= v.tol) { s->status = ICCG_OK; done = 1; }
    else if (k + 1 >= v.maxit) { s->status = ICCG_NOT_CONVERGED; done = 1; }
    else { s->beta = beta; s->rz = rz; }
    P.hist[k + 1] = rn;
    s->iter = k + 1;
    s->rr = sum;
    s->done = done;
    if (done) s->skip = 1.0;
    set_condition(s, !done, k + 1);
  }
}

// After r0 = b - A x0 and z0 = M^-1 r0: ||b||, history[0], stop test.
// init_bb holds <b,b> partials, part_a the <r0,r0> partials; rz valid in
// thread 0.
__device__ void finish_init(const Params &P, double rz, double *red) {
  const double bb = cta_sum_array(P.init_bb, P.nbb, red, false);
  const double rr = cta_sum_array(P.part_a, P.npart_a, red, false);
  if (threadIdx.x == 0) {
    Scalars *s = P.sc;
    const double bn = sqrt(bb);
    s->bb = bb;
    s->bnorm = bn;
    s->iter = 0;
    s->beta = 0.0;
    s->rz = rz;
    s->rr = rr;
    int done = 0;
    if (s->status == ICCG_ERR_TIMEOUT) done = 1;
    else if (bn == 0.0) { P.hist[0] = 0.0; s->status = ICCG_OK; done = 1; }
    else {
      const double rn = sqrt(rr) / bn;
      P.hist[0] = rn;
      if (!isfinite(rn) || !isfinite(rz)) { s->status = ICCG_ERR_NONFINITE; done = 1; }
      else if (rn <= s->tol) { s->status = ICCG_OK; done = 1; }
      else if (s->maxit <= 0) { s->status = ICCG_NOT_CONVERGED; done = 1; }
      else s->status = ICCG_NOT_CONVERGED;
    }
    s->done = done;
    s->skip = done ? 1.0 : 0.0;
    set_condition(s, !done, 0);
  }
}

enum Fin { FIN_NONE = 0, FIN_ITER = 1, FIN_INIT = 2 };

// ---------------------------------------------------------------------------
// color kernel: MODE = forward sweep of one color, backward sweep of one
// color, or both for the last color (fused); one CTA per group
// ---------------------------------------------------------------------------
// groups a warp of the final launch's last CTA sums itself at most, instead of
// the groups' own last CTAs (that level costs an atomic and a trip to L2, about
// 1 us); the same sums in the same order
constexpr int kOneLevel = 2;

struct SlotArgs {
  int off;      // this launch's first slot (-1: no sums wanted)
  int last;     // final launch: slots of the sweep's earlier launches
  int iter;     // 1: a launch of an iteration, which the graph may run after the last one
};

// A backward launch's own look at the end of the solve (forward launches read it
// with alpha), in the kernels of warps on their own.  The load goes out before
// griddepcontrol.wait and is looked at after it: loaded after the wait, the
// sweep's loads would have to wait for it; looked at before, the wait itself
// would, with which the next launch may start.  When a launch starts, everything
// up to two launches before it is complete, the last iteration's end included; a
// value set by the launch just before (a wait that ran out) may be seen or not.
// Either way the launch's sums are dropped (launch_epilogue).  Where a CTA would
// have to agree on it (lane tiles, groups) every launch would pay more than the
// solve's last ones save (27-point 56^3, 40 iterations: blocks of four rows in
// FP32 7.0 against 6.6 ms, blocks of 64 32.4 against 31.6): those run once more.
__device__ __forceinline__ bool sweep_ended(const Params &P, const SlotArgs &sa) {
  return sa.iter != 0 && __ldcg(&P.sc->skip) != 0.0;
}

// End of a launch with a backward sweep: this CTA's <r,r> / <r,z> partials.  A
// non-final launch stores them in its slot region (plain stores: the sweep's
// last launch sums them).  In the last launch every CTA adds a fixed chunk of
// the earlier launches' slots (complete: griddepcontrol.wait before) to its own
// partials; then groups of CTAs, then the last group runs the epilogue.
// (COOP: the cooperative sweep has decided at its start whether the solve goes on)
template <bool COOP = false>
__device__ __forceinline__ void launch_epilogue(const Params &P, int fin, const SlotArgs &sa, double rr_acc,
                                                double rz_acc, double *red, int *flag) {
  if (sa.off < 0) return;
  if (!COOP && fin == FIN_ITER && __ldcg(&P.sc->done)) return;   // an iteration after the last one
  if (fin == FIN_NONE) {
    const double v = cta_sum2(rr_acc, rz_acc, red);
    if (threadIdx.x == 0) P.slot_rr[sa.off + blockIdx.x] = v;
    if (threadIdx.x == 16) P.slot_rz[sa.off + blockIdx.x] = v;
    return;
  }
  const int nb = gridDim.x, chunk = (sa.last + nb - 1) / nb;
  for (int k = threadIdx.x; k < chunk; k += blockDim.x) {
    const int idx = blockIdx.x * chunk + k;
    if (idx < sa.last) {
      rr_acc += __ldcg(P.slot_rr + idx);
      rz_acc += __ldcg(P.slot_rz + idx);
    }
  }
  double v = cta_sum2(rr_acc, rz_acc, red);
  const int ng = (nb + kGroup - 1) / kGroup;
  const double *p0 = P.gsum0, *p1 = P.gsum1;
  if (ng <= kOneLevel * int(blockDim.x >> 5)) {
    // few CTAs: the last of them forms the groups' sums itself, a warp a group
    if (threadIdx.x == 0) P.part0[blockIdx.x] = v;
    if (threadIdx.x == 16) {
      P.part1[blockIdx.x] = v;
      __threadfence();
    }
    if (!arrive_last(&P.sc->ticket, uint32_t(nb), flag)) return;
    const int nw = int(blockDim.x >> 5);
    double *gs = red + 2 * nw;
    for (int g = threadIdx.x >> 5; g < ng; g += int(blockDim.x >> 5)) {
      const int k = g * kGroup + int(threadIdx.x & 31);
      v = warp_sum2(k < nb ? __ldcg(P.part0 + k) : 0.0, k < nb ? __ldcg(P.part1 + k) : 0.0);
      if ((threadIdx.x & 15) == 0) gs[((threadIdx.x >> 4) & 1) * 2 * nw + g] = v;
    }
    __syncthreads();
    p0 = gs;
    p1 = gs + 2 * nw;
  } else {
    double gv;
    if (!group_reduce(P, v, red, flag, gv)) return;
    if (threadIdx.x == 0) P.gsum0[blockIdx.x / kGroup] = gv;
    if (threadIdx.x == 16) {
      P.gsum1[blockIdx.x / kGroup] = gv;
      __threadfence();
    }
    if (!launch_last(P, flag)) return;
  }
  const IterScalars is = load_iter(P.sc);
  double a = 0.0, b = 0.0;
  for (int k = threadIdx.x; k < ng; k += blockDim.x) {
    a += p0 == P.gsum0 ? __ldcg(p0 + k) : p0[k];
    b += p0 == P.gsum0 ? __ldcg(p1 + k) : p1[k];
  }
  v = cta_sum2(a, b, red);
  if (fin == FIN_ITER) {
    finish_iteration(P, v, is);
  } else {
    const double rz = threadIdx.x < kWarp ? __shfl_sync(0xffffffffu, v, 16) : 0.0;
    finish_init(P, rz, red);
  }
}

template <typename PT, int MODE, bool UPDATE>
__global__ void __launch_bounds__(kMaxWarpsPerCta * kWarp)
color_kernel(Params P, int g0, int g1, GroupSmemPlan plan, int fin, SlotArgs sa) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[kRed];
  __shared__ int flag;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const GroupSmem<PT> m = group_smem<PT>(smem, plan);
  double rr_acc = 0.0, rz_acc = 0.0;
  const int g = g0 + blockIdx.x;
  if (g < g1) {
    const GroupDesc d = load_group(P.groups + g);
    const Sweep<PT> sw = sweep_static<PT>(P, d, MODE == M_BWD, m, tid, nthr);
    cp_wait_all();
    __syncthreads();
    pdl_wait();
    if (MODE == M_BWD) {
      group_sweep<PT, true, false>(P, d, sw, m, tid, nthr, 0.0, nullptr, false, true, rr_acc, rz_acc);
    } else {
      double alpha = 0.0;
      const double *pn = P.p0;
      if (UPDATE && !load_alpha(P, alpha)) return;
      group_sweep<PT, false, UPDATE>(P, d, sw, m, tid, nthr, alpha, pn, false, MODE == M_FWD || !sw.fit,
                                     rr_acc, rz_acc);
      if (MODE == M_FUSED) {
        // the last color: y of a fitting group stays in shared memory; the
        // backward sweep restages the U side (the schedule changes, 1/L_ii
        // stays)
        const bool keep = sw.fit;
        const Sweep<PT> su = sweep_static<PT>(P, d, true, m, tid, nthr);
        cp_wait_all();
        __syncthreads();
        group_sweep<PT, true, false>(P, d, su, m, tid, nthr, 0.0, nullptr, keep, true, rr_acc, rz_acc);
      }
    }
  } else {
    pdl_wait();
  }
  if (MODE != M_FWD) launch_epilogue(P, fin, sa, rr_acc, rz_acc, red, &flag);
}

// ---------------------------------------------------------------------------
// lane-tile kernels: one CTA per tile of up to 32 blocks of one color, one
// block per lane (Alg. 1: blocks of a color in parallel, rows of a block in
// sequence).  Step k of the tile is the k-th row of every block; its 32 rows
// are consecutive.
//   A  all warps, steps in parallel: the x / r update, the entries to other
//      colors (gathers of y or z), 1/L_ii and the step's in-block entries
//      into shared memory;
//   B  one warp: the in-block recurrence, step after step, every lane on its
//      own block, shared memory only (no barrier inside);
//   C  all warps: results to global memory, <r,z>.
// ---------------------------------------------------------------------------
template <typename PT> __device__ __forceinline__ const PT *slv(const Params &P);
template <> __device__ __forceinline__ const double *slv<double>(const Params &P) { return P.sl_val; }
template <> __device__ __forceinline__ const float *slv<float>(const Params &P) { return P.sl_val32; }
template <typename PT> __device__ __forceinline__ const PT *suv(const Params &P);
template <> __device__ __forceinline__ const double *suv<double>(const Params &P) { return P.su_val; }
template <> __device__ __forceinline__ const float *suv<float>(const Params &P) { return P.su_val32; }
template <typename PT> __device__ __forceinline__ const PT *siv(const Params &P);
template <> __device__ __forceinline__ const double *siv<double>(const Params &P) { return P.si_val; }
template <> __device__ __forceinline__ const float *siv<float>(const Params &P) { return P.si_val32; }
template <typename PT> __device__ __forceinline__ const PT *uiv(const Params &P);
template <> __device__ __forceinline__ const double *uiv<double>(const Params &P) { return P.ui_val; }
template <> __device__ __forceinline__ const float *uiv<float>(const Params &P) { return P.ui_val32; }

__device__ __forceinline__ TileDesc load_tile(const TileDesc *t) {
  const int4 *p = reinterpret_cast<const int4 *>(t);
  const int4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), d = __ldg(p + 3);
  TileDesc r;
  r.row0 = a.x; r.nrows = a.y; r.nsteps = a.z; r.step0 = a.w;
  r.lo0 = b.x; r.lo1 = b.y; r.li0 = b.z; r.li1 = b.w;
  r.uo0 = c.x; r.uo1 = c.y; r.ui0 = c.z; r.ui1 = c.w;
  r.wl = d.x; r.wu = d.y; r.lw0 = d.z; r.uw0 = d.w;
  return r;
}

// One staged buffer of a tile: step descriptors, 1/L_ii (index row - bdv),
// in-block entries of the first and second set (index entry - base).
template <typename PT>
struct TileBuf {
  const StepDesc *st;
  const PT *dv;
  const int32_t *ic, *ic2;
  const PT *iv, *iv2;
  const int32_t *oc;     // other-color entries (cap_o > 0)
  const PT *ov;
  const double *vec;     // four row vectors of (cap_r + 8) doubles each
  int vstride;
};

template <typename PT>
__device__ __forceinline__ TileBuf<PT> tile_buf(unsigned char *smem, const TilePlan &pl, int size, int k) {
  unsigned char *b = smem + k * size;
  TileBuf<PT> t;
  t.st = reinterpret_cast<const StepDesc *>(b + pl.o_steps);
  t.dv = reinterpret_cast<const PT *>(b + pl.o_dv);
  t.ic = reinterpret_cast<const int32_t *>(b + pl.o_ic);
  t.iv = reinterpret_cast<const PT *>(b + pl.o_iv);
  t.ic2 = reinterpret_cast<const int32_t *>(b + pl.o_ic2);
  t.iv2 = reinterpret_cast<const PT *>(b + pl.o_iv2);
  t.oc = reinterpret_cast<const int32_t *>(b + pl.o_oc);
  t.ov = reinterpret_cast<const PT *>(b + pl.o_ov);
  t.vec = reinterpret_cast<const double *>(b + pl.o_vec);
  t.vstride = r16b((pl.cap_r + 8) * 8) / 8;
  return t;
}

// Whether tile t's other-color entries and row vectors are (to be) staged
__device__ __forceinline__ bool ext_staged(const TilePlan &pl, const TileDesc &t, bool upper) {
  const int n = upper ? t.uo1 - t.uo0 : t.lo1 - t.lo0;
  return pl.cap_o > 0 && n <= pl.cap_o && t.nrows <= pl.cap_r;
}

// Issue (no commit) the copies of tile t's static data into buffer tb:
// steps, 1/L_ii, in-block entries of L (FIRST_UPPER = false) or U, and of U
// as the second set when TWO; an in-block range larger than the capacity
// stays in global memory.
template <typename PT, bool FIRST_UPPER, bool TWO>
__device__ __forceinline__ void tile_stage(const Params &P, const TileDesc &t, const TileBuf<PT> &tb,
                                           const TilePlan &pl, int tid, int nthr) {
  const int cap_i = pl.cap_i, cap_i2 = pl.cap_i2;
  int4 *st = reinterpret_cast<int4 *>(const_cast<StepDesc *>(tb.st));
  const int4 *gs = reinterpret_cast<const int4 *>(P.steps + t.step0);
  for (int k = tid; k < t.nsteps * 3; k += nthr) cp_async16(st + k, gs + k);
  stage_cover<PT>(invds<PT>(P), t.row0, t.row0 + t.nrows, const_cast<PT *>(tb.dv), tid, nthr);
  // entries to other colors of the first sweep (static, like the above)
  if (ext_staged(pl, t, FIRST_UPPER)) {
    const int o0 = FIRST_UPPER ? t.uo0 : t.lo0, o1 = FIRST_UPPER ? t.uo1 : t.lo1;
    if (o1 > o0) {
      stage_cover<int32_t>(FIRST_UPPER ? P.su_col : P.sl_col, o0, o1, const_cast<int32_t *>(tb.oc), tid, nthr);
      stage_cover<PT>(FIRST_UPPER ? suv<PT>(P) : slv<PT>(P), o0, o1, const_cast<PT *>(tb.ov), tid, nthr);
    }
  }
  // a set is copied only into a region the launch has (capacity > 0) and
  // only when non-empty (the cover of an empty range is still 16 bytes)
  const int i0 = FIRST_UPPER ? t.ui0 : t.li0, i1 = FIRST_UPPER ? t.ui1 : t.li1;
  if (i1 > i0 && i1 - i0 <= cap_i) {
    stage_cover<int32_t>(FIRST_UPPER ? P.ui_col : P.si_col, i0, i1, const_cast<int32_t *>(tb.ic), tid, nthr);
    stage_cover<PT>(FIRST_UPPER ? uiv<PT>(P) : siv<PT>(P), i0, i1, const_cast<PT *>(tb.iv), tid, nthr);
  }
  if (TWO && t.ui1 > t.ui0 && t.ui1 - t.ui0 <= cap_i2) {
    stage_cover<int32_t>(P.ui_col, t.ui0, t.ui1, const_cast<int32_t *>(tb.ic2), tid, nthr);
    stage_cover<PT>(uiv<PT>(P), t.ui0, t.ui1, const_cast<PT *>(tb.iv2), tid, nthr);
  }
}

// Issue (no commit) the copies of the row vectors tile t's first sweep reads
// (r, q, x, p forward; y, r backward) when its entries are staged.  They come
// from earlier launches, so the first tile's are issued after
// griddepcontrol.wait; each tile's rows are written by that tile alone.
template <typename PT, bool FIRST_UPPER, bool UPD>
__device__ __forceinline__ void tile_stage_vec(const Params &P, const TileDesc &t, const TileBuf<PT> &tb,
                                               const TilePlan &pl, int tid, int nthr) {
  if (!ext_staged(pl, t, FIRST_UPPER)) return;
  double *v = const_cast<double *>(tb.vec);
  const int r0 = t.row0, r1 = t.row0 + t.nrows, vs = tb.vstride;
  if (FIRST_UPPER) {
    stage_cover<PT>(reinterpret_cast<const PT *>(P.y), r0, r1, reinterpret_cast<PT *>(v), tid, nthr);
    stage_cover<double>(P.r, r0, r1, v + vs, tid, nthr);
  } else {
    stage_cover<double>(P.r, r0, r1, v, tid, nthr);
    if (UPD) {
      stage_cover<double>(P.q, r0, r1, v + vs, tid, nthr);
      stage_cover<double>(P.xh, r0, r1, v + 2 * vs, tid, nthr);
      stage_cover<double>(P.p0, r0, r1, v + 3 * vs, tid, nthr);
    }
  }
}

// The in-block entries a tile's chain reads: staged (index entry - base) or
// the global arrays.
template <typename PT>
struct InBlock {
  const int32_t *ic;
  const PT *iv;
};

template <typename PT>
__device__ __forceinline__ InBlock<PT> in_block(const int32_t *sc, const PT *sv, const int32_t *gc, const PT *gv,
                                               int i0, int i1, int cap_i) {
  if (i1 > i0 && i1 - i0 <= cap_i) return InBlock<PT>{sc - cover_base<int32_t>(i0), sv - cover_base<PT>(i0)};
  return InBlock<PT>{gc, gv};
}

// acc -= sum over a step's sliced-ELL entries to other colors of v * g[col]
// (coalesced loads of the entries, then the gathers; FMAs only for the
// step's real width, a warp-uniform count; padding entries are (kPadCol, 0))
// (NC: col / val in global memory, read through the read-only path; else
// shared-memory copies, plain loads)
template <typename PT, bool NC = true>
__device__ __forceinline__ PT ext_sub(const int32_t *col, const PT *val, int e, int stride, int width, PT acc,
                                      const PT *g) {
  for (int j0 = 0; j0 < width; j0 += kChunk) {
    const int nj = min(kChunk, width - j0);
    int cc[kChunk];
    PT vv[kChunk], xx[kChunk];
#pragma unroll
    for (int j = 0; j < kChunk; ++j) {
      if (NC) {
        cc[j] = j < nj ? __ldg(col + e + (j0 + j) * stride) : kPadCol;
        vv[j] = j < nj ? __ldg(val + e + (j0 + j) * stride) : PT(0);
      } else {
        cc[j] = j < nj ? col[e + (j0 + j) * stride] : kPadCol;
        vv[j] = j < nj ? val[e + (j0 + j) * stride] : PT(0);
      }
    }
#pragma unroll
    for (int j = 0; j < kChunk; ++j) xx[j] = cc[j] == kPadCol ? PT(0) : __ldcg(g + cc[j]);
#pragma unroll
    for (int j = 0; j < kChunk; ++j)
      if (j < nj) acc -= vv[j] * xx[j];
  }
  return acc;
}

// Phase A: forward (UPPER = false; source r with the x / r update when
// UPDATE, gathers of y) or backward (source y from w or global memory,
// gathers of z); the partial row value goes to w[step][lane].
template <typename PT, bool UPPER, bool UPDATE>
__device__ __forceinline__ void tile_phase_a(const Params &P, const TileDesc &t, const TileBuf<PT> &tb, PT *w,
                                             double alpha, const double *pn, bool y_in_smem, bool staged,
                                             int warp, int W) {
  const int lane = threadIdx.x & 31;
  PT *yv = reinterpret_cast<PT *>(P.y);
  const PT *zv = reinterpret_cast<const PT *>(P.z);
  // entries to other colors and row vectors: the staged copies (indexed by
  // global entry / row) or global memory
  const int o0 = UPPER ? t.uo0 : t.lo0;
  const int32_t *oc_s = tb.oc - cover_base<int32_t>(o0), *oc_g = UPPER ? P.su_col : P.sl_col;
  const PT *ov_s = tb.ov - cover_base<PT>(o0), *ov_g = UPPER ? suv<PT>(P) : slv<PT>(P);
  const int vs = tb.vstride;
  const double *v0 = tb.vec - cover_base<double>(t.row0);
  const PT *ys = reinterpret_cast<const PT *>(tb.vec) - cover_base<PT>(t.row0);
  for (int k = warp; k < t.nsteps; k += W) {
    const StepDesc &s = tb.st[k];
    const int cnt = s.cnt;
    if (lane < cnt) {
      const int i = s.row + lane;
      PT acc;
      if (UPPER) {
        PT src;
        if (y_in_smem) src = w[k * kWarp + lane];
        else if (staged) src = ys[i];
        else src = __ldcg(yv + i);
        if (staged) acc = ext_sub<PT, false>(oc_s, ov_s, s.uo + lane, cnt, s.uw, src, zv);
        else acc = ext_sub<PT>(oc_g, ov_g, s.uo + lane, cnt, s.uw, src, zv);
      } else {
        double ri;
        if (staged) {
          ri = v0[i];
          if (UPDATE) {
            ri -= alpha * v0[vs + i];
            P.r[i] = ri;
            P.xh[i] = v0[2 * vs + i] + alpha * v0[3 * vs + i];
          }
          acc = ext_sub<PT, false>(oc_s, ov_s, s.lo + lane, cnt, s.lw, PT(ri), yv);
        } else {
          ri = __ldcg(P.r + i);
          if (UPDATE) {
            ri -= alpha * __ldcg(P.q + i);
            P.r[i] = ri;
            P.xh[i] = __ldcg(P.xh + i) + alpha * __ldcg(pn + i);
          }
          acc = ext_sub<PT>(oc_g, ov_g, s.lo + lane, cnt, s.lw, PT(ri), yv);
        }
      }
      w[k * kWarp + lane] = acc;
    }
  }
}

// Phase B: warp 0 resolves the in-block recurrence, steps ascending (forward)
// or descending (backward), from shared memory only; a lane reads only its
// own block's values.  In-block padding entries are (step 0, value 0).
template <typename PT, bool UPPER>
__device__ __forceinline__ void tile_phase_b(const TileDesc &t, const StepDesc *st, const PT *dv,
                                             const int32_t *ic, const PT *iv, PT *w, int lane) {
  for (int kk = 0; kk < t.nsteps; ++kk) {
    const int k = UPPER ? t.nsteps - 1 - kk : kk;
    const StepDesc &s = st[k];
    const int cnt = s.cnt, wi = UPPER ? s.uiw : s.liw, e = (UPPER ? s.ui : s.li) + lane;
    if (lane < cnt) {
      PT acc = w[k * kWarp + lane];
      for (int j = 0; j < wi; ++j) acc -= iv[e + j * cnt] * w[ic[e + j * cnt] * kWarp + lane];
      w[k * kWarp + lane] = acc * dv[s.row + lane];
    }
  }
}

// Phase C: the tile's results to global memory (y or z), <r,z> and <r,r>
// (backward; rs: the staged r)
template <typename PT, bool UPPER>
__device__ __forceinline__ void tile_phase_c(const Params &P, const TileDesc &t, const StepDesc *st, const PT *w,
                                             const double *rs, double &rr_acc, double &rz_acc, int warp, int W) {
  const int lane = threadIdx.x & 31;
  PT *res = reinterpret_cast<PT *>(UPPER ? P.z : P.y);
  for (int k = warp; k < t.nsteps; k += W) {
    const StepDesc &s = st[k];
    if (lane < s.cnt) {
      const int i = s.row + lane;
      const PT v = w[k * kWarp + lane];
      if (UPPER) {
        double ri;
        if (rs) ri = rs[i];
        else ri = __ldcg(P.r + i);
        res[i] = v;
        rz_add(ri, v, rr_acc, rz_acc);
      } else {
        res[i] = v;
      }
    }
  }
}

// Static shared memory of a lane-tile launch that reduces (red and flag).  CTAs of
// one warp (ONE; one-row blocks) have only what one warp needs: with 784 bytes they
// lost a place on an SM to it (27-point 124^3, FP32, 40 iterations 17.3 ms, so
// 15.7).  Forward launches reduce nothing; they get the same bytes as dynamic
// shared memory.  The grid is one CTA for every place on the SMs: with room left
// beside a full grid the next launch's first CTAs start there, and some SMs end up
// with more of them than others (110^3, FP64 18.7 ms; so 15.9).
constexpr int tile_red_bytes(bool one) { return (one ? kRedWarp : kRed) * 8 + 16; }

// A lane-tile launch: CTAs walk the color's tiles grid-stride; the static
// data of the next tile is copied into the other buffer while the current one
// is computed (the first tile's before griddepcontrol.wait); one <r,r> /
// <r,z> reduction per CTA at the end.
template <typename PT, int MODE, bool UPDATE, bool ONE>
__global__ void __launch_bounds__(kMaxWarpsPerCta * kWarp)
tile_kernel(Params P, int t0, int t1, TilePlan pl, int fin, SlotArgs sa) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[ONE ? kRedWarp : kRed];
  __shared__ int flag;
  constexpr bool FU = MODE == M_BWD, TWO = MODE == M_FUSED;
  const int bsize = TWO && pl.cap_i2 > 0 ? pl.buf2 : pl.buf1;
  const int nbuf = pl.nbuf;
  PT *w = reinterpret_cast<PT *>(smem + nbuf * bsize);
  double rr_acc = 0.0, rz_acc = 0.0;
  int t = t0 + int(blockIdx.x), buf = 0;
  const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  TileDesc td = load_tile(P.tiles + min(t, t1 - 1));
  if (t < t1) tile_stage<PT, FU, TWO>(P, td, tile_buf<PT>(smem, pl, bsize, 0), pl, threadIdx.x, blockDim.x);
  pdl_wait();
  if (t < t1) tile_stage_vec<PT, FU, UPDATE>(P, td, tile_buf<PT>(smem, pl, bsize, 0), pl, threadIdx.x, blockDim.x);
  cp_commit();
  double alpha = 0.0;
  if (UPDATE && !load_alpha(P, alpha)) {
    cp_wait_all();
    return;
  }
  for (; t < t1; t += gridDim.x) {
    const int tn = t + int(gridDim.x);
    TileDesc tdn = td;
    if (tn < t1) tdn = load_tile(P.tiles + tn);
    if (tn < t1 && nbuf == 2) {
      tile_stage<PT, FU, TWO>(P, tdn, tile_buf<PT>(smem, pl, bsize, buf ^ 1), pl, threadIdx.x, blockDim.x);
      tile_stage_vec<PT, FU, UPDATE>(P, tdn, tile_buf<PT>(smem, pl, bsize, buf ^ 1), pl, threadIdx.x, blockDim.x);
    }
    cp_commit();
    cp_wait_prev();
    __syncthreads();
    const TileBuf<PT> tb = tile_buf<PT>(smem, pl, bsize, buf);
    const PT *dv = tb.dv - cover_base<PT>(td.row0);
    const InBlock<PT> ul = in_block<PT>(tb.ic, tb.iv, P.ui_col, uiv<PT>(P), td.ui0, td.ui1, pl.cap_i);
    const InBlock<PT> ll = in_block<PT>(tb.ic, tb.iv, P.si_col, siv<PT>(P), td.li0, td.li1, pl.cap_i);
    const bool stg = ext_staged(pl, td, MODE == M_BWD);
    if (MODE == M_BWD) {
      tile_phase_a<PT, true, false>(P, td, tb, w, 0.0, nullptr, false, stg, wid, nw);
      __syncthreads();
      if (wid == 0) tile_phase_b<PT, true>(td, tb.st, dv, ul.ic, ul.iv, w, threadIdx.x);
      __syncthreads();
      tile_phase_c<PT, true>(P, td, tb.st, w, stg ? tb.vec + tb.vstride - cover_base<double>(td.row0) : nullptr,
                             rr_acc, rz_acc, wid, nw);
    } else {
      tile_phase_a<PT, false, UPDATE>(P, td, tb, w, alpha, P.p0, false, stg, wid, nw);
      __syncthreads();
      if (wid == 0) tile_phase_b<PT, false>(td, tb.st, dv, ll.ic, ll.iv, w, threadIdx.x);
      __syncthreads();
      if (MODE == M_FWD) {
        tile_phase_c<PT, false>(P, td, tb.st, w, nullptr, rr_acc, rz_acc, wid, nw);
      } else {
        // the last color: y stays in shared memory for the backward sweep
        // (its entries to other colors from global memory: the staged set is L's)
        const InBlock<PT> u2 = in_block<PT>(tb.ic2, tb.iv2, P.ui_col, uiv<PT>(P), td.ui0, td.ui1, pl.cap_i2);
        tile_phase_a<PT, true, false>(P, td, tb, w, 0.0, nullptr, true, false, wid, nw);
        __syncthreads();
        if (wid == 0) tile_phase_b<PT, true>(td, tb.st, dv, u2.ic, u2.iv, w, threadIdx.x);
        __syncthreads();
        tile_phase_c<PT, true>(P, td, tb.st, w, nullptr, rr_acc, rz_acc, wid, nw);
      }
    }
    __syncthreads();   // buffer buf and w are reused by the next tile
    if (nbuf == 1) {
      // one buffer: the next tile's copies start now (waited on by the next
      // pass's cp_wait_prev, which leaves only its own empty group pending)
      if (tn < t1) {
        tile_stage<PT, FU, TWO>(P, tdn, tile_buf<PT>(smem, pl, bsize, 0), pl, threadIdx.x, blockDim.x);
        tile_stage_vec<PT, FU, UPDATE>(P, tdn, tile_buf<PT>(smem, pl, bsize, 0), pl, threadIdx.x, blockDim.x);
      }
      cp_commit();
    } else {
      buf ^= 1;
    }
    td = tdn;
  }
  cp_wait_all();
  if (MODE != M_FWD) launch_epilogue(P, fin, sa, rr_acc, rz_acc, red, &flag);
}

// ---------------------------------------------------------------------------
// warp-tile kernels: one warp per lane tile, all of the tile's steps in order
// by that warp (Alg. 1 again: a lane per block, the block's rows in
// sequence).  For colors of many tiles with few steps (blocks of a few rows)
// this keeps every warp of a CTA busy where the CTA-per-tile kernel spreads
// the steps of one tile over its warps; no barrier, and a lane's in-block
// values stay in its own column of the warp's shared-memory buffer.
// ---------------------------------------------------------------------------
__device__ __forceinline__ StepDesc load_step_g(const StepDesc *s) {
  const int4 *p = reinterpret_cast<const int4 *>(s);
  const int4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
  StepDesc r;
  r.row = a.x; r.cnt = a.y; r.lo = a.z; r.lw = a.w;
  r.li = b.x; r.liw = b.y; r.uo = b.z; r.uw = b.w;
  r.ui = c.x; r.uiw = c.y; r.pad0 = r.pad1 = 0;
  return r;
}

// One sweep over tile t by one warp.  Forward (UPPER = false): source r (with
// the x / r update when UPDATE), entries to earlier colors gathered from y,
// in-block entries from wv; result y.  Backward: source y (from wv when
// y_in_smem, the fused last color), gathers of z, result z, <r,z> and <r,r>.
// wv[step * 32 + lane] keeps the lane's own values of the tile.
template <typename PT, bool UPPER, bool UPDATE>
__device__ __forceinline__ void wtile_sweep(const Params &P, const TileDesc &t, PT *wv, double alpha,
                                            bool y_in_smem, bool store, double &rr_acc, double &rz_acc, int lane) {
  PT *res = reinterpret_cast<PT *>(UPPER ? P.z : P.y);
  const PT *ext = reinterpret_cast<const PT *>(UPPER ? P.z : P.y);
  const PT *yv = reinterpret_cast<const PT *>(P.y);
  const PT *dvg = invds<PT>(P);
  const int32_t *icol = UPPER ? P.ui_col : P.si_col;
  const PT *ival = UPPER ? uiv<PT>(P) : siv<PT>(P);
  // in-block padding entries are (step 0, value 0): a backward sweep reads
  // step 0 before computing it, so it must hold a finite value (forward
  // sweeps and the fused one have written it by then)
  if (UPPER && !y_in_smem) {
    for (int k = 0; k < t.nsteps; ++k) wv[k * kWarp + lane] = PT(0);
    __syncwarp();
  }
  for (int kk = 0; kk < t.nsteps; ++kk) {
    const int k = UPPER ? t.nsteps - 1 - kk : kk;
    StepDesc s;
    if (t.nsteps == 1) {
      s.row = t.row0; s.cnt = t.nrows; s.lo = t.lo0; s.lw = t.lw0; s.li = t.li0; s.liw = t.wl;
      s.uo = t.uo0; s.uw = t.uw0; s.ui = t.ui0; s.uiw = t.wu;
    } else {
      s = load_step_g(P.steps + t.step0 + k);
    }
    if (lane < s.cnt) {
      const int i = s.row + lane;
      PT acc;
      if (UPPER) {
        const PT src = y_in_smem ? wv[k * kWarp + lane] : __ldcg(yv + i);
        acc = ext_sub<PT>(P.su_col, suv<PT>(P), s.uo + lane, s.cnt, s.uw, src, ext);
      } else {
        double ri = __ldcg(P.r + i);
        if (UPDATE) {
          ri -= alpha * __ldcg(P.q + i);
          P.r[i] = ri;
          P.xh[i] = __ldcg(P.xh + i) + alpha * __ldcg(P.p0 + i);
        }
        acc = ext_sub<PT>(P.sl_col, slv<PT>(P), s.lo + lane, s.cnt, s.lw, PT(ri), ext);
      }
      const int wi = UPPER ? s.uiw : s.liw, e = (UPPER ? s.ui : s.li) + lane;
      for (int j = 0; j < wi; ++j) acc -= __ldg(ival + e + j * s.cnt) * wv[__ldg(icol + e + j * s.cnt) * kWarp + lane];
      const PT v = acc * __ldg(dvg + i);
      wv[k * kWarp + lane] = v;
      if (store) res[i] = v;
      if (UPPER) rz_add(__ldcg(P.r + i), v, rr_acc, rz_acc);
    }
  }
}

// A warp-tile launch: the warps walk the color's tiles grid-stride (tile of
// warp w of CTA b: t0 + b * W + w, then + gridDim.x * W); one <r,r> / <r,z>
// reduction per CTA at the end.  Shared memory: cap_s * 32 values per warp.
#ifndef ICCG_TILE_MAXNREG
#define ICCG_TILE_MAXNREG 64
#endif

template <typename PT, int MODE, bool UPDATE>
__global__ void __maxnreg__(ICCG_TILE_MAXNREG)
wtile_kernel(Params P, int t0, int t1, int cap_s, int fin, SlotArgs sa) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[kRed];
  __shared__ int flag;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  PT *wv = reinterpret_cast<PT *>(smem) + size_t(wid) * cap_s * kWarp;
  double rr_acc = 0.0, rz_acc = 0.0;
  int t = t0 + int(blockIdx.x) * nw + wid;
  const bool end = MODE == M_BWD && sweep_ended(P, sa);
  TileDesc td = load_tile(P.tiles + min(t, t1 - 1));
  pdl_wait();
  if (MODE == M_BWD && __any_sync(0xffffffffu, end)) t = t1;
  double alpha = 0.0;
  if (UPDATE && !load_alpha(P, alpha)) return;
  for (; t < t1; t += int(gridDim.x) * nw) {
    const int tn = t + int(gridDim.x) * nw;
    const TileDesc tdn = tn < t1 ? load_tile(P.tiles + tn) : td;
    if (MODE == M_BWD) {
      wtile_sweep<PT, true, false>(P, td, wv, 0.0, false, true, rr_acc, rz_acc, lane);
    } else {
      wtile_sweep<PT, false, UPDATE>(P, td, wv, alpha, false, MODE == M_FWD, rr_acc, rz_acc, lane);
      __syncwarp();
      if (MODE == M_FUSED) wtile_sweep<PT, true, false>(P, td, wv, 0.0, true, true, rr_acc, rz_acc, lane);
    }
    __syncwarp();
    td = tdn;
  }
  if (MODE != M_FWD) launch_epilogue(P, fin, sa, rr_acc, rz_acc, red, &flag);
}

// ---------------------------------------------------------------------------
// pair kernels: colors of blocks of one or two rows (tiles of at most two
// steps).  A warp per tile, a lane per block, the block's rows in registers:
// forward
//   y0 = (r0 - sum_j L0j y_j) / L00
//   y1 = (r1 - sum_j L1j y_j - L10 y0) / L11
// (the sums over earlier colors), backward
//   z1 = (y1 - sum_j Lj1 z_j) / L11
//   z0 = (y0 - sum_j Lj0 z_j - L10 z1) / L00
// (the sums over later colors); a one-row block is its step 0 alone.
// Padding entries (kPadCol, 0) add 0 * an element the sweep has already
// written: y_0 (first color) forward, z_{n-1} (last color) backward.
// ---------------------------------------------------------------------------
// a descriptor whose first 16 bytes (first row, block counts) are already
// in registers
__device__ __forceinline__ PairDesc load_pair_rest(const PairDesc *p, int4 a) {
  const int4 *q = reinterpret_cast<const int4 *>(p);
  const int4 b = __ldg(q + 1), c = __ldg(q + 2), d = __ldg(q + 3);
  PairDesc r;
  r.row0 = a.x; r.c0 = a.y; r.c1 = a.z; r.lo = a.w;
  r.lw0 = b.x; r.lw1 = b.y; r.li = b.z; r.liw1 = b.w;
  r.uo = c.x; r.uw0 = c.y; r.uw1 = c.z; r.ui = c.w;
  r.uiw0 = d.x; r.pad0 = r.pad1 = r.pad2 = 0;
  return r;
}
__device__ __forceinline__ int4 pair_head(const PairDesc *p) { return __ldg(reinterpret_cast<const int4 *>(p)); }
__device__ __forceinline__ PairDesc load_pair(const PairDesc *p) { return load_pair_rest(p, pair_head(p)); }

template <typename PT>
__device__ __forceinline__ PT pair_sub(const int32_t *col, const PT *val, int e, int cnt, int w, PT acc,
                                       const PT *g, int pad) {
#pragma unroll 4
  for (int j = 0; j < w; ++j) {
    const int c = __ldg(col + e + j * cnt);
    const PT v = __ldg(val + e + j * cnt);
    acc -= v * __ldcg(g + (c == kPadCol ? pad : c));
  }
  return acc;
}

// backward over one tile from y0 (and y1 when a1): stores z, adds <r,z>
// and <r,r>
template <typename PT>
__device__ __forceinline__ void pair_bwd(const Params &P, const PairDesc &d, int lane, bool a1, PT y0, PT y1,
                                         PT dv0, PT dv1, double r0, double r1, double &rr_acc,
                                         double &rz_acc) {
  PT *zv = reinterpret_cast<PT *>(P.z);
  const int i0 = d.row0 + lane, i1 = d.row0 + d.c0 + lane;
  // both steps' gathers before any store (a store to z would order the
  // other step's gathers after it)
  PT acc0 = pair_sub<PT>(P.su_col, suv<PT>(P), d.uo + lane, d.c0, d.uw0, y0, zv, P.n - 1);
  PT z1 = PT(0);
  if (a1) z1 = pair_sub<PT>(P.su_col, suv<PT>(P), d.uo + d.uw0 * d.c0 + lane, d.c1, d.uw1, y1, zv, P.n - 1) * dv1;
  for (int j = 0; j < d.uiw0; ++j) acc0 -= __ldg(uiv<PT>(P) + d.ui + j * d.c0 + lane) * z1;
  const PT z0 = acc0 * dv0;
  zv[i0] = z0;
  if (a1) zv[i1] = z1;
  rz_add(r0, z0, rr_acc, rz_acc);
  if (a1) rz_add(r1, z1, rr_acc, rz_acc);
}

// one tile of a pair color, warp-wide (lanes beyond the tile's blocks idle)
template <typename PT, int MODE, bool UPDATE>
__device__ __forceinline__ void pair_tile_h(const Params &P, int t, int4 head, int lane, double alpha,
                                            double &rr_acc, double &rz_acc) {
  PT *yv = reinterpret_cast<PT *>(P.y);
  const PT *dvg = invds<PT>(P);
  const PairDesc d = load_pair_rest(P.pairs + t, head);
  if (lane >= d.c0) return;   // a lane active in step 1 is active in step 0
  const bool a1 = lane < d.c1;
  const int i0 = d.row0 + lane, i1 = d.row0 + d.c0 + lane;
  const PT dv0 = __ldg(dvg + i0), dv1 = a1 ? __ldg(dvg + i1) : PT(0);
  if (MODE == M_BWD) {
    const PT y0 = __ldcg(yv + i0), y1 = a1 ? __ldcg(yv + i1) : PT(0);
    const double r0 = __ldcg(P.r + i0), r1 = a1 ? __ldcg(P.r + i1) : 0.0;
    pair_bwd<PT>(P, d, lane, a1, y0, y1, dv0, dv1, r0, r1, rr_acc, rz_acc);
  } else {
    double r0 = __ldcg(P.r + i0), r1 = a1 ? __ldcg(P.r + i1) : 0.0;
    if (UPDATE) {
      r0 -= alpha * __ldcg(P.q + i0);
      P.r[i0] = r0;
      P.xh[i0] = __ldcg(P.xh + i0) + alpha * __ldcg(P.p0 + i0);
      if (a1) {
        r1 -= alpha * __ldcg(P.q + i1);
        P.r[i1] = r1;
        P.xh[i1] = __ldcg(P.xh + i1) + alpha * __ldcg(P.p0 + i1);
      }
    }
    const PT y0 = pair_sub<PT>(P.sl_col, slv<PT>(P), d.lo + lane, d.c0, d.lw0, PT(r0), yv, 0) * dv0;
    PT y1 = PT(0);
    if (a1) {
      PT acc1 = pair_sub<PT>(P.sl_col, slv<PT>(P), d.lo + d.lw0 * d.c0 + lane, d.c1, d.lw1, PT(r1), yv, 0);
      for (int j = 0; j < d.liw1; ++j) acc1 -= __ldg(siv<PT>(P) + d.li + j * d.c1 + lane) * y0;
      y1 = acc1 * dv1;
    }
    if (MODE == M_FWD) {
      yv[i0] = y0;
      if (a1) yv[i1] = y1;
    } else {
      pair_bwd<PT>(P, d, lane, a1, y0, y1, dv0, dv1, r0, r1, rr_acc, rz_acc);
    }
  }
}

template <typename PT, int MODE, bool UPDATE>
__device__ __forceinline__ void pair_tile(const Params &P, int t, int lane, double alpha, double &rr_acc,
                                          double &rz_acc) {
  pair_tile_h<PT, MODE, UPDATE>(P, t, pair_head(P.pairs + t), lane, alpha, rr_acc, rz_acc);
}

// The staged pair kernel (pair_kernel<.., STAGE = true>, chosen per color
// and sweep on the host) loads each tile's static data ahead of its
// gathers: the descriptor, the pivots' reciprocals and in-block coefficient
// in registers, and the first kPairStage entries of each step (the sums over
// the other colors: lower for the forward sweep, upper for the backward) in
// the warp's shared-memory buffer by cp.async.  The warp's first tile is
// staged before griddepcontrol.wait, so these loads overlap the previous
// launch; after the wait a tile's gathers of both steps and its row vectors
// are in flight together.  Wider steps take their remaining entries from
// global memory.  The unstaged kernel (pair_tile_h) keeps the loads in the
// order the recurrence uses them and serves sweeps with few such entries.
constexpr int kPairStage = 6;   // a 7-point row has at most 6 entries to other blocks

template <typename PT>
struct PairStage {
  int32_t col[2][kPairStage][kWarp];
  PT val[2][kPairStage][kWarp];
};

template <typename PT>
struct PairPre {
  PairDesc d;
  PT dv0, dv1, e;   // 1/L_00, 1/L_11 and the in-block coefficient of the sweep
};

template <typename PT, bool BWD>
__device__ __forceinline__ PairPre<PT> pair_stage(const Params &P, int t, int lane, PairStage<PT> &s) {
  PairPre<PT> q;
  q.d = load_pair(P.pairs + t);
  const PairDesc &d = q.d;
  q.dv0 = q.dv1 = q.e = PT(0);
  if (lane < d.c0) {
    const bool a1 = lane < d.c1;
    const PT *dvg = invds<PT>(P);
    q.dv0 = __ldg(dvg + d.row0 + lane);
    if (a1) q.dv1 = __ldg(dvg + d.row0 + d.c0 + lane);
    const int32_t *col = BWD ? P.su_col : P.sl_col;
    const PT *val = BWD ? suv<PT>(P) : slv<PT>(P);
    const int b0 = BWD ? d.uo : d.lo, w0 = BWD ? d.uw0 : d.lw0, w1 = BWD ? d.uw1 : d.lw1;
    const int n0 = min(w0, kPairStage), n1 = a1 ? min(w1, kPairStage) : 0;
    for (int j = 0; j < n0; ++j) {
      cp_async4(&s.col[0][j][lane], col + b0 + j * d.c0 + lane);
      cp_async_elem<PT>(&s.val[0][j][lane], val + b0 + j * d.c0 + lane);
    }
    const int b1 = b0 + w0 * d.c0;
    for (int j = 0; j < n1; ++j) {
      cp_async4(&s.col[1][j][lane], col + b1 + j * d.c1 + lane);
      cp_async_elem<PT>(&s.val[1][j][lane], val + b1 + j * d.c1 + lane);
    }
    // a block of two rows has at most one in-block entry per row: row 1's
    // to row 0 forward, row 0's to row 1 backward
    if (BWD) {
      if (d.uiw0 > 0) q.e = __ldg(uiv<PT>(P) + d.ui + lane);
    } else {
      if (a1 && d.liw1 > 0) q.e = __ldg(siv<PT>(P) + d.li + lane);
    }
  }
  cp_commit();
  return q;
}

// the staged sums of both steps: every gather issued before the first
// multiply-add; entries past kPairStage from global memory
template <typename PT, bool BWD>
__device__ __forceinline__ void pair_staged_sums(const Params &P, const PairDesc &d, const PairStage<PT> &s,
                                                 int lane, bool a1, PT &acc0, PT &acc1) {
  const PT *g = reinterpret_cast<const PT *>(BWD ? P.z : P.y);
  const int pad = BWD ? P.n - 1 : 0;
  const int w0 = BWD ? d.uw0 : d.lw0, w1 = BWD ? d.uw1 : d.lw1;
  PT g0[kPairStage], g1[kPairStage];
#pragma unroll
  for (int j = 0; j < kPairStage; ++j) {
    g0[j] = PT(0);
    if (j < w0) {
      const int c = s.col[0][j][lane];
      g0[j] = __ldcg(g + (c == kPadCol ? pad : c));
    }
  }
#pragma unroll
  for (int j = 0; j < kPairStage; ++j) {
    g1[j] = PT(0);
    if (a1 && j < w1) {
      const int c = s.col[1][j][lane];
      g1[j] = __ldcg(g + (c == kPadCol ? pad : c));
    }
  }
#pragma unroll
  for (int j = 0; j < kPairStage; ++j)
    if (j < w0) acc0 -= s.val[0][j][lane] * g0[j];
#pragma unroll
  for (int j = 0; j < kPairStage; ++j)
    if (a1 && j < w1) acc1 -= s.val[1][j][lane] * g1[j];
  if (w0 > kPairStage || w1 > kPairStage) {
    const int32_t *col = BWD ? P.su_col : P.sl_col;
    const PT *val = BWD ? suv<PT>(P) : slv<PT>(P);
    const int b0 = BWD ? d.uo : d.lo, b1 = b0 + w0 * d.c0;
    for (int j = kPairStage; j < w0; ++j) {
      const int e = b0 + j * d.c0 + lane, c = __ldg(col + e);
      acc0 -= __ldg(val + e) * __ldcg(g + (c == kPadCol ? pad : c));
    }
    if (a1)
      for (int j = kPairStage; j < w1; ++j) {
        const int e = b1 + j * d.c1 + lane, c = __ldg(col + e);
        acc1 -= __ldg(val + e) * __ldcg(g + (c == kPadCol ? pad : c));
      }
  }
}

template <typename PT, int MODE, bool UPDATE>
__device__ __forceinline__ void pair_tile_staged(const Params &P, const PairPre<PT> &q, const PairStage<PT> &s,
                                                 int lane, double alpha, double &rr_acc, double &rz_acc) {
  const PairDesc &d = q.d;
  if (lane >= d.c0) return;
  const bool a1 = lane < d.c1;
  const int i0 = d.row0 + lane, i1 = d.row0 + d.c0 + lane;
  cp_wait_all();   // the lane's own staged entries (it reads no other lane's)
  if (MODE == M_BWD) {
    const PT *yv = reinterpret_cast<const PT *>(P.y);
    PT acc0 = __ldcg(yv + i0), acc1 = a1 ? __ldcg(yv + i1) : PT(0);
    const double r0 = __ldcg(P.r + i0), r1 = a1 ? __ldcg(P.r + i1) : 0.0;
    pair_staged_sums<PT, true>(P, d, s, lane, a1, acc0, acc1);
    const PT z1 = acc1 * q.dv1;
    acc0 -= q.e * z1;
    for (int j = 1; j < d.uiw0; ++j) acc0 -= __ldg(uiv<PT>(P) + d.ui + j * d.c0 + lane) * z1;
    const PT z0 = acc0 * q.dv0;
    PT *zv = reinterpret_cast<PT *>(P.z);
    zv[i0] = z0;
    if (a1) zv[i1] = z1;
    rz_add(r0, z0, rr_acc, rz_acc);
    if (a1) rz_add(r1, z1, rr_acc, rz_acc);
  } else {
    PT acc0, acc1 = PT(0);
    double r0 = __ldcg(P.r + i0), r1 = a1 ? __ldcg(P.r + i1) : 0.0;
    if (UPDATE) {
      const double q0 = __ldcg(P.q + i0), x0 = __ldcg(P.xh + i0), p0 = __ldcg(P.p0 + i0);
      double q1 = 0.0, x1 = 0.0, p1 = 0.0;
      if (a1) {
        q1 = __ldcg(P.q + i1);
        x1 = __ldcg(P.xh + i1);
        p1 = __ldcg(P.p0 + i1);
      }
      r0 -= alpha * q0;
      if (a1) r1 -= alpha * q1;
      acc0 = PT(r0);
      acc1 = PT(r1);
      pair_staged_sums<PT, false>(P, d, s, lane, a1, acc0, acc1);
      P.r[i0] = r0;
      P.xh[i0] = x0 + alpha * p0;
      if (a1) {
        P.r[i1] = r1;
        P.xh[i1] = x1 + alpha * p1;
      }
    } else {
      acc0 = PT(r0);
      acc1 = PT(r1);
      pair_staged_sums<PT, false>(P, d, s, lane, a1, acc0, acc1);
    }
    const PT y0 = acc0 * q.dv0;
    PT y1 = PT(0);
    if (a1) {
      acc1 -= q.e * y0;
      for (int j = 1; j < d.liw1; ++j) acc1 -= __ldg(siv<PT>(P) + d.li + j * d.c1 + lane) * y0;
      y1 = acc1 * q.dv1;
    }
    PT *yv = reinterpret_cast<PT *>(P.y);
    if (MODE == M_FWD) {
      yv[i0] = y0;
      if (a1) yv[i1] = y1;
    } else {
      pair_bwd<PT>(P, d, lane, a1, y0, y1, q.dv0, q.dv1, r0, r1, rr_acc, rz_acc);
    }
  }
}

template <typename PT>
constexpr int pair_stage_bytes() { return int(sizeof(PairStage<PT>)); }

// Registers a thread: the kernel is bound by the loads in flight, i.e. by the CTAs
// that fit beside one another with the gathers' registers: 9 CTAs of 4 warps an SM
// in FP32 (56 registers), 8 in FP64, fewer for the staged forms with the x / r
// update, which need more.  Left to itself the compiler takes 58 to 64 for some
// FP32 forms (8 CTAs) and 40 for others (fewer loads in flight).  40 iterations in
// FP32, two-row blocks: 27-point 66^3 10.0 ms, so 7.3; graph of degree 16, 200,000
// rows 20.8 and 13.1; FP64 27-point 66^3 8.6 and 8.3.
constexpr int pair_regs(int elem, int mode, bool update, bool stage) {
  if (update && stage) return elem == 8 && mode == M_FUSED ? 96 : 64;
  return elem == 4 ? 56 : 64;
}

template <typename PT, int MODE, bool UPDATE, bool STAGE>
__global__ void __maxnreg__(pair_regs(int(sizeof(PT)), MODE, UPDATE, STAGE))
pair_kernel(Params P, int t0, int t1, int fin, SlotArgs sa) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[kRed];
  __shared__ int flag;
  const int lane = threadIdx.x & 31, wid = int(threadIdx.x >> 5);
  const bool end = MODE == M_BWD && sweep_ended(P, sa);
  const int nw = int(blockDim.x >> 5), stride = int(gridDim.x) * nw;
  double rr_acc = 0.0, rz_acc = 0.0;
  int t = t0 + int(blockIdx.x) * nw + wid;
  if constexpr (STAGE) {
    PairStage<PT> &st = reinterpret_cast<PairStage<PT> *>(smem)[wid];
    PairPre<PT> q;
    if (t < t1) q = pair_stage<PT, MODE == M_BWD>(P, t, lane, st);
    pdl_wait();
    if (MODE == M_BWD && __any_sync(0xffffffffu, end)) {
      cp_wait_all();
      t = t1;
    }
    double alpha = 0.0;
    if (UPDATE && !load_alpha(P, alpha)) {
      cp_wait_all();
      return;
    }
    while (t < t1) {
      pair_tile_staged<PT, MODE, UPDATE>(P, q, st, lane, alpha, rr_acc, rz_acc);
      t += stride;
      __syncwarp();
      if (t < t1) q = pair_stage<PT, MODE == M_BWD>(P, t, lane, st);
    }
  } else {
    // the next tile's first descriptor word (its rows) loads while the
    // current tile runs, the first tile's before the wait
    int4 hn = make_int4(0, 0, 0, 0);
    if (t < t1) hn = pair_head(P.pairs + t);
    pdl_wait();
    if (MODE == M_BWD && __any_sync(0xffffffffu, end)) t = t1;
    double alpha = 0.0;
    if (UPDATE && !load_alpha(P, alpha)) return;
    for (; t < t1; t += stride) {
      const int4 h = hn;
      if (t + stride < t1) hn = pair_head(P.pairs + t + stride);
      pair_tile_h<PT, MODE, UPDATE>(P, t, h, lane, alpha, rr_acc, rz_acc);
    }
  }
  if (MODE != M_FWD) launch_epilogue(P, fin, sa, rr_acc, rz_acc, red, &flag);
}

// ---------------------------------------------------------------------------
// warp-unit kernels: colors of blocks of at most 32 rows.  One warp holds 32 / S
// whole blocks, a lane per row (Alg. 1: the blocks of a color in parallel,
// the rows of a block in order).  A sweep over a unit:
//   A  every lane: its source (r with the x / r update, or y) minus its
//      entries to other colors (sliced-ELL over the warp: coalesced);
//   B  the in-block recurrence as a chain of steps: at every step a lane
//      subtracts at most one in-block term, coefficient x t_k, where t_k is
//      the final value of the term's source row k (read from its lane by a
//      shuffle) and the coefficient is the entry divided by the pivot of
//      row k, so the division of Alg. 1 is applied to each row once, at the
//      end.  The host orders each lane's terms by the step their sources
//      become final, so independent terms of different rows share a step:
//      the chain is about as long as the in-block dependency depth or the
//      widest row, not the block size;
//   C  y = t / L_ii (times 1/L_ii), stored; <r,z> and <r,r> for the backward
//      sweep.
// Every static datum of a unit (descriptor, masks, coefficients, 1/L_ii, the
// first entries to other colors) is loaded before the first dependent access
// (griddepcontrol.wait).  A step at
// which no lane of the warp has a coefficient issues no FP64 instruction.
// ---------------------------------------------------------------------------
template <typename PT> __device__ __forceinline__ const PT *wlv(const Params &P);
template <> __device__ __forceinline__ const double *wlv<double>(const Params &P) { return P.wl_val; }
template <> __device__ __forceinline__ const float *wlv<float>(const Params &P) { return P.wl_val32; }
template <typename PT> __device__ __forceinline__ const PT *wuv(const Params &P);
template <> __device__ __forceinline__ const double *wuv<double>(const Params &P) { return P.wu_val; }
template <> __device__ __forceinline__ const float *wuv<float>(const Params &P) { return P.wu_val32; }

__device__ __forceinline__ WarpUnit load_unit(const WarpUnit *u) {
  const int4 *p = reinterpret_cast<const int4 *>(u);
  const int4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), e = __ldg(p + 3);
  WarpUnit r;
  r.blk0 = a.x; r.nblk = a.y; r.lo = a.z; r.lw = a.w;
  r.uo = b.x; r.uw = b.y; r.li = b.z; r.lm = b.w;
  r.ui = c.x; r.um = c.y; r.row0 = c.z; r.nrows = c.w;
  r.ls = e.x; r.us = e.y; r.lt = e.z; r.ut = e.w;
  return r;
}

constexpr int kUnitChunk = 8;   // entries to other colors per batch of loads

// The first kUnitChunk of a lane's entries to other colors (static: loaded
// before griddepcontrol.wait), their gathers, and the subtraction of all w
// entries (stride 32), the first chunk from x.
template <typename PT>
struct UnitExt {
  int c[kUnitChunk];
  PT v[kUnitChunk];
};
template <typename PT>
__device__ __forceinline__ void unit_ext_load(UnitExt<PT> &q, const int32_t *col, const PT *val, int e, int w) {
#pragma unroll
  for (int j = 0; j < kUnitChunk; ++j) {
    q.c[j] = j < w ? __ldg(col + e + j * kWarp) : kPadCol;
    q.v[j] = j < w ? __ldg(val + e + j * kWarp) : PT(0);
  }
}
template <typename PT>
__device__ __forceinline__ void unit_ext_gather(const UnitExt<PT> &q, PT (&x)[kUnitChunk], const PT *g) {
#pragma unroll
  for (int j = 0; j < kUnitChunk; ++j) x[j] = q.c[j] == kPadCol ? PT(0) : __ldcg(g + q.c[j]);
}
template <typename PT>
__device__ __forceinline__ PT unit_ext_sub(UnitExt<PT> &q, PT (&x)[kUnitChunk], const int32_t *col, const PT *val,
                                           int e, int w, PT acc, const PT *g) {
  for (int j0 = 0;;) {
    const int nj = w - j0;
#pragma unroll
    for (int j = 0; j < kUnitChunk; ++j)
      if (j < nj) acc -= q.v[j] * x[j];
    j0 += kUnitChunk;
    if (j0 >= w) return acc;
    unit_ext_load(q, col, val, e + j0 * kWarp, w - j0);
    unit_ext_gather(q, x, g);
  }
}

constexpr int kUnitWarps = 8;   // warps (units in flight) per CTA of the warp-unit kernels

// A unit's chain coefficients into the warp's shared memory as they lie in
// memory (term-major: lane l's j-th term at j * 32 + l, T terms deep; 16-byte
// cp.async, no registers held while the copies fly) and the lane's source
// lanes into registers.  Compact, the buffer is as deep as the lane with most
// terms (3 for 7-point, 13 for 27-point blocks) and not as the chain (up to 32
// steps, 8 KB a warp in FP64), so that the next launch's CTAs fit beside this
// one's and load their static data early, and the copy is T / 2 instructions
// instead of a test and an address for each of 32 steps.
template <typename PT, int S>
__device__ __forceinline__ void unit_coef(const PT *v, const uint32_t *sw, int off, int T, int soff, int M, int lane,
                                          PT *cfs, uint32_t (&src)[(S + 3) / 4]) {
  constexpr int EV = 16 / sizeof(PT);
  __syncwarp();   // the previous coefficients' readers are done
  for (int k = lane; k < T * (kWarp / EV); k += kWarp) cp_async16(cfs + k * EV, v + off + k * EV);
  cp_commit();
#pragma unroll
  for (int w = 0; w < (S + 3) / 4; ++w) src[w] = 4 * w < M ? __ldg(sw + soff + w * kWarp + lane) : 0u;
}

// phase B of a unit: M chain steps; at step k every lane with a term
// subtracts coefficient x the (final) value of its source lane; wmask = OR
// of the warp's lane masks (a step no lane uses issues no FP64 instruction)
template <typename PT, int S>
__device__ __forceinline__ PT unit_chain(PT t, int M, uint32_t mask, uint32_t wmask, const PT *cfs, int lane,
                                         const uint32_t (&src)[(S + 3) / 4]) {
  cp_wait_all();
  __syncwarp();
  const PT *p = cfs + lane;
  PT c = *p;   // the next term's coefficient (one row of padding after the last)
#pragma unroll
  for (int k = 0; k < S; ++k) {
    if (k < M) {
      const int sl = int((src[k / 4] >> (8 * (k % 4))) & 0xffu);
      const PT tk = __shfl_sync(0xffffffffu, t, sl);
      if ((wmask >> k) & 1u) {
        if ((mask >> k) & 1u) {
          t -= c * tk;
          p += kWarp;
          c = *p;
        }
      }
    }
  }
  return t;
}

// shared memory of a warp-unit CTA, coefficients at most T terms deep
inline int unit_smem_bytes(int T, int elem) { return kUnitWarps * (T + 1) * kWarp * elem; }

// CTAs an SM that a form's registers have to leave room for: those that its loads
// and chain need (72 to 80 registers in FP64 with 32-step chains and in the fused
// forms, 64 otherwise; 48 or 64 in FP32).  Left to itself the compiler takes 64 for
// the FP64 backward form of 32 steps, which has fewer loads in flight then (27-point
// 96^3, blocks of 32 rows, one application with a product: 433 us; so 404).
constexpr int unit_ctas(int elem, int mode, int S) {
  if (elem == 8) return mode == M_FUSED || S == kWarp ? 3 : 4;
  return mode == M_FUSED || (mode == M_BWD && (S == 1 || S == kWarp)) ? 4 : 5;
}

template <typename PT, int MODE, bool UPDATE, int S>
__global__ void __launch_bounds__(kUnitWarps * kWarp, unit_ctas(int(sizeof(PT)), MODE, S))
unit_kernel(Params P, int u0, int u1, int T, int fin, SlotArgs sa) {
  __shared__ double red[kRed];
  extern __shared__ __align__(16) unsigned char usm[];
  __shared__ int flag;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  PT *cfs = reinterpret_cast<PT *>(usm) + wid * (T + 1) * kWarp;
  const int step = lane & (S - 1);
  constexpr bool FWD = MODE != M_BWD;
  PT *yv = reinterpret_cast<PT *>(P.y);
  PT *zv = reinterpret_cast<PT *>(P.z);
  const PT *dvg = invds<PT>(P);
  double rr_acc = 0.0, rz_acc = 0.0;
  const bool end = MODE == M_BWD && sweep_ended(P, sa);
  bool waited = false, live = true;
  double alpha = 0.0;
  for (int u = u0 + int(blockIdx.x) * nw + wid; u < u1; u += int(gridDim.x) * nw) {
    // static data of the unit
    const WarpUnit d = load_unit(P.units + u);
    UnitExt<PT> ext;
    if (FWD) unit_ext_load(ext, P.sl_col, slv<PT>(P), d.lo + lane, d.lw);
    else unit_ext_load(ext, P.su_col, suv<PT>(P), d.uo + lane, d.uw);
    int row = -1;
    if (S == kWarp) {   // one block: its rows are the unit's
      if (lane < d.nrows) row = d.row0 + lane;
    } else if (lane / S < d.nblk) {
      const int b = d.blk0 + lane / S;
      const int r = __ldg(P.bptr + b) + step;
      if (r < __ldg(P.bptr + b + 1)) row = r;
    }
    const bool on = row >= 0;
    const uint32_t mf = FWD ? __ldg(P.wl_mask + size_t(u) * kWarp + lane) : 0u;
    const uint32_t mb = MODE != M_FWD ? __ldg(P.wu_mask + size_t(u) * kWarp + lane) : 0u;
    uint32_t src[(S + 3) / 4];
    if (FWD) unit_coef<PT, S>(wlv<PT>(P), P.wl_src, d.li, d.lt, d.ls, d.lm, lane, cfs, src);
    else unit_coef<PT, S>(wuv<PT>(P), P.wu_src, d.ui, d.ut, d.us, d.um, lane, cfs, src);
    const PT dv = on ? __ldg(dvg + row) : PT(0);
    if (!waited) {
      pdl_wait();
      waited = true;
      if (UPDATE && !(live = load_alpha(P, alpha))) break;
      if (MODE == M_BWD && __any_sync(0xffffffffu, end)) break;
    }
    PT t = PT(0), x[kUnitChunk];
    double ri = 0.0;
    if (FWD) {
      // A: source r (with the x / r update), entries to earlier colors (their
      // gathers before the update's stores)
      ri = on ? __ldcg(P.r + row) : 0.0;
      if (UPDATE) {
        const double qi = on ? __ldcg(P.q + row) : 0.0, xi = on ? __ldcg(P.xh + row) : 0.0;
        const double pi = on ? __ldcg(P.p0 + row) : 0.0;
        unit_ext_gather(ext, x, yv);
        ri -= alpha * qi;
        if (on) {
          P.r[row] = ri;
          P.xh[row] = xi + alpha * pi;
        }
      } else {
        unit_ext_gather(ext, x, yv);
      }
      t = unit_ext_sub(ext, x, P.sl_col, slv<PT>(P), d.lo + lane, d.lw, PT(ri), yv);
      // B, C
      t = unit_chain<PT, S>(t, d.lm, mf, __reduce_or_sync(0xffffffffu, mf), cfs, lane, src);
      const PT y = t * dv;   // 0 in an idle lane
      if (MODE == M_FWD && on) yv[row] = y;
      if (MODE == M_FWD) continue;
      // the last color: its backward sweep at once (y stays in registers)
      unit_ext_load(ext, P.su_col, suv<PT>(P), d.uo + lane, d.uw);
      unit_coef<PT, S>(wuv<PT>(P), P.wu_src, d.ui, d.ut, d.us, d.um, lane, cfs, src);
      t = y;
    } else {
      if (on) {
        t = __ldcg(yv + row);
        if (sa.off >= 0) ri = __ldcg(P.r + row);
      }
    }
    unit_ext_gather(ext, x, zv);
    t = unit_ext_sub(ext, x, P.su_col, suv<PT>(P), d.uo + lane, d.uw, t, zv);
    t = unit_chain<PT, S>(t, d.um, mb, __reduce_or_sync(0xffffffffu, mb), cfs, lane, src);
    const PT z = t * dv;   // 0 in an idle lane
    if (on) zv[row] = z;
    if (sa.off >= 0) rz_add(ri, z, rr_acc, rz_acc);
  }
  if (!waited) {
    pdl_wait();
    if (UPDATE) live = load_alpha(P, alpha);
  }
  cp_wait_all();
  if (!live) return;   // (the whole CTA)
  if (MODE != M_FWD) launch_epilogue(P, fin, sa, rr_acc, rz_acc, red, &flag);
}

// ---------------------------------------------------------------------------
// p = z + beta p (start of an iteration; beta = 0 on the first)
// ---------------------------------------------------------------------------
// (two rows per thread per pass: 16-byte loads of p and, for FP64 z, of z)
template <typename ZT>
__global__ void __launch_bounds__(kVecThreads) pupdate_kernel(Params P) {
  pdl_wait();
  const double beta = __ldcg(&P.sc->beta);
  if (__ldcg(&P.sc->done)) return;
  const ZT *z = reinterpret_cast<const ZT *>(P.z);
  const int n2 = P.n / 2;
  const int stride = gridDim.x * blockDim.x;
  double2 *p2 = reinterpret_cast<double2 *>(P.p0);
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n2; k += stride) {
    const double2 pv = __ldcg(p2 + k);
    double z0, z1;
    if (sizeof(ZT) == 8) {
      const double2 zv = __ldcg(reinterpret_cast<const double2 *>(z) + k);
      z0 = zv.x; z1 = zv.y;
    } else {
      const float2 zv = __ldcg(reinterpret_cast<const float2 *>(z) + k);
      z0 = widen(zv.x); z1 = widen(zv.y);
    }
    p2[k] = make_double2(z0 + beta * pv.x, z1 + beta * pv.y);
  }
  if ((P.n & 1) && blockIdx.x == 0 && threadIdx.x == 0)
    P.p0[P.n - 1] = double(__ldcg(z + P.n - 1)) + beta * __ldcg(P.p0 + P.n - 1);
}

// ---------------------------------------------------------------------------
// SpMV over the 32-row slices of A_hat's sliced-ELL copy, one row per lane:
// coalesced loads of a slice's columns and values straight into registers,
// then the gathers; a full-occupancy grid walks the slices grid-stride (each
// warp one slice at a time; the resident warps keep the loads in flight).
// Off-diagonal entries in column order, then the diagonal.
// ---------------------------------------------------------------------------
// mode 0: q = A p, <p, q>; the last CTA sets alpha = rz / pq
// mode 1: r = b_hat - A x_hat, <r, r> partials in part_a (solve start)
// mode 2: q = A x_hat (plain SpMV)
constexpr int kSpmvChunk = 6;   // entries per predicated batch of the SpMV

// 6 CTAs of 8 warps per SM (at most 40 registers a thread): measured 1%
// faster per PCG iteration than 4 CTAs at 60 registers
template <int MODE>
__global__ void __launch_bounds__(kSpmvWarps * kWarp, 6)
spmv_kernel(Params P) {
  __shared__ double red[kRed];
  __shared__ int flag;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  const int nsl = (P.n + kWarp - 1) / kWarp;
  const double *xin = MODE == 0 ? P.p0 : P.xh;
  double acc = 0.0;
  pdl_wait();
  if (MODE == 0 && __ldcg(&P.sc->done)) return;
  for (int sl = blockIdx.x * W + warp; sl < nsl; sl += gridDim.x * W) {
    const int e0 = __ldg(P.sa_ptr + sl), w = (__ldg(P.sa_ptr + sl + 1) - e0) >> 5;
    const int i = sl * kWarp + lane;
    const int32_t *col = P.sa_col + e0 + lane;
    const double *val = P.sa_val + e0 + lane;
    double s = 0.0;
    for (int j0 = 0; j0 < w; j0 += kSpmvChunk) {
      int cc[kSpmvChunk];
      double vv[kSpmvChunk], xx[kSpmvChunk];
#pragma unroll
      for (int j = 0; j < kSpmvChunk; ++j) {
        const bool ok = j0 + j < w;
        cc[j] = ok ? __ldg(col + (j0 + j) * kWarp) : 0;
        vv[j] = ok ? __ldg(val + (j0 + j) * kWarp) : 0.0;
      }
#pragma unroll
      for (int j = 0; j < kSpmvChunk; ++j) xx[j] = j0 + j < w ? __ldcg(xin + cc[j]) : 0.0;
#pragma unroll
      for (int j = 0; j < kSpmvChunk; ++j)
        if (j0 + j < w) s += vv[j] * xx[j];
    }
    if (i < P.n) {
      const double xi = __ldcg(xin + i);
      s += __ldg(P.adiag + i) * xi;
      if (MODE == 0) {
        P.q[i] = s;
        acc += xi * s;
      } else if (MODE == 1) {
        const double ri = __ldcg(P.bh + i) - s;
        P.r[i] = ri;
        acc += ri * ri;
      } else {
        P.q[i] = s;
      }
    }
  }
  if (MODE == 2) return;
  const double tot = cta_sum(acc, red);
  if (threadIdx.x == 0) P.part_a[blockIdx.x] = tot;
  if (MODE == 0 && arrive_last(&P.sc->ticket, gridDim.x, &flag)) {
    const double rz = __ldcg(&P.sc->rz);
    const double pq = cta_sum_array(P.part_a, gridDim.x, red, false);
    if (threadIdx.x == 0) {
      P.sc->alpha = rz / pq;
      P.sc->pq = pq;
    }
  }
}

// b_hat = b[perm], x_hat = x0[perm], <b, b> partials into init_bb
__global__ void __launch_bounds__(kVecThreads) perm_in_kernel(Params P) {
  __shared__ double red[kRed];
  double acc = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
    const int o = P.perm[i];
    const double b = P.bin[o];
    P.bh[i] = b;
    P.xh[i] = P.xin[o];
    acc += b * b;
  }
  const double tot = cta_sum(acc, red);
  if (threadIdx.x == 0) P.init_bb[blockIdx.x] = tot;
}

// x[perm[i]] = x_hat[i] (x = 0 when b = 0)
__global__ void __launch_bounds__(kVecThreads) perm_out_kernel(Params P) {
  const bool zero = P.sc->bnorm == 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x)
    P.xout[P.perm[i]] = zero ? 0.0 : P.xh[i];
}

__global__ void __launch_bounds__(kVecThreads) permute_kernel(const double *src, double *dst, const int32_t *perm,
                                                              int n, int gather) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (gather) dst[i] = src[perm[i]];
    else dst[perm[i]] = src[i];
  }
}

__global__ void __launch_bounds__(kVecThreads) widen_kernel(const float *src, double *dst, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = double(src[i]);
}

// ---------------------------------------------------------------------------
// IC(0) (up-looking, rows of a group level by level, one row per lane)
// ---------------------------------------------------------------------------
// End of a factor row: L_ii and its reciprocal, which later rows multiply by.
__device__ __forceinline__ double factor_check(const Params &P, int i, double d) {
  if (!(d > 0.0) || !isfinite(d)) {
    atomicMin(P.err_row, (unsigned long long)i);
    d = 1.0;
  }
  return d;
}
__device__ __forceinline__ void factor_pivot(const Params &P, int i, double d) {
  const double lii = sqrt(factor_check(P, i, d));
  P.ldiag[i] = lii;
  P.invd[i] = 1.0 / lii;
}

// Row i of the up-looking IC(0): for every j < i in the pattern, ascending,
//   L_ij = (a_ij - sum_{k < j, k in pat(i) and pat(j)} L_ik L_jk) / L_jj,
// then L_ii = sqrt(a_ii - sum_j L_ij^2); rows j are final when row i runs.
// A finished row also stores 1/L_ii, and later rows multiply by it.
// General form: the common columns by a merge of the two sorted rows (a
// chain of dependent loads).
__device__ __forceinline__ void factor_row_merge(const Params &P, int i) {
  const int rb = P.lrp[i], re = P.lrp[i + 1];
  double d = P.adiag[i];
  for (int p = rb; p < re; ++p) {
    const int j = P.lcol[p];
    double s = P.ainit[p];
    int a = rb, b = P.lrp[j];
    const int be = P.lrp[j + 1];
    while (a < p && b < be) {
      const int ca = P.lcol[a], cb = P.lcol[b];
      if (ca == cb) { s -= P.lval[a] * P.lval[b]; ++a; ++b; }
      else if (ca < cb) ++a;
      else ++b;
    }
    const double lij = s * __ldcg(P.invd + j);
    P.lval[p] = lij;
    d -= lij * lij;
  }
  factor_pivot(P, i, d);
}

// Rows of at most kFacRow strictly-lower entries whose referenced rows have
// at most kFacRow as well: row i's columns and computed values sit in the
// thread's slice of shared memory (sc, sv), each row j is loaded with
// independent loads into registers, and the common columns are found by
// compare-and-select, so no load waits on another.  The terms are
// subtracted in ascending k, as in the general form.
constexpr int kFacRow = 32;

__device__ __forceinline__ void factor_row(const Params &P, int i, int32_t *sc, double *sv) {
  const int rb = P.lrp[i], ni = P.lrp[i + 1] - rb;
  if (ni > kFacRow) { factor_row_merge(P, i); return; }
  // the row's columns and the longest referenced row (all loads issued at once)
  int nmax = 0;
#pragma unroll
  for (int t = 0; t < kFacRow; ++t) {
    if (t < ni) {
      const int j = __ldg(P.lcol + rb + t);
      sc[t] = j;
      nmax = max(nmax, __ldg(P.lrp + j + 1) - __ldg(P.lrp + j));
    }
  }
  if (nmax > kFacRow) { factor_row_merge(P, i); return; }
  double d = P.adiag[i];
  for (int p = 0; p < ni; ++p) {
    const int j = sc[p];
    const int jb = __ldg(P.lrp + j), nj = __ldg(P.lrp + j + 1) - jb;
    int cj[kFacRow];
    double vj[kFacRow];
#pragma unroll
    for (int u = 0; u < kFacRow; ++u) {
      cj[u] = u < nj ? __ldg(P.lcol + jb + u) : -2;
      vj[u] = u < nj ? __ldcg(P.lval + jb + u) : 0.0;
    }
    double s = __ldg(P.ainit + rb + p);
    for (int t = 0; t < p; ++t) {
      const int c = sc[t];
      double v = 0.0;
      bool hit = false;
#pragma unroll
      for (int u = 0; u < kFacRow; ++u) {
        const bool m = cj[u] == c;
        v = m ? vj[u] : v;
        hit = hit || m;
      }
      if (hit) s -= sv[t] * v;
    }
    // times 1/L_jj (one division per row, at its end, instead of one per
    // entry: FP64 division is a multi-instruction sequence on this GPU)
    const double lij = s * __ldcg(P.invd + j);
    sv[p] = lij;
    d -= lij * lij;
  }
  for (int t = 0; t < ni; ++t) P.lval[rb + t] = sv[t];
  factor_pivot(P, i, d);
}

// One in-block level of a lane-tile or warp-unit color, a warp per row (rows
// of 9..32 strictly-lower entries with precomputed update pairs).
// Lane p holds entry p of the row; the pairs' values L_jk are gathered by the
// whole warp into shared memory, then
//   s_p = a_ip - sum_{k < p} L_ik L_pk,   L_ip = s_p / L_pp
// in steps: at each, every lane whose next term's L_ik is final (lane k has no
// term left) takes it from lane k by a shuffle, k ascending per entry as in
// the general form.
//
// Bound by latency: a level has few rows (27-point, blocks of 32: about 1000
// rows in each of 200 levels), so what counts is the chain of one row.  A
// thread per row walked its 60 pairs one FP64 multiply-add after another
// (64 cycles each) behind staged copies, 44 us a level; the warp's steps are
// as many as the deepest chain of terms or the longest list (about 10) and
// its loads are all in flight at once.  Static data (record, columns, a_ij,
// pair indices) is read before griddepcontrol.wait, while the previous level
// runs.  Square
// root and division are FP64 sequences that cost a whole warp however few
// lanes run them, so one warp does them for the CTA's rows together.
constexpr int kFacWarps = 8;
constexpr int kFacPairs = kFacRow * (kFacRow - 1) / 2;   // most pairs of a row
constexpr int kFacBatch = 4;                             // pair loads in flight per lane
constexpr int kFacWarpBytes = kFacPairs * 8 + ((kFacPairs + 15) & ~15);

// The steps of one row of ni entries: lane p holds s_p = a_ip, iv_p = 1/L_pp and
// its terms pv / ps [c, ce); l_p = L_ip on return.  Lane 31 carries the pivot
// a_ii - sum_p l_p^2 as one more entry, whose terms are the entries themselves
// (returned in every lane; a row of 32 entries forms it afterwards).  Every sum
// runs in the order of the general form, so the factor is the same to the bit.
__device__ __forceinline__ double factor_steps(double s, double iv, int c, int ce, int ni, double dg, const double *pv,
                                               const uint8_t *ps, int lane, double &l) {
  const bool piv = lane == 31 && ni < 32;
  if (piv) {
    s = dg;
    c = 0;
    ce = ni;
  }
  int src = c < ce ? (piv ? 0 : int(ps[c])) : lane;
  double nv = c < ce && !piv ? pv[c] : 0.0;
  for (uint32_t left = __ballot_sync(0xffffffffu, c < ce); left;) {
    l = s * iv;
    const double lk = __shfl_sync(0xffffffffu, l, src);
    if (c < ce && !((left >> src) & 1u)) {
      s -= lk * (piv ? lk : nv);
      ++c;
      if (c < ce) {
        src = piv ? c : int(ps[c]);
        if (!piv) nv = pv[c];
      }
    }
    left = __ballot_sync(0xffffffffu, c < ce);
  }
  l = s * iv;
  if (ni < 32) return __shfl_sync(0xffffffffu, s, 31);
  double d = dg;
  for (int p = 0; p < 32; ++p) {
    const double lp = __shfl_sync(0xffffffffu, l, p);
    d -= lp * lp;
  }
  return d;
}

// the pivots of a CTA's rows (d in sd, row in srow)
__device__ __forceinline__ void factor_pivots(const Params &P, const double *sd, const int *srow, int rows, int w,
                                              int lane) {
  if (w == 0 && lane < rows) factor_pivot(P, srow[lane], sd[lane]);
}

__global__ void __launch_bounds__(kFacWarps * kWarp) factor_warp_kernel(Params P, int k0, int k1) {
  extern __shared__ __align__(16) unsigned char fsm[];
  __shared__ double sd[kFacWarps];
  __shared__ int srow[kFacWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double *pv = reinterpret_cast<double *>(fsm + size_t(w) * kFacWarpBytes);
  uint8_t *ps = reinterpret_cast<uint8_t *>(pv + kFacPairs);
  bool waited = false;
  for (int kb = k0 + int(blockIdx.x) * kFacWarps; kb < k1; kb += int(gridDim.x) * kFacWarps) {
    const int k = kb + w;
    const int4 rec = k < k1 ? __ldg(P.fac_rec + k) : make_int4(0, 0, 0, 0);
    const int i = rec.x, rb = rec.y, q0 = rec.z, ni = rec.w & 0xff, np = rec.w >> 8;
    const bool on = lane < ni;
    const int col = on ? __ldg(P.lcol + rb + lane) : 0;
    const double s = on ? __ldg(P.ainit + rb + lane) : 0.0;
    const int c = on ? __ldg(P.fp_ptr + rb + lane) - q0 : 0;
    const int ce = on ? __ldg(P.fp_ptr + rb + lane + 1) - q0 : 0;
    const double dg = k < k1 ? __ldg(P.adiag + i) : 1.0;
    int fb[kFacBatch], fp[kFacBatch];
#pragma unroll
    for (int u = 0; u < kFacBatch; ++u) {
      const int q = u * kWarp + lane;
      fb[u] = q < np ? __ldg(P.fp_b + q0 + q) : 0;
      fp[u] = q < np ? int(__ldg(P.fp_pos + q0 + q)) : 0;
    }
    if (!waited) {
      pdl_wait();
      waited = true;
    }
    const double iv = on ? __ldcg(P.invd + col) : 0.0;
    for (int qa = 0; qa < np; qa += kFacBatch * kWarp) {
      if (qa > 0) {
#pragma unroll
        for (int u = 0; u < kFacBatch; ++u) {
          const int q = qa + u * kWarp + lane;
          fb[u] = q < np ? __ldg(P.fp_b + q0 + q) : 0;
          fp[u] = q < np ? int(__ldg(P.fp_pos + q0 + q)) : 0;
        }
      }
      double v[kFacBatch];
#pragma unroll
      for (int u = 0; u < kFacBatch; ++u) v[u] = qa + u * kWarp + lane < np ? __ldcg(P.lval + fb[u]) : 0.0;
#pragma unroll
      for (int u = 0; u < kFacBatch; ++u) {
        const int q = qa + u * kWarp + lane;
        if (q < np) {
          pv[q] = v[u];
          ps[q] = uint8_t(fp[u]);
        }
      }
    }
    __syncwarp();
    double l;
    const double d = factor_steps(s, iv, c, ce, ni, dg, pv, ps, lane, l);
    if (on) P.lval[rb + lane] = l;
    if (lane == 0) {
      sd[w] = d;
      srow[w] = i;
    }
    __syncthreads();
    factor_pivots(P, sd, srow, min(kFacWarps, k1 - kb), w, lane);
    __syncthreads();
  }
}

// A warp-unit color in one launch, a CTA per unit (at most 32 rows of whole
// blocks, their L entries one range), for rows above kFacShort.  Blocks of one color share no
// edge, so a row waits only for rows of its own block: the CTA's warps take
// the rows in turn (first rows of all blocks, second rows, ...), a warp per
// row as above, and a finished row is announced through a flag in shared
// memory, where its entries and 1/L_ii also stay for the rows that
// follow.  A wait that lasts longer than P.wait_ns gives up: the CTA ends, and
// the host reports ICCG_ERR_TIMEOUT (err_row[1]), not a pivot.  A warp loads its next row's indices and its entries of other
// colors while the others work.
//
// Why: with a launch per level every level of a block cost a launch boundary
// and a trip of its values through L2 (27-point 61x67x59, blocks of 32: 205
// launches of 7-9 us); the launch count falls to one per color.  IC(0) and one
// application together there: 7.40 ms with a thread per row, 1.58 ms now, about
// half of it the FP64 pipe.  (Reciprocal square roots, pre-scaled terms and a
// tree for the pivot's sum took 1.15 ms, but moved the factor's last bit; ill-
// conditioned solves then differ by 1e-9.)
constexpr int kFacUnitWarps = 4;
constexpr int kFacSpin = 1 << 22;   // polls of a row's flags before giving up, whatever the clock says

inline int fac_unit_bytes(int cap) { return kFacUnitWarps * kFacWarpBytes + cap * 8; }

__global__ void __launch_bounds__(kFacUnitWarps * kWarp) factor_unit_kernel(Params P, int u0, int S) {
  extern __shared__ __align__(16) unsigned char fsm[];
  __shared__ double ivs[kWarp], ds[kWarp];
  __shared__ volatile int ready[kWarp];
  __shared__ volatile int gave_up;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double *pv = reinterpret_cast<double *>(fsm + size_t(w) * kFacWarpBytes);
  uint8_t *ps = reinterpret_cast<uint8_t *>(pv + kFacPairs);
  double *us = reinterpret_cast<double *>(fsm + kFacUnitWarps * kFacWarpBytes);
  const WarpUnit d = load_unit(P.units + u0 + int(blockIdx.x));
  const int row0 = d.row0, row1 = d.row0 + d.nrows;
  const int l0 = __ldg(P.lrp + row0), l1 = __ldg(P.lrp + row1);
  if (threadIdx.x < kWarp) ready[threadIdx.x] = 0;
  if (threadIdx.x == 0) gave_up = 0;
  __syncthreads();
  bool waited = false;
  for (int t = w; t < S * d.nblk; t += kFacUnitWarps) {
    const int b = d.blk0 + t % d.nblk, i = __ldg(P.bptr + b) + t / d.nblk;
    if (i >= __ldg(P.bptr + b + 1)) continue;
    const int rb = __ldg(P.lrp + i), ni = __ldg(P.lrp + i + 1) - rb;
    const int q0 = __ldg(P.fp_ptr + rb), np = __ldg(P.fp_ptr + rb + ni) - q0;
    const bool on = lane < ni;
    const int col = on ? __ldg(P.lcol + rb + lane) : 0;
    const double s = on ? __ldg(P.ainit + rb + lane) : 0.0;
    const int c = on ? __ldg(P.fp_ptr + rb + lane) - q0 : 0;
    const int ce = on ? __ldg(P.fp_ptr + rb + lane + 1) - q0 : 0;
    const double dg = __ldg(P.adiag + i);
    int fb[kFacBatch], fp[kFacBatch];
#pragma unroll
    for (int u = 0; u < kFacBatch; ++u) {
      const int q = u * kWarp + lane;
      fb[u] = q < np ? __ldg(P.fp_b + q0 + q) : 0;
      fp[u] = q < np ? int(__ldg(P.fp_pos + q0 + q)) : 0;
    }
    if (!waited) {
      pdl_wait();
      waited = true;
    }
    // values of other colors, before the wait for the block's own rows
    const bool in = on && col >= row0;
    double iv = on && !in ? __ldcg(P.invd + col) : 0.0;
    double v[kFacBatch];
#pragma unroll
    for (int u = 0; u < kFacBatch; ++u) {
      const int q = u * kWarp + lane;
      v[u] = q < np && (fb[u] < l0 || fb[u] >= l1) ? __ldcg(P.lval + fb[u]) : 0.0;
    }
    // (the clock is read at the first poll and every 32 polls)
    bool ok = true;
    unsigned long long t0 = 0;
    for (int spin = 0; ok && !__all_sync(0xffffffffu, !in || ready[col - row0] != 0); ++spin) {
      if ((spin & 31) != 0) continue;
      const unsigned long long now = global_ns();
      if (spin == 0) t0 = now;
      ok = !__any_sync(0xffffffffu, now - t0 > P.wait_ns || spin > kFacSpin || gave_up != 0);
    }
    if (!ok) {
      gave_up = 1;
      if (lane == 0) atomicMin(P.err_row + 1, (unsigned long long)i);
      break;
    }
    __threadfence_block();
    if (in) iv = ivs[col - row0];
#pragma unroll
    for (int u = 0; u < kFacBatch; ++u) {
      const int q = u * kWarp + lane;
      if (q < np) {
        pv[q] = fb[u] >= l0 && fb[u] < l1 ? us[fb[u] - l0] : v[u];
        ps[q] = uint8_t(fp[u]);
      }
    }
    for (int q = kFacBatch * kWarp + lane; q < np; q += kWarp) {
      const int e = __ldg(P.fp_b + q0 + q);
      pv[q] = e >= l0 && e < l1 ? us[e - l0] : __ldcg(P.lval + e);
      ps[q] = __ldg(P.fp_pos + q0 + q);
    }
    __syncwarp();
    double l;
    const double dd = factor_steps(s, iv, c, ce, ni, dg, pv, ps, lane, l);
    if (on) us[rb - l0 + lane] = l;
    if (lane == 0) {
      const double lii = sqrt(factor_check(P, i, dd));
      ds[i - row0] = lii;
      ivs[i - row0] = 1.0 / lii;
    }
    __threadfence_block();
    __syncwarp();
    if (lane == 0) ready[i - row0] = 1;
    if (on) P.lval[rb + lane] = l;
  }
  if (!waited) pdl_wait();
  __syncthreads();
  if (gave_up == 0 && threadIdx.x < d.nrows) {
    P.invd[row0 + threadIdx.x] = ivs[threadIdx.x];
    P.ldiag[row0 + threadIdx.x] = ds[threadIdx.x];
  }
}

// The same for rows of 9..64 strictly-lower entries without precomputed
// pairs (a matrix with any row above 32): two entries per lane, and the
// values L_pk as the strictly-lower triangle of a dense matrix in the warp's
// shared memory (column k: entries p = k + 1 .. ni - 1 consecutive, so the
// lanes of a column read without bank conflicts).  The warp reads row j of
// every entry (i, j) coalesced and finds its columns in row i by a binary
// search in shared memory, then resolves the row column by column, every sum in
// the order of the general form (the same bits).  Bound by the FP64 pipe (about
// 3 warp instructions per column of a row).  IC(0) and one application for a
// 3-unknown 27-neighbour 33^3 network with one-row blocks: 3.24 ms with a thread
// per row merging index lists, 1.22 ms so.
constexpr int kFacWide = 64;
constexpr int kFacWideWarps = 4;

__host__ __device__ inline int fac_wide_bytes(int cap) { return r16b(cap * (cap - 1) / 2 * 8 + cap * 4); }

__global__ void __launch_bounds__(kFacWideWarps * kWarp) factor_wide_kernel(Params P, int k0, int k1, int cap) {
  extern __shared__ __align__(16) unsigned char fsm[];
  __shared__ double sd[kFacWideWarps];
  __shared__ int srow[kFacWideWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int bytes = fac_wide_bytes(cap);
  double *M = reinterpret_cast<double *>(fsm + size_t(w) * bytes);
  int32_t *cs = reinterpret_cast<int32_t *>(M + cap * (cap - 1) / 2);
  bool waited = false;
  for (int kb = k0 + int(blockIdx.x) * kFacWideWarps; kb < k1; kb += int(gridDim.x) * kFacWideWarps) {
    const int k = kb + w;
    const int i = k < k1 ? __ldg(P.fac_rows + k) : 0;
    const int rb = k < k1 ? __ldg(P.lrp + i) : 0, ni = k < k1 ? __ldg(P.lrp + i + 1) - rb : 0;
    const bool on0 = lane < ni, on1 = lane + kWarp < ni;
    const int c0 = on0 ? __ldg(P.lcol + rb + lane) : 0, c1 = on1 ? __ldg(P.lcol + rb + kWarp + lane) : 0;
    double s0 = on0 ? __ldg(P.ainit + rb + lane) : 0.0, s1 = on1 ? __ldg(P.ainit + rb + kWarp + lane) : 0.0;
    const int b0 = on0 ? __ldg(P.lrp + c0) : 0, b1 = on1 ? __ldg(P.lrp + c1) : 0;
    const int n0 = on0 ? __ldg(P.lrp + c0 + 1) - b0 : 0, n1 = on1 ? __ldg(P.lrp + c1 + 1) - b1 : 0;
    const double dg = k < k1 ? __ldg(P.adiag + i) : 1.0;
    const int tri = ni * (ni - 1) / 2;
    for (int e = lane; e < tri; e += kWarp) M[e] = 0.0;
    if (on0) cs[lane] = c0;
    if (on1) cs[lane + kWarp] = c1;
    if (!waited) {
      pdl_wait();
      waited = true;
    }
    const double iv0 = on0 ? __ldcg(P.invd + c0) : 0.0, iv1 = on1 ? __ldcg(P.invd + c1) : 0.0;
    __syncwarp();
    // entry p's row j against the columns before p
    auto place = [&](int p, int cu, double v) {
      int lo = 0, hi = p;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cs[mid] < cu) lo = mid + 1;
        else hi = mid;
      }
      if (lo < p && cs[lo] == cu) M[lo * (ni - 1) - lo * (lo - 1) / 2 + (p - lo - 1)] = v;
    };
    for (int p0 = 1; p0 < ni; p0 += kFacBatch) {
      int cu[kFacBatch], nj[kFacBatch], jb[kFacBatch];
      double v[kFacBatch];
#pragma unroll
      for (int u = 0; u < kFacBatch; ++u) {
        const int p = p0 + u;
        jb[u] = __shfl_sync(0xffffffffu, p < kWarp ? b0 : b1, p & 31);
        nj[u] = __shfl_sync(0xffffffffu, p < kWarp ? n0 : n1, p & 31);
        if (p >= ni) nj[u] = 0;
        cu[u] = lane < nj[u] ? __ldg(P.lcol + jb[u] + lane) : 0;
        v[u] = lane < nj[u] ? __ldcg(P.lval + jb[u] + lane) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kFacBatch; ++u) {
        if (lane < nj[u]) place(p0 + u, cu[u], v[u]);
        for (int q = kWarp + lane; q < nj[u]; q += kWarp)
          place(p0 + u, __ldg(P.lcol + jb[u] + q), __ldcg(P.lval + jb[u] + q));
      }
    }
    __syncwarp();
    // lane 31's spare entry carries the pivot a_ii - sum_p l_p^2 (a row of 64
    // entries forms it afterwards)
    const bool piv0 = lane == 31 && ni < kWarp, piv1 = lane == 31 && ni >= kWarp && ni < kFacWide;
    if (piv0) s0 = dg;
    if (piv1) s1 = dg;
    int off = -1;   // column kk's entry p at off + p - kk
    for (int kk = 0; kk < ni; ++kk) {
      const double lk = __shfl_sync(0xffffffffu, kk < kWarp ? s0 * iv0 : s1 * iv1, kk & 31);
      if (kk < kWarp - 1) {
        const double m = piv0 ? lk : (lane > kk && on0 ? M[off + lane - kk] : 0.0);
        if (__double_as_longlong(m) != 0) s0 -= lk * m;
      }
      if (ni >= kWarp) {
        const double m = piv1 ? lk : (lane + kWarp > kk && on1 ? M[off + lane + kWarp - kk] : 0.0);
        if (__double_as_longlong(m) != 0) s1 -= lk * m;
      }
      off += ni - 1 - kk;
    }
    const double l0 = s0 * iv0, l1 = s1 * iv1;
    if (on0) P.lval[rb + lane] = l0;
    if (on1) P.lval[rb + kWarp + lane] = l1;
    double d = __shfl_sync(0xffffffffu, ni < kWarp ? s0 : s1, 31);
    if (ni == kFacWide) {
      d = dg;
      for (int p = 0; p < kFacWide; ++p) {
        const double lp = __shfl_sync(0xffffffffu, p < kWarp ? l0 : l1, p & 31);
        d -= lp * lp;
      }
    }
    if (lane == 0) {
      sd[w] = d;
      srow[w] = i;
    }
    __syncthreads();
    factor_pivots(P, sd, srow, min(kFacWideWarps, k1 - kb), w, lane);
    __syncthreads();
  }
}

// Levels of short rows (at most kFacShort lower entries) with precomputed
// pairs: one row per thread (a warp per row would leave 24 lanes idle in
// every FP64 instruction).  Static data before griddepcontrol.wait; a stencil
// without triangles (5- and 7-point) has no pairs at all.
constexpr int kFacShort = 8;
__global__ void __launch_bounds__(kVecThreads) factor_short_kernel(Params P, int k0, int k1) {
  bool waited = false;
  for (int k = k0 + int(blockIdx.x * blockDim.x + threadIdx.x); k < k1; k += int(gridDim.x * blockDim.x)) {
    const int4 rec = __ldg(P.fac_rec + k);
    const int i = rec.x, rb = rec.y, q0 = rec.z, ni = rec.w & 0xff, np = rec.w >> 8;
    int col[kFacShort], qe[kFacShort];
    double l[kFacShort], iv[kFacShort];
#pragma unroll
    for (int p = 0; p < kFacShort; ++p) {
      col[p] = p < ni ? __ldg(P.lcol + rb + p) : 0;
      l[p] = p < ni ? __ldg(P.ainit + rb + p) : 0.0;
      qe[p] = np > 0 && p < ni ? __ldg(P.fp_ptr + rb + p + 1) - q0 : 0;
    }
    double d = __ldg(P.adiag + i);
    if (!waited) {
      pdl_wait();
      waited = true;
    }
#pragma unroll
    for (int p = 0; p < kFacShort; ++p) iv[p] = p < ni ? __ldcg(P.invd + col[p]) : 0.0;
    int q = 0;
#pragma unroll
    for (int p = 0; p < kFacShort; ++p) {
      if (p < ni) {
        double s = l[p];
        for (; q < qe[p]; ++q) {
          const int pos = int(__ldg(P.fp_pos + q0 + q));
          const double v = __ldcg(P.lval + __ldg(P.fp_b + q0 + q));
          double lk = 0.0;
#pragma unroll
          for (int t = 0; t < kFacShort; ++t)
            if (t < p && t == pos) lk = l[t];
          s -= lk * v;
        }
        l[p] = s * iv[p];
        d -= l[p] * l[p];
      }
    }
#pragma unroll
    for (int p = 0; p < kFacShort; ++p)
      if (p < ni) P.lval[rb + p] = l[p];
    factor_pivot(P, i, d);
  }
  if (!waited) pdl_wait();
}

// levels without precomputed pairs of short rows (short merges) or of rows
// above kFacWide: one row per thread, the general form
__global__ void __launch_bounds__(kVecThreads) factor_merge_kernel(Params P, int k0, int k1) {
  pdl_wait();
  for (int k = k0 + int(blockIdx.x * blockDim.x + threadIdx.x); k < k1; k += int(gridDim.x * blockDim.x))
    factor_row_merge(P, __ldg(P.fac_rows + k));
}

// group colors: one CTA per group, its rows level by level of the in-group
// schedule (dynamic shared memory: a kFacRow slice per thread)
__global__ void __launch_bounds__(kMaxWarpsPerCta * kWarp) factor_color_kernel(Params P, int g0, int g1) {
  extern __shared__ __align__(16) unsigned char fsm[];
  int32_t *sc = reinterpret_cast<int32_t *>(fsm) + threadIdx.x * kFacRow;
  double *sv = reinterpret_cast<double *>(fsm + size_t(blockDim.x) * kFacRow * 4) + threadIdx.x * kFacRow;
  const int g = g0 + blockIdx.x;
  if (g >= g1) return;
  const GroupDesc d = P.groups[g];
  for (int lv = 0; lv < d.nlf; ++lv) {
    const int p0 = P.levp[d.lf + lv], p1 = P.levp[d.lf + lv + 1];
    for (int p = p0 + int(threadIdx.x); p < p1; p += blockDim.x) factor_row(P, d.r0 + P.sched_f[d.r0 + p], sc, sv);
    __syncthreads();
  }
}

// invd = 1/L_ii, U values mirrored from L, FP32 copies, sliced-ELL values
__global__ void __launch_bounds__(kVecThreads) factor_finish_kernel(Params P, int nL) {
  const int stride = gridDim.x * blockDim.x;
  // 1/L_ii was stored with each row; its FP32 copy
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += stride) P.invd32[i] = float(P.invd[i]);
  for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < nL; u += stride) {
    const double lv = P.lval[P.umap[u]];
    P.uval[u] = lv;
    P.uval32[u] = float(lv);
    P.lval32[u] = float(P.lval[u]);
  }
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P.nsl; e += stride) {
    const int m = P.sl_map[e];
    const double v = m >= 0 ? P.lval[m] : 0.0;
    P.sl_val[e] = v;
    P.sl_val32[e] = float(v);
  }
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P.nsu; e += stride) {
    const int m = P.su_map[e];
    const double v = m >= 0 ? P.lval[m] : 0.0;
    P.su_val[e] = v;
    P.su_val32[e] = float(v);
  }
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P.nsi; e += stride) {
    const int m = P.si_map[e];
    const double v = m >= 0 ? P.lval[m] : 0.0;
    P.si_val[e] = v;
    P.si_val32[e] = float(v);
  }
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P.nui; e += stride) {
    const int m = P.ui_map[e];
    const double v = m >= 0 ? P.lval[m] : 0.0;
    P.ui_val[e] = v;
    P.ui_val32[e] = float(v);
  }
  // warp-unit coefficients: the entry divided by the pivot of its source row
  // (times the stored 1/L_kk)
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P.nwl; e += stride) {
    const int m = P.wl_map[e];
    const double v = m >= 0 ? P.lval[m] * P.invd[P.wl_srow[e]] : 0.0;
    P.wl_val[e] = v;
    P.wl_val32[e] = float(v);
  }
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P.nwu; e += stride) {
    const int m = P.wu_map[e];
    const double v = m >= 0 ? P.lval[m] * P.invd[P.wu_srow[e]] : 0.0;
    P.wu_val[e] = v;
    P.wu_val32[e] = float(v);
  }
}

// ---------------------------------------------------------------------------
// Persistent solve: the whole PCG solve in one cooperative launch.  The
// phases of an iteration are
//   SpMV     p = z + beta p (into the other p buffer) and q = A p in one pass:
//            a row's q gathers (z_j + beta p_j), the value the owner of row j
//            stores as its new p_j, so no barrier separates the two; <p,q>
//   fwd c    colors 0 .. n_c-2 (x / r update, <r,r>, L y = r)
//   fused    the last color, forward then backward
//   bwd c    colors n_c-2 .. 0 (L^T z = y, <r,z>)
// with one grid barrier after each (2 n_c per iteration).  Every CTA reduces
// the per-CTA partials itself, in index order, right after the barrier that
// completes them, so all CTAs take identical decisions with no broadcast.
// A CTA walks the groups g0_c + blockIdx.x + k * gridDim.x of each color; the
// static data of its next group (next color, next pass) is copied into the
// other of two shared-memory buffers while it computes the current one, and
// across the barriers in between.
// ---------------------------------------------------------------------------

// A barrier wait gives up after P.wait_ns of wall time (default 4 s, settable
// per context) or kSpinLimit polls, whichever comes first: long enough for any
// phase of a solve the shared-memory plan admits, short enough that a missing
// CTA cannot hang the device.
constexpr long long kSpinLimit = 1ll << 27;

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Sense-reversing grid barrier with a bounded wait.  Returns false (for the
// whole CTA) when this CTA or another one gave up; the error word stays set.
__device__ __forceinline__ bool grid_sync(GridBar *bar, unsigned &gen, int *flag, unsigned long long wait_ns) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();
    const unsigned arrived = atomicAdd(&bar->count, 1u);
    if (arrived == gridDim.x - 1) {
      atomicExch(&bar->count, 0u);
      __threadfence();
      atomicExch(&bar->gen, gen + 1);
    } else {
      const unsigned long long t0 = global_ns();
      // the clock is read on every poll (a short limit must take effect at
      // the first poll); the error word of other CTAs every 64 polls
      for (long long k = 1; ld_acquire_u32(&bar->gen) == gen; ++k) {
        if (global_ns() - t0 > wait_ns || k > kSpinLimit ||
            ((k & 63) == 0 && ld_acquire_u32(&bar->err) != 0u)) {
          atomicExch(&bar->err, 1u);
          ok = 0;
          break;
        }
        __nanosleep(32);
      }
    }
    __threadfence();
    gen = gen + 1;
    *flag = ok && ld_acquire_u32(&bar->err) == 0u;
  }
  __syncthreads();
  return *flag != 0;
}

// Barrier state of one CTA plus the optional phase trace (CTA 0 records the
// time it leaves each barrier, tagged with the phase that barrier ends).
struct GridSync {
  GridBar *bar;
  unsigned gen;
  int *flag;
  unsigned long long *trace;
  int tk, cap;
  unsigned long long wait_ns;
};

__device__ __forceinline__ bool phase_end(GridSync &s, int tag) {
  const bool ok = grid_sync(s.bar, s.gen, s.flag, s.wait_ns);
  if (s.trace && blockIdx.x == 0 && threadIdx.x == 0 && s.tk < s.cap)
    s.trace[s.tk++] = (global_ns() << 4) | unsigned(tag);
  return ok;
}

// sum of arr[0 .. count) (fixed order), broadcast to every thread
__device__ __forceinline__ double cta_sum_bcast(const double *arr, int count, double *red, double *bc) {
  const double s = cta_sum_array(const_cast<double *>(arr), count, red, false);
  if (threadIdx.x == 0) *bc = s;
  __syncthreads();
  const double v = *bc;
  __syncthreads();
  return v;
}

// One pass over all 32-row tiles of A_hat, one row per lane, entries staged
// per warp.  INIT: r = b_hat - A x_hat, returns this thread's share of <r,r>.
// Otherwise: p_new = z + beta p_old, q = A p_new, share of <p_new, q>.
template <bool INIT, typename ZT>
__device__ __forceinline__ double spmv_pass(const Params &P, unsigned char *smem, int cap, double beta,
                                            const double *pold, double *pnew) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  double *sv = reinterpret_cast<double *>(smem + warp * (r16((cap + 8) * 8) + r16((cap + 8) * 4)));
  int32_t *sc = reinterpret_cast<int32_t *>(reinterpret_cast<unsigned char *>(sv) + r16((cap + 8) * 8));
  const int ntile = (P.n + kWarp - 1) / kWarp;
  const ZT *z = reinterpret_cast<const ZT *>(P.z);
  double acc = 0.0;
  for (int tile = blockIdx.x * W + warp; tile < ntile; tile += gridDim.x * W) {
    const int t0 = tile * kWarp, t1 = min(P.n, t0 + kWarp);
    const int i = t0 + lane;
    const int rb = i < t1 ? __ldg(P.arp + i) : 0;
    const int re = i < t1 ? __ldg(P.arp + i + 1) : 0;
    const int e0 = __shfl_sync(0xffffffffu, rb, 0);
    const int e1 = __ldg(P.arp + t1);
    Seg<double> S;
    S.gv = P.aval; S.gc = P.acol; S.sv = sv; S.sc = sc;
    S.staged = e1 - e0 <= cap;
    S.bv = S.bc = 0;
    if (S.staged) {
      S.bv = stage_cover<double>(P.aval, e0, e1, sv, lane, kWarp);
      S.bc = stage_cover<int32_t>(P.acol, e0, e1, sc, lane, kWarp);
    }
    cp_commit();
    cp_wait_all();
    __syncwarp();
    if (i < t1) {
      if (INIT) {
        const double s = -row_sub<double, double>(S, rb, re, 0.0, [&](int c) { return __ldcg(P.xh + c); });
        const double ri = __ldcg(P.bh + i) - s;
        P.r[i] = ri;
        acc += ri * ri;
      } else {
        const double s = -row_sub<double, double>(
            S, rb, re, 0.0, [&](int c) { return double(__ldcg(z + c)) + beta * __ldcg(pold + c); });
        const double pi = double(__ldcg(z + i)) + beta * __ldcg(pold + i);
        pnew[i] = pi;
        P.q[i] = s;
        acc += pi * s;
      }
    }
    __syncwarp();
  }
  return acc;
}

// ---- the work items of one preconditioner pass ----------------------------
// Phase ph in [0, 2 n_c - 1): ph < n_c is the forward sweep of color ph (the
// last of them fused with its backward sweep), ph >= n_c the backward sweep
// of color 2 n_c - 2 - ph.  An item is one sweep over one group; the fused
// phase has two per group (sub 0 forward, sub 1 backward).
struct Item {
  int ph, g, sub;
  bool ok, wrap;   // wrap: the item belongs to the next pass
};

__device__ __forceinline__ int ph_color(int ph, int nc) { return ph < nc ? ph : 2 * nc - 2 - ph; }

// first item of this CTA at phase >= ph (group g of phase ph, or its first)
__device__ __forceinline__ Item seek_item(const Params &P, int ph, int g) {
  const int nc = P.n_c;
  for (; ph < 2 * nc - 1; ++ph, g = -1) {
    const int c = ph_color(ph, nc);
    if (g < 0) g = __ldg(P.color_group + c) + int(blockIdx.x);
    if (g < __ldg(P.color_group + c + 1)) return Item{ph, g, 0, true, false};
  }
  return Item{0, 0, 0, false, false};
}

__device__ __forceinline__ Item next_item(const Params &P, const Item &it) {
  if (it.ph == P.n_c - 1 && it.sub == 0) return Item{it.ph, it.g, 1, true, false};
  Item n = seek_item(P, it.ph, it.g + int(gridDim.x));
  if (!n.ok) {
    n = seek_item(P, 0, -1);
    n.wrap = true;
  }
  return n;
}

__device__ __forceinline__ bool item_upper(const Item &it, int nc) { return it.ph >= nc || it.sub == 1; }

// Double-buffered group plan: static data of buffer k at k * o_w, the
// row-work arrays (w, spl) shared by both buffers after them.
template <typename PT>
__device__ __forceinline__ GroupSmem<PT> group_smem_buf(unsigned char *base, const GroupSmemPlan &p, int k) {
  GroupSmem<PT> s = group_smem<PT>(base + k * p.o_w, p);
  s.w = reinterpret_cast<PT *>(base + 2 * p.o_w);
  s.spl = reinterpret_cast<int32_t *>(base + p.o_w + p.o_spl);
  return s;
}

// copies of item it's static data into buffer k, committed as one group
// (an empty group when there is no item)
template <typename PT>
__device__ __forceinline__ void stage_item(const Params &P, const Item &it, unsigned char *smem,
                                           const GroupSmemPlan &plan, int k) {
  if (it.ok) {
    const GroupDesc d = load_group(P.groups + it.g);
    sweep_issue<PT>(P, d, item_upper(it, P.n_c), group_smem_buf<PT>(smem, plan, k), threadIdx.x, blockDim.x);
  }
  cp_commit();
}

// One preconditioner pass (forward colors, fused color, backward colors)
// with a barrier after every phase but the last; `cur` (staged in buffer
// `buf`) is this CTA's first item and becomes the first item of the next
// pass.  Accumulates this thread's <r,r> (UPDATE) and <r,z> shares.
template <typename PT, bool UPDATE>
__device__ __forceinline__ bool precond_pass(const Params &P, const GroupSmemPlan &plan, unsigned char *smem,
                                             Item &cur, int &buf, double alpha, const double *pn, double &rr_acc,
                                             double &rz_acc, GridSync &gs) {
  const int nc = P.n_c, nph = 2 * nc - 1;
  const int tid = threadIdx.x, nthr = blockDim.x;
  cur.wrap = false;
  for (int ph = 0; ph < nph; ++ph) {
    while (cur.ok && !cur.wrap && cur.ph == ph) {
      const Item nx = next_item(P, cur);
      stage_item<PT>(P, nx, smem, plan, buf ^ 1);
      cp_wait_prev();
      __syncthreads();
      const GroupSmem<PT> m = group_smem_buf<PT>(smem, plan, buf);
      const GroupDesc d = load_group(P.groups + cur.g);
      const bool fused = ph == nc - 1;
      if (!item_upper(cur, nc)) {
        const Sweep<PT> sw = sweep_desc<PT>(P, d, false, m);
        group_sweep<PT, false, UPDATE>(P, d, sw, m, tid, nthr, alpha, pn, false, !fused || !sw.fit, rr_acc,
                                       rz_acc);
      } else {
        const Sweep<PT> sw = sweep_desc<PT>(P, d, true, m);
        group_sweep<PT, true, false>(P, d, sw, m, tid, nthr, 0.0, nullptr, fused && sw.fit, true, rr_acc, rz_acc);
      }
      buf ^= 1;
      cur = nx;
    }
    if (ph < nph - 1 && !phase_end(gs, ph < nc - 1 ? PH_FWD : (ph == nc - 1 ? PH_FUSED : PH_BWD))) return false;
  }
  return true;
}

// 64 registers a thread: up to 2 CTAs of 16 warps (or 8 of 4) per SM
#ifndef ICCG_PERSIST_MIN_CTAS
#define ICCG_PERSIST_MIN_CTAS 2
#endif

template <typename PT>
__global__ void __launch_bounds__(kMaxWarpsPerCta * kWarp, ICCG_PERSIST_MIN_CTAS)
persistent_kernel(Params P, GroupSmemPlan plan, int cap_a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[kRed];
  __shared__ double bc;
  __shared__ int flag;
  const int tid = threadIdx.x, nthr = blockDim.x, nb = gridDim.x, b = blockIdx.x;
  const int gstride = nb * nthr, gi = b * nthr + tid;
  unsigned char *smem_a = smem + plan.o_w + plan.total;   // SpMV staging
  GridSync gs{P.bar, 0u, &flag, P.trace, 0, P.trace_cap, P.wait_ns};
  Scalars *S = P.sc;
  const double tol = __ldcg(&S->tol);
  const int maxit = __ldcg(&S->maxit);
  double *pp_a = P.part0, *pp_b = P.part1;   // per-CTA partials [gridDim.x]
  int status = ICCG_ERR_TIMEOUT, it = 0;
  bool ok = true;

  // this CTA's first preconditioner item, staged while the solve starts
  int buf = 0;
  Item cur = seek_item(P, 0, -1);
  stage_item<PT>(P, cur, smem, plan, 0);

  // solve start: b_hat, x_hat, p = 0, <b,b>
  double acc = 0.0;
  for (int i = gi; i < P.n; i += gstride) {
    const int o = __ldg(P.perm + i);
    const double bi = __ldcg(P.bin + o);
    P.bh[i] = bi;
    P.xh[i] = __ldcg(P.xin + o);
    P.p0[i] = 0.0;
    acc += bi * bi;
  }
  acc = cta_sum(acc, red);
  if (tid == 0) P.init_bb[b] = acc;
  ok = phase_end(gs, PH_INIT);
  // r0 = b_hat - A x_hat, <r0, r0>
  if (ok) {
    acc = cta_sum(spmv_pass<true, PT>(P, smem_a, cap_a, 0.0, nullptr, nullptr), red);
    if (tid == 0) pp_a[b] = acc;
    ok = phase_end(gs, PH_INIT);
  }
  // z0 = M^-1 r0, <r0, z0>
  double rr_acc = 0.0, rz_acc = 0.0;
  if (ok) ok = precond_pass<PT, false>(P, plan, smem, cur, buf, 0.0, nullptr, rr_acc, rz_acc, gs);
  if (ok) {
    acc = cta_sum(rz_acc, red);
    if (tid == 0) pp_b[b] = acc;
    ok = phase_end(gs, PH_INIT);
  }
  double bnorm = 0.0, rz = 0.0;
  bool done = false;
  if (ok) {
    const double bb = cta_sum_bcast(P.init_bb, nb, red, &bc);
    const double rr0 = cta_sum_bcast(pp_a, nb, red, &bc);
    rz = cta_sum_bcast(pp_b, nb, red, &bc);
    bnorm = sqrt(bb);
    if (bnorm == 0.0) {
      done = true;
      status = ICCG_OK;
      if (b == 0 && tid == 0) P.hist[0] = 0.0;
    } else {
      const double rn = sqrt(rr0) / bnorm;
      if (b == 0 && tid == 0) P.hist[0] = rn;
      if (!isfinite(rn) || !isfinite(rz)) { done = true; status = ICCG_ERR_NONFINITE; }
      else if (rn <= tol) { done = true; status = ICCG_OK; }
      else if (maxit <= 0) { done = true; status = ICCG_NOT_CONVERGED; }
    }
    // pp_a is next written by the SpMV, read after its barrier; pp_b after at
    // least one color barrier: every CTA has read both by then
  }
  double beta = 0.0;
  while (ok && !done) {
    // p_new = z + beta p_old, q = A p_new, <p_new, q>, alpha
    const double *pold = (it & 1) ? P.p1 : P.p0;
    double *pnew = (it & 1) ? P.p0 : P.p1;
    acc = cta_sum(spmv_pass<false, PT>(P, smem_a, cap_a, beta, pold, pnew), red);
    if (tid == 0) pp_a[b] = acc;
    if (!(ok = phase_end(gs, PH_SPMV))) break;
    const double pq = cta_sum_bcast(pp_a, nb, red, &bc);
    const double alpha = rz / pq;
    // x / r update, forward and backward substitution
    rr_acc = 0.0;
    rz_acc = 0.0;
    if (!(ok = precond_pass<PT, true>(P, plan, smem, cur, buf, alpha, pnew, rr_acc, rz_acc, gs))) break;
    const double rrc = cta_sum(rr_acc, red);
    const double rzc = cta_sum(rz_acc, red);
    if (tid == 0) { pp_a[b] = rrc; pp_b[b] = rzc; }
    if (!(ok = phase_end(gs, PH_BWD))) break;
    const double rr = cta_sum_bcast(pp_a, nb, red, &bc);
    const double rz_new = cta_sum_bcast(pp_b, nb, red, &bc);
    ++it;
    const double rn = sqrt(rr) / bnorm;
    if (b == 0 && tid == 0) P.hist[it] = rn;
    if (!isfinite(rn) || !isfinite(rz_new)) { done = true; status = ICCG_ERR_NONFINITE; }
    else if (rn <= tol) { done = true; status = ICCG_OK; }
    else if (it >= maxit) { done = true; status = ICCG_NOT_CONVERGED; }
    else {
      beta = rz_new / rz;
      rz = rz_new;
    }
  }
  cp_wait_all();
  if (ok) {
    for (int i = gi; i < P.n; i += gstride) P.xout[__ldg(P.perm + i)] = bnorm == 0.0 ? 0.0 : __ldcg(P.xh + i);
  }
  if (b == 0 && tid == 0) {
    S->iter = it;
    S->status = ok ? status : ICCG_ERR_TIMEOUT;
    S->bnorm = bnorm;
    S->done = 1;
    if (P.trace && gs.tk < P.trace_cap) P.trace[gs.tk++] = (global_ns() << 4) | unsigned(PH_ALL);
    if (P.trace_len) *P.trace_len = gs.tk;
  }
}

// ---------------------------------------------------------------------------
// Cooperative sweep: a whole preconditioner application in one launch for a
// layout whose colors are all pair tiles (blocks of one or two rows): the
// forward colors, the fused last color and the backward colors (Alg. 1 and
// the reverse sweep) one after another, each color's tiles taken grid-stride
// by every warp of the grid, a bounded grid barrier where a color needs the
// previous one's results; one reduction closes the launch.  It replaces the
// 2 n_c - 1 color launches of the sweep, whose fixed cost (launch, ramp-up,
// tail, per-launch reduction) dominates colors of few rows.
// ---------------------------------------------------------------------------
constexpr int kCoopWarps = 8;

// c_lo > 0: the tail of a sweep (forward colors c_lo .. n_c - 2, the fused
// last color, backward colors n_c - 2 .. c_lo), between per-color launches.
// The <r,r> / <r,z> partials of a tail go to the slot regions of its colors
// (from rr0; one per CTA in the first of the ntail regions, zeros in the others).
template <typename PT, bool UPDATE>
__global__ void __launch_bounds__(kCoopWarps * kWarp)
coop_sweep_kernel(Params P, int c_lo, int fin, int rr0, int ntail) {
  __shared__ double red[kRed];
  __shared__ int flag;
  const int lane = threadIdx.x & 31;
  const int nw = int(blockDim.x >> 5), gw = int(blockIdx.x) * nw + int(threadIdx.x >> 5);
  const int NW = int(gridDim.x) * nw, nc = P.n_c;
  double rr_acc = 0.0, rz_acc = 0.0;
  pdl_wait();
  // one decision per CTA: a CTA of this launch whose wait runs out may end the
  // solve at any time
  __shared__ double alpha_s;
  if (threadIdx.x == 0) {
    double a = 0.0;
    flag = UPDATE ? int(load_alpha(P, a)) : 1;
    alpha_s = a;
  }
  __syncthreads();
  const double alpha = alpha_s;
  if (!flag) return;
  __syncthreads();   // flag is reused by the barriers
  GridSync gs{P.bar, 0u, &flag, nullptr, 0, 0, P.wait_ns};
  bool ok = true;
  for (int c = c_lo; c < nc - 1 && ok; ++c) {
    const int t1 = __ldg(P.ctile + c + 1);
    for (int t = __ldg(P.ctile + c) + gw; t < t1; t += NW) pair_tile<PT, M_FWD, UPDATE>(P, t, lane, alpha, rr_acc, rz_acc);
    ok = phase_end(gs, PH_FWD);
  }
  if (ok) {
    const int t1 = __ldg(P.ctile + nc);
    for (int t = __ldg(P.ctile + nc - 1) + gw; t < t1; t += NW)
      pair_tile<PT, M_FUSED, UPDATE>(P, t, lane, alpha, rr_acc, rz_acc);
  }
  for (int c = nc - 2; c >= c_lo && ok; --c) {
    if (!(ok = phase_end(gs, PH_BWD))) break;
    const int t1 = __ldg(P.ctile + c + 1);
    for (int t = __ldg(P.ctile + c) + gw; t < t1; t += NW) pair_tile<PT, M_BWD, false>(P, t, lane, alpha, rr_acc, rz_acc);
  }
  if (!ok) {
    // a barrier wait gave up: the solve stops with ICCG_ERR_TIMEOUT
    if (threadIdx.x == 0) {
      P.sc->status = ICCG_ERR_TIMEOUT;
      P.sc->done = 1;
      P.sc->skip = 1.0;
      set_condition(P.sc, false, 0);
    }
    return;
  }
  if (rr0 < 0) return;   // no sums wanted
  launch_epilogue<true>(P, fin, SlotArgs{rr0, 0, 0}, rr_acc, rz_acc, red, &flag);
  const int G = int(gridDim.x), b = int(blockIdx.x);
  if (threadIdx.x == 0)
    for (int k = 1; k < ntail; ++k) P.slot_rr[rr0 + k * G + b] = P.slot_rz[rr0 + k * G + b] = 0.0;
}

// ---------------------------------------------------------------------------
// launch helpers
// ---------------------------------------------------------------------------
template <typename... KArgs, typename... Args>
cudaError_t launch_coop(void (*kernel)(KArgs...), int grid, int threads, int smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = size_t(smem);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), int grid, int threads, int smem, const Plan &L, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = size_t(smem);
  cfg.stream = L.stream;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (L.carve >= 0) {
    attr[na].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[na++].val.sharedMemCarveout = unsigned(L.carve);
  }
  if (L.pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na++].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = unsigned(na);
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename PT>
GroupSmemPlan plan_of(const Params &P, bool fused, bool upper) {
  const int cap = fused ? max(P.cap_l, P.cap_u) : (upper ? P.cap_u : P.cap_l);
  return group_smem_plan(cap, P.cap_rows, P.cap_lev, int(sizeof(PT)));
}

template <typename PT>
TilePlan tile_plan_of(const Params &P, bool stage_ext = true) {
  TilePlan p = tile_plan(P.lane_max, P.tcap_r, P.tcap_i, int(sizeof(PT)), stage_ext ? P.tcap_o : 0);
  p.nbuf = P.tnbuf;
  p.cap_i2 = P.tcap_i2;
  return p;
}

template <typename PT, bool ONE>
cudaError_t launch_tile_w(const Params &P, const Plan &L, int c, int mode, bool update, int fin, const SlotArgs &sa) {
  const TilePlan pl = tile_plan_of<PT>(P, L.stage_ext[c] != 0);
  const int g = L.grid_c[c], t0 = L.tile0[c], t1 = L.tile1[c], th = L.Wt * kWarp;
  const int sm = tile_launch_bytes(pl, mode == M_FUSED) + (mode == M_FWD ? tile_red_bytes(ONE) : 0);
  if (mode == M_BWD) return launch(tile_kernel<PT, M_BWD, false, ONE>, g, th, sm, L, P, t0, t1, pl, fin, sa);
  if (update) {
    if (mode == M_FUSED) return launch(tile_kernel<PT, M_FUSED, true, ONE>, g, th, sm, L, P, t0, t1, pl, fin, sa);
    return launch(tile_kernel<PT, M_FWD, true, ONE>, g, th, sm, L, P, t0, t1, pl, fin, sa);
  }
  if (mode == M_FUSED) return launch(tile_kernel<PT, M_FUSED, false, ONE>, g, th, sm, L, P, t0, t1, pl, fin, sa);
  return launch(tile_kernel<PT, M_FWD, false, ONE>, g, th, sm, L, P, t0, t1, pl, fin, sa);
}

template <typename PT>
cudaError_t launch_tile(const Params &P, const Plan &L, int c, int mode, bool update, int fin, const SlotArgs &sa) {
  return L.Wt == 1 ? launch_tile_w<PT, true>(P, L, c, mode, update, fin, sa)
                   : launch_tile_w<PT, false>(P, L, c, mode, update, fin, sa);
}

template <typename PT>
cudaError_t launch_wtile(const Params &P, const Plan &L, int c, int mode, bool update, int fin, const SlotArgs &sa) {
  const int g = L.grid_c[c], t0 = L.tile0[c], t1 = L.tile1[c], th = L.Ww * kWarp, sm = L.smem_wt, cs = L.cap_ws;
  if (mode == M_BWD) return launch(wtile_kernel<PT, M_BWD, false>, g, th, sm, L, P, t0, t1, cs, fin, sa);
  if (update) {
    if (mode == M_FUSED) return launch(wtile_kernel<PT, M_FUSED, true>, g, th, sm, L, P, t0, t1, cs, fin, sa);
    return launch(wtile_kernel<PT, M_FWD, true>, g, th, sm, L, P, t0, t1, cs, fin, sa);
  }
  if (mode == M_FUSED) return launch(wtile_kernel<PT, M_FUSED, false>, g, th, sm, L, P, t0, t1, cs, fin, sa);
  return launch(wtile_kernel<PT, M_FWD, false>, g, th, sm, L, P, t0, t1, cs, fin, sa);
}

template <typename PT, bool STAGE>
cudaError_t launch_pair_s(const Params &P, const Plan &L, int c, int mode, bool update, int fin,
                          const SlotArgs &sa) {
  const int g = L.grid_c[c], t0 = L.tile0[c], t1 = L.tile1[c], th = L.Wp * kWarp;
  const int sm = STAGE ? L.Wp * pair_stage_bytes<PT>() : 0;
  if (mode == M_BWD) return launch(pair_kernel<PT, M_BWD, false, STAGE>, g, th, sm, L, P, t0, t1, fin, sa);
  if (update) {
    if (mode == M_FUSED) return launch(pair_kernel<PT, M_FUSED, true, STAGE>, g, th, sm, L, P, t0, t1, fin, sa);
    return launch(pair_kernel<PT, M_FWD, true, STAGE>, g, th, sm, L, P, t0, t1, fin, sa);
  }
  if (mode == M_FUSED) return launch(pair_kernel<PT, M_FUSED, false, STAGE>, g, th, sm, L, P, t0, t1, fin, sa);
  return launch(pair_kernel<PT, M_FWD, false, STAGE>, g, th, sm, L, P, t0, t1, fin, sa);
}

template <typename PT>
cudaError_t launch_pair(const Params &P, const Plan &L, int c, int mode, bool update, int fin, const SlotArgs &sa) {
  const bool stage = mode == M_BWD ? L.pstage_b[c] != 0 : L.pstage_f[c] != 0;
  return stage ? launch_pair_s<PT, true>(P, L, c, mode, update, fin, sa)
               : launch_pair_s<PT, false>(P, L, c, mode, update, fin, sa);
}

template <typename PT, int S>
cudaError_t launch_unit_s(const Params &P, const Plan &L, int c, int mode, bool update, int fin, const SlotArgs &sa) {
  const int g = L.grid_c[c], t0 = L.unit0[c], t1 = L.unit1[c], th = kUnitWarps * kWarp;
  const int T = L.unit_T[c], sm = unit_smem_bytes(T, int(sizeof(PT)));
  if (mode == M_BWD) return launch(unit_kernel<PT, M_BWD, false, S>, g, th, sm, L, P, t0, t1, T, fin, sa);
  if (update) {
    if (mode == M_FUSED) return launch(unit_kernel<PT, M_FUSED, true, S>, g, th, sm, L, P, t0, t1, T, fin, sa);
    return launch(unit_kernel<PT, M_FWD, true, S>, g, th, sm, L, P, t0, t1, T, fin, sa);
  }
  if (mode == M_FUSED) return launch(unit_kernel<PT, M_FUSED, false, S>, g, th, sm, L, P, t0, t1, T, fin, sa);
  return launch(unit_kernel<PT, M_FWD, false, S>, g, th, sm, L, P, t0, t1, T, fin, sa);
}

template <typename PT>
cudaError_t launch_unit(const Params &P, const Plan &L, int c, int mode, bool update, int fin, const SlotArgs &sa) {
  switch (L.unit_S[c]) {
    case 1: return launch_unit_s<PT, 1>(P, L, c, mode, update, fin, sa);
    case 2: return launch_unit_s<PT, 2>(P, L, c, mode, update, fin, sa);
    case 4: return launch_unit_s<PT, 4>(P, L, c, mode, update, fin, sa);
    case 8: return launch_unit_s<PT, 8>(P, L, c, mode, update, fin, sa);
    case 16: return launch_unit_s<PT, 16>(P, L, c, mode, update, fin, sa);
    default: return launch_unit_s<PT, 32>(P, L, c, mode, update, fin, sa);
  }
}

// Forward launch of color c, with its backward sweep when fused; sums: <r,r> and
// <r,z> are wanted.
template <typename PT>
cudaError_t launch_fwd(const Params &P, const Plan &L, int c, bool update, bool fused, bool sums, int fin) {
  const SlotArgs sa{sums ? L.off[c] : -1, 0, update};   // a final fused launch (one color) has no earlier slots
  const int mode = fused ? M_FUSED : M_FWD;
  if (L.unit1[c] > L.unit0[c]) return launch_unit<PT>(P, L, c, mode, update, fin, sa);
  if (L.tile1[c] > L.tile0[c] && L.wtile[c] == 2) return launch_pair<PT>(P, L, c, mode, update, fin, sa);
  if (L.tile1[c] > L.tile0[c] && L.wtile[c]) return launch_wtile<PT>(P, L, c, mode, update, fin, sa);
  if (L.tile1[c] > L.tile0[c]) return launch_tile<PT>(P, L, c, mode, update, fin, sa);
  const int threads = L.W * kWarp;
  const GroupSmemPlan pl = plan_of<PT>(P, fused, false);
  const int smem = pl.total;
  const int g = L.grid_c[c], t0 = L.task0[c], t1 = L.task1[c];
  if (update) {
    if (fused) return launch(color_kernel<PT, M_FUSED, true>, g, threads, smem, L, P, t0, t1, pl, fin, sa);
    return launch(color_kernel<PT, M_FWD, true>, g, threads, smem, L, P, t0, t1, pl, fin, sa);
  }
  if (fused) return launch(color_kernel<PT, M_FUSED, false>, g, threads, smem, L, P, t0, t1, pl, fin, sa);
  return launch(color_kernel<PT, M_FWD, false>, g, threads, smem, L, P, t0, t1, pl, fin, sa);
}

template <typename PT>
cudaError_t launch_bwd(const Params &P, const Plan &L, int c, bool update, bool sums, int fin) {
  const GroupSmemPlan pl = plan_of<PT>(P, false, true);
  const SlotArgs sa{sums ? L.off[c] : -1, L.off[c], update};
  if (L.unit1[c] > L.unit0[c]) return launch_unit<PT>(P, L, c, M_BWD, false, fin, sa);
  if (L.tile1[c] > L.tile0[c] && L.wtile[c] == 2) return launch_pair<PT>(P, L, c, M_BWD, false, fin, sa);
  if (L.tile1[c] > L.tile0[c] && L.wtile[c]) return launch_wtile<PT>(P, L, c, M_BWD, false, fin, sa);
  if (L.tile1[c] > L.tile0[c]) return launch_tile<PT>(P, L, c, M_BWD, false, fin, sa);
  return launch(color_kernel<PT, M_BWD, false>, L.grid_c[c], L.W * kWarp, pl.total, L, P, L.task0[c], L.task1[c], pl,
                fin, sa);
}

// Forward sweep (with or without the x/r update), fused last color, backward
// sweep.  fin_last: the epilogue run by the last launch.
template <typename PT>
cudaError_t launch_coop_sweep(const Params &P, const Plan &L, bool update, int fin) {
  cudaError_t e = cudaMemsetAsync(P.bar, 0, sizeof(GridBar), L.stream);
  if (e != cudaSuccess) return e;
  const int rr0 = fin == FIN_NONE ? -1 : 0;
  if (update) return launch_coop(coop_sweep_kernel<PT, true>, L.grid_coop, kCoopWarps * kWarp, 0, L.stream, P, 0, fin, rr0, 1);
  return launch_coop(coop_sweep_kernel<PT, false>, L.grid_coop, kCoopWarps * kWarp, 0, L.stream, P, 0, fin, rr0, 1);
}

// the sweep's tail colors (tail_c .. n_c - 1) in one cooperative launch
template <typename PT>
cudaError_t launch_coop_tail(const Params &P, const Plan &L, bool update, bool sums) {
  cudaError_t e = cudaMemsetAsync(P.bar, 0, sizeof(GridBar), L.stream);
  if (e != cudaSuccess) return e;
  const int ct = L.tail_c, nt = L.n_c - ct, rr0 = sums ? L.off[L.n_c - 1] : -1;
  if (update)
    return launch_coop(coop_sweep_kernel<PT, true>, L.grid_tail, kCoopWarps * kWarp, 0, L.stream, P, ct, int(FIN_NONE), rr0, nt);
  return launch_coop(coop_sweep_kernel<PT, false>, L.grid_tail, kCoopWarps * kWarp, 0, L.stream, P, ct, int(FIN_NONE), rr0, nt);
}

template <typename PT>
cudaError_t sweep(const Params &P, const Plan &L, bool update, int fin_last, PhaseHook h, void *u) {
  cudaError_t e = cudaSuccess;
  const int nc = L.n_c, ct = L.tail_c > 0 ? L.tail_c : nc - 1;   // forward launches of their own
  const bool sums = fin_last != FIN_NONE;
  if (L.coop) {
    if (h) h(u, PH_FWD, 1);
    e = launch_coop_sweep<PT>(P, L, update, fin_last);
    if (h) h(u, PH_FWD, 0);
    return e;
  }
  for (int c = 0; c < ct && e == cudaSuccess; ++c) {
    if (h) h(u, PH_FWD, 1);
    e = launch_fwd<PT>(P, L, c, update, false, false, FIN_NONE);
    if (h) h(u, PH_FWD, 0);
  }
  if (e != cudaSuccess) return e;
  if (h) h(u, PH_FUSED, 1);
  e = L.tail_c > 0 ? launch_coop_tail<PT>(P, L, update, sums)
                   : launch_fwd<PT>(P, L, nc - 1, update, true, sums, nc == 1 ? fin_last : FIN_NONE);
  if (h) h(u, PH_FUSED, 0);
  for (int c = ct - 1; c >= 0 && e == cudaSuccess; --c) {
    if (h) h(u, PH_BWD, 1);
    e = launch_bwd<PT>(P, L, c, update, sums, c == 0 ? fin_last : FIN_NONE);
    if (h) h(u, PH_BWD, 0);
  }
  return e;
}

template <int MODE>
cudaError_t launch_spmv(const Params &P, const Plan &L) {
  return launch(spmv_kernel<MODE>, L.grid_a, L.Wa * kWarp, 0, L, P);
}

template <typename K>
cudaError_t allow_smem(K kernel) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024);
}

template <typename PT, int S>
cudaError_t allow_unit() {
  cudaError_t e = allow_smem(unit_kernel<PT, M_FWD, true, S>);
  if (e == cudaSuccess) e = allow_smem(unit_kernel<PT, M_FWD, false, S>);
  if (e == cudaSuccess) e = allow_smem(unit_kernel<PT, M_FUSED, true, S>);
  if (e == cudaSuccess) e = allow_smem(unit_kernel<PT, M_FUSED, false, S>);
  if (e == cudaSuccess) e = allow_smem(unit_kernel<PT, M_BWD, false, S>);
  return e;
}

template <typename PT>
cudaError_t configure_pt() {
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = allow_smem(color_kernel<PT, M_FUSED, true>);
  if (e == cudaSuccess) e = allow_smem(color_kernel<PT, M_FWD, true>);
  if (e == cudaSuccess) e = allow_smem(color_kernel<PT, M_FUSED, false>);
  if (e == cudaSuccess) e = allow_smem(color_kernel<PT, M_FWD, false>);
  if (e == cudaSuccess) e = allow_smem(color_kernel<PT, M_BWD, false>);
  if (e == cudaSuccess) e = allow_smem(persistent_kernel<PT>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_FUSED, true, false>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_FUSED, true, true>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_FWD, true, false>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_FWD, true, true>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_FUSED, false, false>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_FUSED, false, true>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_FWD, false, false>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_FWD, false, true>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_BWD, false, false>);
  if (e == cudaSuccess) e = allow_smem(tile_kernel<PT, M_BWD, false, true>);
  if (e == cudaSuccess) e = allow_smem(pair_kernel<PT, M_FUSED, true, true>);
  if (e == cudaSuccess) e = allow_smem(pair_kernel<PT, M_FWD, true, true>);
  if (e == cudaSuccess) e = allow_smem(pair_kernel<PT, M_FUSED, false, true>);
  if (e == cudaSuccess) e = allow_smem(pair_kernel<PT, M_FWD, false, true>);
  if (e == cudaSuccess) e = allow_smem(pair_kernel<PT, M_BWD, false, true>);
  if (e == cudaSuccess) e = allow_smem(wtile_kernel<PT, M_FUSED, true>);
  if (e == cudaSuccess) e = allow_smem(wtile_kernel<PT, M_FWD, true>);
  if (e == cudaSuccess) e = allow_smem(wtile_kernel<PT, M_FUSED, false>);
  if (e == cudaSuccess) e = allow_smem(wtile_kernel<PT, M_FWD, false>);
  if (e == cudaSuccess) e = allow_smem(wtile_kernel<PT, M_BWD, false>);
  if (e == cudaSuccess) e = allow_unit<PT, 1>();
  if (e == cudaSuccess) e = allow_unit<PT, 2>();
  if (e == cudaSuccess) e = allow_unit<PT, 4>();
  if (e == cudaSuccess) e = allow_unit<PT, 8>();
  if (e == cudaSuccess) e = allow_unit<PT, 16>();
  if (e == cudaSuccess) e = allow_unit<PT, 32>();
  return e;
}

}  // namespace

int group_smem_bytes(int cap, int rows, int levs, int elem) { return group_smem_plan(cap, rows, levs, elem).total; }
int spmv_smem_bytes(int cap) { return r16((cap + 8) * 8) + r16((cap + 8) * 4); }

int tile_resident_ctas(bool fp32, int threads, int smem) {
  int nb = 0;
  const auto kernel = threads == kWarp
                          ? (fp32 ? tile_kernel<float, M_FUSED, true, true> : tile_kernel<double, M_FUSED, true, true>)
                          : (fp32 ? tile_kernel<float, M_FUSED, true, false> : tile_kernel<double, M_FUSED, true, false>);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, size_t(smem)) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return nb > 0 ? nb : 1;
}

int wtile_resident_ctas(bool fp32, int threads, int smem) {
  int nb = 0;
  const cudaError_t e =
      fp32 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, wtile_kernel<float, M_FWD, true>, threads, size_t(smem))
           : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, wtile_kernel<double, M_FWD, true>, threads, size_t(smem));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return nb > 0 ? nb : 1;
}

int pair_resident_ctas(bool fp32, int threads) {
  int nb = 0;
  const cudaError_t e =
      fp32 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pair_kernel<float, M_FWD, true, true>, threads,
                                                           size_t(threads / kWarp) * pair_stage_bytes<float>())
           : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pair_kernel<double, M_FWD, true, true>, threads,
                                                           size_t(threads / kWarp) * pair_stage_bytes<double>());
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return nb > 0 ? nb : 1;
}

int coop_sweep_resident_ctas(bool fp32) {
  int nb = 0;
  const cudaError_t e =
      fp32 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, coop_sweep_kernel<float, true>, kCoopWarps * kWarp, 0)
           : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, coop_sweep_kernel<double, true>, kCoopWarps * kWarp, 0);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}

int unit_resident_ctas(bool fp32, int S, int T, int threads) {
  int nb = 0;
  cudaError_t e;
  const size_t sm = size_t(unit_smem_bytes(T, fp32 ? 4 : 8));
  if (fp32) {
    e = S <= 8 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, unit_kernel<float, M_FWD, true, 8>, threads, sm)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, unit_kernel<float, M_FWD, true, 32>, threads, sm);
  } else {
    e = S <= 8 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, unit_kernel<double, M_FWD, true, 8>, threads, sm)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, unit_kernel<double, M_FWD, true, 32>, threads, sm);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return nb > 0 ? nb : 1;
}

int spmv_resident_ctas(int Wa, int smem) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, spmv_kernel<0>, Wa * kWarp, size_t(smem)) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return nb > 0 ? nb : 1;
}

int solve_body_iterations(const Plan &L) {
  const int64_t launches = 2 + (L.coop ? 1 : 2 * int64_t(L.n_c) - 1);
  return int(std::max<int64_t>(1, std::min<int64_t>(L.body, 160 / std::max<int64_t>(launches, 1))));
}

int persistent_smem_bytes(const Params &P, bool fp32, int W, int budget, int *cap_spmv) {
  const GroupSmemPlan pl = fp32 ? plan_of<float>(P, true, false) : plan_of<double>(P, true, false);
  // two buffers of static group data, the shared row-work arrays, then the
  // SpMV staging; a tile larger than the staging capacity that fits the
  // budget reads global memory instead
  const int groups = pl.o_w + pl.total;
  int cap = P.cap_a;
  while (cap > 4 && W * spmv_smem_bytes(cap) > budget) cap = std::max(4, (cap / 2) & ~3);
  *cap_spmv = cap;
  return groups + W * spmv_smem_bytes(cap);
}

int persistent_resident_ctas(bool fp32, int W, int smem) {
  int nb = 0;
  const cudaError_t e =
      fp32 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, persistent_kernel<float>, W * kWarp, size_t(smem))
           : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, persistent_kernel<double>, W * kWarp, size_t(smem));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}

cudaError_t launch_solve_persistent(const Params &P, const Plan &L, bool fp32) {
  cudaError_t e = cudaMemsetAsync(P.bar, 0, sizeof(GridBar), L.stream);
  if (e != cudaSuccess) return e;
  const int threads = L.W * kWarp;
  if (fp32)
    return launch_coop(persistent_kernel<float>, L.grid_p, threads, L.smem_p, L.stream, P,
                       plan_of<float>(P, true, false), L.cap_p);
  return launch_coop(persistent_kernel<double>, L.grid_p, threads, L.smem_p, L.stream, P,
                     plan_of<double>(P, true, false), L.cap_p);
}

cudaError_t configure_kernels() {
  cudaError_t e = cudaFuncSetAttribute(factor_color_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMaxWarpsPerCta * kWarp * kFacRow * 12);
  if (e == cudaSuccess) e = allow_smem(factor_wide_kernel);
  if (e == cudaSuccess) e = allow_smem(factor_unit_kernel);
  if (e == cudaSuccess) e = configure_pt<double>();
  if (e == cudaSuccess) e = configure_pt<float>();
  return e;
}

// IC(0) of color c as one launch (factor_unit_kernel): warp units of several
// levels with precomputed pairs and rows above kFacShort entries; shorter
// rows would fill too few lanes of a warp (a launch per level, a thread per
// row: 7-point 99x90x85 in blocks of 32 0.62 ms; a warp per row spends 32
// lanes of the scarce FP64 pipe on 3 entries)
bool fac_unit_color(const Plan &L, int c) {
  if (L.unit1[c] <= L.unit0[c] || L.fac_unit_cap <= 0 || L.fac_nlev[c] < 2) return false;
  int wide = 0;
  for (int v = 0; v < L.fac_nlev[c]; ++v) wide = std::max(wide, L.fac_wide[size_t(L.fac_lev0[c] + v)]);
  return wide > kFacShort;
}

cudaError_t launch_factor(const Params &P, const Plan &L, int nL) {
  for (int c = 0; c < L.n_c; ++c) {
    if (fac_unit_color(L, c)) {
      cudaError_t e = launch(factor_unit_kernel, L.unit1[c] - L.unit0[c], kFacUnitWarps * kWarp,
                             fac_unit_bytes(L.fac_unit_cap), L, P, L.unit0[c], L.unit_S[c]);
      if (e != cudaSuccess) return e;
    } else if (L.tile1[c] > L.tile0[c] || L.unit1[c] > L.unit0[c]) {
      // other lane-tile and warp-unit colors: one launch per in-block level
      for (int v = 0; v < L.fac_nlev[c]; ++v) {
        const int k0 = L.fac_ptr[size_t(L.fac_lev0[c] + v)], k1 = L.fac_ptr[size_t(L.fac_lev0[c] + v + 1)];
        // consecutive levels overlap through programmatic dependent launch:
        // a level's static loads run while the previous level finishes
        cudaError_t e;
        const int rows = k1 - k0, wide = L.fac_wide[size_t(L.fac_lev0[c] + v)];
        const bool pairs = P.fac_rec != nullptr;
        if (pairs && wide > kFacShort) {
          const int grid = std::max(1, std::min((rows + kFacWarps - 1) / kFacWarps, 4 * L.grid_v));
          e = launch(factor_warp_kernel, grid, kFacWarps * kWarp, kFacWarps * kFacWarpBytes, L, P, k0, k1);
        } else if (!pairs && wide > kFacShort && wide <= kFacWide) {
          const int grid = std::max(1, std::min((rows + kFacWideWarps - 1) / kFacWideWarps, 4 * L.grid_v));
          const int sm = kFacWideWarps * fac_wide_bytes(wide);
          e = launch(factor_wide_kernel, grid, kFacWideWarps * kWarp, sm, L, P, k0, k1, wide);
        } else {
          const int grid = std::max(1, std::min((rows + kVecThreads - 1) / kVecThreads, L.grid_v));
          e = launch(pairs ? factor_short_kernel : factor_merge_kernel, grid, kVecThreads, 0, L, P, k0, k1);
        }
        if (e != cudaSuccess) return e;
      }
    } else {
      const int threads = L.W * kWarp;
      factor_color_kernel<<<L.grid_c[c], threads, size_t(threads) * kFacRow * 12, L.stream>>>(P, L.task0[c], L.task1[c]);
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
  }
  factor_finish_kernel<<<L.grid_v, kVecThreads, 0, L.stream>>>(P, nL);
  return cudaGetLastError();
}

cudaError_t launch_solve_init(const Params &P, const Plan &L, bool fp32, PhaseHook h, void *u) {
  if (h) h(u, PH_INIT, 1);
  cudaError_t e = cudaMemsetAsync(P.gticket, 0, sizeof(uint32_t) * size_t(P.ngroup), L.stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(P.p0, 0, sizeof(double) * size_t(P.n > 0 ? P.n : 1), L.stream);
  if (e == cudaSuccess) {
    perm_in_kernel<<<L.grid_v, kVecThreads, 0, L.stream>>>(P);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = launch_spmv<1>(P, L);
  if (h) h(u, PH_INIT, 0);
  if (e != cudaSuccess) return e;
  if (h) h(u, PH_INIT, 1);
  e = fp32 ? sweep<float>(P, L, false, FIN_INIT, nullptr, nullptr) : sweep<double>(P, L, false, FIN_INIT, nullptr, nullptr);
  if (h) h(u, PH_INIT, 0);
  return e;
}

cudaError_t launch_spmv_phase(const Params &P, const Plan &L, bool fp32) {
  cudaError_t e = fp32 ? launch(pupdate_kernel<float>, L.grid_v, kVecThreads, 0, L, P)
                       : launch(pupdate_kernel<double>, L.grid_v, kVecThreads, 0, L, P);
  if (e == cudaSuccess) e = launch_spmv<0>(P, L);
  return e;
}

cudaError_t launch_solve_body(const Params &P, const Plan &L, bool fp32, PhaseHook h, void *u) {
  if (h) h(u, PH_SPMV, 1);
  cudaError_t e = launch_spmv_phase(P, L, fp32);
  if (h) h(u, PH_SPMV, 0);
  if (e != cudaSuccess) return e;
  return fp32 ? sweep<float>(P, L, true, FIN_ITER, h, u) : sweep<double>(P, L, true, FIN_ITER, h, u);
}

cudaError_t launch_solve_final(const Params &P, const Plan &L) {
  perm_out_kernel<<<L.grid_v, kVecThreads, 0, L.stream>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_precond(const Params &P, const Plan &L, bool fp32) {
  return fp32 ? sweep<float>(P, L, false, FIN_NONE, nullptr, nullptr) : sweep<double>(P, L, false, FIN_NONE, nullptr, nullptr);
}

cudaError_t launch_spmv_plain(const Params &P, const Plan &L) { return launch_spmv<2>(P, L); }

cudaError_t launch_permute(const double *src, double *dst, const int32_t *perm, int32_t n, bool gather,
                           int32_t grid, cudaStream_t s) {
  permute_kernel<<<grid, kVecThreads, 0, s>>>(src, dst, perm, n, gather ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_widen(const float *src, double *dst, int32_t n, int32_t grid, cudaStream_t s) {
  widen_kernel<<<grid, kVecThreads, 0, s>>>(src, dst, n);
  return cudaGetLastError();
}

}  // namespace iccg
