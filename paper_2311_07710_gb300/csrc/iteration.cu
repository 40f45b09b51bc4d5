// The inner iteration of Algorithm 1 (Section 2) as two fused row-block
// kernels per iteration:
//   k_dual   : rows of A   -- v = A x_tilde, y+ = proj_Y(y - sigma (v - b)),
//              y_bar+ = (1 - 1/beta) y_bar + y+/beta
//   k_primal : rows of P = [Q | -A'] gathering [x_md ; y+] -- g = Q x_md + c - A'y+,
//              x+ = proj_[l,u](x - tau g), x_bar+ = (1 - 1/beta) x_bar + x+/beta,
//              and the next iteration's x_md and x_tilde
// with their pipelined persistent variants, the kernels of a row per thread on
// the slice layout, the member-interleaved family kernels, the segment sums of
// long rows, and the host loop that launches a chunk of iterations (a whole chunk
// in one launch: chunk.cu).
#include <algorithm>

#include "rowblock.cuh"
#include "rowupdate.cuh"

namespace pdqp {

// --------------------------------------------------------------------------
// One inner iteration of Algorithm 1: the dual half-step (rows of A)
// --------------------------------------------------------------------------
template <typename V>
struct DualB {
  BCsr<V> A;
  const V* xt;      // extrapolated primal point x_tilde
  const V* yold;    // y^k
  V* ynew;          // y^{k+1}
  V* ybar;
  const V* b;
  const V* ylo;     // lower bound of inequality duals (mixed-mode shift) or null (0)
  const StepEntry* tab;    // [instance][C]
  const int* __restrict__ blk_inst;     // instance of each row block
  const DevState* st;      // per instance
  const unsigned char* __restrict__ ineq;   // per row: inequality
  int C;
  const int2* __restrict__ blk_seg;     // long rows: {first segment, segments} per block (null: none)
  const V* lpart;          // segment sums of the long rows
  const int* act;          // row block of each CUDA block (null: the block index)
  int early;                            // launched by launch_early: no state read before grid_wait()
};

template <typename V>
__device__ __forceinline__ void dual_row(const DualB<V>& a, const StepEntry& e, int r, V s, V yo, V bi, V yb,
                                         V lo) {
  V yn, ybn;
  dual_update<V>(e, s, yo, bi, yb, lo, a.ineq[r] != 0, yn, ybn);
  a.ybar[r] = ybn;
  a.ynew[r] = yn;
}

__device__ __forceinline__ float staged_sum(const float* prod, const float*, int e, int end) {
  float s = 0.f;
  for (; e < end; ++e) s += prod[e];
  return s;
}
__device__ __forceinline__ double staged_sum(const double* sval, const double* sx, int e, int end) {
  double s = 0.0;
  for (; e < end; ++e) s = r_dot(sval[e], sx[e], s);
  return s;
}

// The dual half-step of row block bk (one CUDA block): prod, sx and srp are the
// block's staging buffers.
template <typename V, int NT>
__device__ __forceinline__ void dual_block(const DualB<V>& a, int bk, int j, V* prod, V* sx, int* srp) {
  const int tid = threadIdx.x;
  const int inst = a.blk_inst[bk];
  if (!a.early && a.st[inst].status != ST_RUNNING) return;    // uniform over the block
  const int r0 = a.A.blk[bk], r1 = a.A.blk[bk + 1];
  const int nr = r1 - r0;
  const int e0 = a.A.rp[r0];
  const int ne = a.A.rp[r1] - e0;
  // operands of this thread's first row, fetched before the gathers
  V yo = V(0), bi = V(0), yb = V(0), lo = V(0);
  auto mid = [&]() {
    grid_wait();
    if (a.early && a.st[inst].status != ST_RUNNING) return false;
    if (tid < nr) {
      const int r = r0 + tid;
      yo = a.yold[r]; bi = a.b[r]; yb = a.ybar[r];
      if (a.ylo) lo = a.ylo[r];
    }
    return true;
  };
  if (ne > BNNZ && !mid()) return;
  if (ne <= BNNZ) {
    if (!stage_rows<NT>(a.A, a.xt, e0, ne, r0, nr, prod, sx, srp, mid)) return;
    __syncthreads();
    const StepEntry& es = a.tab[inst * a.C + j];
    for (int t = tid; t < nr; t += NT) {
      const V s = staged_sum(prod, sx, srp[t], srp[t + 1]);
      const int r = r0 + t;
      if (t >= BNT) {
        yo = a.yold[r]; bi = a.b[r]; yb = a.ybar[r];
        lo = a.ylo ? a.ylo[r] : V(0);
      }
      dual_row(a, es, r, s, yo, bi, yb, lo);
    }
  } else if (a.blk_seg) {   // a long row: the sum of its segments (k_long_partials), in order
    if (tid == 0) {
      const int2 sg = a.blk_seg[bk];
      V s = V(0);
      for (int q = 0; q < sg.y; ++q) s += a.lpart[sg.x + q];
      dual_row(a, a.tab[inst * a.C + j], r0, s, yo, bi, yb, lo);
    }
  } else {   // a single row longer than a block
    V s = V(0);
    for (int e = e0 + tid; e < e0 + ne; e += NT)
      s += a.A.val[e] * a.xt[a.A.col[e]];
    s = block_sum(s);
    if (tid == 0) dual_row(a, a.tab[inst * a.C + j], r0, s, yo, bi, yb, lo);
  }
}

template <typename V, int NT>
__global__ void __launch_bounds__(NT, MinBlocks<V, NT>::value) k_dual(DualB<V> a, int j) {
  __shared__ V prod[BNNZ];
  __shared__ V sx[sizeof(V) == 8 ? BNNZ : 1];
  __shared__ int srp[BROWS + 1];
  grid_trigger();
  const int bk = a.act ? a.act[blockIdx.x] : (int)blockIdx.x;   // compacted batches: running blocks only
  if (bk < 0) return;                                             // padding of a compacted grid
  dual_block<V, NT>(a, bk, j, prod, sx, srp);
}

// --------------------------------------------------------------------------
// One inner iteration of Algorithm 1: the primal half-step (rows of P)
// --------------------------------------------------------------------------
template <typename V>
struct PrimalB {
  BCsr<V> P;
  const V* zin;     // [x_md ; y^{k+1}] of this iteration
  V* zout;          // x_md of the next iteration -> zout[0:n]
  V* x;
  V* xbar;
  V* xt;            // x_tilde of the next iteration
  const V* c;
  const V* l;
  const V* u;
  const StepEntry* tab;    // [instance][C]
  const int* __restrict__ blk_inst;
  const DevState* st;
  int C;
  const V* F;              // low-rank factor F~ (null: none)
  const V* wlr;            // F~' x_md of this iteration
  int r;
  const int2* __restrict__ blk_seg;     // long rows: {first segment, segments} per block (null: none)
  const V* lpart;          // segment sums of the long rows
  const int* act;          // row block of each CUDA block (null: the block index)
  int early;                            // launched by launch_early: no state read before grid_wait()
};

template <typename V, bool LR = false>
__device__ __forceinline__ void primal_row(const PrimalB<V>& a, const StepEntry& e, int r, V s, V xo, V xb0,
                                           V cr, V lr, V ur) {
  V g = r_add(s, cr);
  if constexpr (LR) g = r_add(g, lr_row<V, V, V>(a.F, a.wlr, a.r, r));
  V xn, xb, zo, xtn;
  primal_update<V>(e, g, xo, xb0, lr, ur, xn, xb, zo, xtn);
  a.xbar[r] = xb;
  a.zout[r] = zo;
  a.xt[r] = xtn;
  a.x[r] = xn;
}

// The primal half-step of row block bk (one CUDA block), as dual_block.
template <typename V, int NT, bool LR>
__device__ __forceinline__ void primal_block(const PrimalB<V>& a, int bk, int j, V* prod, V* sx, int* srp) {
  const int tid = threadIdx.x;
  const int inst = a.blk_inst[bk];
  if (!a.early && a.st[inst].status != ST_RUNNING) return;    // uniform over the block
  const int r0 = a.P.blk[bk], r1 = a.P.blk[bk + 1];
  const int nr = r1 - r0;
  const int e0 = a.P.rp[r0];
  const int ne = a.P.rp[r1] - e0;
  V xo = V(0), xb = V(0), cr = V(0), lr = V(0), ur = V(0);
  auto mid = [&]() {
    grid_wait();
    if (a.early && a.st[inst].status != ST_RUNNING) return false;
    if (tid < nr) {
      const int r = r0 + tid;
      xo = a.x[r]; xb = a.xbar[r]; cr = a.c[r]; lr = a.l[r]; ur = a.u[r];
    }
    return true;
  };
  if (ne > BNNZ && !mid()) return;
  if (ne <= BNNZ) {
    if (!stage_rows<NT>(a.P, a.zin, e0, ne, r0, nr, prod, sx, srp, mid)) return;
    __syncthreads();
    const StepEntry& es = a.tab[inst * a.C + j];
    for (int t = tid; t < nr; t += NT) {
      const V s = staged_sum(prod, sx, srp[t], srp[t + 1]);
      const int r = r0 + t;
      if (t >= BNT) { xo = a.x[r]; xb = a.xbar[r]; cr = a.c[r]; lr = a.l[r]; ur = a.u[r]; }
      primal_row<V, LR>(a, es, r, s, xo, xb, cr, lr, ur);
    }
  } else if (a.blk_seg) {
    if (tid == 0) {
      const int2 sg = a.blk_seg[bk];
      V s = V(0);
      for (int q = 0; q < sg.y; ++q) s += a.lpart[sg.x + q];
      primal_row<V, LR>(a, a.tab[inst * a.C + j], r0, s, xo, xb, cr, lr, ur);
    }
  } else {
    V s = V(0);
    for (int e = e0 + tid; e < e0 + ne; e += NT)
      s += a.P.val[e] * a.zin[a.P.col[e]];
    s = block_sum(s);
    if (tid == 0) primal_row<V, LR>(a, a.tab[inst * a.C + j], r0, s, xo, xb, cr, lr, ur);
  }
}

// LR: the problem has a low-rank term (its row term gets its own instantiation
// so that the plain kernel keeps its 32 registers)
template <typename V, int NT, bool LR = false>
__global__ void __launch_bounds__(NT, MinBlocks<V, NT, LR>::value) k_primal(PrimalB<V> a, int j) {
  __shared__ V prod[BNNZ];
  __shared__ V sx[sizeof(V) == 8 ? BNNZ : 1];
  __shared__ int srp[BROWS + 1];
  grid_trigger();
  const int bk = a.act ? a.act[blockIdx.x] : (int)blockIdx.x;
  if (bk < 0) return;
  // (the dual half-step measured no gain from it: 202.6 -> 203.9 ms of a control-QP
  // batch solve, against 225.4 -> 219.9 here)
  prefetch_ahead(a.P, a.act, (int)blockIdx.x, (int)gridDim.x);
  primal_block<V, NT, LR>(a, bk, j, prod, sx, srp);
}

// Segment sums of the long rows: one CUDA block per segment of LSEG nonzeros
// of M v (skipping instances that stopped); the iteration kernels add a row's
// segments in order.
template <typename V>
__global__ void __launch_bounds__(256) k_long_partials(BCsr<V> M, const V* __restrict__ vec,
                                                       const int4* __restrict__ lseg, const int* __restrict__ blk_inst,
                                                       const DevState* __restrict__ st, V* __restrict__ out) {
  const int4 g = lseg[blockIdx.x];
  if (st[blk_inst[g.w]].status != ST_RUNNING) return;
  long_segment_sum(M, vec, g, out + blockIdx.x);
}


// ==========================================================================
// One row per thread on a slice layout (one instance without long rows): 32 rows a
// slice, entry pairs of a slice's rows side by side, so that a warp's index and
// value loads are contiguous and nothing is staged in shared memory.
// The staged row blocks fill 2.4 (P) and 1.2 (A) waves of an n = 300007 problem
// and wait at a barrier each; here all warps of an SM have gathers in flight and
// L2's sectors (one of 32 bytes for a value) are the bound.
// ==========================================================================
constexpr int SL_U = 2;                  // pairs of a row in flight
// Warps per SM against pairs in flight, n = 1e6 in float32 / 300007 in float64:
// 64 / 32 warps and two pairs 115 / 52 us an iteration, 48 / 40 and two 118 / 58,
// 48 / 32 and three 115 / 54, 40 / 24 and four 120 / 64.
template <typename V> struct Sl;
template <> struct Sl<float> { static constexpr int NT = 128, MINB = 16; };
template <> struct Sl<double> { static constexpr int NT = 64, MINB = 16; };

template <typename V> struct V2;
template <> struct V2<float> { using T = float2; };
template <> struct V2<double> { using T = double2; };

// the matrix passes through once: not kept in L1, which the gathered vector needs
__device__ __forceinline__ int2 ld_once(const int2* p) {
  int2 v;
  asm("ld.global.nc.L1::no_allocate.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ld_once(const float2* p) {
  float2 v;
  asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ double2 ld_once(const double2* p) {
  double2 v;
  asm("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}

template <typename V>
struct SliceM {
  const int* __restrict__ rp;            // the CSR row pointers
  const int* __restrict__ sp;            // slice starts, in groups of 32 pairs
  const int2* __restrict__ idx;
  const typename V2<V>::T* __restrict__ val;
};
// a thread's row: its length and its first pairs
template <typename V>
struct SliceRow {
  int len;
  const int2* c;
  const typename V2<V>::T* v;
  int2 hc[SL_U];
  typename V2<V>::T hv[SL_U];
};
template <typename V>
__device__ __forceinline__ void slice_head(const SliceM<V>& M, int r, bool on, SliceRow<V>& h) {
  h.len = on ? M.rp[r + 1] - M.rp[r] : 0;
  const size_t at = on ? (size_t)M.sp[r >> 5] * 32 + (r & 31) : 0;
  h.c = M.idx + at;
  h.v = M.val + at;
#pragma unroll
  for (int k = 0; k < SL_U; ++k)
    if (2 * k < h.len) { h.hc[k] = ld_once(h.c + 32 * k); h.hv[k] = ld_once(h.v + 32 * k); }
}
// the row's sum, its entries in CSR order by r_dot as in every variant
template <typename V>
__device__ __forceinline__ V slice_sum(SliceRow<V>& h, const V* vec) {
  V s = V(0);
  for (int e = 0; e < h.len; e += 2 * SL_U) {
    V x[2 * SL_U];
    typename V2<V>::T v[SL_U];
#pragma unroll
    for (int k = 0; k < SL_U; ++k) {
      x[2 * k] = e + 2 * k < h.len ? vec[h.hc[k].x] : V(0);
      x[2 * k + 1] = e + 2 * k + 1 < h.len ? vec[h.hc[k].y] : V(0);
      v[k] = h.hv[k];
    }
#pragma unroll
    for (int k = 0; k < SL_U; ++k) {
      const int p = (e >> 1) + SL_U + k;
      if (2 * p < h.len) { h.hc[k] = ld_once(h.c + 32 * p); h.hv[k] = ld_once(h.v + 32 * p); }
    }
#pragma unroll
    for (int k = 0; k < SL_U; ++k) {
      if (e + 2 * k < h.len) s = r_dot(v[k].x, x[2 * k], s);
      if (e + 2 * k + 1 < h.len) s = r_dot(v[k].y, x[2 * k + 1], s);
    }
  }
  return s;
}

template <typename V>
__global__ void __launch_bounds__(Sl<V>::NT, Sl<V>::MINB) k_dual_sl(DualB<V> a, SliceM<V> M, int m, int j) {
  grid_trigger();
  const int r = blockIdx.x * Sl<V>::NT + threadIdx.x;
  const bool on = r < m;
  SliceRow<V> h;
  slice_head(M, r, on, h);
  grid_wait();
  if (!on || a.st->status != ST_RUNNING) return;
  const V s = slice_sum(h, a.xt);
  dual_row(a, a.tab[j], r, s, a.yold[r], a.b[r], a.ybar[r], a.ylo ? a.ylo[r] : V(0));
}
template <typename V>
__global__ void __launch_bounds__(Sl<V>::NT, Sl<V>::MINB) k_primal_sl(PrimalB<V> a, SliceM<V> M, int n, int j) {
  grid_trigger();
  const int r = blockIdx.x * Sl<V>::NT + threadIdx.x;
  const bool on = r < n;
  SliceRow<V> h;
  slice_head(M, r, on, h);
  grid_wait();
  if (!on || a.st->status != ST_RUNNING) return;
  const V s = slice_sum(h, a.zin);
  primal_row<V, false>(a, a.tab[j], r, s, a.x[r], a.xbar[r], a.c[r], a.l[r], a.u[r]);
}

template <typename V>
static void run_chunk_sl(Work& w, int j0, int len, V* xt, V* const* Z, V* ybar, const V* b, const V* ylo, V* x, V* xbar,
                         const V* c, const V* l, const V* u, cudaStream_t s) {
  using T = typename V2<V>::T;
  Profiler& Pr = w.prof;
  const SlicePlan& q = w.slices;
  const T* val = sizeof(V) == 4 ? (const T*)q.valf : (const T*)q.vald;
  DualB<V> da{};
  da.xt = xt; da.ybar = ybar; da.b = b; da.ylo = ylo; da.tab = w.tab; da.st = w.st; da.ineq = w.row_ineq;
  PrimalB<V> pa{};
  pa.x = x; pa.xbar = xbar; pa.xt = xt; pa.c = c; pa.l = l; pa.u = u; pa.tab = w.tab; pa.st = w.st;
  const SliceM<V> A{w.A.rp, q.sp, q.idx, val}, P{w.P.rp, q.sp + q.nsA, q.idx, val};
  for (int j = j0; j < j0 + len; ++j) {
    if (w.m > 0) {
      da.yold = Z[(j + 1) & 1] + w.n;
      da.ynew = Z[j & 1] + w.n;
      if (Pr.on) Pr.begin(0, s, launch_bytes(w, 0, sizeof(V)));
      launch_early(k_dual_sl<V>, cdiv(w.m, Sl<V>::NT), Sl<V>::NT, 0, s, da, A, w.m, j);
      if (Pr.on) Pr.end(s);
    }
    pa.zin = Z[j & 1];
    pa.zout = Z[(j + 1) & 1];
    if (Pr.on) Pr.begin(1, s, launch_bytes(w, 1, sizeof(V)));
    launch_early(k_primal_sl<V>, cdiv(w.n, Sl<V>::NT), Sl<V>::NT, 0, s, pa, P, w.n, j);
    if (Pr.on) Pr.end(s);
  }
}

// The slice layout from the CSR arrays: A's slices, then P's.
// width of a slice in pairs: its longest row, rounded up
__global__ void __launch_bounds__(256) k_slice_width(const int* __restrict__ arp, int m, int nsA,
                                                     const int* __restrict__ prp, int n, int ns,
                                                     int* __restrict__ wid) {
  const int s = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (s >= ns) return;
  const bool isA = s < nsA;
  const int r = 32 * (isA ? s : s - nsA) + lane;
  const int* rp = isA ? arp : prp;
  const int len = __reduce_max_sync(0xffffffffu, r < (isA ? m : n) ? rp[r + 1] - rp[r] : 0);
  if (lane == 0) wid[s] = (len + 1) >> 1;
}
// columns (val null) or values; the second half of a row's last pair may be a pad
template <typename V, bool VALUES>
__global__ void __launch_bounds__(256) k_slice_fill(BCsr<V> A, int m, int nsA, BCsr<V> P, int n, int ns,
                                                    const int* __restrict__ sp, int2* __restrict__ idx,
                                                    typename V2<V>::T* __restrict__ val) {
  const int s = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (s >= ns) return;
  const bool isA = s < nsA;
  const int r = 32 * (isA ? s : s - nsA) + lane;
  if (r >= (isA ? m : n)) return;
  const int* rp = isA ? A.rp : P.rp;
  const int e1 = rp[r + 1];
  size_t at = (size_t)sp[s] * 32 + lane;
  for (int e = rp[r]; e < e1; e += 2, at += 32) {
    if constexpr (VALUES) {
      const V* v = isA ? A.val : P.val;
      typename V2<V>::T q;
      q.x = v[e];
      q.y = e + 1 < e1 ? v[e + 1] : V(0);
      val[at] = q;
    } else {
      const int* c = isA ? A.col : P.col;
      idx[at] = make_int2(c[e], e + 1 < e1 ? c[e + 1] : 0);
    }
  }
}
// One row per thread has a longer chain than a staged row block: below some 24 MB
// of matrix the row blocks are faster (n = 60000 in float64: 22.5 against 30.2 us
// an iteration, n = 300007 in float32: 41.1 against 49.6), above it the solve's
// tuning decides (n = 300007 in float64: 85.1 against 51.9, n = 1e6 in float32:
// 123.9 against 115.0).
bool slices_ok(const Work& w, bool mixed) {
  return w.count == 1 && w.r == 0 && w.A.nlseg == 0 && w.P.nlseg == 0 && w.P.nblk > 0 &&
         (w.A.nnz + w.P.nnz) * (mixed ? 8 : 12) >= 24LL << 20;
}
void slices_width(Work& w, int* wid, cudaStream_t s) {
  const SlicePlan& q = w.slices;
  launch(k_slice_width, cdiv(q.nsA + q.nsP, 8), 256, 0, s, (const int*)w.A.rp, w.m, q.nsA, (const int*)w.P.rp, w.n,
         q.nsA + q.nsP, wid);
}
void slices_fill_index(Work& w, cudaStream_t s) {
  const SlicePlan& q = w.slices;
  launch(k_slice_fill<float, false>, cdiv(q.nsA + q.nsP, 8), 256, 0, s, w.A.bscaled_f(), w.m, q.nsA, w.P.bscaled_f(),
         w.n, q.nsA + q.nsP, (const int*)q.sp, q.idx, (float2*)nullptr);
}
void slices_fill_values(Work& w, bool mixed, cudaStream_t s) {
  const SlicePlan& q = w.slices;
  if (mixed)
    launch(k_slice_fill<float, true>, cdiv(q.nsA + q.nsP, 8), 256, 0, s, w.A.bscaled_f(), w.m, q.nsA, w.P.bscaled_f(),
           w.n, q.nsA + q.nsP, (const int*)q.sp, (int2*)nullptr, q.valf);
  else
    launch(k_slice_fill<double, true>, cdiv(q.nsA + q.nsP, 8), 256, 0, s, w.A.bscaled(), w.m, q.nsA, w.P.bscaled(),
           w.n, q.nsA + q.nsP, (const int*)q.sp, (int2*)nullptr, q.vald);
}

// ==========================================================================
// Pipelined persistent variants of the two half-steps.  Each CUDA block loops
// over row blocks b = blockIdx.x, blockIdx.x + gridDim.x, ...; while it
// gathers and finishes block b, the index, value and row-pointer ranges of its
// next block stream into the other shared-memory stage with cp.async (16-byte
// copies of the 16-byte aligned superset of each range).  Block bounds come
// from one int4 {r0, r1, e0, e1} per block.  Global index/value/rowptr arrays
// carry 8 elements of padding so the aligned superset never leaves them.
// ==========================================================================
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::); }

template <typename V>
struct PipeSmem {
  int col[2][BNNZ + 8];
  V val[2][BNNZ + 8];
  int rp[2][BROWS + 8];
  V prod[BNNZ];
};

// Queue the copies of block m = {r0, r1, e0, e1} into stage s (no copy for a long row).
template <int NT, typename V>
__device__ __forceinline__ void pipe_issue(PipeSmem<V>& sm, int s, const int4 m, const int* __restrict__ col,
                                           const V* __restrict__ val, const int* __restrict__ rp) {
  const int tid = threadIdx.x;
  if (m.w - m.z <= BNNZ) {
    const int a0 = m.z & ~3, a1 = (m.w + 3) & ~3;
    for (int c = tid; c < (a1 - a0) >> 2; c += NT) cp_async16(&sm.col[s][c << 2], col + a0 + (c << 2));
    constexpr int PER = 16 / sizeof(V);
    for (int c = tid; c < (a1 - a0) / PER; c += NT) cp_async16(&sm.val[s][c * PER], val + a0 + c * PER);
    const int q0 = m.x & ~3, q1 = (m.y + 1 + 3) & ~3;
    for (int c = tid; c < (q1 - q0) >> 2; c += NT) cp_async16(&sm.rp[s][c << 2], rp + q0 + (c << 2));
  }
  cp_async_commit();
}

// what prod holds, and one term of a row sum from it (float32: the product;
// float64: the gathered entry, fused with its value)
__device__ __forceinline__ float pipe_entry(float v, float x) { return v * x; }
__device__ __forceinline__ double pipe_entry(double, double x) { return x; }
__device__ __forceinline__ float pipe_add(float s, float, float p) { return s + p; }
__device__ __forceinline__ double pipe_add(double s, double v, double x) { return r_dot(v, x, s); }

template <typename V, int NT>
__global__ void __launch_bounds__(NT) k_dual_pipe(DualB<V> a, const int4* __restrict__ meta, int nblk, int j) {
  extern __shared__ __align__(16) unsigned char smraw[];
  PipeSmem<V>& sm = *reinterpret_cast<PipeSmem<V>*>(smraw);
  const int tid = threadIdx.x;
  int b = blockIdx.x;
  if (b >= nblk) return;
  int4 mc = meta[b];
  pipe_issue<NT>(sm, 0, mc, a.A.col, a.A.val, a.A.rp);
  for (int s = 0; b < nblk; b += gridDim.x, s ^= 1) {
    const int bn = b + gridDim.x;
    int4 mn = make_int4(0, 0, 0, 0);
    if (bn < nblk) mn = meta[bn];
    pipe_issue<NT>(sm, s ^ 1, mn, a.A.col, a.A.val, a.A.rp);
    const int r0 = mc.x, nr = mc.y - mc.x, e0 = mc.z, ne = mc.w - mc.z;
    const int inst = a.blk_inst[b];
    const bool live = a.st[inst].status == ST_RUNNING;
    const StepEntry& es = a.tab[inst * a.C + j];
    V yo = V(0), bi = V(0), yb = V(0), lo = V(0);
    if (live && tid < nr) {
      const int r = r0 + tid;
      yo = a.yold[r]; bi = a.b[r]; yb = a.ybar[r];
      if (a.ylo) lo = a.ylo[r];
    }
    cp_async_wait1();
    __syncthreads();
    if (!live) {
    } else if (ne <= BNNZ) {
      const int off = e0 - (e0 & ~3), roff = r0 - (r0 & ~3);
#pragma unroll
      for (int k = 0; k < BNNZ / NT; ++k) {
        const int e = tid + k * NT;
        if (e < ne) sm.prod[e] = pipe_entry(sm.val[s][e + off], a.xt[sm.col[s][e + off]]);
      }
      __syncthreads();
      for (int t = tid; t < nr; t += NT) {
        V acc = V(0);
        const int eb = sm.rp[s][t + roff] - e0, ee = sm.rp[s][t + 1 + roff] - e0;
        for (int e = eb; e < ee; ++e) acc = pipe_add(acc, sm.val[s][e + off], sm.prod[e]);
        const int r = r0 + t;
        if (t >= NT) {
          yo = a.yold[r]; bi = a.b[r]; yb = a.ybar[r];
          lo = a.ylo ? a.ylo[r] : V(0);
        }
        dual_row(a, es, r, acc, yo, bi, yb, lo);
      }
    } else if (a.blk_seg) {   // a long row: the sum of its segments (k_long_partials), as k_dual
      if (tid == 0) {
        const int2 sg = a.blk_seg[b];
        V acc = V(0);
        for (int q = 0; q < sg.y; ++q) acc += a.lpart[sg.x + q];
        dual_row(a, es, r0, acc, yo, bi, yb, lo);
      }
    } else {
      V acc = V(0);
      for (int e = e0 + tid; e < e0 + ne; e += NT) acc += a.A.val[e] * a.xt[a.A.col[e]];
      acc = block_sum(acc);
      if (tid == 0) dual_row(a, es, r0, acc, yo, bi, yb, lo);
    }
    __syncthreads();
    mc = mn;
  }
}

template <typename V, int NT>
__global__ void __launch_bounds__(NT) k_primal_pipe(PrimalB<V> a, const int4* __restrict__ meta, int nblk, int j) {
  extern __shared__ __align__(16) unsigned char smraw[];
  PipeSmem<V>& sm = *reinterpret_cast<PipeSmem<V>*>(smraw);
  const int tid = threadIdx.x;
  int b = blockIdx.x;
  if (b >= nblk) return;
  int4 mc = meta[b];
  pipe_issue<NT>(sm, 0, mc, a.P.col, a.P.val, a.P.rp);
  for (int s = 0; b < nblk; b += gridDim.x, s ^= 1) {
    const int bn = b + gridDim.x;
    int4 mn = make_int4(0, 0, 0, 0);
    if (bn < nblk) mn = meta[bn];
    pipe_issue<NT>(sm, s ^ 1, mn, a.P.col, a.P.val, a.P.rp);
    const int r0 = mc.x, nr = mc.y - mc.x, e0 = mc.z, ne = mc.w - mc.z;
    const int inst = a.blk_inst[b];
    const bool live = a.st[inst].status == ST_RUNNING;
    const StepEntry& es = a.tab[inst * a.C + j];
    V xo = V(0), xb = V(0), cr = V(0), lr = V(0), ur = V(0);
    if (live && tid < nr) {
      const int r = r0 + tid;
      xo = a.x[r]; xb = a.xbar[r]; cr = a.c[r]; lr = a.l[r]; ur = a.u[r];
    }
    cp_async_wait1();
    __syncthreads();
    if (!live) {
    } else if (ne <= BNNZ) {
      const int off = e0 - (e0 & ~3), roff = r0 - (r0 & ~3);
#pragma unroll
      for (int k = 0; k < BNNZ / NT; ++k) {
        const int e = tid + k * NT;
        if (e < ne) sm.prod[e] = pipe_entry(sm.val[s][e + off], a.zin[sm.col[s][e + off]]);
      }
      __syncthreads();
      for (int t = tid; t < nr; t += NT) {
        V acc = V(0);
        const int eb = sm.rp[s][t + roff] - e0, ee = sm.rp[s][t + 1 + roff] - e0;
        for (int e = eb; e < ee; ++e) acc = pipe_add(acc, sm.val[s][e + off], sm.prod[e]);
        const int r = r0 + t;
        if (t >= NT) { xo = a.x[r]; xb = a.xbar[r]; cr = a.c[r]; lr = a.l[r]; ur = a.u[r]; }
        if (a.F) primal_row<V, true>(a, es, r, acc, xo, xb, cr, lr, ur);
        else primal_row<V, false>(a, es, r, acc, xo, xb, cr, lr, ur);
      }
    } else if (a.blk_seg) {   // a long row: the sum of its segments, as k_primal
      if (tid == 0) {
        const int2 sg = a.blk_seg[b];
        V acc = V(0);
        for (int q = 0; q < sg.y; ++q) acc += a.lpart[sg.x + q];
        if (a.F) primal_row<V, true>(a, es, r0, acc, xo, xb, cr, lr, ur);
        else primal_row<V, false>(a, es, r0, acc, xo, xb, cr, lr, ur);
      }
    } else {
      V acc = V(0);
      for (int e = e0 + tid; e < e0 + ne; e += NT) acc += a.P.val[e] * a.zin[a.P.col[e]];
      acc = block_sum(acc);
      if (tid == 0) {
        if (a.F) primal_row<V, true>(a, es, r0, acc, xo, xb, cr, lr, ur);
        else primal_row<V, false>(a, es, r0, acc, xo, xb, cr, lr, ur);
      }
    }
    __syncthreads();
    mc = mn;
  }
}

// resident blocks per SM of a pipelined kernel (its shared-memory limit set
// once; a function-local static is initialised once, thread-safely)
template <typename K>
static int pipe_blocks(K kern, int nt, size_t smem) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem);
  return per_sm > 0 ? per_sm : 1;
}
template <typename V, int NT>
static int pipe_grid(void (*kern)(DualB<V>, const int4*, int, int)) {
  static const int blocks = pipe_blocks(kern, NT, sizeof(PipeSmem<V>));
  return blocks;
}
template <typename V, int NT>
static int pipe_grid_p(void (*kern)(PrimalB<V>, const int4*, int, int)) {
  static const int blocks = pipe_blocks(kern, NT, sizeof(PipeSmem<V>));
  return blocks;
}

// Algorithmic bytes of one dual (kind 0) or primal (kind 1) launch over the
// instances running at the last check: the matrix streams (index + value),
// the row pointers, each vector read or written once (the gathered vector
// counted once); sv = bytes per value.
double launch_bytes(const Work& w, int kind, double sv) {
  const BatchState& b = *w.bst_host;
  if (kind == 0) return b.run_nnzA * (sv + 4.0) + 4.0 * (b.run_m + 1.0) + sv * (b.run_n + 5.0 * b.run_m);
  return b.run_nnzP * (sv + 4.0) + 4.0 * (b.run_n + 1.0) + sv * (10.0 * b.run_n + b.run_m);
}

template <typename V, int NT>
static void run_chunk_pipe(Work& w, int j0, int len, BCsr<V> A, BCsr<V> P, V* xt, V* const* Z, V* ybar, const V* b,
                           const V* ylo, V* x, V* xbar, const V* c, const V* l, const V* u, cudaStream_t s) {
  Profiler& Pr = w.prof;
  DualB<V> da{A, xt, nullptr, nullptr, ybar, b, ylo, w.tab, w.blk_inst_A, w.st, w.row_ineq, w.tab_stride};
  PrimalB<V> pa{P, nullptr, nullptr, x, xbar, xt, c, l, u, w.tab, w.blk_inst_P, w.st, w.tab_stride,
                w.r > 0 ? lr_factor<V>(w) : nullptr, lr_weights<V>(w), w.r};
  const int gd = std::min(w.A.nblk, w.num_sms * pipe_grid<V, NT>(k_dual_pipe<V, NT>));
  const int gp = std::min(w.P.nblk, w.num_sms * pipe_grid_p<V, NT>(k_primal_pipe<V, NT>));
  const size_t smem = sizeof(PipeSmem<V>);
  // long rows: segment sums first, the same as the row-block variants
  V* lpA = sizeof(V) == 4 ? (V*)w.A.lpart_f : (V*)w.A.lpart_d;
  V* lpP = sizeof(V) == 4 ? (V*)w.P.lpart_f : (V*)w.P.lpart_d;
  if (w.A.nlseg) { da.blk_seg = w.A.blk_seg; da.lpart = lpA; }
  if (w.P.nlseg) { pa.blk_seg = w.P.blk_seg; pa.lpart = lpP; }
  for (int j = j0; j < j0 + len; ++j) {
    if (w.r > 0) lowrank_ft1(w, pa.F, (const V*)Z[j & 1], s);
    if (w.m > 0) {
      da.yold = Z[(j + 1) & 1] + w.n;
      da.ynew = Z[j & 1] + w.n;
      if (Pr.on) Pr.begin(0, s, launch_bytes(w, 0, sizeof(V)));
      if (w.A.nlseg)
        launch(k_long_partials<V>, w.A.nlseg, 256, 0, s, A, (const V*)xt, (const int4*)w.A.lseg,
               (const int*)w.blk_inst_A, (const DevState*)w.st, lpA);
      launch(k_dual_pipe<V, NT>, gd, NT, smem, s, da, (const int4*)w.A.meta, w.A.nblk, j);
      if (Pr.on) Pr.end(s);
    }
    pa.zin = Z[j & 1];
    pa.zout = Z[(j + 1) & 1];
    if (Pr.on) Pr.begin(1, s, launch_bytes(w, 1, sizeof(V)));
    if (w.P.nlseg)
      launch(k_long_partials<V>, w.P.nlseg, 256, 0, s, P, (const V*)pa.zin, (const int4*)w.P.lseg,
             (const int*)w.blk_inst_P, (const DevState*)w.st, lpP);
    launch(k_primal_pipe<V, NT>, gp, NT, smem, s, pa, (const int4*)w.P.meta, w.P.nblk, j);
    if (Pr.on) Pr.end(s);
  }
}

// The dual half-step beside the reduction of F' x_md from its tiles' partials (the
// low-rank half-step, lowrank.cu): blocks [0, r) sum a column each, the next take
// a segment of a long row of A each, the others a row block of short rows.  The
// last segment of a row to finish (ticket, back at zero for the next launch) adds
// them in order and updates the row, as dual_block does.  A portfolio has two
// long rows and nothing else: with the segments and the two rows in launches of
// their own a solve (n = 1e5, r = 64) took 48.2 ms, so 40.6.
template <typename V>
struct LrColumns {
  const double* part;            // [nparts][r]
  int nparts, r;
  double* w;
  float* wf;
  const int4* __restrict__ lseg;
  int nlseg;
  V* lpart;
  unsigned* ticket;              // [nlseg], at a row's first segment
};
template <typename V>
__global__ void __launch_bounds__(256, MinBlocks<V, 256>::value == 8 ? 4 : MinBlocks<V, 256>::value)
    k_dual_lr(DualB<V> a, LrColumns<V> q, int j) {
  __shared__ V prod[BNNZ];
  __shared__ V sx[sizeof(V) == 8 ? BNNZ : 1];
  __shared__ int srp[BROWS + 1];
  grid_trigger();
  int b = blockIdx.x;
  if (b < q.r) {
    grid_wait();
    if (a.st->status == ST_RUNNING) lr_reduce_column(q.part, q.nparts, q.r, 1, b, q.w, q.wf);
    return;
  }
  b -= q.r;
  if (b >= q.nlseg) {
    b -= q.nlseg;
    if (a.blk_seg && a.blk_seg[b].y > 0) grid_wait();          // a long row
    else dual_block<V, 256>(a, b, j, prod, sx, srp);
    return;
  }
  // long_segment_sum with the segment's entries fetched before the wait
  constexpr int PER = (LSEG + 255) / 256;
  const int4 g = q.lseg[b];                                     // {row, first nonzero, end, row block}
  const int2 sg = a.blk_seg[g.w];
  V v[PER];
  int c[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int e = g.y + threadIdx.x + 256 * k;
    v[k] = e < g.z ? a.A.val[e] : V(0);
    c[k] = e < g.z ? a.A.col[e] : 0;
  }
  grid_wait();
  if (a.st->status != ST_RUNNING) return;
  V z[PER], s = V(0);
#pragma unroll
  for (int k = 0; k < PER; ++k) z[k] = g.y + (int)threadIdx.x + 256 * k < g.z ? a.xt[c[k]] : V(0);
  V yo = V(0), bi = V(0), yb = V(0), lo = V(0);
  if (threadIdx.x == 0) {
    yo = a.yold[g.x]; bi = a.b[g.x]; yb = a.ybar[g.x];
    if (a.ylo) lo = a.ylo[g.x];
  }
#pragma unroll
  for (int k = 0; k < PER; ++k)
    if (g.y + (int)threadIdx.x + 256 * k < g.z) s += v[k] * z[k];
  s = block_sum(s);
  if (threadIdx.x != 0) return;
  q.lpart[b] = s;
  __threadfence();
  if (atomicAdd(q.ticket + sg.x, 1u) != (unsigned)sg.y - 1u) return;
  __threadfence();
  q.ticket[sg.x] = 0u;
  s = V(0);
  for (int k = 0; k < sg.y; ++k) s += __ldcg(q.lpart + sg.x + k);
  dual_row(a, a.tab[j], g.x, s, yo, bi, yb, lo);
}

template <typename V>
void run_dual_lr(Work& w, int j, int nparts, BCsr<V> A, V* xt, V* const* Z, V* ybar, const V* b, const V* ylo,
                 cudaStream_t s) {
  DualB<V> da{A, xt, nullptr, nullptr, ybar, b, ylo, w.tab, w.blk_inst_A, w.st, w.row_ineq, w.tab_stride};
  da.yold = Z[(j + 1) & 1] + w.n;
  da.ynew = Z[j & 1] + w.n;
  V* lp = sizeof(V) == 4 ? (V*)w.A.lpart_f : (V*)w.A.lpart_d;
  if (w.A.nlseg) { da.blk_seg = w.A.blk_seg; da.lpart = lp; }
  da.early = 1;
  const LrColumns<V> q{w.lr_part, nparts, w.r, w.wlr, w.wlr_f, w.A.lseg, w.A.nlseg, lp, w.lr_ticket};
  launch_early(k_dual_lr<V>, w.r + w.A.nlseg + (w.m > 0 ? w.A.nblk : 0), 256, 0, s, da, q, j);
}
template void run_dual_lr<float>(Work&, int, int, BCsr<float>, float*, float* const*, float*, const float*,
                                 const float*, cudaStream_t);
template void run_dual_lr<double>(Work&, int, int, BCsr<double>, double*, double* const*, double*, const double*,
                                  const double*, cudaStream_t);

template <typename V, int NT>
static void run_chunk(Work& w, int j0, int len, BCsr<V> A, BCsr<V> P, V* xt, V* const* Z, V* ybar, const V* b,
                      const V* ylo, V* x, V* xbar, const V* c, const V* l, const V* u, cudaStream_t s,
                      bool compact) {
  Profiler& Pr = w.prof;
  DualB<V> da{A, xt, nullptr, nullptr, ybar, b, ylo, w.tab, w.blk_inst_A, w.st, w.row_ineq, w.tab_stride};
  PrimalB<V> pa{P, nullptr, nullptr, x, xbar, xt, c, l, u, w.tab, w.blk_inst_P, w.st, w.tab_stride,
                w.r > 0 ? lr_factor<V>(w) : nullptr, lr_weights<V>(w), w.r};
  // long rows: segment sums first (float or float64 buffers by V)
  V* lpA = sizeof(V) == 4 ? (V*)w.A.lpart_f : (V*)w.A.lpart_d;
  V* lpP = sizeof(V) == 4 ? (V*)w.P.lpart_f : (V*)w.P.lpart_d;
  if (w.A.nlseg) { da.blk_seg = w.A.blk_seg; da.lpart = lpA; }
  if (w.P.nlseg) { pa.blk_seg = w.P.blk_seg; pa.lpart = lpP; }
  int gA = w.A.nblk, gP = w.P.nblk;
  if (compact) {   // only the running instances' row blocks (counts of the last check)
    da.act = w.act_A;
    pa.act = w.act_P;
    // a grid padded for a replayed graph (entries past the count are -1), or
    // the counts themselves
    gA = w.act_grid_A > 0 ? w.act_grid_A : w.bst_host->act_A;
    gP = w.act_grid_P > 0 ? w.act_grid_P : w.bst_host->act_P;
  }
  // One instance: its half-steps follow each other without a gap (a batch's
  // blocks look at their instance's status before they load anything).
  const bool early = w.count == 1 && w.r == 0 && w.A.nlseg == 0 && w.P.nlseg == 0;
  da.early = pa.early = early;
  for (int j = j0; j < j0 + len; ++j) {
    if (w.r > 0) lowrank_ft1(w, pa.F, (const V*)Z[j & 1], s);
    if (w.m > 0) {
      da.yold = Z[(j + 1) & 1] + w.n;
      da.ynew = Z[j & 1] + w.n;
      if (Pr.on) Pr.begin(0, s, launch_bytes(w, 0, sizeof(V)));
      if (w.A.nlseg)
        launch(k_long_partials<V>, w.A.nlseg, 256, 0, s, A, (const V*)xt, (const int4*)w.A.lseg,
               (const int*)w.blk_inst_A, (const DevState*)w.st, lpA);
      if (early) launch_early(k_dual<V, NT>, gA, NT, 0, s, da, j);
      else launch(k_dual<V, NT>, gA, NT, 0, s, da, j);
      if (Pr.on) Pr.end(s);
    }
    pa.zin = Z[j & 1];
    pa.zout = Z[(j + 1) & 1];
    if (Pr.on) Pr.begin(1, s, launch_bytes(w, 1, sizeof(V)));
    if (w.P.nlseg)
      launch(k_long_partials<V>, w.P.nlseg, 256, 0, s, P, (const V*)pa.zin, (const int4*)w.P.lseg,
             (const int*)w.blk_inst_P, (const DevState*)w.st, lpP);
    if (w.r > 0) launch(k_primal<V, NT, true>, gP, NT, 0, s, pa, j);
    else if (early) launch_early(k_primal<V, NT, false>, gP, NT, 0, s, pa, j);
    else launch(k_primal<V, NT, false>, gP, NT, 0, s, pa, j);
    if (Pr.on) Pr.end(s);
  }
}

// ==========================================================================
// Family handles: members that share the matrix, run on member-interleaved
// vectors v[j * ld + member] (ld = members rounded up to 32).  A warp takes
// one row for 32 members: each matrix entry is read once for them and meets
// their 32 values of the gathered vector in one coalesced load, where the
// member-major layout gathers 32 scattered sectors.  The row sum runs over
// the row's entries in CSR order by r_dot, as the row-block kernels sum their
// staged entries, and the row update is
// the same function: a member's iterates are bitwise those of its standalone
// solve.  The vectors are transposed into this layout at the start of a
// chunk and back at its end, so the checks, restarts and rebases run on the
// member-major layout as for any batch.  Only the members that still run are
// laid out, densely (il_slots), and lanes without one load nothing: padding 300
// members to 384 and keeping those that stopped took 170.1 ms of a solve
// instead of 158.7.
// ==========================================================================
constexpr int IL_NT = 256;
constexpr int IL_RPB = IL_NT / 32;     // rows per CUDA block (one warp each)


template <typename V>
struct FamIL {
  const int* __restrict__ rp;          // one member's CSR (A, or P with local columns)
  const int* __restrict__ col;
  const V* __restrict__ val;           // scaled values (the same for every member)
  int rows, ld;
  const V* steps;         // [k][IL_STEPS][ld] step scalars of up to IL_STEP_ITERS iterations (k_il_steps)
  const int* slot;        // [ld] member, or -1
  const V* zin;           // gathered vector (x_tilde, or [x_md ; y+])
  // dual: yold, ynew, ybar, b, ylo (may be null), ineq;  primal: x, xbar, zout, xt, c, l, u
  const V* v0;
  V* w0;
  V* w1;
  V* w2;
  V* w3;
  const V* r0;
  const V* r1;
  const V* r2;
  const unsigned char* __restrict__ ineq;
};

// 16 bytes of consecutive members per lane: 4 float or 2 double
template <typename V> struct IlVec;
template <> struct IlVec<float> { using T = float4; static constexpr int W = 4; };
template <> struct IlVec<double> { using T = double2; static constexpr int W = 2; };
constexpr int IL_LD_ALIGN = 128;       // members per warp in float32 (the leading dimension's unit)

template <typename V>
__device__ __forceinline__ void il_load(const V* p, V (&v)[IlVec<V>::W]) {
  const typename IlVec<V>::T q = *reinterpret_cast<const typename IlVec<V>::T*>(p);
  if constexpr (IlVec<V>::W == 4) { v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w; }
  else { v[0] = q.x; v[1] = q.y; }
}
template <typename V>
__device__ __forceinline__ void il_load_rw(const V* p, V (&v)[IlVec<V>::W]) {   // a vector the kernel writes
  const typename IlVec<V>::T q = *reinterpret_cast<const typename IlVec<V>::T*>(p);
  if constexpr (IlVec<V>::W == 4) { v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w; }
  else { v[0] = q.x; v[1] = q.y; }
}
template <typename V>
__device__ __forceinline__ void il_store(V* p, const V (&v)[IlVec<V>::W]) {
  typename IlVec<V>::T q;
  if constexpr (IlVec<V>::W == 4) { q.x = v[0]; q.y = v[1]; q.z = v[2]; q.w = v[3]; }
  else { q.x = v[0]; q.y = v[1]; }
  *reinterpret_cast<typename IlVec<V>::T*>(p) = q;
}

// The row sums of this lane's W members: for each, sequential over the row's
// entries by r_dot, as the row-block kernels sum their staged entries.  The warp reads
// the row's indices and values 32 at a time in one coalesced load and hands
// each entry to all lanes by shuffle, so that the L1 data pipe (the bound of
// this kernel) moves only the gathered members' values, those of lanes that
// hold members (on).  Every lane of the warp runs it (the shuffles need the
// whole warp).
template <typename V>
__device__ __forceinline__ void il_row_sum(const FamIL<V>& a, int e0, int e1, int m0, bool on, V (&s)[IlVec<V>::W]) {
  constexpr int W = IlVec<V>::W;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < W; ++q) s[q] = V(0);
  for (int base = e0; base < e1; base += 32) {
    int cl = 0;
    V vl = V(0);
    if (base + lane < e1) { cl = __ldg(a.col + base + lane); vl = __ldg(a.val + base + lane); }
    const int cnt = min(32, e1 - base);
    int k = 0;
    for (; k + 4 <= cnt; k += 4) {
      int c[4];
      V v[4], z[4][W];
#pragma unroll
      for (int i = 0; i < 4; ++i) { c[i] = __shfl_sync(0xffffffffu, cl, k + i); v[i] = __shfl_sync(0xffffffffu, vl, k + i); }
      if (!on) continue;
#pragma unroll
      for (int i = 0; i < 4; ++i) il_load(a.zin + (size_t)c[i] * a.ld + m0, z[i]);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < W; ++q) s[q] = r_dot(v[i], z[i][q], s[q]);
    }
    for (; k < cnt; ++k) {
      const int c = __shfl_sync(0xffffffffu, cl, k);
      const V v = __shfl_sync(0xffffffffu, vl, k);
      if (!on) continue;
      V z[W];
      il_load(a.zin + (size_t)c * a.ld + m0, z);
#pragma unroll
      for (int q = 0; q < W; ++q) s[q] = r_dot(v, z[q], s[q]);
    }
  }
}

// The step scalars of a chunk's iterations in slot order, so that a lane loads
// those of its members in one 16-byte access.  (Each CUDA block staging its members' 64-byte table entries and
// statuses cost 12 KB of scattered loads and a barrier before its eight rows'
// 65 KB (A) could start.)
enum { IL_SIGMA = 0, IL_TAU, IL_IB, IL_IBN, IL_THN, IL_STEPS };
template <typename V>
__global__ void __launch_bounds__(128) k_il_steps(const StepEntry* __restrict__ tab, int C, const int* __restrict__ slot,
                                                  int ld, int j0, V* __restrict__ steps) {
  const int m = blockIdx.x * 128 + threadIdx.x, k = blockIdx.y;
  if (m >= ld) return;
  const int mem = slot[m];
  V v[IL_STEPS] = {V(0), V(0), V(0), V(0), V(0)};
  if (mem >= 0) {
    const StepEntry e = tab[(size_t)mem * C + j0 + k];
    v[IL_SIGMA] = step_sigma<V>(e); v[IL_TAU] = step_tau<V>(e); v[IL_IB] = step_ib<V>(e);
    v[IL_IBN] = step_ibn<V>(e); v[IL_THN] = step_thn<V>(e);
  }
#pragma unroll
  for (int q = 0; q < IL_STEPS; ++q) steps[((size_t)k * IL_STEPS + q) * ld + m] = v[q];
}

template <typename V>
__device__ __forceinline__ void il_steps(const FamIL<V>& a, int k, int q, int m0, V (&v)[IlVec<V>::W]) {
  il_load(a.steps + ((size_t)k * IL_STEPS + q) * a.ld + m0, v);
}
// this lane's members: run[q] where slot q holds one, and whether any does
template <typename V>
__device__ __forceinline__ bool il_running(const FamIL<V>& a, int m0, int (&run)[IlVec<V>::W]) {
  int any = 0;
#pragma unroll
  for (int q = 0; q < IlVec<V>::W; ++q) {
    run[q] = a.slot[m0 + q] >= 0;
    any |= run[q];
  }
  return any != 0;
}

// k: the iteration among those whose step scalars are laid out
template <typename V>
__global__ void __launch_bounds__(IL_NT, 4) k_dual_il(FamIL<V> a, int k) {
  constexpr int W = IlVec<V>::W;
  grid_trigger();
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * IL_RPB + (threadIdx.x >> 5);
  if (r >= a.rows) return;
  const int m0 = blockIdx.y * 32 * W + lane * W;
  const int e0 = __ldg(a.rp + r), e1 = __ldg(a.rp + r + 1);
  grid_wait();
  int run[W];
  const bool on = il_running(a, m0, run);
  if (!__any_sync(0xffffffffu, on)) return;
  const size_t idx = (size_t)r * a.ld + m0;
  V yo[W], bi[W], yb[W], lo[W], s[W], sg[W], ib[W], yn[W], ybn[W];
#pragma unroll
  for (int q = 0; q < W; ++q) lo[q] = V(0);
  if (on) {
    il_load_rw(a.v0 + idx, yo);
    il_load(a.r0 + idx, bi);
    il_load_rw(a.w1 + idx, yb);
    if (a.r1) il_load(a.r1 + idx, lo);
  }
  il_row_sum(a, e0, e1, m0, on, s);
  if (!on) return;
  const bool ineq = a.ineq[r] != 0;
  il_steps(a, k, IL_SIGMA, m0, sg);
  il_steps(a, k, IL_IB, m0, ib);
#pragma unroll
  for (int q = 0; q < W; ++q) {
    if (run[q]) dual_update<V>(sg[q], ib[q], s[q], yo[q], bi[q], yb[q], lo[q], ineq, yn[q], ybn[q]);
    else { ybn[q] = yb[q]; yn[q] = a.w0[idx + q]; }    // an empty slot
  }
  il_store(a.w1 + idx, ybn);   // y_bar
  il_store(a.w0 + idx, yn);    // y+
}

template <typename V>
__global__ void __launch_bounds__(IL_NT, 4) k_primal_il(FamIL<V> a, int k) {
  constexpr int W = IlVec<V>::W;
  grid_trigger();
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * IL_RPB + (threadIdx.x >> 5);
  if (r >= a.rows) return;
  const int m0 = blockIdx.y * 32 * W + lane * W;
  const int e0 = __ldg(a.rp + r), e1 = __ldg(a.rp + r + 1);
  grid_wait();
  int run[W];
  const bool on = il_running(a, m0, run);
  if (!__any_sync(0xffffffffu, on)) return;
  const size_t idx = (size_t)r * a.ld + m0;
  V s[W], xo[W], xb0[W], cr[W], lr[W], ur[W], tau[W], ib[W], ibn[W], thn[W], xn[W], xb[W], zo[W], xtn[W];
  if (on) {
    il_load_rw(a.w0 + idx, xo);
    il_load_rw(a.w1 + idx, xb0);
    il_load(a.r0 + idx, cr);
    il_load(a.r1 + idx, lr);
    il_load(a.r2 + idx, ur);
  }
  il_row_sum(a, e0, e1, m0, on, s);
  if (!on) return;
  il_steps(a, k, IL_TAU, m0, tau);
  il_steps(a, k, IL_IB, m0, ib);
  il_steps(a, k, IL_IBN, m0, ibn);
  il_steps(a, k, IL_THN, m0, thn);
#pragma unroll
  for (int q = 0; q < W; ++q) {
    if (run[q]) {
      const V g = r_add(s[q], cr[q]);
      primal_update<V>(tau[q], ib[q], ibn[q], thn[q], g, xo[q], xb0[q], lr[q], ur[q], xn[q], xb[q], zo[q], xtn[q]);
    } else {   // an empty slot
      xn[q] = xo[q]; xb[q] = xb0[q]; zo[q] = a.w2[idx + q]; xtn[q] = a.w3[idx + q];
    }
  }
  il_store(a.w1 + idx, xb);    // x_bar
  il_store(a.w2 + idx, zo);    // x_md of the next iteration
  il_store(a.w3 + idx, xtn);   // x_tilde of the next iteration
  il_store(a.w0 + idx, xn);    // x
}

// Algorithmic bytes of one family launch: the shared matrix once, the vectors
// of each running member once (kind 0 dual, 1 primal; sv = bytes per value).
static double il_launch_bytes(const Work& w, int kind, double sv) {
  const double members = w.fam_n > 0 ? w.bst_host->run_n / w.fam_n : 0.0;
  if (kind == 0)
    return w.fam_nnzA * (sv + 4.0) + 4.0 * (w.fam_m + 1.0) + sv * members * (w.fam_n + 5.0 * w.fam_m);
  return w.fam_nnzP * (sv + 4.0) + 4.0 * (w.fam_n + 1.0) + sv * members * (10.0 * w.fam_n + w.fam_m);
}

template <typename V>
static void run_chunk_il(Work& w, int j0, int len, const V* Aval, const V* Pval, V* xt, V* const* Z, V* ybar,
                         const V* b, const V* ylo, V* x, V* xbar, const V* c, const V* l, const V* u,
                         cudaStream_t s) {
  Profiler& Pr = w.prof;
  V* const* I = reinterpret_cast<V* const*>(sizeof(V) == 4 ? (void* const*)w.ilf : (void* const*)w.ild);
  const int n = w.fam_n, m = w.fam_m, cnt = w.fam_count, ld = w.fam_ld;
  const long long N = (long long)cnt * n;
  auto tin = [&](const V* src, long long stride, int L, V* dst) { to_il<V>(src, stride, L, w.il_slot, cnt, dst, ld, s); };
  il_slots(w, s);
  // member-major -> interleaved: everything the iterations read
  for (int p = 0; p < 2; ++p) {
    tin(Z[p], n, n, I[IL_Z0 + p]);
    tin(Z[p] + N, m, m, I[IL_Z0 + p] + (size_t)n * ld);
  }
  tin(x, n, n, I[IL_X]);
  tin(xbar, n, n, I[IL_XBAR]);
  tin(xt, n, n, I[IL_XT]);
  tin(ybar, m, m, I[IL_YBAR]);
  tin(c, n, n, I[IL_C]);
  tin(l, n, n, I[IL_L]);
  tin(u, n, n, I[IL_U]);
  tin(b, m, m, I[IL_B]);
  tin(ylo, m, m, I[IL_YLO]);
  const int groups = ld / (32 * IlVec<V>::W);
  V* steps = sizeof(V) == 4 ? (V*)w.il_steps_f : (V*)w.il_steps_d;
  FamIL<V> da{};
  da.rp = w.A.rp; da.col = w.A.col; da.val = Aval;
  da.rows = m; da.ld = ld; da.steps = steps; da.slot = w.il_slot;
  da.zin = I[IL_XT];
  da.w1 = I[IL_YBAR]; da.r0 = I[IL_B]; da.r1 = ylo ? I[IL_YLO] : nullptr; da.ineq = w.row_ineq;
  FamIL<V> pa{};
  pa.rp = w.P.rp; pa.col = w.famP_col; pa.val = Pval;
  pa.rows = n; pa.ld = ld; pa.steps = steps; pa.slot = w.il_slot;
  pa.w0 = I[IL_X]; pa.w1 = I[IL_XBAR]; pa.w3 = I[IL_XT]; pa.r0 = I[IL_C]; pa.r1 = I[IL_L]; pa.r2 = I[IL_U];
  for (int j = j0; j < j0 + len; ++j) {
    const int k = (j - j0) % IL_STEP_ITERS;
    if (k == 0)
      launch(k_il_steps<V>, dim3(cdiv(ld, 128), std::min(IL_STEP_ITERS, j0 + len - j)), 128, 0, s,
             (const StepEntry*)w.tab, w.tab_stride, (const int*)w.il_slot, ld, j, steps);
    if (m > 0) {
      da.v0 = I[IL_Z0 + ((j + 1) & 1)] + (size_t)n * ld;   // y^k
      da.w0 = I[IL_Z0 + (j & 1)] + (size_t)n * ld;         // y^{k+1}
      if (Pr.on) Pr.begin(0, s, il_launch_bytes(w, 0, sizeof(V)));
      launch_early(k_dual_il<V>, dim3(cdiv(m, IL_RPB), groups), IL_NT, 0, s, da, k);
      if (Pr.on) Pr.end(s);
    }
    pa.zin = I[IL_Z0 + (j & 1)];
    pa.w2 = I[IL_Z0 + ((j + 1) & 1)];
    if (Pr.on) Pr.begin(1, s, il_launch_bytes(w, 1, sizeof(V)));
    launch_early(k_primal_il<V>, dim3(cdiv(n, IL_RPB), groups), IL_NT, 0, s, pa, k);
    if (Pr.on) Pr.end(s);
  }
  // interleaved -> member-major: everything the iterations wrote
  auto back = [&](const V* src, int L, V* dst, long long stride) { from_il<V>(src, ld, L, w.il_slot, cnt, dst, stride, s); };
  for (int p = 0; p < 2; ++p) {
    back(I[IL_Z0 + p], n, Z[p], n);
    back(I[IL_Z0 + p] + (size_t)n * ld, m, Z[p] + N, m);
  }
  back(I[IL_X], n, x, n);
  back(I[IL_XBAR], n, xbar, n);
  back(I[IL_XT], n, xt, n);
  back(I[IL_YBAR], m, ybar, m);
}

void iterate_chunk(Work& w, int len, bool mixed, int nt, cudaStream_t s, int j0, bool compact) {
  if (nt == 3) {   // a family handle on member-interleaved vectors
    if (len <= 0) return;
    if (mixed) {
      run_chunk_il<float>(w, j0, len, w.A.sval_f, w.P.sval_f, w.fxt, w.fZ, w.fybar, w.fb, w.fylo, w.fx, w.fxbar, w.fc,
                          w.fl, w.fu, s);
      w.fy = w.fZ[(j0 + len - 1) & 1] + w.n;
    } else {
      run_chunk_il<double>(w, j0, len, w.A.sval, w.P.sval, w.xt, w.Z, w.ybar, w.bs, nullptr, w.x, w.xbar, w.cs, w.ls,
                           w.us, s);
      w.y = w.Z[(j0 + len - 1) & 1] + w.n;
    }
    return;
  }
  if (nt == 2) {   // the whole chunk in one launch (small instances)
    chunk_run(w, len, mixed, s, j0);
    return;
  }
  if (nt == 4) {   // a low-rank term over short rows
    lowrank_run(w, len, mixed, s, j0);
    return;
  }
  if (nt == 5) {   // a row per thread on the slice layout
    if (mixed) {
      run_chunk_sl<float>(w, j0, len, w.fxt, w.fZ, w.fybar, w.fb, w.fylo, w.fx, w.fxbar, w.fc, w.fl, w.fu, s);
      w.fy = w.fZ[(j0 + len - 1) & 1] + w.n;
    } else {
      run_chunk_sl<double>(w, j0, len, w.xt, w.Z, w.ybar, w.bs, nullptr, w.x, w.xbar, w.cs, w.ls, w.us, s);
      w.y = w.Z[(j0 + len - 1) & 1] + w.n;
    }
    return;
  }
  if (nt == 1) {   // pipelined persistent kernels, 256 threads
    if (mixed) {
      run_chunk_pipe<float, 256>(w, j0, len, w.A.bscaled_f(), w.P.bscaled_f(), w.fxt, w.fZ, w.fybar, w.fb, w.fylo, w.fx,
                                 w.fxbar, w.fc, w.fl, w.fu, s);
      w.fy = w.fZ[(j0 + len - 1) & 1] + w.n;
    } else {
      run_chunk_pipe<double, 256>(w, j0, len, w.A.bscaled(), w.P.bscaled(), w.xt, w.Z, w.ybar, w.bs, nullptr, w.x,
                                  w.xbar, w.cs, w.ls, w.us, s);
      w.y = w.Z[(j0 + len - 1) & 1] + w.n;
    }
    return;
  }
  if (mixed) {
    if (nt != 512)
      run_chunk<float, 256>(w, j0, len, w.A.bscaled_f(), w.P.bscaled_f(), w.fxt, w.fZ, w.fybar, w.fb, w.fylo, w.fx,
                            w.fxbar, w.fc, w.fl, w.fu, s, compact);
    else
      run_chunk<float, 512>(w, j0, len, w.A.bscaled_f(), w.P.bscaled_f(), w.fxt, w.fZ, w.fybar, w.fb, w.fylo, w.fx,
                            w.fxbar, w.fc, w.fl, w.fu, s, compact);
    w.fy = w.fZ[(j0 + len - 1) & 1] + w.n;
  } else {
    if (nt != 512)
      run_chunk<double, 256>(w, j0, len, w.A.bscaled(), w.P.bscaled(), w.xt, w.Z, w.ybar, w.bs, nullptr, w.x, w.xbar,
                             w.cs, w.ls, w.us, s, compact);
    else
      run_chunk<double, 512>(w, j0, len, w.A.bscaled(), w.P.bscaled(), w.xt, w.Z, w.ybar, w.bs, nullptr, w.x, w.xbar,
                             w.cs, w.ls, w.us, s, compact);
    w.y = w.Z[(j0 + len - 1) & 1] + w.n;
  }
}

}  // namespace pdqp
