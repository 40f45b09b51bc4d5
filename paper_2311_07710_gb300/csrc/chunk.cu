// A whole chunk of iterations of Algorithm 1 (Section 2) in one launch: a CTA
// (or, where a handle holds fewer problems than the chip has SMs, a
// thread-block cluster) per instance keeps the instance's vectors and as much
// of its matrices as fits in shared memory and runs every iteration of the
// chunk there, with one barrier after each half-step.
//
// What bounds the per-iteration kernels on small instances is not their
// arithmetic: every iteration streams each matrix from memory once more (a
// batch of 4096 control QPs: 0.55 GB per iteration) or, with few instances,
// waits out two launches and the row blocks' dependent load chains.  Here the
// matrix is read once per chunk and the half-steps run at the shared-memory
// rate of the SM that holds it.
//
// Matrix layout: slices of 32 consecutive rows of one instance; a slice's
// entries are stored pair by pair, 32 lanes wide (lane = row), columns as two
// 16-bit local indices per pair, so that a warp's loads are contiguous and a
// thread walks its row in order.  Rows shorter than the slice's width are
// padded with value 0 at a column that holds 0 (one slot behind the vector);
// the sum starts at +0 and is never -0 afterwards (x + y = -0 needs both
// -0), so adding the pads' +0 changes no bit.  The products and sums are
// rounded in the row's order (r_dot) and the row updates are the shared ones
// (rowupdate.cuh): the iterates are bitwise those of k_dual / k_primal.
#include <cooperative_groups.h>

#include <algorithm>
#include <functional>
#include <mutex>

#include "rowblock.cuh"
#include "rowupdate.cuh"

namespace cg = cooperative_groups;

namespace pdqp {

constexpr int CHUNK_TAB = 64;                     // step-table entries staged at a time
constexpr int CHUNK_SMEM_MAX = 226 * 1024;

template <typename V> struct Pair;
template <> struct Pair<float> { using T = float2; };
template <> struct Pair<double> { using T = double2; };

template <typename V>
struct ChunkArgs {
  const ChunkInst* __restrict__ inst;   // launch order
  const int* __restrict__ sp;           // slice starts, in groups of 32 pairs (A's slices, then P's)
  const unsigned* __restrict__ idx;     // [groups][32] two 16-bit columns
  const typename Pair<V>::T* __restrict__ val;   // [groups][32]
  V* __restrict__ xt;
  V* __restrict__ z0;
  V* __restrict__ z1;
  V* __restrict__ x;
  V* __restrict__ xbar;
  V* __restrict__ ybar;
  const V* __restrict__ b;
  const V* __restrict__ ylo;            // may be null (0)
  const V* __restrict__ c;
  const V* __restrict__ l;
  const V* __restrict__ u;
  const unsigned char* __restrict__ ineq;
  const StepEntry* __restrict__ tab;    // [instance][C]
  const DevState* __restrict__ st;
  int C, N;                             // step-table stride, variables of the whole handle
  int smem;                             // dynamic shared memory of the launch
};

__host__ __device__ inline int chunk_r4(int v) { return (v + 3) & ~3; }

// Shared memory of one CTA without the matrix: the staged step table, x~ and
// both [x_md ; y] buffers (each with the pads' zero slot), x, x_bar, c, l, u of
// the CTA's rows of P, y_bar, b, the lower bound and the inequality flag of its
// rows of A, its slice starts.
template <typename V>
__host__ __device__ inline size_t chunk_fixed_bytes(int n, int m, int ownA, int ownP) {
  const size_t v = 5 * CHUNK_TAB + (size_t)chunk_r4(n + 1) + 2 * (size_t)chunk_r4(n + m + 1) + 160 * (size_t)ownP +
                   128 * (size_t)ownA;
  return v * sizeof(V) + (size_t)chunk_r4(ownA + ownP + 2) * sizeof(int);
}
template <typename V>
constexpr size_t chunk_group_bytes() { return 32 * (sizeof(unsigned) + 2 * sizeof(V)); }

__device__ __forceinline__ void chunk_cp16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}

// every thread of the cluster (or CTA) arrives (release) and waits (acquire)
template <bool CL>
__device__ __forceinline__ void chunk_barrier() {
  if constexpr (CL) {
    asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");
  } else {
    __syncthreads();
  }
}

// v into slot p of every CTA's copy (p: this CTA's shared address)
template <bool CL, typename V>
__device__ __forceinline__ void chunk_put(cg::cluster_group& cl, int ctas, V* p, V v) {
  if constexpr (CL) {
    for (int q = 0; q < ctas; ++q) *cl.map_shared_rank(p, q) = v;
  } else {
    *p = v;
  }
}

// s plus the terms of N consecutive groups of this lane: the columns and values
// of all of them, then the gathers, then the chain of adds.
template <typename V, bool SM, int N>
__device__ __forceinline__ V chunk_batch(V s, const V* z, const unsigned* pi, const typename Pair<V>::T* pv) {
  unsigned ii[N];
  typename Pair<V>::T vv[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if constexpr (SM) {
      ii[k] = pi[k * 32];
      vv[k] = pv[k * 32];
    } else {
      ii[k] = __ldg(pi + k * 32);
      vv[k] = __ldg(pv + k * 32);
    }
  }
  V a[N], b[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    a[k] = z[ii[k] & 0xFFFFu];
    b[k] = z[ii[k] >> 16];
  }
#pragma unroll
  for (int k = 0; k < N; ++k) s = r_dot(vv[k].y, b[k], r_dot(vv[k].x, a[k], s));
  return s;
}
// Four groups at a time; what is left (the slices' widths are uniform over the
// warp) in one batch of its own size, not group by group: a batch costs two
// shared-memory latencies however short it is.  (A double-buffered form, the next
// batch fetched ahead, was slower: 5.1 against 4.0 us per iteration at horizon
// 100; with 32 warps the shared-memory pipe and the issue slots bind.)
template <typename V, bool SM>
__device__ __forceinline__ V chunk_span_sum(V s, const V* z, int g0, int g1, const unsigned* pi,
                                            const typename Pair<V>::T* pv) {
  const int lane = threadIdx.x & 31;
  pi += (size_t)g0 * 32 + lane;
  pv += (size_t)g0 * 32 + lane;
  int left = g1 - g0;
  for (; left >= 4; left -= 4, pi += 128, pv += 128) s = chunk_batch<V, SM, 4>(s, z, pi, pv);
  if (left == 3) s = chunk_batch<V, SM, 3>(s, z, pi, pv);
  else if (left == 2) s = chunk_batch<V, SM, 2>(s, z, pi, pv);
  else if (left == 1) s = chunk_batch<V, SM, 1>(s, z, pi, pv);
  return s;
}
// The row sum of this lane over the slice's groups [g0, g1): the first `res`
// groups of this CTA's range are resident (si, sv), the others stream from
// global memory (gi, gv: L2, since the CTA walks them every iteration).
template <typename V>
__device__ __forceinline__ V chunk_slice_sum(const V* z, int g0, int g1, int res, const unsigned* si,
                                             const typename Pair<V>::T* sv, const unsigned* __restrict__ gi,
                                             const typename Pair<V>::T* __restrict__ gv) {
  V s = V(0);
  if (g0 < res) s = chunk_span_sum<V, true>(s, z, g0, min(g1, res), si, sv);
  if (g1 > res) s = chunk_span_sum<V, false>(s, z, max(g0, res), g1, gi, gv);
  return s;
}

// CTA `rank` of the instance's `ctas` takes a contiguous share of its slices
// of A and of P; every CTA of a cluster holds whole copies of the gathered
// vectors, which the row updates write through distributed shared memory.
// Every thread of a cluster takes the same number of barriers (an instance
// that stopped leaves before the first one).
template <typename V, bool CL>
__global__ void __launch_bounds__(1024, 1) k_chunk(ChunkArgs<V> a, int first, int j0, int len) {
  using P2 = typename Pair<V>::T;
  extern __shared__ __align__(16) unsigned char chunk_sm[];
  cg::cluster_group cl = cg::this_cluster();
  const int ctas = CL ? (int)cl.num_blocks() : 1, rank = CL ? (int)cl.block_rank() : 0;
  const ChunkInst in = a.inst[first + (int)blockIdx.x / ctas];
  if (a.st[in.id].status != ST_RUNNING) return;   // uniform over the cluster
  const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, NW = NT >> 5;
  const int n = in.n, m = in.m;
  const int a0 = (int)((long long)in.nsA * rank / ctas), a1 = (int)((long long)in.nsA * (rank + 1) / ctas);
  const int p0 = (int)((long long)in.nsP * rank / ctas), p1 = (int)((long long)in.nsP * (rank + 1) / ctas);
  V* tabs = reinterpret_cast<V*>(chunk_sm);
  V* xs = tabs + 5 * CHUNK_TAB;
  V* const zs = xs + chunk_r4(n + 1);               // both [x_md ; y] buffers, zstep apart
  const int zstep = chunk_r4(n + m + 1);
  const int rowsP = 32 * (p1 - p0), rowsA = 32 * (a1 - a0);   // the CTA's rows, whole slices
  V* own_x = zs + 2 * zstep;                        // x, x_bar, c, l, u, rowsP apart
  V* own_yb = own_x + 5 * rowsP;                    // y_bar, b, lower bound, inequality (1 or 0), rowsA apart
  int* spA = reinterpret_cast<int*>(own_yb + 4 * rowsA);
  int* spP = spA + (a1 - a0 + 1);
  const size_t fixed = chunk_fixed_bytes<V>(n, m, a1 - a0, p1 - p0);
  const int baseA = a.sp[in.sA + a0], baseP = a.sp[in.sP + p0];
  const int gA = a.sp[in.sA + a1] - baseA, gP = a.sp[in.sP + p1] - baseP;
  const int room = (int)((a.smem - fixed) / chunk_group_bytes<V>());
  const int resA = min(gA, room), resP = min(gP, room - resA);
  P2* sval = reinterpret_cast<P2*>(chunk_sm + fixed);           // [resA + resP][32]
  unsigned* sidx = reinterpret_cast<unsigned*>(sval + 32 * (resA + resP));
  const unsigned* giA = a.idx + (size_t)baseA * 32;
  const unsigned* giP = a.idx + (size_t)baseP * 32;
  const P2* gvA = a.val + (size_t)baseA * 32;
  const P2* gvP = a.val + (size_t)baseP * 32;
  // the resident matrix (every piece a multiple of 16 bytes, 16-byte aligned)
  for (int i = tid; i < resA * 8; i += NT) chunk_cp16(sidx + 4 * i, giA + 4 * i);
  for (int i = tid; i < resP * 8; i += NT) chunk_cp16(sidx + 32 * resA + 4 * i, giP + 4 * i);
  constexpr int VP = 32 * (int)sizeof(P2) / 16;                 // 16-byte pieces of a group's values
  for (int i = tid; i < resA * VP; i += NT)
    chunk_cp16(reinterpret_cast<char*>(sval) + 16 * i, reinterpret_cast<const char*>(gvA) + 16 * (size_t)i);
  for (int i = tid; i < resP * VP; i += NT)
    chunk_cp16(reinterpret_cast<char*>(sval + 32 * resA) + 16 * i, reinterpret_cast<const char*>(gvP) + 16 * (size_t)i);
  asm volatile("cp.async.commit_group;\n" ::);
  // the vectors: x~, x_md of the first iteration, y of the one before
  {
    const V* zj = (j0 & 1) ? a.z1 : a.z0;
    const V* zo = (j0 & 1) ? a.z0 : a.z1;
    for (int i = tid; i < n; i += NT) {
      xs[i] = a.xt[in.xoff + i];
      zs[(j0 & 1) * zstep + i] = zj[in.xoff + i];
    }
    for (int i = tid; i < m; i += NT) zs[((j0 + 1) & 1) * zstep + n + i] = zo[(size_t)a.N + in.yoff + i];
    if (tid == 0) xs[n] = zs[n + m] = zs[zstep + n + m] = V(0);
    for (int i = tid; i < rowsP; i += NT) {
      const int r = 32 * p0 + i;
      if (r >= n) continue;
      own_x[i] = a.x[in.xoff + r];
      own_x[rowsP + i] = a.xbar[in.xoff + r];
      own_x[2 * rowsP + i] = a.c[in.xoff + r];
      own_x[3 * rowsP + i] = a.l[in.xoff + r];
      own_x[4 * rowsP + i] = a.u[in.xoff + r];
    }
    for (int i = tid; i < rowsA; i += NT) {
      const int r = 32 * a0 + i;
      if (r >= m) continue;
      own_yb[i] = a.ybar[in.yoff + r];
      own_yb[rowsA + i] = a.b[in.yoff + r];
      own_yb[2 * rowsA + i] = a.ylo ? a.ylo[in.yoff + r] : V(0);
      own_yb[3 * rowsA + i] = a.ineq[in.yoff + r] ? V(1) : V(0);
    }
    for (int i = tid; i <= a1 - a0; i += NT) spA[i] = a.sp[in.sA + a0 + i] - baseA;
    for (int i = tid; i <= p1 - p0; i += NT) spP[i] = a.sp[in.sP + p0 + i] - baseP;
  }
  asm volatile("cp.async.wait_all;\n" ::);
  chunk_barrier<CL>();                            // every copy is whole before anyone writes into it
  for (int j = j0; j < j0 + len; ++j) {
    const int t = (j - j0) % CHUNK_TAB;
    if (t == 0) {                                 // the next iterations' steps (their readers met at a barrier)
      if (tid < min(CHUNK_TAB, j0 + len - j)) {
        const StepEntry e = a.tab[(size_t)in.id * a.C + j + tid];
        V* q = tabs + 5 * tid;
        q[0] = step_sigma<V>(e); q[1] = step_tau<V>(e); q[2] = step_ib<V>(e); q[3] = step_ibn<V>(e);
        q[4] = step_thn<V>(e);
      }
      __syncthreads();
    }
    const V sigma = tabs[5 * t], tau = tabs[5 * t + 1], ib = tabs[5 * t + 2], ibn = tabs[5 * t + 3],
            thn = tabs[5 * t + 4];
    V* zj = zs + (j & 1) * zstep;
    V* zn = zs + ((j + 1) & 1) * zstep;
    for (int s = a0 + warp; s < a1; s += NW) {    // dual half-step
      const int r = 32 * s + lane, q = 32 * (s - a0) + lane;
      const V sum = chunk_slice_sum<V>(xs, spA[s - a0], spA[s - a0 + 1], resA, sidx, sval, giA, gvA);
      if (r < m) {
        V yn, ybn;
        dual_update<V>(sigma, ib, sum, zn[n + r], own_yb[rowsA + q], own_yb[q], own_yb[2 * rowsA + q],
                       own_yb[3 * rowsA + q] != V(0), yn, ybn);
        own_yb[q] = ybn;
        chunk_put<CL>(cl, ctas, zj + n + r, yn);
      }
    }
    chunk_barrier<CL>();
    for (int s = p0 + warp; s < p1; s += NW) {    // primal half-step
      const int r = 32 * s + lane, q = 32 * (s - p0) + lane;
      const V sum = chunk_slice_sum<V>(zj, spP[s - p0], spP[s - p0 + 1], resP, sidx + 32 * resA,
                                       sval + 32 * resA, giP, gvP);
      if (r < n) {
        V xn, xb, zo, xtn;
        primal_update<V>(tau, ib, ibn, thn, r_add(sum, own_x[2 * rowsP + q]), own_x[q], own_x[rowsP + q],
                         own_x[3 * rowsP + q], own_x[4 * rowsP + q], xn, xb, zo, xtn);
        own_x[q] = xn;
        own_x[rowsP + q] = xb;
        chunk_put<CL>(cl, ctas, zn + r, zo);
        chunk_put<CL>(cl, ctas, xs + r, xtn);
      }
    }
    chunk_barrier<CL>();
  }
  // the CTA's rows back to global memory: what the checks and the next chunk read
  const int jl = j0 + len - 1;
  V* gzj = (jl & 1) ? a.z1 : a.z0;
  V* gzn = (jl & 1) ? a.z0 : a.z1;
  for (int i = tid; i < rowsP; i += NT) {
    const int r = 32 * p0 + i;
    if (r >= n) continue;
    a.x[in.xoff + r] = own_x[i];
    a.xbar[in.xoff + r] = own_x[rowsP + i];
    a.xt[in.xoff + r] = xs[r];
    gzn[in.xoff + r] = zs[((jl + 1) & 1) * zstep + r];
  }
  for (int i = tid; i < rowsA; i += NT) {
    const int r = 32 * a0 + i;
    if (r >= m) continue;
    a.ybar[in.yoff + r] = own_yb[i];
    gzj[(size_t)a.N + in.yoff + r] = zs[(jl & 1) * zstep + n + r];
  }
}

// --------------------------------------------------------------------------
// The slice layout, built from the handle's CSR arrays (blockIdx.x = the
// instance's place in the plan's order; the slices of an instance over blockIdx.y)
// --------------------------------------------------------------------------
// width of every slice in pairs (its longest row, rounded up to a pair) and {the
// width were its rows all of their mean length, the entries of its longest row past that}
__global__ void __launch_bounds__(256) k_chunk_width(const ChunkInst* __restrict__ inst, const int* __restrict__ arp,
                                                     const int* __restrict__ prp, int* __restrict__ wid,
                                                     int2* __restrict__ even) {
  const ChunkInst in = inst[blockIdx.x];
  const int lane = threadIdx.x & 31, step = gridDim.y * 8;
  for (int s = blockIdx.y * 8 + (threadIdx.x >> 5); s < in.nsA + in.nsP; s += step) {
    const bool isA = s < in.nsA;
    const int r0 = 32 * (isA ? s : s - in.nsA), r = r0 + lane;
    const int rows = min(32, (isA ? in.m : in.n) - r0);
    int len = 0;
    if (lane < rows) {
      const int* rp = isA ? arp + in.yoff : prp + in.xoff;
      len = rp[r + 1] - rp[r];
    }
    const int width = (__reduce_max_sync(0xffffffffu, len) + 1) >> 1;
    const int mean = (__reduce_add_sync(0xffffffffu, len) + 2 * rows - 1) / (2 * rows);
    if (lane == 0) {
      const int gs = isA ? in.sA + s : in.sP + s - in.nsA;
      wid[gs] = width;
      even[gs] = make_int2(mean, 2 * (width - mean));
    }
  }
}

// {groups of A, groups of P, groups were the rows of every slice of its mean
// length, the most entries of a row past that} of every instance, in the order of
// inst; a warp each
__global__ void __launch_bounds__(256) k_chunk_shape(const ChunkInst* __restrict__ inst, int count,
                                                     const int* __restrict__ sp, const int2* __restrict__ even,
                                                     int4* __restrict__ out) {
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= count) return;
  const ChunkInst in = inst[i];
  int sum = 0, most = 0;
  for (int s = lane; s < in.nsA + in.nsP; s += 32) {
    const int2 e = even[s < in.nsA ? in.sA + s : in.sP + s - in.nsA];
    sum += e.x;
    most = max(most, e.y);
  }
  sum = __reduce_add_sync(0xffffffffu, sum);
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 0) out[i] = make_int4(sp[in.sA + in.nsA] - sp[in.sA], sp[in.sP + in.nsP] - sp[in.sP], sum, most);
}

// Columns (val null) or values of every slice; pads: the zero slot, value 0.
template <typename V, bool VALUES>
__global__ void __launch_bounds__(256)
    k_chunk_fill(const ChunkInst* __restrict__ inst, const int* __restrict__ sp, BCsr<V> A, BCsr<V> P, int N,
                 unsigned* __restrict__ idx, typename Pair<V>::T* __restrict__ val) {
  const ChunkInst in = inst[blockIdx.x];
  const int lane = threadIdx.x & 31, step = gridDim.y * 8;
  for (int s = blockIdx.y * 8 + (threadIdx.x >> 5); s < in.nsA + in.nsP; s += step) {
    const bool isA = s < in.nsA;
    const int gs = isA ? in.sA + s : in.sP + s - in.nsA;
    const int g0 = sp[gs], g1 = sp[gs + 1];
    const int r = 32 * (isA ? s : s - in.nsA) + lane;
    int e0 = 0, e1 = 0;
    if (r < (isA ? in.m : in.n)) {
      const int* rp = isA ? A.rp + in.yoff : P.rp + in.xoff;
      e0 = rp[r];
      e1 = rp[r + 1];
    }
    const int zero = isA ? in.n : in.n + in.m;
    for (int g = g0; g < g1; ++g) {
      const int e = e0 + 2 * (g - g0);
      if constexpr (VALUES) {
        const V* v = isA ? A.val : P.val;
        typename Pair<V>::T q;
        q.x = e < e1 ? v[e] : V(0);
        q.y = e + 1 < e1 ? v[e + 1] : V(0);
        val[(size_t)g * 32 + lane] = q;
      } else {
        unsigned c[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          int cc = zero;
          if (e + k < e1) {
            if (isA) cc = A.col[e + k] - in.xoff;
            else {
              cc = P.col[e + k];
              cc = cc < N ? cc - in.xoff : in.n + (cc - N - in.yoff);
            }
          }
          c[k] = (unsigned)cc;
        }
        idx[(size_t)g * 32 + lane] = c[0] | (c[1] << 16);
      }
    }
  }
}

static dim3 chunk_grid(const Work& w) {
  int big = 1;
  for (const Inst& I : w.inst_host) big = std::max(big, cdiv(I.n, 32) + cdiv(I.m, 32));
  return dim3(w.count, std::max(1, std::min(cdiv(big, 8), cdiv(8 * w.num_sms, w.count))));
}

void chunk_widths(Work& w, int* wid, int2* even, cudaStream_t s) {
  launch(k_chunk_width, chunk_grid(w), 256, 0, s, (const ChunkInst*)w.chunk.inst, (const int*)w.A.rp,
         (const int*)w.P.rp, wid, even);
}
void chunk_shapes(Work& w, const int2* even, int4* out, cudaStream_t s) {
  launch(k_chunk_shape, cdiv(w.count, 8), 256, 0, s, (const ChunkInst*)w.chunk.inst, w.count,
         (const int*)w.chunk.sp, even, out);
}
void chunk_fill_index(Work& w, cudaStream_t s) {
  launch(k_chunk_fill<float, false>, chunk_grid(w), 256, 0, s, (const ChunkInst*)w.chunk.inst, (const int*)w.chunk.sp,
         w.A.bscaled_f(), w.P.bscaled_f(), w.n, w.chunk.idx, (float2*)nullptr);
}
void chunk_fill_values(Work& w, bool mixed, cudaStream_t s) {
  if (mixed)
    launch(k_chunk_fill<float, true>, chunk_grid(w), 256, 0, s, (const ChunkInst*)w.chunk.inst,
           (const int*)w.chunk.sp, w.A.bscaled_f(), w.P.bscaled_f(), w.n, (unsigned*)nullptr, w.chunk.valf);
  else
    launch(k_chunk_fill<double, true>, chunk_grid(w), 256, 0, s, (const ChunkInst*)w.chunk.inst,
           (const int*)w.chunk.sp, w.A.bscaled(), w.P.bscaled(), w.n, (unsigned*)nullptr, w.chunk.vald);
}

// --------------------------------------------------------------------------
// host side
// --------------------------------------------------------------------------
static int g_chunk_max_ctas = 8;   // 16 where a 16-CTA cluster of the largest footprint can be resident

template <typename V>
static cudaLaunchConfig_t chunk_cfg(int ctas, int clusters, int threads, size_t smem, cudaStream_t s,
                                    cudaLaunchAttribute* at) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas * clusters);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = ctas > 1 ? 1 : 0;
  return cfg;
}

template <typename V>
static int chunk_resident_ctas() {
  cudaFuncSetAttribute(k_chunk<V, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, CHUNK_SMEM_MAX);
  cudaFuncSetAttribute(k_chunk<V, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, CHUNK_SMEM_MAX);
  cudaFuncSetAttribute(k_chunk<V, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = chunk_cfg<V>(16, 1, 1024, CHUNK_SMEM_MAX, nullptr, at);
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, k_chunk<V, true>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 8;
  }
  return clusters >= 1 ? 16 : 8;
}

static void prepare_chunk() {   // once per process
  static std::once_flag once;
  std::call_once(once, [] { g_chunk_max_ctas = std::min(chunk_resident_ctas<float>(), chunk_resident_ctas<double>()); });
}

// CTAs of every instance: one each with at least as many instances as SMs.
// Fewer instances share out the SMs by their rows, so that no CTA has much more to
// do than another and all run at once: the least bound on a CTA's rows under which
// the clusters fit the SMs (a cluster lies within one GPC, taken as 19 SMs of which
// pairs give 18 to clusters; without that, 30 control QPs in float64 took 9.0 us an
// iteration, with it 5.9).  A power of two of CTAs for all, as before, leaves the
// launch waiting for the largest: 77 control QPs of horizons 10 to 100 took 12.7 us
// in float64 and 5.4 in mixed precision against 9.8 and 4.1.
// In float64, more than half as many instances as SMs keep two CTAs each where that
// finishes earlier (pairs dealt out largest first to the SMs as they fall free): the
// float64 pipes bind there, and a second round of small instances costs less than
// idle pipes (151 of them 17.7 us against 23.2, 120 of them 14.1 against 17.2).
static const int kChunkSizes[] = {1, 2, 3, 4, 6, 8, 12, 16};
static std::vector<int> chunk_ctas(const Work& w, bool mixed) {
  std::vector<int> out(w.count, 1);
  if (w.count >= w.num_sms) return out;
  const int gpcs = std::max(1, w.num_sms / 19);
  // larger clusters pay with their barriers: 1500 rows (n = 1000) take 3.26 us an
  // iteration on 8 CTAs, 3.45 on 16; 2824 (a control QP of horizon 100) 3.15, 3.30 on
  // 12 and 3.46; 1000 rows 2.69 on 4 and 2.96 on 16; 6000 rows 4.69 on 12 and 4.90, in
  // float64 10.0 on 16 and 11.6 on 12.  Rows much longer than these (15 to 43 thousand
  // nonzeros in all) pay for more: 5000 nonzeros a CTA, counted by the rows.
  const double per_row = (double)(w.A.nnz + w.P.nnz) / std::max<long long>(1, (long long)w.n + w.m);
  auto cap = [&](const Inst& I) {
    int k = 1;
    for (int q : kChunkSizes) {
      const int rows = q <= 4 ? 100 : q <= 8 ? 187 : q <= 12 || !mixed ? 250 : 500;   // at least, a CTA
      const bool enough = (long long)q * rows <= I.n + I.m || q * 5000.0 <= per_row * (I.n + I.m);
      if (q <= g_chunk_max_ctas && 32 * (q - 1) < I.n && enough) k = q;
    }
    return k;
  };
  auto split = [&](long long rows) {              // at most `rows` rows per CTA: whether all CTAs fit
    int all = 0, of_size[17] = {};
    for (int i = 0; i < w.count; ++i) {
      const Inst& I = w.inst_host[i];
      int k = 1;
      for (int q : kChunkSizes)
        if (q <= cap(I) && (long long)k * rows < I.n + I.m) k = q;
      all += out[i] = k;
      ++of_size[k];
    }
    std::vector<int> room(gpcs, 18);
    for (int k = 16; k > 1; --k)
      for (int c = 0; c < of_size[k]; ++c) {
        auto g = std::find_if(room.begin(), room.end(), [&](int r) { return r >= k; });
        if (g == room.end()) return false;
        *g -= k;
      }
    return all <= w.num_sms;
  };
  long long lo = 1, hi = 1;
  for (const Inst& I : w.inst_host) hi = std::max<long long>(hi, I.n + I.m);
  while (lo < hi) {
    const long long mid = (lo + hi) / 2;
    if (split(mid)) hi = mid;
    else lo = mid + 1;
  }
  split(hi);
  if (mixed || 2 * w.count <= w.num_sms) return out;
  double most = 0.0;                               // rows of the fullest CTA
  std::vector<int> rows(w.count);
  for (int i = 0; i < w.count; ++i) {
    rows[i] = w.inst_host[i].n + w.inst_host[i].m;
    most = std::max(most, (double)rows[i] / out[i]);
  }
  constexpr int k = 2;
  std::sort(rows.begin(), rows.end(), std::greater<int>());
  std::vector<double> busy(w.num_sms, 0.0);
  for (int r : rows) {
    std::partial_sort(busy.begin(), busy.begin() + k, busy.end());
    std::fill(busy.begin(), busy.begin() + k, busy[k - 1] + (double)r / k);
  }
  if (*std::max_element(busy.begin(), busy.end()) < 0.9 * most)
    for (int i = 0; i < w.count; ++i) out[i] = std::min(k, cap(w.inst_host[i]));
  return out;
}

// Whether the vectors of an instance on k CTAs fit shared memory.
static bool chunk_fits(const Inst& I, int k, bool mixed) {
  const int oA = cdiv(cdiv(I.m, 32), k), oP = cdiv(cdiv(I.n, 32), k);
  return I.n + I.m <= 65535 &&                     // 16-bit columns, the pads' slot included
         (mixed ? chunk_fixed_bytes<float>(I.n, I.m, oA, oP) : chunk_fixed_bytes<double>(I.n, I.m, oA, oP)) <=
             (size_t)CHUNK_SMEM_MAX;
}
// Asked for, an instance that chunk_ctas gives too few CTAs for its vectors (rows
// of few variables: n = 100, m = 10000 in float64) takes the fewest that hold them.
static std::vector<int> chunk_ctas_asked(const Work& w, bool mixed) {
  std::vector<int> k = chunk_ctas(w, mixed);
  for (int i = 0; i < w.count && w.count < w.num_sms; ++i)
    for (int q : kChunkSizes)
      if (q > k[i] && q <= g_chunk_max_ctas && !chunk_fits(w.inst_host[i], k[i], mixed)) k[i] = q;
  return k;
}

bool chunk_ok(const Work& w, bool mixed, bool asked) {
  if (w.r != 0 || w.A.nlseg != 0 || w.P.nlseg != 0 || w.n < 1) return false;
  prepare_chunk();
  const std::vector<int> k = asked ? chunk_ctas_asked(w, mixed) : chunk_ctas(w, mixed);
  for (int i = 0; i < w.count; ++i)
    if (!chunk_fits(w.inst_host[i], k[i], mixed)) return false;
  return true;
}

// Whether the chunk beats the per-iteration kernels where the rows are even
// (chunk_even).  From 20 instances on it always did: 1200 control QPs 17 us per
// iteration against 88, 160 of them 3.8 against 12, 77 in float64 9.8 against 16;
// random patterns, 20 of n = 1e4 (3e5 nonzeros each) 13.1 against 28.7, 80 of
// n = 5000 22.7 against 46.4, 304 of n = 2500 28.5 against 77.3, in float64 20 of
// n = 5000 16.1 against 37.1 and 304 of n = 2500 92.9 against 185.
// A few instances on many CTAs pay for the cluster barriers and, on random
// patterns, for bank conflicts: random sparse QPs, per iteration in float32,
// 2.7 us (n = 1000, 4e3 nonzeros per CTA) against 7.5, 8.1 (n = 1e4, 19e3) against
// 8.0; in float64 10.5 (n = 4000, 8e3) against 13.
bool chunk_pays(const Work& w, bool mixed) {
  if (w.count >= 20) return true;
  long long k = 0;
  for (int c : chunk_ctas(w, mixed)) k += c;
  return (w.A.nnz + w.P.nnz) / k <= (mixed ? 18000 : 8000);
}

// Whether the rows are even enough for the slices (the plan's shapes known).  A
// slice is as wide as its longest row: one long row is walked by one warp, mostly on
// pads and past some length from L2, and many of them make the streams mostly pads.
// Measured, us an iteration, chunk against the faster row-block kernel:
// - one long row among rows of 10.  Float32, n = 1000 alone: 5.5 / 6.7 at 256 entries,
//   6.5 / 7.0 at 320, 8.7 / 7.0 at 384, 23.0 / 9.3 at 1000; n = 4000 at 2000 45.7 / 13.8;
//   a batch hides more of it: 160 of n = 1000 13.0 / 16.4 at 256, 29.0 / 19.5 at 1000.
//   Float64, n = 1000 alone: 23.3 / 24.5 at 384, 30.4 / 29.3 at 512; 24 of them
//   13.6 / 14.7 at 64, 19.2 / 17.5 at 128, 30.4 / 22.0 at 256; 160 of n = 300 19.2 / 22.2
//   at 128, 24.7 / 24.2 at 192; 160 of n = 2000 71.8 / 70.2 at 256.
// - a long row in every slice of A (groups over even groups).  Float32, where the
//   matrices stay in shared memory: n = 1000 alone 5.9 / 7.2 (6.5), 160 of n = 300 6.9 /
//   10.5 (4.7); where they do not: 160 of n = 2000 21.5 / 27.0 (2.7), 41.5 / 32.2 (4.3),
//   1200 of n = 300 28.9 / 30.5 (4.7), 47.7 / 38.6 (6.3).  Float64, which has time for
//   the streams: 160 of n = 1000 60.6 / 60.8 (4.4), 100 / 91 (6.5), 1200 of n = 300 74 /
//   125 (4.7).
bool chunk_even(const Work& w, bool mixed) {
  const ChunkPlan& ck = w.chunk;
  const std::vector<int> ctas = chunk_ctas(w, mixed);
  const size_t cap = w.count >= 2 * w.num_sms ? 112 * 1024 : CHUNK_SMEM_MAX;
  long long groups = 0, even = 0;
  int most = 0;
  bool resident = true;
  for (int i = 0; i < w.count; ++i) {
    const Inst& I = w.inst_host[i];
    const int4 g = ck.shape[i];
    const int k = ctas[i], oA = cdiv(cdiv(I.m, 32), k), oP = cdiv(cdiv(I.n, 32), k);
    const size_t fixed = mixed ? chunk_fixed_bytes<float>(I.n, I.m, oA, oP) : chunk_fixed_bytes<double>(I.n, I.m, oA, oP);
    resident = resident && fixed + ((size_t)g.x + g.y) / k * (mixed ? chunk_group_bytes<float>() : chunk_group_bytes<double>()) <= cap;
    groups += (long long)g.x + g.y;
    even += g.z;
    most = std::max(most, g.w);
  }
  const double millions = 1e-6 * (double)(w.A.nnz + w.P.nnz);
  const double row = mixed ? 320 + 50 * millions : (w.count < 20 ? 384 : 128) + 30 * millions;
  return most <= row && groups <= (mixed ? (resident ? 8 : 4) : 6) * even;
}

// The launches of one precision, one a class: the instances by the shared memory
// their vectors and matrices take, largest first within a class, so that
// smaller ones share an SM: up to 64 KB four a SM, up to 130 KB two (the part
// that does not fit streams from L2).  A batch of at least two instances an SM
// takes two a SM however large they are (two half-resident instances hide each
// other's barriers: horizon 100 alone 99.6 us per iteration of 4096 against
// 103.7); with fewer, a larger one keeps its SM to itself (160 instances: 3.8
// against 6.1).
template <typename V>
static void chunk_classes(Work& w, std::vector<ChunkClass>& out, std::vector<ChunkInst>& launch) {
  ChunkPlan& ck = w.chunk;
  const size_t gb = chunk_group_bytes<V>();
  constexpr int CLASSES = 3 + 16;                  // by what shares an SM (0..2), by the cluster's CTAs
  std::vector<ChunkInst> of[CLASSES];
  ChunkClass cls[CLASSES] = {};
  std::vector<int> seen;                           // in the order of their largest instances
  for (const ChunkInst& I : ck.order) {
    const int ctas = ck.ctas[I.id];
    const int oA = cdiv(I.nsA, ctas), oP = cdiv(I.nsP, ctas);
    const size_t fixed = chunk_fixed_bytes<V>(I.n, I.m, oA, oP);
    // a CTA's share of the groups, rounded up by a slice's worth
    const size_t own = ((size_t)ck.shape[I.id].x + ck.shape[I.id].y) / ctas;
    const size_t need = fixed + (ctas > 1 ? own + own / 8 + 64 : own) * gb;
    int c = 0;
    if (ctas > 1) c = 2 + ctas;
    else if (w.count >= w.num_sms)
      c = need <= 64 * 1024 && fixed <= 48 * 1024 ? 2
          : (need <= 130 * 1024 || w.count >= 2 * w.num_sms) && fixed <= 108 * 1024 ? 1 : 0;
    if (of[c].empty()) seen.push_back(c);
    of[c].push_back(I);
    ChunkClass& k = cls[c];
    k.ctas = ctas;
    const size_t cap = c == 2 ? 55 * 1024 : c == 1 ? 112 * 1024 : (size_t)CHUNK_SMEM_MAX;
    k.smem = std::max(k.smem, std::min(need, cap));
    const int own_slices = std::max(oA, oP);
    k.threads = std::max(k.threads, std::min(c == 2 ? 256 : c == 1 ? 512 : 1024, 32 * std::max(4, own_slices)));
  }
  out.clear();
  launch.clear();
  for (int c : seen) {
    cls[c].first = (int)launch.size();
    cls[c].count = (int)of[c].size();
    out.push_back(cls[c]);
    launch.insert(launch.end(), of[c].begin(), of[c].end());
  }
}

void chunk_plan_instances(Work& w) {
  ChunkPlan& ck = w.chunk;
  ck.order.resize(w.count);
  int sA = 0, sP = 0;
  for (const Inst& I : w.inst_host) sP += cdiv(I.m, 32);   // P's slices follow A's
  for (int i = 0; i < w.count; ++i) {
    const Inst& I = w.inst_host[i];
    ck.order[i] = ChunkInst{I.n, I.m, I.xoff, I.yoff, sA, cdiv(I.m, 32), sP, cdiv(I.n, 32), i};
    sA += cdiv(I.m, 32);
    sP += cdiv(I.n, 32);
  }
  ck.slices = sP;
}
void chunk_plan_order(Work& w) {
  ChunkPlan& ck = w.chunk;
  auto total = [&](const ChunkInst& p) { return (long long)ck.shape[p.id].x + ck.shape[p.id].y; };
  std::stable_sort(ck.order.begin(), ck.order.end(),
                   [&](const ChunkInst& p, const ChunkInst& q) {
                     const int rp = p.n + p.m, rq = q.n + q.m;   // with few instances the rows set the CTAs
                     return w.count < w.num_sms && rp != rq ? rp > rq : total(p) > total(q);
                   });
}
void chunk_plan_classes(Work& w, bool mixed) {
  w.chunk.ctas = chunk_ctas_asked(w, mixed);       // (chunk_ctas' where these fit)
  if (mixed) chunk_classes<float>(w, w.chunk.cls[1], w.chunk.launch_host[1]);
  else chunk_classes<double>(w, w.chunk.cls[0], w.chunk.launch_host[0]);
}

template <typename V>
static void run_chunk(Work& w, int j0, int len, const typename Pair<V>::T* val, V* xt, V* const* Z, V* ybar,
                      const V* b, const V* ylo, V* x, V* xbar, const V* c, const V* l, const V* u, cudaStream_t s) {
  Profiler& Pr = w.prof;
  ChunkPlan& ck = w.chunk;
  ChunkArgs<V> a{ck.launch[sizeof(V) == 4 ? 1 : 0], ck.sp, ck.idx, val, xt, Z[0], Z[1], x, xbar, ybar, b, ylo, c, l, u, w.row_ineq, w.tab, w.st,
                 w.tab_stride, w.n, 0};
  // kind 3: one launch holds both half-steps of `len` iterations
  if (Pr.on) Pr.begin(3, s, len * (launch_bytes(w, 0, sizeof(V)) + launch_bytes(w, 1, sizeof(V))));
  const std::vector<ChunkClass>& cls = ck.cls[sizeof(V) == 4 ? 1 : 0];
  // the classes run side by side (forked onto the plan's own streams), so that
  // their CTAs share the SMs and no class's last wave leaves the chip idle
  const size_t sides = std::min<size_t>(cls.size() - 1, ChunkPlan::SIDES);
  if (sides) cudaEventRecord(ck.fork, s);
  for (size_t k = 0; k < sides; ++k) cudaStreamWaitEvent(ck.side[k], ck.fork, 0);
  for (size_t k = 0; k < cls.size(); ++k) {
    const ChunkClass& q = cls[k];
    a.smem = (int)q.smem;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg =
        chunk_cfg<V>(q.ctas, q.count, q.threads, q.smem, k == 0 ? s : ck.side[(k - 1) % ChunkPlan::SIDES], at);
    if (q.ctas > 1) cudaLaunchKernelEx(&cfg, k_chunk<V, true>, a, q.first, j0, len);
    else cudaLaunchKernelEx(&cfg, k_chunk<V, false>, a, q.first, j0, len);
    count_launch();
  }
  for (size_t k = 0; k < sides; ++k) {
    cudaEventRecord(ck.join[k], ck.side[k]);
    cudaStreamWaitEvent(s, ck.join[k], 0);
  }
  if (Pr.on) Pr.end(s);
}

void chunk_run(Work& w, int len, bool mixed, cudaStream_t s, int j0) {
  if (len <= 0) return;
  if (mixed) {
    run_chunk<float>(w, j0, len, w.chunk.valf, w.fxt, w.fZ, w.fybar, w.fb, w.fylo, w.fx, w.fxbar, w.fc, w.fl, w.fu, s);
    w.fy = w.fZ[(j0 + len - 1) & 1] + w.n;
  } else {
    run_chunk<double>(w, j0, len, w.chunk.vald, w.xt, w.Z, w.ybar, w.bs, nullptr, w.x, w.xbar, w.cs, w.ls, w.us, s);
    w.y = w.Z[(j0 + len - 1) & 1] + w.n;
  }
}

}  // namespace pdqp
