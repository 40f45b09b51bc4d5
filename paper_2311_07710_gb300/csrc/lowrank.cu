// The half-steps of a problem with a low-rank term Q + F F' whose rows of
// P are short (a portfolio: a diagonal Q and a few dense rows of A).
//
// The general path reads F twice per iteration: k_lr_ft for F' x_md and, in
// k_primal, every thread its own row for F w (one row per lane: 32 lines per
// load, 196 CUDA blocks of 512 rows at n = 1e5).  Here one CUDA block takes the
// row tile of one k_lr_ft block, brings its rows of F to shared memory in
// contiguous 16-byte copies, finishes its rows and, with x_md of the next
// iteration in hand, forms the tile's partial of F' x_md from the same copy:
// F is read once.  The reduction of the partials runs beside the dual half-step
// (k_dual_lr), and both kernels of an iteration start early (launch_early): the
// tiles' copies of F run while that kernel, a few blocks, finishes.  Every sum keeps k_lr_ft's, k_lr_reduce's
// and lr_row's order and rounding, so the iterates are bitwise the general
// path's.
#include <algorithm>

#include "rowblock.cuh"
#include "rowupdate.cuh"

namespace pdqp {

constexpr int LRF_NT = 256;
constexpr int LRF_PRE = 4;     // entries of a thread's first row fetched ahead

// shared memory of a tile of `per` rows: F with rows padded so that 16-byte
// accesses of consecutive rows meet different banks, x_md of the rows, w
template <typename V>
__host__ __device__ inline int lrf_ld(int r) {
  constexpr int W = 16 / (int)sizeof(V);
  return r % W == 0 ? r + W : r | 1;
}
template <typename V>
static size_t lrf_smem(int per, int r) {
  return ((size_t)per * lrf_ld<V>(r) + ((per + 3) & ~3) + ((r + 3) & ~3)) * sizeof(V);
}

template <typename V>
struct LrPrimal {
  const int* __restrict__ rp;
  const int* __restrict__ col;
  const V* __restrict__ val;
  const V* zin;
  V* zout;
  V* x;
  V* xbar;
  V* xt;
  const V* c;
  const V* l;
  const V* u;
  const StepEntry* tab;
  const DevState* st;
  const V* __restrict__ F;
  const V* w;          // F' x_md of this iteration
  double* part;        // [tiles][r] partials of the next iteration's
  int n, r, per;
};

template <typename V>
__device__ __forceinline__ void lrf_stage(V* fs, const V* __restrict__ F, int rows, int r) {
  constexpr int W = 16 / (int)sizeof(V);
  const int ld = lrf_ld<V>(r);
  if (r % W == 0) {
    const int pr = r / W;                          // 16-byte pieces per row
    for (int i = threadIdx.x; i < rows * pr; i += LRF_NT) {
      const int j = i / pr, k = i - j * pr;
      const unsigned d = (unsigned)__cvta_generic_to_shared(fs + (size_t)j * ld + k * W);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(F + (size_t)i * W));
    }
  } else {
    for (int i = threadIdx.x; i < rows * r; i += LRF_NT) {
      const int j = i / r, k = i - j * r;
      fs[(size_t)j * ld + k] = F[i];
    }
  }
  asm volatile("cp.async.commit_group;\n" ::);
}

template <typename V>
__global__ void __launch_bounds__(LRF_NT) k_primal_lr(LrPrimal<V> a, int j) {
  extern __shared__ __align__(16) unsigned char lrf_sm[];
  grid_trigger();
  const int j0 = blockIdx.x * a.per, rows = min(a.per, a.n - j0), r = a.r, ld = lrf_ld<V>(r), tid = threadIdx.x;
  V* fs = reinterpret_cast<V*>(lrf_sm);
  V* zs = fs + (size_t)a.per * ld;
  V* ws = zs + ((a.per + 3) & ~3);
  lrf_stage<V>(fs, a.F + (size_t)j0 * r, rows, r);
  // what no kernel of the chunk writes (F, P, c, l, u; the chunk's first kernel
  // is launched normally) is on its way before the wait
  V cr0 = V(0), lr0 = V(0), ur0 = V(0), pv[LRF_PRE];
  int e0 = 0, e1 = 0, pc[LRF_PRE];
  if (tid < rows) {
    const int row = j0 + tid;
    e0 = a.rp[row]; e1 = a.rp[row + 1];
    cr0 = a.c[row]; lr0 = a.l[row]; ur0 = a.u[row];
  }
#pragma unroll
  for (int k = 0; k < LRF_PRE; ++k) {
    pc[k] = e0 + k < e1 ? a.col[e0 + k] : 0;
    pv[k] = e0 + k < e1 ? a.val[e0 + k] : V(0);
  }
  grid_wait();
  if (a.st->status != ST_RUNNING) {
    asm volatile("cp.async.wait_all;\n" ::);
    return;
  }
  for (int k = tid; k < r; k += LRF_NT) ws[k] = a.w[k];
  const StepEntry& e = a.tab[j];
  const V tau = step_tau<V>(e), ib = step_ib<V>(e), ibn = step_ibn<V>(e), thn = step_thn<V>(e);
  for (int base = 0; base < rows; base += LRF_NT) {
    const int t = base + tid, row = j0 + t;
    V s = V(0), xo = V(0), xb0 = V(0), cr = V(0), lr = V(0), ur = V(0);
    if (t < rows) {
      xo = a.x[row]; xb0 = a.xbar[row];
      if (base == 0) {
        V z[LRF_PRE];
#pragma unroll
        for (int k = 0; k < LRF_PRE; ++k) z[k] = e0 + k < e1 ? a.zin[pc[k]] : V(0);
        cr = cr0; lr = lr0; ur = ur0;
#pragma unroll
        for (int k = 0; k < LRF_PRE; ++k)
          if (e0 + k < e1) s = r_dot(pv[k], z[k], s);
        for (int k = e0 + LRF_PRE; k < e1; ++k) s = r_dot(a.val[k], a.zin[a.col[k]], s);
      } else {
        cr = a.c[row]; lr = a.l[row]; ur = a.u[row];
        const int q1 = a.rp[row + 1];
        for (int k = a.rp[row]; k < q1; ++k) s = r_dot(a.val[k], a.zin[a.col[k]], s);
      }
    }
    if (base == 0) {
      asm volatile("cp.async.wait_all;\n" ::);
      __syncthreads();
    }
    if (t < rows) {
      const V g = r_add(r_add(s, cr),
                        lr_row<V, V, V>(fs + (size_t)t * ld, ws, r, 0));
      V xn, xb, zo, xtn;
      primal_update<V>(tau, ib, ibn, thn, g, xo, xb0, lr, ur, xn, xb, zo, xtn);
      a.xbar[row] = xb;
      a.zout[row] = zo;
      a.xt[row] = xtn;
      a.x[row] = xn;
      zs[t] = zo;
    }
  }
  __syncthreads();
  // the tile's partial of F' x_md (k_lr_ft: thread (g, k) sums column k over
  // every G-th row in its factor's precision, then the G sums in order)
  __shared__ V sh[LRF_NT];
  const int G = LRF_NT / r, g = tid / r, k = tid % r;
  V acc = V(0);
  if (g < G)
    for (int t = g; t < rows; t += G) acc = r_fma(fs[(size_t)t * ld + k], zs[t], acc);
  sh[tid] = acc;
  __syncthreads();
  if (tid < r) {
    V s = V(0);
    for (int gg = 0; gg < G; ++gg) s = r_add(s, sh[gg * r + tid]);
    a.part[(size_t)blockIdx.x * r + tid] = (double)s;
  }
}

// Low-rank row terms (F w0)_j and (F w1)_j of a float64 check: 64 rows of F
// through shared memory, one thread per (row, iterate).
__global__ void __launch_bounds__(128) k_lr_rows(const double* __restrict__ F, int n, int r,
                                                 const double* __restrict__ w, int nit, double* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char lrf_sm[];
  const int ld = lrf_ld<double>(r), j0 = blockIdx.x * 64, rows = min(64, n - j0);
  double* fs = reinterpret_cast<double*>(lrf_sm);
  double* ws = fs + (size_t)64 * ld;
  for (int i = threadIdx.x; i < rows * r; i += 128) {
    const int j = i / r, k = i - j * r;
    fs[(size_t)j * ld + k] = F[(size_t)j0 * r + i];
  }
  const int wld = (r + 1) & ~1;
  for (int i = threadIdx.x; i < nit * r; i += 128) ws[(i / r) * wld + i % r] = w[i];
  __syncthreads();
  const int t = threadIdx.x & 63, it = threadIdx.x >> 6;
  if (t < rows && it < nit) 
    out[(size_t)it * n + j0 + t] = lr_row<double, double, double>(fs + (size_t)t * ld, ws + it * wld, r, 0);
}

void lowrank_rows(Work& w, const double* F, int nit, cudaStream_t s) {
  const size_t smem = ((size_t)64 * lrf_ld<double>(w.r) + 2 * ((w.r + 1) & ~1)) * sizeof(double);
  static const bool attr = cudaFuncSetAttribute(k_lr_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024) ==
                           cudaSuccess;
  (void)attr;
  launch(k_lr_rows, cdiv(w.n, 64), 128, smem, s, F, w.n, w.r, (const double*)w.wlr, nit, w.lr_rows);
}

constexpr int LRF_SMEM_MAX = 220 * 1024;

// Rows of P are short, on average and each of them: a thread walks a row, entry
// after entry, while its block waits.  With one variable in K rows of A, us an iteration
// against the faster general kernel: n = 2000, r = 16 in float32 15.3 / 21.9 (K = 0),
// 19.6 / 22.3 (128), 32.8 / 24.1 (512), 82.8 / 28.8 (2000), in float64 103 / 107 (128),
// 136 / 123 (512); n = 20000, r = 32 in float32 12.8 / 19.8 (128), 27.0 / 22.1 (512);
// n = 1e5, r = 64 31.3 / 33.5 (512), 82.9 / 33.6 (2000).
constexpr int LRF_ROW_MAX = 192;
bool lowrank_fused_ok(const Work& w, bool mixed) {
  if (w.r < 1 || w.count != 1 || w.P.nnz > 8LL * w.n || w.longest_P > LRF_ROW_MAX) return false;
  const int grid = lr_ft_grid(w), per = cdiv(w.n, grid);
  return (mixed ? lrf_smem<float>(per, w.r) : lrf_smem<double>(per, w.r)) <= (size_t)LRF_SMEM_MAX;
}

template <typename V>
static void run_chunk_lr(Work& w, int j0, int len, BCsr<V> A, BCsr<V> P, V* xt, V* const* Z, V* ybar, const V* b,
                         const V* ylo, V* x, V* xbar, const V* c, const V* l, const V* u, cudaStream_t s) {
  static const bool attr = cudaFuncSetAttribute(k_primal_lr<V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                LRF_SMEM_MAX) == cudaSuccess;
  (void)attr;
  Profiler& Pr = w.prof;
  const int grid = lr_ft_grid(w), per = cdiv(w.n, grid);
  LrPrimal<V> pa{P.rp, P.col, P.val, nullptr, nullptr, x, xbar, xt, c, l, u, w.tab, w.st, lr_factor<V>(w),
                 lr_weights<V>(w), w.lr_part, w.n, w.r, per};
  for (int j = j0; j < j0 + len; ++j) {
    if (Pr.on) Pr.begin(0, s, launch_bytes(w, 0, sizeof(V)));
    if (j == j0) lowrank_ft_part(w, pa.F, (const V*)Z[j & 1], s);   // later ones come from k_primal_lr
    run_dual_lr(w, j, grid, A, xt, Z, ybar, b, ylo, s);
    if (Pr.on) Pr.end(s);
    pa.zin = Z[j & 1];
    pa.zout = Z[(j + 1) & 1];
    if (Pr.on) Pr.begin(1, s, launch_bytes(w, 1, sizeof(V)));
    launch_early(k_primal_lr<V>, grid, LRF_NT, lrf_smem<V>(per, w.r), s, pa, j);
    if (Pr.on) Pr.end(s);
  }
}

void lowrank_run(Work& w, int len, bool mixed, cudaStream_t s, int j0) {
  if (len <= 0) return;
  if (mixed) {
    run_chunk_lr<float>(w, j0, len, w.A.bscaled_f(), w.P.bscaled_f(), w.fxt, w.fZ, w.fybar, w.fb, w.fylo, w.fx,
                        w.fxbar, w.fc, w.fl, w.fu, s);
    w.fy = w.fZ[(j0 + len - 1) & 1] + w.n;
  } else {
    run_chunk_lr<double>(w, j0, len, w.A.bscaled(), w.P.bscaled(), w.xt, w.Z, w.ybar, w.bs, nullptr, w.x, w.xbar, w.cs,
                         w.ls, w.us, s);
    w.y = w.Z[(j0 + len - 1) & 1] + w.n;
  }
}

}  // namespace pdqp
