// Learned warm start: a tensor-core (tcgen05) BF16 GEMM and the forward,
// backward and Adam kernels of the warm-start network (sm_103a).
//
// The paper has no learned component; Algorithm 1 takes its starting point
// (x^{0,0}, y^{0,0}) as an input and this network produces one for a member of
// a parameterised QP family from its data (c, b).  Network: per-feature
// normalisation u = (v - mean) * scale of v = [c; b], h_0 = u P' with a fixed
// random projection P (d x F), depth hidden layers h_j = relu(h_{j-1} W_j' + b_j)
// of width w, output o = h W_out' + b_out, prediction [x0; y0] = omean + ostd * o.
// Training minimises the mean squared error to the normalised solver outputs
// [x*; y*] with Adam.  Weights and activations are stored in bfloat16, every
// product accumulates in float32 in tensor memory, master weights, gradients
// and Adam moments are float32.
//
// GEMM: D[M x N] = A[M x K] * B[N x K]^T with A and B row-major bfloat16 (both
// K-major), persistent: one CUDA block per SM walks 128 x 256 tiles (128 x 128
// when N < 256) and k splits.  Thread 0 of warp 0 streams 64-wide K slices of
// A and B into a 4-stage shared-memory ring with TMA (128-byte swizzle),
// thread 0 of warp 1 issues tcgen05.mma (M=128, N=256, K=16, kind::f16 with
// bf16 A and B) on each stage into one of two float32 accumulators in tensor
// memory and releases the stage with tcgen05.commit, and warps 2..9 drain the
// other accumulator with tcgen05.ld into the fused epilogue (warp w reads TMEM
// lanes 32 (w mod 4) .. +32), so a tile's epilogue overlaps the next tile's
// main loop.  Split-K: a unit takes a range of k slices and writes raw float32
// partials that a second kernel sums in a fixed order.  Every mbarrier wait is
// bounded; a wait that gives up sets the error flag, the roles leave their
// loops, the copies still in flight land (bounded), the tensor memory is freed.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "pdqp.h"
#include "pdqp_ws.h"

typedef __nv_bfloat16 bf16;

namespace mlp {

// Tile: BM = 128 rows of A, BN = 128 or 256 rows of B (the N width of the MMA
// and of the tensor-memory accumulator), BK = 64 (one 128-byte swizzle row).
constexpr int BM = 128, BK = 64, STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;                    // 16 KiB
template <int BN> struct Tile {
  static constexpr int B_BYTES = BN * BK * 2;           // 16 or 32 KiB
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int EPI_BYTES = 8 * 32 * 32 * 4;     // the epilogue warps' stages
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /* alignment */ + 256 /* barriers */ + EPI_BYTES;
};
constexpr uint64_t WAIT_NS = 200000000ULL;            // a wait gives up after 0.2 s without progress

struct Epi {
  float* out_f;                  // float32 output [M x ldo] or null
  bf16* out_b;                   // bf16 output [M x ldo] or null
  const float* bias;             // [N] or null
  const bf16* mask;              // [M x ldm]: keep where mask > 0, else 0 (ReLU derivative), or null
  int ldo, ldm;
  int relu;
  int vec;                       // the outputs and the mask start on 16 (8) bytes: 4 columns per access
  // The network's last product writes its prediction [px | py] = pmean + pstd * value
  // in float64 (row lengths pn, N - pn; either array may be null) and nothing else.
  const float *pmean = nullptr, *pstd = nullptr;
  double *px = nullptr, *py = nullptr;
  int pn = 0, pm = 0;
  int pvec = 0;                  // pn and pm even, both arrays on 16 bytes: 2 columns per access
};

// A kernel of the network starts with early_start() and is launched by early():
// its blocks are set up while the last blocks of the kernel before it still run
// (every block of that kernel has started by then), and wait for its end before
// they touch memory (plain loads through pointers without __restrict__, which
// the compiler cannot move above the wait).  A training step is about 40 launches of a few microseconds:
// the gaps between them were 0.8 of 5.0 ms for 2048 samples.
__device__ __forceinline__ void early_start() {
  asm volatile("griddepcontrol.launch_dependents;\ngriddepcontrol.wait;\n" ::: "memory");
}
template <typename... KArgs, typename... Args>
static void early(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait for the completion of the phase with the given parity: gives up
// (false) after WAIT_NS without progress (progress = a counter another thread
// of the block advances, or null) or as soon as the error flag is set.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, const volatile int* err,
                                          const volatile int* progress = nullptr) {
  const uint32_t a = smem_u32(bar);
  uint64_t start = 0;
  int seen = progress ? *progress : 0;
  for (uint32_t i = 0;; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if ((i & 255) == 255) {
      const uint64_t now = global_ns();
      if (start == 0) start = now;
      if (progress && *progress != seen) {
        seen = *progress;
        start = now;
      }
      if (now - start > WAIT_NS || *err) return false;
    }
  }
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n" ::
          "r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile written by TMA
// with 128-byte swizzle: rows of 64 bf16 (128 B), 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t smem_desc(const void* p) {
  const uint64_t addr = (uint64_t)(smem_u32(p) & 0x3FFFF) >> 4;
  uint64_t d = 0;
  d |= addr;                         // bits 0-13: start address / 16
  d |= (uint64_t)1 << 16;            // bits 16-29: leading byte offset / 16 (ignored with this swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;  // bits 32-45: stride byte offset / 16
  d |= (uint64_t)1 << 46;            // bits 46-48: descriptor version 1
  d |= (uint64_t)2 << 61;            // bits 61-63: 128-byte swizzle
  return d;
}

// Instruction descriptor of kind::f16: bf16 A and B, both K-major, float32 D.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n) {
  return (1u << 4)                      // D format: f32
         | (1u << 7)                    // A format: bf16
         | (1u << 10)                   // B format: bf16
         | ((uint32_t)(n >> 3) << 17)   // N / 8
         | ((uint32_t)(m >> 4) << 24);  // M / 16
}

__device__ __forceinline__ float epi_value(float r, int row, int col, const Epi& e) {
  if (e.bias) r += e.bias[col];
  if (e.relu) r = fmaxf(r, 0.f);
  if (e.mask && !(__bfloat162float(e.mask[(size_t)row * e.ldm + col]) > 0.f)) r = 0.f;
  return r;
}

// An epilogue warp's stage: 32 rows of 32 floats, the eight 16-byte pieces of a
// row exchanged by its number so that a column of pieces meets all banks.
__device__ __forceinline__ int epi_at(int row, int piece) { return row * 32 + ((piece ^ (row & 7)) << 2); }
constexpr int EPI_WARPS = 8;
constexpr int GEMM_NT = 64 + 32 * EPI_WARPS;   // TMA, MMA and epilogue warps

// float -> double by integer instructions (the conversion instruction issues on
// the float64 pipe): the same value for every float (NaN payloads aside)
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xFFu;
  if (e - 1u >= 254u) return (double)x;           // zero, subnormal, infinite, NaN
  return __hiloint2double((int)((u & 0x80000000u) | (((u >> 3) & 0x0FFFFFFFu) + 0x38000000u)), (int)(u << 29));
}

// Where the prediction of (row, col) goes, or null.  Its value is
// pmean + pstd * v: the product of two floats is exact in float64, so one fused
// multiply-add rounds like the separate addition.
__device__ __forceinline__ double* pred_at(const Epi& e, int row, int col) {
  double* d = col < e.pn ? e.px : e.py;
  return d ? d + (size_t)row * (col < e.pn ? e.pn : e.pm) + (col < e.pn ? col : col - e.pn) : nullptr;
}
__device__ __forceinline__ void put_value(const Epi& e, int row, int col, float x) {
  if (e.pstd) {
    if (double* d = pred_at(e, row, col)) *d = __fma_rn((double)e.pstd[col], (double)x, (double)e.pmean[col]);
    return;
  }
  const size_t o = (size_t)row * e.ldo + col;
  if (e.out_f) e.out_f[o] = x;
  if (e.out_b) e.out_b[o] = __float2bfloat16_rn(x);
}

// The predictions of 32 rows x 32 columns staged as in store_chunk: 16 lanes
// store a row's 256 contiguous bytes, two columns each.  Two columns per lane
// widen their statistics once for their 16 rows; the value itself is widened
// by integer instructions, which leaves the float64 pipe one operation a value.
__device__ __forceinline__ void store_pred(const float* stg, int row0, int cb, int nend, const Epi& e) {
  const int lane = threadIdx.x & 31, cl = (lane & 15) * 2, col = cb + cl, r0 = lane >> 4;
  if (col >= nend) return;
  double* d = pred_at(e, row0 + r0, col);
  if (!d) return;
  const size_t ld = 2 * (size_t)(col < e.pn ? e.pn : e.pm);
  const double s0 = widen(e.pstd[col]), s1 = widen(e.pstd[col + 1]);
  const double m0 = widen(e.pmean[col]), m1 = widen(e.pmean[col + 1]);
  const float b0 = e.bias ? e.bias[col] : 0.f, b1 = e.bias ? e.bias[col + 1] : 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float2 v = *reinterpret_cast<const float2*>(stg + epi_at(2 * i + r0, cl >> 2) + (cl & 3));
    if (e.bias) { v.x += b0; v.y += b1; }
    *reinterpret_cast<double2*>(d + i * ld) = make_double2(__fma_rn(s0, widen(v.x), m0), __fma_rn(s1, widen(v.y), m1));
  }
}

// Epilogue of a warp's 32 x 32 accumulator values (rows row0.., columns cb..
// below nend), staged in `stg`: the raw float32 split-K partial of split z (ld =
// N), or the fused epilogue into the outputs.  A lane holds one accumulator row,
// so storing from its registers touches 32 rows at a time in 16-byte pieces;
// through shared memory eight lanes store a row's 128 contiguous bytes, four rows
// an instruction.  The short-K products of the network are bound by this path
// (its shared-memory and store wavefronts and its chain of dependent
// instructions), so the common case reads all its values first, takes its
// branches outside the loops, and eight warps drain an accumulator, two per 32
// TMEM lanes: 512 x 30000 x 64 took 31 us with four warps, 19.1 with eight and 16
// columns a chunk, 17.9 so; 30000 x 1024 x 256 went from 48.0 to 43.4.
__device__ __forceinline__ void store_chunk(const float* stg, int row0, int cb, int z, int M, int N, int nend,
                                            const Epi& epi, float* partial) {
  const int lane = threadIdx.x & 31;
  const bool whole = row0 + 32 <= M;            // whole rows; the last chunk may hold fewer than 32 columns
  const bool vec = whole && ((nend - cb) & 3) == 0 && epi.vec &&
                   (partial ? (N & 3) == 0 : (epi.ldo & 3) == 0 && (!epi.mask || (epi.ldm & 3) == 0));
  if (epi.pvec && !partial && whole && ((nend - cb) & 1) == 0) {
    store_pred(stg, row0, cb, nend, epi);
    return;
  }
  if (vec && (partial || !epi.pstd)) {
    const int col = cb + (lane & 7) * 4, r0 = lane >> 3, row = row0 + r0;
    if (col >= nend) return;
    float4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = *reinterpret_cast<const float4*>(stg + epi_at(4 * i + r0, lane & 7));
    if (partial) {
      float* d = partial + ((size_t)z * M + row) * N + col;
#pragma unroll
      for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(d + (size_t)(4 * i) * N) = v[i];
      return;
    }
    if (epi.bias) {
      const float4 b = make_float4(epi.bias[col], epi.bias[col + 1], epi.bias[col + 2], epi.bias[col + 3]);
#pragma unroll
      for (int i = 0; i < 8; ++i) { v[i].x += b.x; v[i].y += b.y; v[i].z += b.z; v[i].w += b.w; }
    }
    if (epi.relu) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        v[i].x = fmaxf(v[i].x, 0.f); v[i].y = fmaxf(v[i].y, 0.f);
        v[i].z = fmaxf(v[i].z, 0.f); v[i].w = fmaxf(v[i].w, 0.f);
      }
    }
    if (epi.mask) {
      const bf16* mk = epi.mask + (size_t)row * epi.ldm + col;
      uint2 q[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) q[i] = *reinterpret_cast<const uint2*>(mk + (size_t)(4 * i) * epi.ldm);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&q[i].x);
        const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&q[i].y);
        if (!(__low2float(a) > 0.f)) v[i].x = 0.f;
        if (!(__high2float(a) > 0.f)) v[i].y = 0.f;
        if (!(__low2float(b) > 0.f)) v[i].z = 0.f;
        if (!(__high2float(b) > 0.f)) v[i].w = 0.f;
      }
    }
    const size_t o = (size_t)row * epi.ldo + col;
    if (epi.out_f) {
#pragma unroll
      for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(epi.out_f + o + (size_t)(4 * i) * epi.ldo) = v[i];
    }
    if (epi.out_b) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[i].x, v[i].y), h1 = __floats2bfloat162_rn(v[i].z, v[i].w);
        uint2 q;
        q.x = *reinterpret_cast<const uint32_t*>(&h0);
        q.y = *reinterpret_cast<const uint32_t*>(&h1);
        *reinterpret_cast<uint2*>(epi.out_b + o + (size_t)(4 * i) * epi.ldo) = q;
      }
    }
    return;
  }
  // ragged rows or columns, unaligned rows: one column per lane
  const int col = cb + lane;
  if (col >= nend) return;
  for (int i = 0; i < 32; ++i) {
    const int row = row0 + i;
    if (row >= M) return;
    const float v = stg[epi_at(i, lane >> 2) + (lane & 3)];
    if (partial) {
      partial[((size_t)z * M + row) * N + col] = v;
      continue;
    }
    put_value(epi, row, col, epi_value(v, row, col, epi));
  }
}

// 32 float32 accumulator columns of this warp's TMEM lanes, from column address
// taddr: the load, and the wait after which v holds them
__device__ __forceinline__ void tmem_ld32(uint32_t (&v)[32], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait(uint32_t (&v)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]),
                 "+r"(v[15]), "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]),
                 "+r"(v[22]), "+r"(v[23]), "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]),
                 "+r"(v[29])
               :
               : "memory");
  asm volatile("" : "+r"(v[30]), "+r"(v[31])::"memory");
}

// One warp's share of an accumulator (TMEM base address of its lanes, columns
// 32 half, 32 half + 64, ... of width) through its stage into the outputs.  The
// last chunk of a width that 32 does not divide reads columns past it, which lie
// in this CTA's 512 allocated ones and are not stored.
__device__ __forceinline__ void drain(float* stg, uint32_t tmem, int half, int width, int row0, int n0, int z, int M,
                                      int N, const Epi& epi, float* partial) {
  const int lane = threadIdx.x & 31, nend = min(n0 + width, N);
  uint32_t v[32];
  int c0 = 32 * half;
  if (c0 < width && n0 + c0 < N) tmem_ld32(v, tmem + (uint32_t)c0);
  for (; c0 < width && n0 + c0 < N; c0 += 64) {
    tmem_wait(v);
    __syncwarp();                             // the previous chunk has left the stage
#pragma unroll
    for (int i = 0; i < 8; ++i)
      *reinterpret_cast<float4*>(stg + epi_at(lane, i)) =
          make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]), __uint_as_float(v[4 * i + 2]),
                      __uint_as_float(v[4 * i + 3]));
    __syncwarp();
    if (c0 + 64 < width && n0 + c0 + 64 < N) tmem_ld32(v, tmem + (uint32_t)(c0 + 64));   // lands while this one goes out
    store_chunk(stg, row0, n0 + c0, z, M, N, nend, epi, partial);
  }
}

// D = A B' (bf16 A, B K-major, float32 accumulation in tensor memory), persistent:
// one CTA per SM takes work units u = blockIdx.x,
// blockIdx.x + gridDim.x, ... (a unit is one BM x BN tile of one k split;
// the tiles in bands of tile rows, see `unit`).
// Warp roles: warp 0 lane 0 issues the TMA loads of every unit through the
// STAGES ring, warp 1 lane 0 the MMAs, warps 2..9 drain the accumulators
// (warp w reads TMEM lanes 32 (w mod 4) .. +32).  Two accumulators of BN
// columns: the epilogue of one unit overlaps the main loop of the next.
// Every wait is bounded (WAIT_NS without progress, or the error flag), after
// which the roles leave their loops, the copies in flight land, and the TMEM
// is freed.
template <int BN>
__global__ void __launch_bounds__(GEMM_NT, 1)
    k_gemm_tn_p(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, int M, int N,
                int K, int ktps, int splits, Epi epi, float* partial, int* err) {
  constexpr int STAGE_BYTES = Tile<BN>::STAGE_BYTES;
  extern __shared__ __align__(1024) unsigned char smraw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(sm + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;       // [2]: the MMAs of a unit are done
  uint64_t* acc_empty = acc_full + 2;        // [2]: the epilogue has read the accumulator
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
  float* epi_stage = (float*)(sm + STAGES * STAGE_BYTES + 256);
  __shared__ volatile int s_fail;
  __shared__ int s_issued;                   // stage loads issued, for the cleanup
  __shared__ volatile int s_progress;        // stages consumed by the MMA issuer
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tn = (N + BN - 1) / BN, tm = (M + BM - 1) / BM;
  const int KT = (K + BK - 1) / BK;
  const int units = tm * tn * splits;

  if (threadIdx.x == 0) {
    s_fail = 0;
    s_issued = 0;
    s_progress = 0;
    for (int q = 0; q < STAGES; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&acc_full[q], 1);
      mbar_init(&acc_empty[q], EPI_WARPS);   // one arrival per epilogue warp
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {   // two accumulators: 128 lanes x 2 BN float32 columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"(2 * BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = *tmem_slot;
  early_start();

  // tiles in bands of GROUP tile rows, column-major inside a band: the CTAs
  // running together cover about GROUP rows of A and gridDim / GROUP columns of
  // B tiles, a working set that stays in L2
  constexpr int GROUP = 8;
  auto unit = [&](int u, int& m0, int& n0, int& kt0, int& nk, int& z) {
    z = u / (tm * tn);
    const int t = u - z * (tm * tn);
    const int band = t / (GROUP * tn), first = band * GROUP;
    const int rows = min(tm - first, GROUP);
    const int q = t - band * GROUP * tn;
    m0 = (first + q % rows) * BM;
    n0 = (q / rows) * BN;
    kt0 = z * ktps;
    nk = min(KT, kt0 + ktps) - kt0;
  };

  if (warp == 0 && lane == 0) {   // TMA producer
    int i = 0;
    for (int u = blockIdx.x; u < units && !s_fail; u += gridDim.x) {
      int m0, n0, kt0, nk, z;
      unit(u, m0, n0, kt0, nk, z);
      for (int k = 0; k < nk; ++k, ++i) {
        const int q = i % STAGES;
        if (i >= STAGES && !mbar_wait(&empty[q], ((i / STAGES) - 1) & 1, err, &s_progress)) {
          s_fail = 1;
          break;
        }
        unsigned char* a = sm + q * STAGE_BYTES;
        mbar_expect_tx(&full[q], STAGE_BYTES);
        tma_load_2d(a, &mapA, &full[q], (kt0 + k) * BK, m0);
        tma_load_2d(a + A_BYTES, &mapB, &full[q], (kt0 + k) * BK, n0);
        s_issued = i + 1;
      }
    }
  } else if (warp == 1 && lane == 0) {   // MMA issuer
    const uint32_t idesc = instr_desc(BM, BN);
    int i = 0, lt = 0;
    for (int u = blockIdx.x; u < units && !s_fail; u += gridDim.x, ++lt) {
      int m0, n0, kt0, nk, z;
      unit(u, m0, n0, kt0, nk, z);
      const int buf = lt & 1;
      // the epilogue has drained this accumulator (its first use passes at once)
      if (!mbar_wait(&acc_empty[buf], ((lt >> 1) & 1) ^ 1, err)) {
        s_fail = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n");
      const uint32_t acc_tm = tmem + (uint32_t)(buf * BN);
      for (int k = 0; k < nk; ++k, ++i) {
        const int q = i % STAGES;
        if (!mbar_wait(&full[q], (i / STAGES) & 1, err)) {
          s_fail = 1;
          break;
        }
        s_progress = i + 1;
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        const unsigned char* a = sm + q * STAGE_BYTES;
        const uint64_t da = smem_desc(a), db = smem_desc(a + A_BYTES);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) {
          const uint64_t step = (uint64_t)((kk * 16 * 2) >> 4);   // 32 bytes further along K
          const uint32_t acc = (k > 0 || kk > 0) ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc_tm),
              "l"(da + step), "l"(db + step), "r"(idesc), "r"(acc));
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
            smem_u32(&empty[q])));
      }
      if (s_fail) break;
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
          smem_u32(&acc_full[buf])));
    }
  } else if (warp >= 2) {   // epilogue
    const int sp = warp & 3;
    int lt = 0;
    for (int u = blockIdx.x; u < units; u += gridDim.x, ++lt) {
      int m0, n0, kt0, nk, z;
      unit(u, m0, n0, kt0, nk, z);
      const int buf = lt & 1;
      if (s_fail || !mbar_wait(&acc_full[buf], (lt >> 1) & 1, err, &s_progress)) {
        s_fail = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n");
      drain(epi_stage + (warp - 2) * 32 * 32, tmem + ((uint32_t)(sp * 32) << 16) + (uint32_t)(buf * BN),
            (warp - 2) >> 2, BN, m0 + sp * 32, n0, z, M, N, epi, splits > 1 ? partial : nullptr);
      asm volatile("tcgen05.fence::before_thread_sync;\n");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&acc_empty[buf])) : "memory");
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  if (s_fail && threadIdx.x == 0) {   // record the failure; let the copies in flight land
    atomicExch(err, 1);
    const int issued = s_issued;
    for (int i = max(0, issued - STAGES); i < issued; ++i) {
      int never = 0;
      mbar_wait(&full[i % STAGES], (i / STAGES) & 1, &never);
    }
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(2 * BN));
}

// --------------------------------------------------------------------------
// The same product on CTA pairs (cta_group::2): a cluster of two CTAs works on
// one 256 x bn tile.  Each CTA loads its 128 rows of A and its half of the bn rows of
// B, the even CTA's thread issues M = 256 MMAs that read both CTAs' shared memory,
// and each CTA drains the 128 rows that its tensor memory holds.  Per MMA step a
// CTA then moves 16 KB through shared memory (TMA write and tensor-core read of
// 4 KB of A and 4 KB of B) instead of 24 KB: with one CTA per tile the 192 bytes
// a clock exceed the 128 of the shared memory, which bound k_gemm_tn_p.
// bn (a multiple of 16, <= 256) is chosen so that the tiles fill the waves
// (plan_pairs).  Barriers: `full` lives in the even CTA and counts both CTAs'
// bytes; `empty` and `acc_full` are signalled in both CTAs by a multicast commit;
// `acc_empty` in the even CTA takes an arrival of each CTA's epilogue warps.
// Every wait is bounded as in k_gemm_tn_p; both CTAs meet at a cluster barrier
// before they leave, so no signal reaches shared memory that is gone.
constexpr int P_STAGES = 6;
constexpr int P_B_BYTES = 128 * BK * 2;                 // at most 128 rows of B per CTA
constexpr int P_STAGE_BYTES = A_BYTES + P_B_BYTES;      // 32 KiB
constexpr int P_SMEM_BYTES = P_STAGES * P_STAGE_BYTES + 1024 + 256 + EPI_WARPS * 32 * 32 * 4;

__device__ __forceinline__ uint32_t mapa_u32(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// a load into this CTA whose bytes count on the barrier at cluster address bar
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];\n" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void commit_pair(uint64_t* bar) {   // arrives on this barrier in both CTAs
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3));
}

__global__ void __launch_bounds__(GEMM_NT, 1) __cluster_dims__(2, 1, 1)
    k_gemm_tn_pair(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, int M, int N,
                   int K, int bn, int ktps, int splits, Epi epi, float* partial, int* err) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(sm + P_STAGES * P_STAGE_BYTES);
  uint64_t* empty = full + P_STAGES;
  uint64_t* acc_full = empty + P_STAGES;     // [2]
  uint64_t* acc_empty = acc_full + 2;        // [2]
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
  float* epi_stage = (float*)(sm + P_STAGES * P_STAGE_BYTES + 256);
  __shared__ volatile int s_fail;
  __shared__ int s_issued;
  __shared__ volatile int s_progress;        // stages consumed (even CTA), stages granted (odd CTA)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = blockIdx.x & 1;
  const bool leader = rank == 0;
  const int tn = (N + bn - 1) / bn, tm = (M + 2 * BM - 1) / (2 * BM);
  const int KT = (K + BK - 1) / BK;
  const int units = tm * tn * splits;
  const int u0 = blockIdx.x >> 1, du = gridDim.x >> 1;
  const uint32_t half_bytes = (uint32_t)(bn / 2) * BK * 2;

  if (threadIdx.x == 0) {
    s_fail = 0;
    s_issued = 0;
    s_progress = 0;
    for (int q = 0; q < P_STAGES; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&acc_full[q], 1);
      mbar_init(&acc_empty[q], 2 * EPI_WARPS);   // the epilogue warps of both CTAs
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {   // both CTAs: two accumulators of 256 float32 columns
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  cluster_sync();                            // the peer's barriers are initialised
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = *tmem_slot;
  early_start();

  // tiles in bands of tile rows, as k_gemm_tn_p (4 x 256 rows)
  constexpr int GROUP = 4;
  auto unit = [&](int u, int& m0, int& n0, int& kt0, int& nk, int& z) {
    z = u / (tm * tn);
    const int t = u - z * (tm * tn);
    const int band = t / (GROUP * tn), first = band * GROUP;
    const int rows = min(tm - first, GROUP);
    const int q = t - band * GROUP * tn;
    m0 = (first + q % rows) * 2 * BM;
    n0 = (q / rows) * bn;
    kt0 = z * ktps;
    nk = min(KT, kt0 + ktps) - kt0;
  };

  if (warp == 0 && lane == 0) {   // TMA producer of this CTA's halves
    int i = 0;
    for (int u = u0; u < units && !s_fail; u += du) {
      int m0, n0, kt0, nk, z;
      unit(u, m0, n0, kt0, nk, z);
      for (int k = 0; k < nk; ++k, ++i) {
        const int q = i % P_STAGES;
        if (i >= P_STAGES && !mbar_wait(&empty[q], ((i / P_STAGES) - 1) & 1, err, &s_progress)) {
          s_fail = 1;
          break;
        }
        if (!leader) s_progress = i + 1;
        unsigned char* a = sm + q * P_STAGE_BYTES;
        if (leader) mbar_expect_tx(&full[q], 2 * (A_BYTES + half_bytes));
        const uint32_t bar = mapa_u32(smem_u32(&full[q]), 0);
        tma_load_2d_pair(a, &mapA, bar, (kt0 + k) * BK, m0 + (int)rank * BM);
        tma_load_2d_pair(a + A_BYTES, &mapB, bar, (kt0 + k) * BK, n0 + (int)rank * (bn / 2));
        s_issued = i + 1;
      }
    }
  } else if (warp == 1 && lane == 0 && leader) {   // MMA issuer
    const uint32_t idesc = instr_desc(2 * BM, bn);
    int i = 0, lt = 0;
    for (int u = u0; u < units && !s_fail; u += du, ++lt) {
      int m0, n0, kt0, nk, z;
      unit(u, m0, n0, kt0, nk, z);
      const int buf = lt & 1;
      if (!mbar_wait(&acc_empty[buf], ((lt >> 1) & 1) ^ 1, err)) {
        s_fail = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n");
      const uint32_t acc_tm = tmem + (uint32_t)(buf * 256);
      for (int k = 0; k < nk; ++k, ++i) {
        const int q = i % P_STAGES;
        if (!mbar_wait(&full[q], (i / P_STAGES) & 1, err)) {
          s_fail = 1;
          break;
        }
        s_progress = i + 1;
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        const unsigned char* a = sm + q * P_STAGE_BYTES;
        const uint64_t da = smem_desc(a), db = smem_desc(a + A_BYTES);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) {
          const uint64_t step = (uint64_t)((kk * 16 * 2) >> 4);
          const uint32_t acc = (k > 0 || kk > 0) ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc_tm),
              "l"(da + step), "l"(db + step), "r"(idesc), "r"(acc));
        }
        commit_pair(&empty[q]);
      }
      if (s_fail) break;
      commit_pair(&acc_full[buf]);
    }
  } else if (warp >= 2) {   // epilogue of this CTA's 128 rows
    const int sp = warp & 3;
    const uint32_t ae0 = mapa_u32(smem_u32(&acc_empty[0]), 0), ae1 = mapa_u32(smem_u32(&acc_empty[1]), 0);
    int lt = 0;
    for (int u = u0; u < units; u += du, ++lt) {
      int m0, n0, kt0, nk, z;
      unit(u, m0, n0, kt0, nk, z);
      const int buf = lt & 1;
      if (s_fail || !mbar_wait(&acc_full[buf], (lt >> 1) & 1, err, &s_progress)) {
        s_fail = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n");
      drain(epi_stage + (warp - 2) * 32 * 32, tmem + ((uint32_t)(sp * 32) << 16) + (uint32_t)(buf * 256),
            (warp - 2) >> 2, bn, m0 + (int)rank * BM + sp * 32, n0, z, M, N, epi, splits > 1 ? partial : nullptr);
      asm volatile("tcgen05.fence::before_thread_sync;\n");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(buf ? ae1 : ae0)
                     : "memory");
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  cluster_sync();
  if (s_fail && threadIdx.x == 0) {   // record the failure; let the copies in flight land (both CTAs' count on the leader)
    atomicExch(err, 1);
    const int issued = s_issued;
    if (leader)
      for (int i = max(0, issued - P_STAGES); i < issued; ++i) {
        int never = 0;
        mbar_wait(&full[i % P_STAGES], (i / P_STAGES) & 1, &never);
      }
  }
  __syncthreads();
  cluster_sync();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512));
}

// The bounded wait of the tensor-core kernels on an mbarrier that nothing
// completes: it gives up after WAIT_NS and raises the error flag, as a GEMM
// whose copies or MMAs never landed would (the host then reads
// PDQP_DEVICE_TIMEOUT and the context stays usable).
__global__ void k_wait_probe(int* err) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait(&bar, 0, err)) atomicExch(err, 1);
}

// Sum of the split-K partials in a fixed order, then the epilogue: W columns
// per thread (4 where N and the leading dimensions allow), a row per grid y.
template <int W>
__global__ void __launch_bounds__(128) k_splitk_epi(const float* part, int splits, int M, int N, Epi epi) {
  early_start();
  const size_t MN = (size_t)M * N;
  const int col = (blockIdx.x * 128 + threadIdx.x) * W;
  if (col >= N) return;
  for (int row = blockIdx.y; row < M; row += gridDim.y) {
    const float* p = part + (size_t)row * N + col;
    float r[W];
#pragma unroll
    for (int i = 0; i < W; ++i) r[i] = 0.f;
    for (int z = 0; z < splits; ++z) {
      if constexpr (W == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p + z * MN);
        r[0] += q.x; r[1] += q.y; r[2] += q.z; r[3] += q.w;
      } else {
        r[0] += p[z * MN];
      }
    }
#pragma unroll
    for (int i = 0; i < W; ++i) put_value(epi, row, col + i, epi_value(r[i], row, col + i, epi));
  }
}

// --------------------------------------------------------------------------
// network kernels
// --------------------------------------------------------------------------
__device__ __forceinline__ long long visit(long long a, long long s, long long count, long long i) {
  return (a * i + s) % count;
}

// The elementwise kernels below take W columns per thread (two, in 16-byte
// accesses, where n and m are even) and ROWS_PER rows per grid y: the
// per-feature constants are read (and converted) once, no index is divided,
// and the rows' loads are in flight together.  What bounds them is memory or,
// where a value is converted, GB300's float64 pipe (two lanes per clock per
// SM, conversions included).
constexpr int ROWS_PER = 16;
constexpr int BATCH = 8;            // rows loaded before the first is used

template <int W>
__device__ __forceinline__ void load_cols(const double* p, double (&v)[W]) {
  if constexpr (W == 2) {
    const double2 q = __ldcs(reinterpret_cast<const double2*>(p));
    v[0] = q.x;
    v[1] = q.y;
  } else {
    v[0] = __ldcs(p);
  }
}

// u = bf16((fl32(v) - mean) * scale) for rows [row0, row0+rows) of v = [C | B]
template <int W>
__global__ void __launch_bounds__(256)
    k_prep_input(const double* C, const double* B, int n, int m, long long row0, int rows,
                 const float* mean, const float* scale, bf16* U, int ldu) {
  early_start();
  const int f = (blockIdx.x * 256 + threadIdx.x) * W;
  if (f >= n + m) return;
  const double* src = f < n ? C + (size_t)row0 * n + f : B + (size_t)row0 * m + (f - n);
  const size_t ld = f < n ? n : m;
  float mu[W], sc[W];
#pragma unroll
  for (int i = 0; i < W; ++i) { mu[i] = mean[f + i]; sc[i] = scale[f + i]; }
  const int r1 = min(rows, (int)(blockIdx.y + 1) * ROWS_PER);
  for (int r = blockIdx.y * ROWS_PER; r < r1; r += BATCH) {
    double v[BATCH][W];
#pragma unroll
    for (int k = 0; k < BATCH; ++k)
      if (r + k < r1) load_cols<W>(src + (r + k) * ld, v[k]);
#pragma unroll
    for (int k = 0; k < BATCH; ++k) {
      if (r + k >= r1) break;
      bf16 h[W];
#pragma unroll
      for (int i = 0; i < W; ++i) h[i] = __float2bfloat16_rn(__fmul_rn(__fsub_rn((float)v[k][i], mu[i]), sc[i]));
      bf16* d = U + (size_t)(r + k) * ldu + f;
      if constexpr (W == 2) *reinterpret_cast<__nv_bfloat162*>(d) = __nv_bfloat162(h[0], h[1]);
      else *d = h[0];
    }
  }
}

// t = (fl32(v) - omean) * oinv, float32, for rows [0, count) of [X | Y]
template <int W>
__global__ void __launch_bounds__(256)
    k_prep_target(const double* X, const double* Y, int n, int m, long long count,
                  const float* omean, const float* oinv, float* T, int ldt) {
  early_start();
  const int f = (blockIdx.x * 256 + threadIdx.x) * W;
  if (f >= n + m) return;
  const double* src = f < n ? X + f : Y + (f - n);
  const size_t ld = f < n ? n : m;
  float mu[W], sc[W];
#pragma unroll
  for (int i = 0; i < W; ++i) { mu[i] = omean[f + i]; sc[i] = oinv[f + i]; }
  for (long long b = blockIdx.y; b * ROWS_PER < count; b += gridDim.y) {
    const long long r1 = min(count, (b + 1) * ROWS_PER);
    for (long long r = b * ROWS_PER; r < r1; r += BATCH) {
      double v[BATCH][W];
#pragma unroll
      for (int k = 0; k < BATCH; ++k)
        if (r + k < r1) load_cols<W>(src + (r + k) * ld, v[k]);
#pragma unroll
      for (int k = 0; k < BATCH; ++k) {
        if (r + k >= r1) break;
        float t[W];
#pragma unroll
        for (int i = 0; i < W; ++i) t[i] = __fmul_rn(__fsub_rn((float)v[k][i], mu[i]), sc[i]);
        if constexpr (W == 2) *reinterpret_cast<float2*>(T + (r + k) * ldt + f) = make_float2(t[0], t[1]);
        else T[(r + k) * ldt + f] = t[0];
      }
    }
  }
}

// The sum of (hi, lo) and x, the rounding error kept (Knuth's two-sum), plus a
// low-order term.
__device__ __forceinline__ void pair_add(float& hi, float& lo, float x, float xl) {
  const float t = __fadd_rn(hi, x), b = __fsub_rn(t, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, b)), __fsub_rn(x, b));
  hi = t;
  lo = __fadd_rn(lo, __fadd_rn(e, xl));
}

// Per-feature mean and sum of squared deviations of a range of rows, one pass:
// deviations from the range's first row.  That row is one of the data, so its
// squared distance from the mean is at most FIT_ROWS times the range's
// variance, and the cancellation in M2 costs at most about that factor of a
// rounding.  In float64 the pass takes three float64-pipe operations a value
// (1.27 ms for 4096 x 60000 values at that pipe's rate); it takes the difference
// there, and the sums run on float32 pairs: the difference's bits split into
// 24 + 23 (truncated at 2^-46 of it), products and sums with their exact
// rounding errors.  Values whose square, its error or a range's sum of squares
// leaves float32's range take the float64 sums.  Two arrays per launch (grid z) and short ranges, so
// that the blocks fill whole waves (ranges of 256 rows, one array a launch: a
// little over two waves, 1.48 ms; the two-pass form before, 157 blocks of one
// column per thread: 4.8 ms).
constexpr int FIT_ROWS = 64;
struct FitPair {
  const double* v[2];
  double* mean[2];       // [ranges x nf]
  double* m2[2];
};
__global__ void __launch_bounds__(256) k_fit_part(FitPair a, long long count, int nf) {
  const int f = blockIdx.x * 256 + threadIdx.x;
  if (f >= nf) return;
  const double* V = a.v[blockIdx.z];
  for (long long b = blockIdx.y; b * FIT_ROWS < count; b += gridDim.y) {
    const long long r0 = b * FIT_ROWS;
    const int rows = (int)min((long long)FIT_ROWS, count - r0);
    const double* p = V + (size_t)r0 * nf + f;
    const double K = isfinite(p[0]) ? p[0] : 0.0;
    float sh = 0.f, sl = 0.f, qh = 0.f, ql = 0.f;
    double sd = 0.0, qd = 0.0;
    for (int r = 0; r < rows; r += BATCH) {
      double v[BATCH];                             // all in flight before the first is used
#pragma unroll
      for (int k = 0; k < BATCH; ++k) v[k] = r + k < rows ? __ldcs(p + (size_t)(r + k) * nf) : K;
#pragma unroll
      for (int k = 0; k < BATCH; ++k) {            // (a row past the end adds 0)
        const double d = v[k] - K;
        const unsigned hw = (unsigned)__double2hiint(d), lw = (unsigned)__double2loint(d);
        const unsigned e = (hw >> 20) & 0x7FFu, sg = hw & 0x80000000u;
        if (e - 973u <= 109u) {                    // 2^-50 <= |d| < 2^60: FIT_ROWS squares stay below 2^126
          const float hi = __uint_as_float(sg | ((e - 896u) << 23) | (__funnelshift_l(lw, hw, 3) & 0x7FFFFFu));
          const float lo = __fmul_rn(__fsub_rn(__uint_as_float(0x4B000000u | ((lw >> 6) & 0x7FFFFFu)), 8388608.f),
                                     __uint_as_float(sg | ((e - 942u) << 23)));
          pair_add(sh, sl, hi, lo);
          const float q = __fmul_rn(hi, hi);
          pair_add(qh, ql, q, __fmaf_rn(__fadd_rn(hi, hi), lo, __fmaf_rn(hi, hi, -q)));
        } else if (((hw << 1) | lw) != 0u) {       // not a zero
          sd += d;
          qd = fma(d, d, qd);
        }
      }
    }
    const double s = (double)sh + (double)sl + sd, q = (double)qh + (double)ql + qd;
    const double c = s * (1.0 / (double)rows), t = fma(-s, c, q);
    a.mean[blockIdx.z][(size_t)b * nf + f] = K + c;
    a.m2[blockIdx.z][(size_t)b * nf + f] = t < 0.0 ? 0.0 : t;    // (a NaN stays one)
  }
}

// the ranges merged in order (Chan, Golub & LeVeque 1983): per-feature mean and
// population std over all rows; std below 1e-8 counts as 1.  The merge weights
// are the same for every feature: the block's threads form 128 at a time.
struct FitOut {
  float* mean[2];
  float* scale[2];
  float* stdv[2];        // null: not kept
};
__global__ void __launch_bounds__(128) k_fit_merge(FitPair a, long long count, int nf, FitOut o) {
  __shared__ double sw[128], sv[128];
  const int f = blockIdx.x * 128 + threadIdx.x;
  const double *pm = a.mean[blockIdx.z], *p2 = a.m2[blockIdx.z];
  const long long nb = (count + FIT_ROWS - 1) / FIT_ROWS;
  double mu = 0.0, q = 0.0;
  if (f < nf) { mu = pm[f]; q = p2[f]; }
  for (long long b0 = 1; b0 < nb; b0 += 128) {
    const long long b = b0 + threadIdx.x;
    __syncthreads();
    if (b < nb) {
      const double na = (double)(b * FIT_ROWS), c = (double)min((long long)FIT_ROWS, count - b * FIT_ROWS);
      sw[threadIdx.x] = c / (na + c);
      sv[threadIdx.x] = na * c / (na + c);
    }
    __syncthreads();
    if (f >= nf) continue;
    const int n = (int)min(128LL, nb - b0);
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
      const double mb = pm[(size_t)(b0 + i) * nf + f], d = mb - mu;
      mu = isfinite(d) ? fma(d, sw[i], mu) : mu + mb;    // an infinite mean stays one
      q = fma(d * d, sv[i], q + p2[(size_t)(b0 + i) * nf + f]);
    }
  }
  if (f >= nf) return;
  double sd = sqrt(q / (double)count);
  if (sd < 1e-8) sd = 1.0;
  const int z = blockIdx.z;
  o.mean[z][f] = (float)mu;
  o.scale[z][f] = (float)(1.0 / sd);
  if (o.stdv[z]) o.stdv[z][f] = (float)sd;
}

__global__ void k_gather_rows(const bf16* src, int ld, long long a, long long s, long long count,
                              long long row0, int rows, int d, bf16* dst, int ldd) {
  early_start();
  const int vec = d / 8;   // d is a multiple of 8
  const long long total = (long long)rows * vec;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / vec), k = (int)(i % vec) * 8;
    const long long smp = visit(a, s, count, row0 + r);
    *(uint4*)(dst + (size_t)r * ldd + k) = *(const uint4*)(src + (size_t)smp * ld + k);
  }
}

// Gradient tiles (32 rows x 64 features per block of 256 threads: a warp per
// row, two features per lane).
// MODE 0 (output layer): g = (o - t) * scale with t the target row of sample
// visit(row0 + r); also the squared-error partial of the block.
// MODE 1 (hidden layer): g = in.
// Writes g as bf16 row-major [rows x ldg] and transposed [F x ldgt], and the
// float32 column sums of the tile (rows in order) to colpart[blockIdx.y][f].
// Every leading dimension is even.
constexpr int GT_F = 64;
template <int MODE>
__global__ void __launch_bounds__(256) k_grad_tiles(const float* in, int ldi, const float* T,
                                                    int ldt, long long a, long long sft, long long count,
                                                    long long row0, int rows, int F, float scale, bf16* gb,
                                                    int ldg, bf16* gt, int ldgt,
                                                    float* colpart, int ldc, double* lossp) {
  early_start();
  __shared__ float tile[32][GT_F + 1];
  __shared__ double red[8];
  __shared__ long long smp_of[32];
  const int f0 = blockIdx.x * GT_F, r0 = blockIdx.y * 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int f = f0 + 2 * lane;
  const bool on0 = f < F, on1 = f + 1 < F;
  // the squared error in float32 pairs (product and sum with their exact
  // rounding errors, about 2^-48 relative): in float64 each term would take
  // two operations of that pipe, conversion included; terms whose square or
  // its error leaves float32's range go to ld
  float lh = 0.f, ll = 0.f;
  double ld = 0.0;
  if (MODE == 0) {   // the rows' samples, one 64-bit remainder each
    if (w == 0 && r0 + lane < rows) smp_of[lane] = visit(a, sft, count, row0 + r0 + lane);
    __syncthreads();
  }
  float2 o[4], t[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int i = w + 8 * k, r = r0 + i;
    o[k] = t[k] = make_float2(0.f, 0.f);
    if (r < rows && on0) {
      const float* po = in + (size_t)r * ldi + f;
      const float* pt = MODE == 0 ? T + (size_t)smp_of[i] * ldt + f : nullptr;
      if (on1) {
        o[k] = *reinterpret_cast<const float2*>(po);
        if (MODE == 0) t[k] = *reinterpret_cast<const float2*>(pt);
      } else {
        o[k].x = *po;
        if (MODE == 0) t[k].x = *pt;
      }
    }
  }
  auto square = [&](float d) {
    if (fabsf(d) > 1e-10f && fabsf(d) < 1e15f) {
      const float ph = __fmul_rn(d, d);
      pair_add(lh, ll, ph, __fmaf_rn(d, d, -ph));
    } else if (d != 0.f) {
      ld += (double)d * (double)d;
    }
  };
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int i = w + 8 * k, r = r0 + i;
    float2 g = o[k];
    if (MODE == 0) {
      const float2 d = make_float2(__fsub_rn(o[k].x, t[k].x), __fsub_rn(o[k].y, t[k].y));   // 0 outside the tile
      square(d.x);
      square(d.y);
      g = make_float2(__fmul_rn(d.x, scale), __fmul_rn(d.y, scale));
    }
    if (r < rows && on0) {
      bf16* p = gb + (size_t)r * ldg + f;
      if (on1) *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(g.x, g.y);
      else *p = __float2bfloat16_rn(g.x);
    }
    tile[i][2 * lane] = g.x;
    tile[i][2 * lane + 1] = g.y;
  }
  __syncthreads();
  if (threadIdx.x < GT_F && f0 + threadIdx.x < F) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 32; ++i) s += tile[i][threadIdx.x];
    colpart[(size_t)blockIdx.y * ldc + f0 + threadIdx.x] = s;
  }
  const int rp = 2 * (lane & 15), rr = r0 + rp;    // ldgt is even: pairs of rows in 4 bytes
#pragma unroll
  for (int k = 0; k < GT_F / 16; ++k) {
    const int fl = 2 * (w + 8 * k) + (lane >> 4);
    if (f0 + fl >= F || rr >= rows) continue;
    bf16* p = gt + (size_t)(f0 + fl) * ldgt + rr;
    if (rr + 1 < rows) *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(tile[rp][fl], tile[rp + 1][fl]);
    else *p = __float2bfloat16_rn(tile[rp][fl]);
  }
  if (MODE == 0) {
    for (int s = 16; s > 0; s >>= 1) {
      const float xh = __shfl_down_sync(0xffffffffu, lh, s), xl = __shfl_down_sync(0xffffffffu, ll, s);
      pair_add(lh, ll, xh, xl);
    }
    if (__any_sync(0xffffffffu, ld != 0.0))       // warp-uniform (a NaN too)
      for (int s = 16; s > 0; s >>= 1) ld += __shfl_down_sync(0xffffffffu, ld, s);
    if (lane == 0) red[w] = (double)lh + (double)ll + ld;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int i = 0; i < 8; ++i) s += red[i];
      lossp[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
  }
}

__global__ void k_colsum(const float* part, int ntiles, int F, int ld, float* out) {
  early_start();
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  float s = 0.f;
  for (int t = 0; t < ntiles; ++t) s += part[(size_t)t * ld + f];
  out[f] = s;
}

// acc += inv * sum(parts) (one block of 1024 threads, fixed order)
__global__ void __launch_bounds__(1024) k_loss_acc(const double* parts, int n, double inv,
                                                   double* acc) {
  early_start();
  __shared__ double red[32];
  double s = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += 1024) s += parts[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = red[threadIdx.x];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *acc += inv * s;
  }
}

__global__ void k_transpose_bf16(const bf16* in, int ldi, int rows, int cols, bf16* out,
                                 int ldo) {
  early_start();
  __shared__ bf16 t[32][34];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < rows && c < cols) t[i][threadIdx.x] = in[(size_t)r * ldi + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < rows && c < cols) out[(size_t)c * ldo + r] = t[threadIdx.x][i];
  }
}

struct AdamArgs {
  float lr, b1, b2, eps, c1, c2;   // c1 = 1/(1-b1^t), c2 = 1/(1-b2^t)
  int update;                      // 0: only refresh the bf16 copies
};

__device__ __forceinline__ float adam_one(float w, float g, float& m, float& v, const AdamArgs& a) {
  m = a.b1 * m + (1.f - a.b1) * g;
  v = a.b2 * v + (1.f - a.b2) * g * g;
  return w - a.lr * (m * a.c1) / (sqrtf(v * a.c2) + a.eps);
}

// Adam on a rows x cols weight (all float32 arrays row-major, ld = cols, a
// multiple of 4), then the bf16 copy [rows x ldb] and the transposed bf16 copy
// [cols x ldt].  Bound by memory (28 bytes read and written per weight and 4
// for the copies): 64 x 64 tiles, four columns per thread in 16-byte accesses,
// the transposed copy in 128-byte runs.
constexpr int ADAM_T = 64;
__global__ void __launch_bounds__(256) k_adam_mat(float* W, float* mW,
                                                  float* vW, const float* g, int rows,
                                                  int cols, AdamArgs a, bf16* Wb, int ldb,
                                                  bf16* Wt, int ldt) {
  early_start();
  __shared__ bf16 t[ADAM_T][ADAM_T + 2];          // [column][row]
  const int c0 = blockIdx.x * ADAM_T, r0 = blockIdx.y * ADAM_T;
  const int cl = (threadIdx.x & 15) * 4, c = c0 + cl;
#pragma unroll
  for (int k = 0; k < ADAM_T / 16; ++k) {
    const int rl = (threadIdx.x >> 4) + 16 * k, r = r0 + rl;
    if (r < rows && c < cols) {
      const size_t o = (size_t)r * cols + c;
      float4 w = *reinterpret_cast<const float4*>(W + o);
      if (a.update) {
        float4 m = *reinterpret_cast<const float4*>(mW + o), v = *reinterpret_cast<const float4*>(vW + o);
        const float4 gg = *reinterpret_cast<const float4*>(g + o);
        w.x = adam_one(w.x, gg.x, m.x, v.x, a);
        w.y = adam_one(w.y, gg.y, m.y, v.y, a);
        w.z = adam_one(w.z, gg.z, m.z, v.z, a);
        w.w = adam_one(w.w, gg.w, m.w, v.w, a);
        *reinterpret_cast<float4*>(W + o) = w;
        *reinterpret_cast<float4*>(mW + o) = m;
        *reinterpret_cast<float4*>(vW + o) = v;
      }
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(w.x, w.y), h1 = __floats2bfloat162_rn(w.z, w.w);
      uint2 q;
      q.x = *reinterpret_cast<const uint32_t*>(&h0);
      q.y = *reinterpret_cast<const uint32_t*>(&h1);
      *reinterpret_cast<uint2*>(Wb + (size_t)r * ldb + c) = q;
      t[cl][rl] = h0.x;
      t[cl + 1][rl] = h0.y;
      t[cl + 2][rl] = h1.x;
      t[cl + 3][rl] = h1.y;
    }
  }
  __syncthreads();
  const int rp = (threadIdx.x & 31) * 2;          // ldt is even and r0 + rp too: 4-byte stores
#pragma unroll
  for (int k = 0; k < ADAM_T / 8; ++k) {
    const int cc = (threadIdx.x >> 5) + 8 * k;
    if (c0 + cc >= cols || r0 + rp >= rows) continue;
    bf16* d = Wt + (size_t)(c0 + cc) * ldt + r0 + rp;
    if (r0 + rp + 1 < rows) *reinterpret_cast<uint32_t*>(d) = *reinterpret_cast<const uint32_t*>(&t[cc][rp]);
    else *d = t[cc][rp];
  }
}

__global__ void k_adam_vec(float* b, float* mb, float* vb,
                           const float* g, int n, AdamArgs a) {
  early_start();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || !a.update) return;
  float m = mb[i], v = vb[i];
  b[i] = adam_one(b[i], g[i], m, v, a);
  mb[i] = m;
  vb[i] = v;
}

__global__ void k_f32_to_bf16_2d(const float* __restrict__ in, int rows, int cols, bf16* __restrict__ out, int ldo) {
  const long long total = (long long)rows * cols;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / cols), c = (int)(i % cols);
    out[(size_t)r * ldo + c] = __float2bfloat16_rn(in[i]);
  }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  });
  return fn;
}

// Tensor map of a row-major rows x cols bf16 matrix with leading dimension ld
// (elements): boxes of box_rows rows x 64 columns, 128-byte swizzle, zero fill
// outside the matrix.
static bool make_map(CUtensorMap* map, const void* base, int rows, int cols, int ld, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  if (((uintptr_t)base & 15) || (((size_t)ld * 2) & 15) || cols > ld) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {BK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static int num_sms() {   // of the current device, read once (a thread-safe static)
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
  }();
  return n;
}

// the B tile width: 256 when N fills it, else 128
inline int tile_n(int N) { return N >= 256 ? 256 : 128; }

// How a product runs: on CTA pairs (256 x bn tiles) or single CTAs (128 x bn),
// and in how many splits of K.
struct GemmPlan {
  int pair, bn, splits;
};

// Splits: with fewer 128 x 256 (128) tiles than SMs, enough to cover the SMs,
// at least 4 k-tiles each.  Pairs where M and N fill their tiles (a pair on
// M <= 128 would idle one CTA).  A product on pairs takes the tile width whose
// waves cost least: per k-tile a tile lasts as long as it is wide (plus about 32
// columns' worth of the A side), its epilogue about six k-tiles (against ten: 256 x
// 1024 x 30000 28.9 -> 23.9 us); the epilogue
// of all but the last tile hides behind the next tile's main loop or the other
// way round.  So 256 for long products with many tiles, less where that
// leaves the last wave nearly empty or the epilogue of a single wave shows.
GemmPlan plan_gemm(int M, int N, int K, int requested) {
  GemmPlan p;
  p.bn = tile_n(N);
  const int KT = (K + BK - 1) / BK;
  int splits = requested;
  if (splits <= 0) {
    const long long t = (long long)((M + BM - 1) / BM) * ((N + p.bn - 1) / p.bn);
    splits = 1;
    if (t < num_sms()) splits = (int)std::min<long long>(KT / 4, (num_sms() + t - 1) / t);
  }
  splits = std::max(1, std::min(splits, KT));
  const int ktps = (KT + splits - 1) / splits;
  p.splits = (KT + ktps - 1) / ktps;
  p.pair = M > 128 && N >= 256;
  if (p.pair) {
    const long long tm = (M + 2 * BM - 1) / (2 * BM), pairs = std::max(1, num_sms() / 2);
    const long long kt = (KT + p.splits - 1) / p.splits;
    long long best = 0;
    for (int bn = 256; bn >= 128; bn -= 16) {
      const long long waves = (tm * ((N + bn - 1) / bn) * p.splits + pairs - 1) / pairs;
      const long long main = kt * (bn + 32), epi = 6LL * bn;
      const long long cost = waves * std::max(main, epi) + std::min(main, epi);
      if (best == 0 || cost < best) {
        best = cost;
        p.bn = bn;
      }
    }
  }
  return p;
}
int plan_splits(int M, int N, int K, int requested) { return plan_gemm(M, N, K, requested).splits; }

size_t splitk_floats(int M, int N, int K, int splits) {
  const int s = plan_splits(M, N, K, splits);
  return s > 1 ? (size_t)s * M * N : 0;
}

// D = A B^T (+ epilogue).  A: M x K (lda), B: N x K (ldb), bf16 row-major.
// `work` holds at least splitk_floats(M, N, K, splits) floats, else no split.
cudaError_t gemm_tn(const bf16* A, int lda, const bf16* B, int ldb, int M, int N, int K, const Epi& epi, int splits,
                    float* work, size_t work_floats, int* err, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaErrorInvalidValue;
  const GemmPlan plan = plan_gemm(M, N, K, splits);
  const int BN = plan.bn;
  CUtensorMap ma, mb;
  if (!make_map(&ma, A, M, K, lda, BM) || !make_map(&mb, B, N, K, ldb, plan.pair ? BN / 2 : BN))
    return cudaErrorInvalidValue;
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(k_gemm_tn_p<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile<128>::SMEM_BYTES);
    cudaFuncSetAttribute(k_gemm_tn_p<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile<256>::SMEM_BYTES);
    cudaFuncSetAttribute(k_gemm_tn_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, P_SMEM_BYTES);
  });
  Epi ep = epi;
  ep.vec = ((uintptr_t)epi.out_f & 15) == 0 && ((uintptr_t)epi.out_b & 7) == 0 && ((uintptr_t)epi.mask & 7) == 0 &&
           ((uintptr_t)work & 15) == 0;
  const int KT = (K + BK - 1) / BK;
  int sp = plan.splits;
  if (sp > 1 && (!work || work_floats < (size_t)sp * M * N)) sp = 1;
  const int ktps = (KT + sp - 1) / sp;
  const int bm = plan.pair ? 2 * BM : BM;
  const long long units = (long long)((N + BN - 1) / BN) * ((M + bm - 1) / bm) * sp;
  if (plan.pair)
    early(k_gemm_tn_pair, 2 * (int)std::min<long long>(units, num_sms() / 2), GEMM_NT, P_SMEM_BYTES, s, ma, mb, M, N,
          K, BN, ktps, sp, ep, work, err);
  else if (BN == 256)
    early(k_gemm_tn_p<256>, (int)std::min<long long>(units, num_sms()), GEMM_NT, Tile<256>::SMEM_BYTES, s, ma, mb, M,
          N, K, ktps, sp, ep, work, err);
  else
    early(k_gemm_tn_p<128>, (int)std::min<long long>(units, num_sms()), GEMM_NT, Tile<128>::SMEM_BYTES, s, ma, mb, M,
          N, K, ktps, sp, ep, work, err);
  if (sp > 1) {
    const int rows = std::min(M, 32768);
    if ((N & 3) == 0 && ((uintptr_t)work & 15) == 0)
      early(k_splitk_epi<4>, dim3((N / 4 + 127) / 128, rows), 128, 0, s, work, sp, M, N, epi);
    else
      early(k_splitk_epi<1>, dim3((N + 127) / 128, rows), 128, 0, s, work, sp, M, N, epi);
  }
  return cudaGetLastError();
}

inline int grid_for(long long total, int threads = 256) {
  return (int)std::max<long long>(1, std::min<long long>((total + threads - 1) / threads, 16LL * num_sms()));
}
// two columns per thread: pairs do not straddle [n | m] and every row of both
// arrays starts on 16 bytes
inline bool two_columns(int n, int m, const void* p, const void* q) {
  return n % 2 == 0 && m % 2 == 0 && ((uintptr_t)p & 15) == 0 && ((uintptr_t)q & 15) == 0;
}
inline int r8(long long v) { return (int)((v + 7) / 8 * 8); }

}  // namespace mlp

// ==========================================================================
// the network handle
// ==========================================================================
using namespace mlp;

struct WsLayer {
  int out = 0, in = 0;
  float *W = nullptr, *b = nullptr, *mW = nullptr, *vW = nullptr, *mb = nullptr, *vb = nullptr, *gW = nullptr,
        *gb = nullptr;
  bf16 *Wb = nullptr, *Wt = nullptr;   // [out x in] and [in x ldt]
  int ldt = 0;
};

struct pdqp_ws_s {
  int n = 0, m = 0, F = 0, Fp = 0, d = 0, width = 0, depth = 0, maxb = 0;
  int ldc = 0;                         // leading dimension of colpart: max(Fp, width)
  std::vector<WsLayer> L;              // depth hidden layers, then the output layer
  bf16* P = nullptr;                   // [d x Fp], fixed projection
  float *in_mean = nullptr, *in_scale = nullptr, *out_mean = nullptr, *out_std = nullptr, *out_inv = nullptr;
  bool have_norm = false, have_proj = false;
  long long step = 0;                  // Adam steps taken
  std::vector<bf16*> H, Ht;            // activations [maxb x ld] and transposes [ld x maxb]
  bf16* U = nullptr;                   // normalised inputs [maxb x Fp]
  float* O = nullptr;                  // outputs [maxb x Fp]
  float* G = nullptr;                  // hidden gradients [maxb x width]
  bf16 *dOb = nullptr, *dOt = nullptr, *dZb = nullptr, *dZt = nullptr;
  float* colpart = nullptr;            // [(maxb/32 + 1) x ldc]
  double* lossp = nullptr;             // [(maxb/32 + 1) x (Fp/32 + 1)]
  double* lossacc = nullptr;
  float* work = nullptr;               // split-K partials
  size_t work_floats = 0;
  int* err = nullptr;
  // training set
  long long tcount = 0;
  bf16* H0all = nullptr;               // [count x d]
  float* Tall = nullptr;               // [count x Fp]
  std::vector<void*> allocs;
  std::string last_error;
};

namespace {

struct WsFail {
  pdqp_status st;
  std::string msg;
};

thread_local std::string g_ws_error;

#define WCK(x)                                                                                          \
  do {                                                                                                  \
    cudaError_t e_ = (x);                                                                               \
    if (e_ != cudaSuccess)                                                                              \
      throw WsFail{e_ == cudaErrorMemoryAllocation ? PDQP_ERR_OOM : PDQP_ERR_CUDA,                      \
                   std::string(#x) + ": " + cudaGetErrorString(e_)};                                    \
  } while (0)

template <class T>
T* walloc(pdqp_ws_s* w, size_t count) {
  void* p = nullptr;
  WCK(cudaMalloc(&p, std::max<size_t>(count, 1) * sizeof(T)));
  w->allocs.push_back(p);
  return (T*)p;
}

void wfree(pdqp_ws_s* w, void* p) {
  if (!p) return;
  cudaFree(p);
  auto it = std::find(w->allocs.begin(), w->allocs.end(), p);
  if (it != w->allocs.end()) w->allocs.erase(it);
}

bool is_device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

void check_space(const void* p, int mem, const char* what) {
  if (mem != PDQP_MEM_HOST && mem != PDQP_MEM_DEVICE) throw WsFail{PDQP_ERR_INVALID, "mem_space"};
  if (!p) return;
  if ((mem == PDQP_MEM_DEVICE) != is_device_ptr(p))
    throw WsFail{PDQP_ERR_INVALID, std::string(what) + " does not live in the given mem_space"};
}

// A device view of `count` elements: the pointer itself, or a temporary copy.
template <class T>
struct DevView {
  T* p = nullptr;
  bool owned = false;
  DevView(const T* src, size_t count, int mem, cudaStream_t s) {
    if (!src || mem == PDQP_MEM_DEVICE || count == 0) {
      p = const_cast<T*>(src);
      return;
    }
    WCK(cudaMalloc(&p, count * sizeof(T)));
    owned = true;
    const cudaError_t e = cudaMemcpyAsync(p, src, count * sizeof(T), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) {
      cudaFree(p);
      p = nullptr;
      owned = false;
      WCK(e);
    }
  }
  ~DevView() {
    if (owned) cudaFree(p);   // cudaFree waits for the work queued on the copy
  }
  DevView(const DevView&) = delete;
  DevView& operator=(const DevView&) = delete;
};

void gemm(pdqp_ws_s* w, const bf16* A, int lda, const bf16* B, int ldb, int M, int N, int K, const Epi& e,
          cudaStream_t s) {
  const size_t need = splitk_floats(M, N, K, 0);
  if (need > w->work_floats) {
    WCK(cudaStreamSynchronize(s));
    wfree(w, w->work);
    w->work = nullptr;
    w->work_floats = 0;
    w->work = walloc<float>(w, need);
    w->work_floats = need;
  }
  WCK(gemm_tn(A, lda, B, ldb, M, N, K, e, 0, w->work, w->work_floats, w->err, s));
}

Epi epi_of(float* of, bf16* ob, int ldo, const float* bias, int relu, const bf16* mask = nullptr, int ldm = 0) {
  Epi e;
  e.out_f = of;
  e.out_b = ob;
  e.ldo = ldo;
  e.bias = bias;
  e.relu = relu;
  e.mask = mask;
  e.ldm = ldm;
  return e;
}

// forward from H[0] (rows x d) to O; hidden activations in H[1..depth]
// (with x0 or y0: to the prediction of rows from those pointers on)
void forward(pdqp_ws_s* w, int rows, cudaStream_t s, double* x0 = nullptr, double* y0 = nullptr) {
  for (int j = 0; j < w->depth; ++j) {
    const WsLayer& l = w->L[j];
    gemm(w, w->H[j], l.in, l.Wb, l.in, rows, l.out, l.in, epi_of(nullptr, w->H[j + 1], l.out, l.b, 1), s);
  }
  const WsLayer& o = w->L[w->depth];
  Epi e = epi_of(w->O, nullptr, w->Fp, o.b, 0);
  if (x0 || y0) {
    e.out_f = nullptr;
    e.pmean = w->out_mean; e.pstd = w->out_std;
    e.px = x0; e.py = y0; e.pn = w->n; e.pm = w->m;
    e.pvec = two_columns(w->n, w->m, x0, y0);
  }
  gemm(w, w->H[w->depth], o.in, o.Wb, o.in, rows, w->F, o.in, e, s);
}

// Backward of the mean squared error against targets T (the target of row r
// is row visit(a, sft, count, row0 + r) of T); leaves the gradients in gW/gb
// and adds loss / (rows F) to *lossacc.
void backward(pdqp_ws_s* w, int rows, const float* T, long long a, long long sft, long long count, long long row0,
              cudaStream_t s) {
  const int F = w->F, Fp = w->Fp, mb = w->maxb;
  const int rt = (rows + 31) / 32;
  {
    dim3 grid((F + GT_F - 1) / GT_F, rt);
    const float scale = (float)(2.0 / ((double)rows * F));
    early(k_grad_tiles<0>, grid, 256, 0, s, w->O, Fp, T, Fp, a, sft, count, row0, rows, F, scale, w->dOb, Fp, w->dOt,
          mb, w->colpart, w->ldc, w->lossp);
    early(k_loss_acc, 1, 1024, 0, s, w->lossp, (int)(grid.x * grid.y), 1.0 / ((double)rows * F), w->lossacc);
  }
  WsLayer& o = w->L[w->depth];
  early(k_colsum, (F + 255) / 256, 256, 0, s, w->colpart, rt, F, w->ldc, o.gb);
  {
    const int c = o.in;
    dim3 grid((c + 31) / 32, rt), blk(32, 8);
    early(k_transpose_bf16, grid, blk, 0, s, w->H[w->depth], c, rows, c, w->Ht[w->depth], mb);
  }
  // gW_out = dO' H_depth  (F x width), K = rows
  gemm(w, w->dOt, mb, w->Ht[w->depth], mb, F, o.in, rows, epi_of(o.gW, nullptr, o.in, nullptr, 0), s);
  // dZ of the last hidden layer = (dO W_out) * (H_depth > 0)
  gemm(w, w->dOb, Fp, o.Wt, o.ldt, rows, o.in, F, epi_of(w->G, nullptr, o.in, nullptr, 0, w->H[w->depth], o.in), s);
  for (int j = w->depth - 1; j >= 0; --j) {
    WsLayer& l = w->L[j];
    {
      dim3 grid((l.out + GT_F - 1) / GT_F, rt);
      early(k_grad_tiles<1>, grid, 256, 0, s, w->G, l.out, nullptr, 0, 1, 0, 1LL << 62, 0, rows, l.out, 1.f, w->dZb,
            l.out, w->dZt, mb, w->colpart, w->ldc, nullptr);
    }
    early(k_colsum, (l.out + 255) / 256, 256, 0, s, w->colpart, rt, l.out, w->ldc, l.gb);
    {
      dim3 grid((l.in + 31) / 32, rt), blk(32, 8);
      early(k_transpose_bf16, grid, blk, 0, s, w->H[j], l.in, rows, l.in, w->Ht[j], mb);
    }
    gemm(w, w->dZt, mb, w->Ht[j], mb, l.out, l.in, rows, epi_of(l.gW, nullptr, l.in, nullptr, 0), s);
    if (j > 0)
      gemm(w, w->dZb, l.out, l.Wt, l.ldt, rows, l.in, l.out, epi_of(w->G, nullptr, l.in, nullptr, 0, w->H[j], l.in),
           s);
  }
}

void adam(pdqp_ws_s* w, float lr, float b1, float b2, float eps, cudaStream_t s) {
  w->step += 1;
  AdamArgs a;
  a.lr = lr;
  a.b1 = b1;
  a.b2 = b2;
  a.eps = eps;
  a.c1 = (float)(1.0 / (1.0 - std::pow((double)b1, (double)w->step)));
  a.c2 = (float)(1.0 / (1.0 - std::pow((double)b2, (double)w->step)));
  a.update = 1;
  for (WsLayer& l : w->L) {
    dim3 grid((l.in + ADAM_T - 1) / ADAM_T, (l.out + ADAM_T - 1) / ADAM_T);
    early(k_adam_mat, grid, 256, 0, s, l.W, l.mW, l.vW, l.gW, l.out, l.in, a, l.Wb, l.in, l.Wt, l.ldt);
    early(k_adam_vec, (l.out + 255) / 256, 256, 0, s, l.b, l.mb, l.vb, l.gb, l.out, a);
  }
}

void refresh_copies(WsLayer& l, cudaStream_t s) {
  AdamArgs a{};
  a.update = 0;
  dim3 grid((l.in + ADAM_T - 1) / ADAM_T, (l.out + ADAM_T - 1) / ADAM_T);
  early(k_adam_mat, grid, 256, 0, s, l.W, l.mW, l.vW, l.gW, l.out, l.in, a, l.Wb, l.in, l.Wt, l.ldt);
}

// the elementwise kernels' grid over `rows` rows of arrays p, q
dim3 row_grid(const pdqp_ws_s* w, const void* p, const void* q, long long rows) {
  const int per = two_columns(w->n, w->m, p, q) ? 512 : 256;
  return dim3((w->F + per - 1) / per, (unsigned)std::min<long long>((rows + ROWS_PER - 1) / ROWS_PER, 32768));
}

// normalised inputs of rows [row0, row0+rows) -> U -> H0 = U P'
void project(pdqp_ws_s* w, const double* C, const double* B, long long row0, int rows, bf16* H0, cudaStream_t s) {
  auto prep = two_columns(w->n, w->m, C, B) ? k_prep_input<2> : k_prep_input<1>;
  early(prep, row_grid(w, C, B, rows), 256, 0, s, C, B, w->n, w->m, row0, rows, w->in_mean, w->in_scale, w->U, w->Fp);
  gemm(w, w->U, w->Fp, w->P, w->Fp, rows, w->d, w->F, epi_of(nullptr, H0, w->d, nullptr, 0), s);
}

void finish(pdqp_ws_s* w, cudaStream_t s) {
  int herr = 0;
  WCK(cudaGetLastError());
  WCK(cudaMemcpyAsync(&herr, w->err, sizeof(int), cudaMemcpyDeviceToHost, s));
  WCK(cudaStreamSynchronize(s));
  if (herr) {
    cudaMemsetAsync(w->err, 0, sizeof(int), s);
    cudaStreamSynchronize(s);
    throw WsFail{PDQP_DEVICE_TIMEOUT, "a tensor-core GEMM wait gave up (device timeout)"};
  }
}

template <class Fn>
pdqp_status guard(pdqp_ws_s* w, Fn fn) {
  try {
    fn();
    return PDQP_OK;
  } catch (const WsFail& f) {
    (w ? w->last_error : g_ws_error) = f.msg;
    return f.st;
  } catch (const std::bad_alloc&) {
    (w ? w->last_error : g_ws_error) = "host allocation failed";
    return PDQP_ERR_OOM;
  }
}

void need_ready(const pdqp_ws_s* w) {
  if (!w->have_norm) throw WsFail{PDQP_ERR_INVALID, "normalisation not set: call pdqp_ws_fit or pdqp_ws_set_normalization"};
  if (!w->have_proj) throw WsFail{PDQP_ERR_INVALID, "projection not set: call pdqp_ws_set_params with layer -1"};
}

void need_data(const pdqp_ws_s* w, const void* C, const void* B, const void* X, const void* Y, int mem, bool targets) {
  if (!C || (w->m > 0 && !B) || (targets && (!X || (w->m > 0 && !Y))))
    throw WsFail{PDQP_ERR_INVALID, "null C, B, X or Y"};
  for (const void* p : {C, B, X, Y}) check_space(p, mem, "data array");
}

// visit order of an epoch: i -> (a i + sft) mod count, (a, sft) from SplitMix64
// (Steele, Lea & Flood 2014) of the seed and the epoch
void visit_order(uint64_t seed, int epoch, long long count, long long* a_out, long long* s_out) {
  auto mix = [](uint64_t z) {
    z += 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
  };
  auto gcd = [](long long p, long long q) {
    while (q) {
      const long long t = p % q;
      p = q;
      q = t;
    }
    return p;
  };
  const uint64_t z = mix(seed * 0x9E3779B97F4A7C15ULL + (uint64_t)epoch * 0xD1B54A32D192ED03ULL);
  long long a = (long long)(z % (uint64_t)count) | 1;
  while (gcd(a, count) != 1) a += 2;
  a %= count;
  if (a == 0) a = 1;
  *a_out = a;
  *s_out = (long long)((z >> 32) % (uint64_t)count);
}

}  // namespace

// ==========================================================================
// C ABI
// ==========================================================================
extern "C" {

pdqp_status pdqp_ws_create(pdqp_ws_handle* out, int64_t n, int64_t m, int32_t d, int32_t width, int32_t depth,
                           int32_t max_batch, void* stream) {
  if (!out) return PDQP_ERR_INVALID;
  *out = nullptr;
  return guard(nullptr, [&] {
    if (n < 1 || m < 0 || n + m > (1LL << 26)) throw WsFail{PDQP_ERR_INVALID, "sizes: need n >= 1, m >= 0, n + m <= 2^26"};
    if (d < 8 || width < 8 || d % 8 || width % 8 || d > 16384 || width > 16384)
      throw WsFail{PDQP_ERR_INVALID, "d and width: multiples of 8 in [8, 16384]"};
    if (depth < 1 || depth > 16) throw WsFail{PDQP_ERR_INVALID, "depth in [1, 16]"};
    if (max_batch < 8 || max_batch % 8 || max_batch > 8192)
      throw WsFail{PDQP_ERR_INVALID, "max_batch: multiple of 8 in [8, 8192]"};
    cudaStream_t s = (cudaStream_t)stream;
    pdqp_ws_s* w = new pdqp_ws_s();
    try {
      w->n = (int)n;
      w->m = (int)m;
      w->F = (int)(n + m);
      w->Fp = r8(w->F);
      w->d = d;
      w->width = width;
      w->depth = depth;
      w->maxb = max_batch;
      const int Fp = w->Fp, mb = max_batch;
      w->L.resize(depth + 1);
      for (int j = 0; j <= depth; ++j) {
        WsLayer& l = w->L[j];
        l.in = j == 0 ? d : width;
        l.out = j == depth ? w->F : width;
        l.ldt = r8(l.out);
        const size_t ne = (size_t)l.out * l.in;
        l.W = walloc<float>(w, ne);
        l.mW = walloc<float>(w, ne);
        l.vW = walloc<float>(w, ne);
        l.gW = walloc<float>(w, ne);
        l.b = walloc<float>(w, l.out);
        l.mb = walloc<float>(w, l.out);
        l.vb = walloc<float>(w, l.out);
        l.gb = walloc<float>(w, l.out);
        l.Wb = walloc<bf16>(w, ne);
        l.Wt = walloc<bf16>(w, (size_t)l.in * l.ldt);
        for (void* p : {(void*)l.W, (void*)l.mW, (void*)l.vW, (void*)l.gW})
          WCK(cudaMemsetAsync(p, 0, ne * sizeof(float), s));
        for (void* p : {(void*)l.b, (void*)l.mb, (void*)l.vb, (void*)l.gb})
          WCK(cudaMemsetAsync(p, 0, l.out * sizeof(float), s));
        WCK(cudaMemsetAsync(l.Wb, 0, ne * sizeof(bf16), s));
        WCK(cudaMemsetAsync(l.Wt, 0, (size_t)l.in * l.ldt * sizeof(bf16), s));
      }
      w->P = walloc<bf16>(w, (size_t)d * Fp);
      WCK(cudaMemsetAsync(w->P, 0, (size_t)d * Fp * sizeof(bf16), s));
      for (float** p : {&w->in_mean, &w->in_scale, &w->out_mean, &w->out_std, &w->out_inv}) {
        *p = walloc<float>(w, Fp);
        WCK(cudaMemsetAsync(*p, 0, (size_t)Fp * sizeof(float), s));
      }
      w->H.resize(depth + 1);
      w->Ht.resize(depth + 1);
      for (int j = 0; j <= depth; ++j) {
        const int c = j == 0 ? d : width;
        w->H[j] = walloc<bf16>(w, (size_t)mb * c);
        w->Ht[j] = walloc<bf16>(w, (size_t)c * mb);
      }
      w->U = walloc<bf16>(w, (size_t)mb * Fp);
      WCK(cudaMemsetAsync(w->U, 0, (size_t)mb * Fp * sizeof(bf16), s));
      w->O = walloc<float>(w, (size_t)mb * Fp);
      w->G = walloc<float>(w, (size_t)mb * width);
      w->dOb = walloc<bf16>(w, (size_t)mb * Fp);
      w->dOt = walloc<bf16>(w, (size_t)Fp * mb);
      w->dZb = walloc<bf16>(w, (size_t)mb * width);
      w->dZt = walloc<bf16>(w, (size_t)width * mb);
      w->ldc = std::max(Fp, width);
      w->colpart = walloc<float>(w, (size_t)(mb / 32 + 1) * w->ldc);
      w->lossp = walloc<double>(w, (size_t)(mb / 32 + 1) * (Fp / 32 + 1));
      w->lossacc = walloc<double>(w, 1);
      w->err = walloc<int>(w, 1);
      WCK(cudaMemsetAsync(w->err, 0, sizeof(int), s));
      WCK(cudaMemsetAsync(w->lossacc, 0, sizeof(double), s));
      WCK(cudaStreamSynchronize(s));
    } catch (...) {
      pdqp_ws_destroy(w);
      throw;
    }
    *out = w;
  });
}

void pdqp_ws_destroy(pdqp_ws_handle w) {
  if (!w) return;
  cudaDeviceSynchronize();
  for (void* p : w->allocs) cudaFree(p);
  delete w;
}

const char* pdqp_ws_last_error(pdqp_ws_handle w) { return w ? w->last_error.c_str() : g_ws_error.c_str(); }

pdqp_status pdqp_ws_set_params(pdqp_ws_handle w, int32_t layer, const float* W, const float* b, int32_t mem,
                               void* stream) {
  if (!w) return PDQP_ERR_INVALID;
  return guard(w, [&] {
    cudaStream_t s = (cudaStream_t)stream;
    if (layer < -1 || layer > w->depth) throw WsFail{PDQP_ERR_INVALID, "layer out of range"};
    if (!W) throw WsFail{PDQP_ERR_INVALID, "null W"};
    check_space(W, mem, "W");
    check_space(b, mem, "b");
    if (layer == -1) {
      DevView<float> v(W, (size_t)w->d * w->F, mem, s);
      k_f32_to_bf16_2d<<<grid_for((long long)w->d * w->F), 256, 0, s>>>(v.p, w->d, w->F, w->P, w->Fp);
      WCK(cudaGetLastError());
      WCK(cudaStreamSynchronize(s));
      w->have_proj = true;
      return;
    }
    const cudaMemcpyKind kind = mem == PDQP_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    WsLayer& l = w->L[layer];
    WCK(cudaMemcpyAsync(l.W, W, (size_t)l.out * l.in * sizeof(float), kind, s));
    if (b) WCK(cudaMemcpyAsync(l.b, b, (size_t)l.out * sizeof(float), kind, s));
    else WCK(cudaMemsetAsync(l.b, 0, (size_t)l.out * sizeof(float), s));
    refresh_copies(l, s);
    WCK(cudaGetLastError());
    WCK(cudaStreamSynchronize(s));
  });
}

pdqp_status pdqp_ws_get_params(pdqp_ws_handle w, int32_t layer, int32_t what, float* W, float* b, int32_t mem,
                               void* stream) {
  if (!w) return PDQP_ERR_INVALID;
  return guard(w, [&] {
    cudaStream_t s = (cudaStream_t)stream;
    if (layer < 0 || layer > w->depth) throw WsFail{PDQP_ERR_INVALID, "layer out of range"};
    if (what < 0 || what > 3)
      throw WsFail{PDQP_ERR_INVALID, "what: 0 parameters, 1 gradients, 2 first moments, 3 second moments"};
    check_space(W, mem, "W");
    check_space(b, mem, "b");
    const WsLayer& l = w->L[layer];
    const float* srcW[4] = {l.W, l.gW, l.mW, l.vW};
    const float* srcb[4] = {l.b, l.gb, l.mb, l.vb};
    const cudaMemcpyKind kind = mem == PDQP_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    if (W) WCK(cudaMemcpyAsync(W, srcW[what], (size_t)l.out * l.in * sizeof(float), kind, s));
    if (b) WCK(cudaMemcpyAsync(b, srcb[what], (size_t)l.out * sizeof(float), kind, s));
    WCK(cudaStreamSynchronize(s));
  });
}

pdqp_status pdqp_ws_set_normalization(pdqp_ws_handle w, const float* in_mean, const float* in_scale,
                                      const float* out_mean, const float* out_std, const float* out_inv, int32_t mem,
                                      void* stream) {
  if (!w) return PDQP_ERR_INVALID;
  return guard(w, [&] {
    cudaStream_t s = (cudaStream_t)stream;
    const float* src[5] = {in_mean, in_scale, out_mean, out_std, out_inv};
    float* dst[5] = {w->in_mean, w->in_scale, w->out_mean, w->out_std, w->out_inv};
    for (int i = 0; i < 5; ++i) {
      if (!src[i]) throw WsFail{PDQP_ERR_INVALID, "null normalisation vector"};
      check_space(src[i], mem, "normalisation vector");
    }
    const cudaMemcpyKind kind = mem == PDQP_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    for (int i = 0; i < 5; ++i) WCK(cudaMemcpyAsync(dst[i], src[i], (size_t)w->F * sizeof(float), kind, s));
    WCK(cudaStreamSynchronize(s));
    w->have_norm = true;
  });
}

pdqp_status pdqp_ws_get_normalization(pdqp_ws_handle w, float* in_mean, float* in_scale, float* out_mean,
                                      float* out_std, float* out_inv, int32_t mem, void* stream) {
  if (!w) return PDQP_ERR_INVALID;
  return guard(w, [&] {
    cudaStream_t s = (cudaStream_t)stream;
    float* dst[5] = {in_mean, in_scale, out_mean, out_std, out_inv};
    const float* src[5] = {w->in_mean, w->in_scale, w->out_mean, w->out_std, w->out_inv};
    const cudaMemcpyKind kind = mem == PDQP_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    for (int i = 0; i < 5; ++i) {
      check_space(dst[i], mem, "normalisation vector");
      if (dst[i]) WCK(cudaMemcpyAsync(dst[i], src[i], (size_t)w->F * sizeof(float), kind, s));
    }
    WCK(cudaStreamSynchronize(s));
  });
}

pdqp_status pdqp_ws_fit(pdqp_ws_handle w, const double* C, const double* B, const double* X, const double* Y,
                        int64_t count, int32_t mem, void* stream) {
  if (!w) return PDQP_ERR_INVALID;
  return guard(w, [&] {
    cudaStream_t s = (cudaStream_t)stream;
    if (count < 1) throw WsFail{PDQP_ERR_INVALID, "count >= 1"};
    need_data(w, C, B, X, Y, mem, true);
    const int n = w->n, m = w->m;
    // partials of two arrays at a time: mean and M2 per range of FIT_ROWS rows
    const long long nb = (count + FIT_ROWS - 1) / FIT_ROWS;
    const size_t need = 4 * (size_t)nb * (size_t)std::max(n, m) * (sizeof(double) / sizeof(float));
    if (need > w->work_floats) {
      WCK(cudaStreamSynchronize(s));
      wfree(w, w->work);
      w->work = nullptr;
      w->work_floats = 0;
      w->work = walloc<float>(w, need);
      w->work_floats = need;
    }
    // the statistics of the inputs `in` and of the targets `out`, nf columns each, from feature f0
    auto stats = [&](const double* in, const double* out, int nf, int f0) {
      double* part = reinterpret_cast<double*>(w->work);
      const size_t len = (size_t)nb * nf;
      const FitPair p{{in, out}, {part, part + 2 * len}, {part + len, part + 3 * len}};
      const FitOut o{{w->in_mean + f0, w->out_mean + f0}, {w->in_scale + f0, w->out_inv + f0}, {nullptr, w->out_std + f0}};
      k_fit_part<<<dim3((nf + 255) / 256, (unsigned)std::min<long long>(nb, 32768), 2), 256, 0, s>>>(p, count, nf);
      k_fit_merge<<<dim3((nf + 127) / 128, 1, 2), 128, 0, s>>>(p, count, nf, o);
      WCK(cudaGetLastError());
    };
    {
      DevView<double> c(C, (size_t)count * n, mem, s), x(X, (size_t)count * n, mem, s);
      stats(c.p, x.p, n, 0);
      if (mem != PDQP_MEM_DEVICE) WCK(cudaStreamSynchronize(s));
    }
    if (m > 0) {
      DevView<double> b(B, (size_t)count * m, mem, s), y(Y, (size_t)count * m, mem, s);
      stats(b.p, y.p, m, n);
      if (mem != PDQP_MEM_DEVICE) WCK(cudaStreamSynchronize(s));
    }
    WCK(cudaStreamSynchronize(s));
    w->have_norm = true;
  });
}

pdqp_status pdqp_ws_grad(pdqp_ws_handle w, const double* C, const double* B, const double* X, const double* Y,
                         int64_t count, double* loss, int32_t mem, void* stream) {
  if (!w) return PDQP_ERR_INVALID;
  return guard(w, [&] {
    cudaStream_t s = (cudaStream_t)stream;
    need_ready(w);
    if (count < 1 || count > w->maxb) throw WsFail{PDQP_ERR_INVALID, "count in [1, max_batch]"};
    need_data(w, C, B, X, Y, mem, true);
    const int n = w->n, m = w->m;
    DevView<double> c(C, (size_t)count * n, mem, s), b(B, (size_t)count * m, mem, s),
        x(X, (size_t)count * n, mem, s), y(Y, (size_t)count * m, mem, s);
    float* T = walloc<float>(w, (size_t)count * w->Fp);
    try {
      early((two_columns(n, m, x.p, y.p) ? k_prep_target<2> : k_prep_target<1>), row_grid(w, x.p, y.p, count), 256,
            0, s, x.p, y.p, n, m, count, w->out_mean, w->out_inv, T, w->Fp);
      project(w, c.p, b.p, 0, (int)count, w->H[0], s);
      forward(w, (int)count, s);
      WCK(cudaMemsetAsync(w->lossacc, 0, sizeof(double), s));
      backward(w, (int)count, T, 1, 0, 1LL << 62, 0, s);
      finish(w, s);
      double h = 0.0;
      WCK(cudaMemcpy(&h, w->lossacc, sizeof(double), cudaMemcpyDeviceToHost));
      if (loss) *loss = h;
    } catch (...) {
      cudaStreamSynchronize(s);
      wfree(w, T);
      throw;
    }
    wfree(w, T);
  });
}

pdqp_status pdqp_ws_train(pdqp_ws_handle w, const pdqp_ws_train_options* opt, const double* C, const double* B,
                          const double* X, const double* Y, int64_t count, double* losses, int32_t mem,
                          void* stream) {
  if (!w || !opt) return PDQP_ERR_INVALID;
  return guard(w, [&] {
    cudaStream_t s = (cudaStream_t)stream;
    need_ready(w);
    const int batch = opt->batch;
    if (batch < 8 || batch > w->maxb || batch % 8) throw WsFail{PDQP_ERR_INVALID, "batch: multiple of 8 in [8, max_batch]"};
    if (count < batch) throw WsFail{PDQP_ERR_INVALID, "count >= batch"};
    if (opt->epochs < 0 || !(opt->lr > 0.f) || !(opt->beta1 >= 0.f && opt->beta1 < 1.f) ||
        !(opt->beta2 >= 0.f && opt->beta2 < 1.f) || !(opt->eps >= 0.f))
      throw WsFail{PDQP_ERR_INVALID, "options: epochs >= 0, lr > 0, 0 <= beta < 1, eps >= 0"};
    need_data(w, C, B, X, Y, mem, true);
    const int n = w->n, m = w->m, F = w->F, Fp = w->Fp, d = w->d;
    // the training set: H0 = projected normalised inputs (bf16), T = normalised targets (float32)
    if (w->tcount != count) {
      wfree(w, w->H0all);
      wfree(w, w->Tall);
      w->H0all = nullptr;
      w->Tall = nullptr;
      w->tcount = 0;
      w->H0all = walloc<bf16>(w, (size_t)count * d);
      w->Tall = walloc<float>(w, (size_t)count * Fp);
      w->tcount = count;
    }
    {
      DevView<double> c(C, (size_t)count * n, mem, s), b(B, (size_t)count * m, mem, s);
      for (long long r0 = 0; r0 < count; r0 += w->maxb) {
        const int rows = (int)std::min<long long>(w->maxb, count - r0);
        project(w, c.p, b.p, r0, rows, w->H0all + (size_t)r0 * d, s);
      }
      finish(w, s);
    }
    {
      DevView<double> x(X, (size_t)count * n, mem, s), y(Y, (size_t)count * m, mem, s);
      early((two_columns(n, m, x.p, y.p) ? k_prep_target<2> : k_prep_target<1>), row_grid(w, x.p, y.p, count), 256,
            0, s, x.p, y.p, n, m, count, w->out_mean, w->out_inv, w->Tall, Fp);
      finish(w, s);
    }
    const long long steps = count / batch;
    for (int e = 0; e < opt->epochs; ++e) {
      long long a = 1, sft = 0;
      visit_order(opt->seed, e, count, &a, &sft);
      WCK(cudaMemsetAsync(w->lossacc, 0, sizeof(double), s));
      for (long long st = 0; st < steps; ++st) {
        const long long row0 = st * batch;
        early(k_gather_rows, grid_for((long long)batch * d / 8), 256, 0, s, w->H0all, d, a, sft, count, row0, batch,
              d, w->H[0], d);
        forward(w, batch, s);
        backward(w, batch, w->Tall, a, sft, count, row0, s);
        adam(w, opt->lr, opt->beta1, opt->beta2, opt->eps, s);
      }
      finish(w, s);
      if (losses) {
        double h = 0.0;
        WCK(cudaMemcpy(&h, w->lossacc, sizeof(double), cudaMemcpyDeviceToHost));
        losses[e] = h / (double)steps;
      }
    }
  });
}

pdqp_status pdqp_ws_infer(pdqp_ws_handle w, const double* C, const double* B, int64_t count, double* X0,
                          double* Y0, int32_t mem, void* stream) {
  if (!w) return PDQP_ERR_INVALID;
  return guard(w, [&] {
    cudaStream_t s = (cudaStream_t)stream;
    need_ready(w);
    if (count < 1) throw WsFail{PDQP_ERR_INVALID, "count >= 1"};
    if (!X0 && !Y0) throw WsFail{PDQP_ERR_INVALID, "both outputs null"};
    need_data(w, C, B, X0, Y0, mem, false);
    const int n = w->n, m = w->m;
    DevView<double> c(C, (size_t)count * n, mem, s), b(B, (size_t)count * m, mem, s);
    double *x0 = X0, *y0 = m > 0 ? Y0 : nullptr;
    double *tx = nullptr, *ty = nullptr;
    if (mem == PDQP_MEM_HOST) {
      if (x0) tx = x0 = walloc<double>(w, (size_t)count * n);
      if (y0) ty = y0 = walloc<double>(w, (size_t)count * m);
    }
    try {
      for (long long r0 = 0; r0 < count; r0 += w->maxb) {
        const int rows = (int)std::min<long long>(w->maxb, count - r0);
        project(w, c.p, b.p, r0, rows, w->H[0], s);
        forward(w, rows, s, x0 ? x0 + (size_t)r0 * n : nullptr, y0 ? y0 + (size_t)r0 * m : nullptr);
      }
      finish(w, s);
      if (tx) WCK(cudaMemcpy(X0, tx, (size_t)count * n * sizeof(double), cudaMemcpyDeviceToHost));
      if (ty) WCK(cudaMemcpy(Y0, ty, (size_t)count * m * sizeof(double), cudaMemcpyDeviceToHost));
    } catch (...) {
      cudaStreamSynchronize(s);
      wfree(w, tx);
      wfree(w, ty);
      throw;
    }
    wfree(w, tx);
    wfree(w, ty);
  });
}

// Raw GEMM.  The error flag of its bounded waits lives in device memory of the
// library (no allocation per call); pdqp_gemm_bf16_check reads and clears it.
static __device__ int g_gemm_err;

static int* gemm_err_ptr() {
  static int* p = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* q = nullptr;
    if (cudaGetSymbolAddress(&q, g_gemm_err) == cudaSuccess) p = (int*)q;
  });
  return p;
}

pdqp_status pdqp_gemm_bf16(int32_t M, int32_t N, int32_t K, const void* A, int32_t lda, const void* B, int32_t ldb,
                           const float* bias, int32_t relu, const void* mask, int32_t ldm, float* D_f32, void* D_bf16,
                           int32_t ldd, int32_t splits, float* workspace, int64_t workspace_bytes, void* stream) {
  if (M < 1 || N < 1 || K < 1 || !A || !B || (!D_f32 && !D_bf16) || lda < K || ldb < K || ldd < N || splits < 0)
    return PDQP_ERR_INVALID;
  if ((lda % 8) || (ldb % 8) || ((uintptr_t)A & 15) || ((uintptr_t)B & 15)) return PDQP_ERR_INVALID;
  if (mask && ldm < N) return PDQP_ERR_INVALID;
  for (const void* p : {A, B, (const void*)bias, mask, (const void*)D_f32, (const void*)D_bf16, (const void*)workspace})
    if (p && !is_device_ptr(p)) return PDQP_ERR_INVALID;
  const int sp = plan_splits(M, N, K, splits);
  if (splits > 0 && sp > 1 && (!workspace || (size_t)workspace_bytes < (size_t)sp * M * N * sizeof(float)))
    return PDQP_ERR_INVALID;
  int* err = gemm_err_ptr();
  if (!err) return PDQP_ERR_CUDA;
  Epi e;
  e.out_f = D_f32;
  e.out_b = (bf16*)D_bf16;
  e.bias = bias;
  e.mask = (const bf16*)mask;
  e.ldo = ldd;
  e.ldm = ldm;
  e.relu = relu;
  const size_t wf = workspace ? (size_t)workspace_bytes / sizeof(float) : 0;
  if (gemm_tn((const bf16*)A, lda, (const bf16*)B, ldb, M, N, K, e, splits, workspace, wf, err,
              (cudaStream_t)stream) != cudaSuccess)
    return PDQP_ERR_CUDA;
  return PDQP_OK;
}

pdqp_status pdqp_gemm_bf16_check(void* stream) {
  int* err = gemm_err_ptr();
  if (!err) return PDQP_ERR_CUDA;
  int h = 0;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return PDQP_ERR_CUDA;
  if (h) {
    cudaMemsetAsync(err, 0, sizeof(int), s);
    cudaStreamSynchronize(s);
    return PDQP_DEVICE_TIMEOUT;
  }
  return PDQP_OK;
}

pdqp_status pdqp_gemm_bf16_wait_probe(void* stream) {
  int* err = gemm_err_ptr();
  if (!err) return PDQP_ERR_CUDA;
  k_wait_probe<<<1, 32, 0, (cudaStream_t)stream>>>(err);
  if (cudaGetLastError() != cudaSuccess) return PDQP_ERR_CUDA;
  return pdqp_gemm_bf16_check(stream);
}

int32_t pdqp_gemm_bf16_splits(int32_t M, int32_t N, int32_t K, int32_t splits) {
  if (M < 1 || N < 1 || K < 1 || splits < 0) return 0;
  return plan_splits(M, N, K, splits);
}

}  // extern "C"
