// The step/guess predictor: a small MLP trained on trajectories the
// integrator itself generates, mapping a reactor state to the first internal
// step size and the Newton starting stages of the first step.  Radau keeps
// its error test and step control, so the network can only save rejected
// steps and Newton iterations (it changes no accepted result beyond the
// integrator's tolerance).
//
// Network: x (din) -> 3 x [Linear(width) -> SiLU] -> Linear(dout).
// Two arithmetic modes:
//   BF16  5th-generation tensor cores (tcgen05.mma, BF16 operands, FP32
//         accumulators in tensor memory);
//         activations are rounded to BF16 between layers, master weights and
//         the optimiser stay FP32;
//   FP32  CUDA-core FMA everywhere (a check mode for gradient tests).
// Training: MSE loss, backprop, Adam with bias correction.
// Features for the integrator: log T, log P, log dt, log10(max(Y_k, 1e-12))
// (all species), standardised with caller-given moments; outputs: log h0 and
// the 3 N stage increments, de-standardised.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <vector>

#include "kin_internal.h"

using namespace kin;

namespace {

constexpr int LAYERS = 4;

__device__ __forceinline__ float silu(float a) { return a / (1.0f + __expf(-a)); }
__device__ __forceinline__ float silu_grad(float a) {
  const float s = 1.0f / (1.0f + __expf(-a));
  return s * (1.0f + a * (1.0f - s));
}

// ---------------------------------------------------------------------------
// GEMM, generic strides: C[m][n] (+)= sum_k A(m,k) B(k,n) with
// A(m,k) = A[m*sam + k*sak], B(k,n) = B[k*sbk + n*sbn]; out of range = 0.  It
// serves the weight gradients, and every product of widths that are not
// multiples of 8 (the others' forward and input-gradient products are
// k_gemm_kk's below).
//
// BF16 version on the 5th-generation tensor cores (tcgen05): a CTA of four
// warps owns a 128 x 128 tile of C.  Per 64-wide slice of K, the warps copy
// A (128 x 64) and B (as its transpose, 128 x 64, K contiguous) into shared
// memory in the canonical no-swizzle K-major layout (8-row x 16-byte core
// matrices, 128 B each: core (g, c) of rows 8g.. and K columns 8c.. at
// (8 g + c) * 128 bytes), one thread issues four m128n128k16 MMAs into the
// tile's FP32 accumulator in tensor memory (TMEM, 128 columns), and their
// completion is signalled on an mbarrier before the slice is overwritten.
// The epilogue reads the accumulator back with tcgen05.ld (warp w owns TMEM
// lanes 32w..32w+31, the tile's rows) and writes or adds C.  Every wait is
// bounded: on expiry the kernel sets *err, waits (bounded) for its MMAs and
// loads, frees its TMEM and returns.
// A K-contiguous operand with 16-byte rows (the input layer and the output
// layer's input gradient) is loaded by the tensor memory accelerator: one thread
// issues eight cp.async.bulk.tensor boxes of 8 K x 128 rows per slice, each
// landing as 16 core matrices in a row (core (g, c) at c * 2048 + g * 128
// bytes), completion counted in bytes on a second mbarrier; the TMA fills
// rows and K past the matrix with zeros.
// ---------------------------------------------------------------------------
constexpr int TC_BM = 128, TC_BN = 128, TC_BK = 64;
constexpr int TC_THREADS = 128;
constexpr uint32_t TC_TMEM_COLS = 128;
// 16 KB per operand slice; the dynamic allocation is padded so that at most
// four CTAs share an SM (4 x 128 of its 512 TMEM columns)
constexpr size_t TC_SMEM = 2 * TC_BM * TC_BK * sizeof(__nv_bfloat16) + 20 * 1024;
constexpr long long TC_SPIN_LIMIT = 1ll << 26;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor, no swizzle: start address, leading byte
// offset (next core matrix along K), stride byte offset (next 8 rows), the
// fixed version bits 46-48 = 0b001
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16
// A and B (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bits 17-22, M >> 4 at
// bits 24-28
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t phase) {
  for (long long it = 0; it < TC_SPIN_LIMIT; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

// byte offset of element (r, k) of a 128 x 64 K-major slice
__device__ __forceinline__ int tc_off(int r, int k) {
  return (((r >> 3) * (TC_BK / 8) + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1);
}

// 16-byte copy of a core-matrix row (8 consecutive K) when the operand is
// K-contiguous and the row lies inside the matrix, else element by element
__device__ __forceinline__ void tc_stage_row(unsigned char *dst, const __nv_bfloat16 *src_row,
                                             int64_t sk, bool vec, bool row_ok, int gk, int ke) {
  if (vec && row_ok && gk + 8 <= ke) {
    *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(src_row + gk);
    return;
  }
  __nv_bfloat16 *d = reinterpret_cast<__nv_bfloat16 *>(dst);
#pragma unroll
  for (int e = 0; e < 8; ++e)
    d[e] = (row_ok && gk + e < ke) ? src_row[(int64_t)(gk + e) * sk] : __float2bfloat16(0.0f);
}

// A 128 x 64 slice of an operand contiguous in its rows (element (r, k) at
// src[k * sk + r]): a thread loads eight rows at k and k + 1 and stores the
// eight (k, k + 1) pairs; the pairs' order is rotated by lane, so a warp's
// 32-bit stores fall into 32 banks.  rows: rows left in the matrix.
__device__ __forceinline__ void tc_stage_t(unsigned char *dst, const __nv_bfloat16 *src, int64_t sk,
                                           int rows, int k0, int ke) {
#pragma unroll
  for (int it = 0; it < (TC_BM / 8) * (TC_BK / 2) / TC_THREADS; ++it) {
    const int e = it * TC_THREADS + (int)threadIdx.x;
    // lanes: four k pairs of a core matrix, eight row groups; then the rest
    const int kp = (e & 3) + 4 * ((e >> 6) & 7), rg = (e >> 2) & 15;
    const int k = 2 * kp, gk = k0 + k, r = 8 * rg;
    uint4 a = {0, 0, 0, 0}, b = {0, 0, 0, 0};
    if (r < rows) {
      if (gk < ke) a = *reinterpret_cast<const uint4 *>(src + (int64_t)gk * sk + r);
      if (gk + 1 < ke) b = *reinterpret_cast<const uint4 *>(src + (int64_t)(gk + 1) * sk + r);
    }
    const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
    uint32_t p[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      p[2 * q] = __byte_perm(aw[q], bw[q], 0x5410);
      p[2 * q + 1] = __byte_perm(aw[q], bw[q], 0x7632);
    }
    unsigned char *d = dst + tc_off(r, k);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int x = (q + rg) & 7;
      uint32_t v = p[0];
#pragma unroll
      for (int z = 1; z < 8; ++z) v = x == z ? p[z] : v;
      *reinterpret_cast<uint32_t *>(d + 16 * x) = v;
    }
  }
}

// Split K: CTA z sums K in [z kchunk, min(K, (z + 1) kchunk)) and writes its
// partial tile to C + z cz (the caller reduces the partials).
// tma: bit 0 loads A, bit 1 loads B through the tensor maps (rows x K, K
// innermost, boxes of 8 x 128); the split-K chunks are multiples of the slice
__global__ void __launch_bounds__(TC_THREADS) k_gemm_tc(int M, int N, int K,
                                                       const __nv_bfloat16 *A, int64_t sam,
                                                       int64_t sak, const __nv_bfloat16 *B,
                                                       int64_t sbk, int64_t sbn, float *C,
                                                       int64_t ldc, int accumulate, int *err,
                                                       int kchunk, int64_t cz,
                                                       const __grid_constant__ CUtensorMap tmA,
                                                       const __grid_constant__ CUtensorMap tmB,
                                                       int tma) {
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  __shared__ __align__(8) unsigned long long mbar, mfull;
  __shared__ uint32_t tmem_base;
  unsigned char *sA = tc_smem, *sB = tc_smem + TC_BM * TC_BK * 2;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * TC_BM, n0 = blockIdx.y * TC_BN;
  const uint32_t mb = smem_u32(&mbar), mf = smem_u32(&mfull);
  const bool ta = (tma & 1) != 0, tb = (tma & 2) != 0;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base)),
                 "r"(TC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mf) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
  C += (int64_t)blockIdx.z * cz;
  // K-contiguous operands are staged 16 bytes (a core-matrix row) at a time
  const bool a_k1 = sak == 1, b_k1 = sbk == 1;
  const bool a_vec = a_k1 && sam % 8 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const bool b_vec = b_k1 && sbn % 8 == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  const bool a_kfast = sak <= sam, b_kfast = sbk <= sbn;
  // M- or N-contiguous operands (the weight gradients): 16-byte loads of
  // eight rows, transposed on the way into shared memory
  const bool a_m1 = sam == 1 && sak % 8 == 0 && M % 8 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const bool b_n1 = sbn == 1 && sbk % 8 == 0 && N % 8 == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  uint32_t phase = 0, fphase = 0;
  bool ok = true, tma_pending = false;
  const int nk = (ke - kb + TC_BK - 1) / TC_BK;
  for (int kt = 0; kt < nk && ok; ++kt) {
    const int k0 = kb + kt * TC_BK;
    if ((ta || tb) && tid == 0) {  // x = k0 + 8 j: a multiple of 8 elements (16 bytes)
      const uint32_t bytes = (ta ? TC_BM * TC_BK * 2u : 0u) + (tb ? TC_BN * TC_BK * 2u : 0u);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mf), "r"(bytes)
                   : "memory");
#pragma unroll
      for (int j = 0; j < TC_BK / 8; ++j) {
        if (ta)
          asm volatile(
              "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
              " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(sA) + (uint32_t)(j * TC_BM * 16)),
              "l"(reinterpret_cast<uint64_t>(&tmA)), "r"(k0 + 8 * j), "r"(m0), "r"(mf)
              : "memory");
        if (tb)
          asm volatile(
              "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
              " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(sB) + (uint32_t)(j * TC_BN * 16)),
              "l"(reinterpret_cast<uint64_t>(&tmB)), "r"(k0 + 8 * j), "r"(n0), "r"(mf)
              : "memory");
      }
    }
    tma_pending = ta || tb;
    // stage the other slices (zero outside the matrices and the K range)
    if (ta) {
    } else if (a_k1) {
      for (int e = tid; e < TC_BM * (TC_BK / 8); e += TC_THREADS) {
        const int r = e >> 3, kc = (e & 7) * 8, gm = m0 + r;
        tc_stage_row(sA + tc_off(r, kc), A + (int64_t)(gm < M ? gm : 0) * sam, 1, a_vec,
                     gm < M, k0 + kc, ke);
      }
    } else if (a_m1) {
      tc_stage_t(sA, A + m0, sak, M - m0, k0, ke);
    } else {
      for (int e = tid; e < TC_BM * TC_BK; e += TC_THREADS) {
        const int r = a_kfast ? e / TC_BK : e % TC_BM, k = a_kfast ? e % TC_BK : e / TC_BM;
        const int gm = m0 + r, gk = k0 + k;
        const __nv_bfloat16 v = (gm < M && gk < ke) ? A[(int64_t)gm * sam + (int64_t)gk * sak]
                                                    : __float2bfloat16(0.0f);
        *reinterpret_cast<__nv_bfloat16 *>(sA + tc_off(r, k)) = v;
      }
    }
    if (tb) {
    } else if (b_k1) {
      for (int e = tid; e < TC_BN * (TC_BK / 8); e += TC_THREADS) {
        const int c = e >> 3, kc = (e & 7) * 8, gn = n0 + c;
        tc_stage_row(sB + tc_off(c, kc), B + (int64_t)(gn < N ? gn : 0) * sbn, 1, b_vec,
                     gn < N, k0 + kc, ke);
      }
    } else if (b_n1) {
      tc_stage_t(sB, B + n0, sbk, N - n0, k0, ke);
    } else {
      for (int e = tid; e < TC_BN * TC_BK; e += TC_THREADS) {
        const int c = b_kfast ? e / TC_BK : e % TC_BN, k = b_kfast ? e % TC_BK : e / TC_BN;
        const int gn = n0 + c, gk = k0 + k;
        const __nv_bfloat16 v = (gn < N && gk < ke) ? B[(int64_t)gk * sbk + (int64_t)gn * sbn]
                                                    : __float2bfloat16(0.0f);
        *reinterpret_cast<__nv_bfloat16 *>(sB + tc_off(c, k)) = v;
      }
    }
    // make the generic-proxy writes visible to the tensor core (async proxy)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (ta || tb) {  // the TMA boxes have landed
      ok = __syncthreads_and(tc_wait(mf, fphase)) != 0;
      fphase ^= 1u;
      tma_pending = !ok;
      if (!ok) break;
    }
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t idesc = tc_idesc(TC_BM, TC_BN);
#pragma unroll
      for (int s = 0; s < TC_BK / 16; ++s) {
        // k16 step s covers K cores 2s and 2s + 1
        // K cores 128 B apart, 8-row groups 1024 B (threads' layout); or K
        // cores 2048 B apart, row groups 128 B (the TMA boxes)
        const uint64_t da = ta ? tc_desc(smem_u32(sA) + 4096u * s, 2048u, 128u)
                               : tc_desc(smem_u32(sA) + 256u * s, 128u, (TC_BK / 8) * 128u);
        const uint64_t db = tb ? tc_desc(smem_u32(sB) + 4096u * s, 2048u, 128u)
                               : tc_desc(smem_u32(sB) + 256u * s, 128u, (TC_BK / 8) * 128u);
        const uint32_t acc = (kt > 0 || s > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(acc)
            : "memory");
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mb)
          : "memory");
    }
    // the slice may be overwritten once its MMAs have completed; every
    // thread leaves the loop on the same trip
    ok = tc_wait(mb, phase);
    phase ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    ok = __syncthreads_and(ok) != 0;
  }
  if (ok) {
    const int row = m0 + warp * 32 + lane;
    for (int c0 = 0; c0 < TC_BN; c0 += 16) {
      uint32_t v[16];
      const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
          "%14,%15}, [%16];\n"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
            "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
            "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
          : "r"(taddr)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (row < M) {
        float *dst = C + (int64_t)row * ldc + n0 + c0;
        // whole 16-byte pieces when the rows allow it: a lane's scalar stores
        // touch one sector each
        if (!accumulate && n0 + c0 + 16 <= N && ldc % 4 == 0 &&
            (reinterpret_cast<uintptr_t>(C) & 15) == 0) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            *reinterpret_cast<float4 *>(dst + 4 * q) =
                make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                            __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (n0 + c0 + j < N) {
              const float x = __uint_as_float(v[j]);
              dst[j] = accumulate ? dst[j] + x : x;
            }
        }
      }
    }
  } else {
    if (tid == 0) atomicOr(err, 1);
    if (tma_pending) (void)tc_wait(mf, fphase);  // boxes still landing
    else (void)tc_wait(mb, phase ^ 1u);          // the last commit, if it is still pending
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TC_TMEM_COLS)
                 : "memory");
}

// ---------------------------------------------------------------------------
// The same GEMM for two K-contiguous operands with what follows it fused into
// the epilogue (the forward pass and the input gradients).  What bounded
// k_gemm_tc here were its loads: boxes of 16-byte rows (2048 TMA requests per
// slice) and no overlap of loads and MMAs, 1.7 to 3.1 % of the tensor pipe.
// Here a slice is one 128-byte-row box per operand in the 128-byte swizzle
// (rows of 64 K, 8-row groups 1024 bytes apart), three slices are in flight on
// full / empty mbarriers, and bias, SiLU, its derivative, the loss gradient or
// the prediction's de-standardisation run on the accumulator as it leaves
// tensor memory, so no FP32 product is written and read back.  The MMAs and
// their K order are k_gemm_tc's: the same bits.
// ---------------------------------------------------------------------------
constexpr int KK_STAGES = 3;
// eight warps: warps w and w + 4 share TMEM lanes 32 w .. 32 w + 31 and halve
// the epilogue's columns
constexpr int KK_THREADS = 256;
constexpr int KK_STAGE_BYTES = 2 * TC_BM * TC_BK * 2;
constexpr size_t KK_SMEM = (size_t)KK_STAGES * KK_STAGE_BYTES + 1024;  // two CTAs per SM

enum { EP_HIDDEN = 0, EP_OUT, EP_MSE, EP_BACK, EP_UNPACK };

struct Epilogue {
  int mode;
  const float *bias;       // forward modes
  float *a;                // HIDDEN: pre-activation out (or null); BACK: in
  __nv_bfloat16 *hb;       // HIDDEN: activation
  float *out;              // OUT: [M][dout]
  int dout;
  const float *tgt;        // MSE: targets [.][dout], gathered through rows when given
  const int32_t *rows;
  int64_t nrows;
  float *g;                // MSE, BACK: gradient, FP32 and BF16
  __nv_bfloat16 *gb;
  float *loss;
  const float *mean, *stdv;  // UNPACK
  double dt, *h0, *z0;
};

// exact float -> double on the integer pipe (the conversion unit shares the
// FP64 pipe's rate); zeros kept, subnormals and non-finite values converted
__device__ __forceinline__ double widen(float v) {
  const unsigned u = __float_as_uint(v), e = u & 0x7f800000u;
  if (e == 0x7f800000u || (e == 0 && (u << 1) != 0)) return (double)v;
  const unsigned hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (e ? 0x38000000u : 0u));
  return __hiloint2double((int)hi, (int)(u << 29));
}

// sixteen accumulators of row r, columns c0 .. c0 + 15 (n of them inside)
__device__ __forceinline__ void kk_epilogue(const Epilogue &ep, int64_t M, int N, int64_t r, int c0,
                                            int n, const uint32_t (&v)[16], float &loss) {
  const int64_t o = r * N + c0;
  if (ep.mode == EP_HIDDEN || ep.mode == EP_BACK) {
    __align__(16) float x[16];
    __align__(16) __nv_bfloat16 b[16];
    const bool back = ep.mode == EP_BACK;
#pragma unroll
    for (int q = 0; q < 4; ++q)  // N is a multiple of 8: n is 8 or 16
      if (4 * q < n) {
        const float4 in = back ? *reinterpret_cast<const float4 *>(ep.a + o + 4 * q)
                               : *reinterpret_cast<const float4 *>(ep.bias + c0 + 4 * q);
        const float p[4] = {in.x, in.y, in.z, in.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const float acc = __uint_as_float(v[4 * q + t]);
          x[4 * q + t] = back ? acc * silu_grad(p[t]) : acc + p[t];
          b[4 * q + t] = __float2bfloat16(back ? x[4 * q + t] : silu(x[4 * q + t]));
        }
      }
    float *f = back ? ep.g : ep.a;
    __nv_bfloat16 *h = back ? ep.gb : ep.hb;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (f && 4 * q < n)
        *reinterpret_cast<float4 *>(f + o + 4 * q) = *reinterpret_cast<const float4 *>(x + 4 * q);
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (8 * q < n)
        *reinterpret_cast<uint4 *>(h + o + 8 * q) = *reinterpret_cast<const uint4 *>(b + 8 * q);
    return;
  }
  if (ep.mode == EP_MSE) {
    int64_t tr = r;
    if (ep.rows) {
      const int32_t s = ep.rows[r];
      tr = (s >= 0 && (int64_t)s < ep.nrows) ? (int64_t)s : -1;
    }
    const float scale = (float)(M * ep.dout);
    const float *t = ep.tgt + tr * ep.dout + c0;
    __align__(16) float g[16];
    __align__(16) __nv_bfloat16 b[16];
    float tv[16];
    // a row's targets 16 bytes at a time when its length allows
    const bool vec = tr >= 0 && ep.dout % 4 == 0 && c0 + 16 <= ep.dout &&
                     (reinterpret_cast<uintptr_t>(ep.tgt) & 15) == 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (vec) x = *reinterpret_cast<const float4 *>(t + 4 * q);
      tv[4 * q] = x.x;
      tv[4 * q + 1] = x.y;
      tv[4 * q + 2] = x.z;
      tv[4 * q + 3] = x.w;
    }
    float sq = 0.0f;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      g[j] = 0.0f;
      if (j < n && c0 + j < ep.dout) {
        const float y = __uint_as_float(v[j]) + ep.bias[c0 + j];
        const float d = y - (vec ? tv[j] : tr >= 0 ? t[j] : 0.0f);
        g[j] = 2.0f * d / scale;
        sq += d * d;
      }
      b[j] = __float2bfloat16(g[j]);
    }
    loss += sq / scale;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * q < n)
        *reinterpret_cast<float4 *>(ep.g + o + 4 * q) = *reinterpret_cast<const float4 *>(g + 4 * q);
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (8 * q < n)
        *reinterpret_cast<uint4 *>(ep.gb + o + 8 * q) = *reinterpret_cast<const uint4 *>(b + 8 * q);
    return;
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int c = c0 + j;
    if (j >= n) break;
    const float y = __uint_as_float(v[j]) + ep.bias[c];
    if (ep.mode == EP_OUT) {
      if (c < ep.dout) ep.out[r * ep.dout + c] = y;
    } else if (c < ep.dout) {
      const double sd = widen(ep.stdv[c]), mu = widen(ep.mean[c]);
      if (c == 0) {
        if (ep.h0) ep.h0[r] = fmin(fmax(exp(widen(y) * sd + mu), 1e-14), ep.dt);
      } else if (ep.z0) {
        ep.z0[(int64_t)(c - 1) * M + r] = widen(y) * sd + mu;
      }
    }
  }
}

__device__ __forceinline__ void tma_box(uint32_t dst, const CUtensorMap *tm, int x, int y,
                                        uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(mbar)
      : "memory");
}

__global__ void __launch_bounds__(KK_THREADS) k_gemm_kk(int64_t M, int N, int K, int *err,
                                                       const __grid_constant__ CUtensorMap tmA,
                                                       const __grid_constant__ CUtensorMap tmB,
                                                       const __grid_constant__ Epilogue ep) {
  extern __shared__ unsigned char kk_raw[];
  __shared__ __align__(8) unsigned long long full[KK_STAGES], empty[KK_STAGES], alldone;
  __shared__ uint32_t tmem_base;
  __shared__ int failed;
  const uint32_t base = (smem_u32(kk_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t m0 = (int64_t)blockIdx.x * TC_BM;
  const int n0 = blockIdx.y * TC_BN;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base)),
                 "r"(TC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    failed = 0;
    for (int s = 0; s < KK_STAGES; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&alldone)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const int nk = (K + TC_BK - 1) / TC_BK;
  if (tid == 0) {
    auto load = [&](int kt) {
      const int s = kt % KK_STAGES;
      const uint32_t mb = smem_u32(&full[s]), dst = base + (uint32_t)(s * KK_STAGE_BYTES);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb),
                   "r"((uint32_t)KK_STAGE_BYTES)
                   : "memory");
      // x = 64 kt: a multiple of 8 elements (16 bytes); zero fill past the matrix
      tma_box(dst, &tmA, kt * TC_BK, (int)m0, mb);
      tma_box(dst + KK_STAGE_BYTES / 2, &tmB, kt * TC_BK, n0, mb);
    };
    int loaded = 0;
    for (; loaded < nk && loaded < KK_STAGES; ++loaded) load(loaded);
    bool ok = true;
    int kt = 0;
    for (; kt < nk && ok; ++kt) {
      const int s = kt % KK_STAGES;
      const uint32_t ph = (uint32_t)(kt / KK_STAGES) & 1u;
      ok = tc_wait(smem_u32(&full[s]), ph);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = base + (uint32_t)(s * KK_STAGE_BYTES), sb = sa + KK_STAGE_BYTES / 2;
#pragma unroll
      for (int q = 0; q < TC_BK / 16; ++q) {
        // 128-byte swizzle (layout 2): K advances by 32 bytes inside the row
        const uint64_t sw = (uint64_t)2 << 61;
        const uint64_t da = tc_desc(sa + 32u * q, 16u, 1024u) | sw;
        const uint64_t db = tc_desc(sb + 32u * q, 16u, 1024u) | sw;
        const uint32_t acc = (kt > 0 || q > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(da), "l"(db), "r"(tc_idesc(TC_BM, TC_BN)), "r"(acc)
            : "memory");
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              smem_u32(&empty[s]))
          : "memory");
      if (loaded < nk) {  // the stage is free once its MMAs are done
        ok = tc_wait(smem_u32(&empty[s]), ph);
        if (ok) load(loaded++);
      }
    }
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(&alldone))
        : "memory");
    if (!ok) {  // flagged; wait (bounded) for the boxes still in flight
      failed = 1;
      atomicOr(err, 1);
      for (int q = kt; q < loaded; ++q)
        (void)tc_wait(smem_u32(&full[q % KK_STAGES]), (uint32_t)(q / KK_STAGES) & 1u);
    }
  }
  __syncwarp();
  const bool done = tc_wait(smem_u32(&alldone), 0);
  if (!done) atomicOr(err, 1);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool good = __syncthreads_and(done) && !failed;
  float loss = 0.0f;
  if (good) {
    const int64_t row = m0 + (warp & 3) * 32 + lane;
    const int nc = N - n0 < TC_BN ? N - n0 : TC_BN;
    for (int c0 = (warp >> 2) * 16; c0 < nc; c0 += 32) {
      uint32_t v[16];
      const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
          "%14,%15}, [%16];\n"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
            "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
            "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
          : "r"(taddr)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (row < M) kk_epilogue(ep, M, N, row, n0 + c0, min(16, nc - c0), v, loss);
    }
    if (ep.mode == EP_MSE) {
      for (int o = 16; o > 0; o >>= 1) loss += __shfl_down_sync(0xffffffffu, loss, o);
      if (lane == 0 && loss != 0.0f) atomicAdd(ep.loss, loss);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TC_TMEM_COLS)
                 : "memory");
}

// FP32 CUDA-core version (check mode): one output per thread.
__global__ void k_gemm_f32(int M, int N, int K, const float *A, int64_t sam, int64_t sak,
                           const float *B, int64_t sbk, int64_t sbn, float *C, int64_t ldc,
                           int accumulate) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)M * N) return;
  const int m = (int)(idx / N), n = (int)(idx % N);
  float s = 0.0f;
  for (int k = 0; k < K; ++k) s = fmaf(A[m * sam + k * sak], B[k * sbk + n * sbn], s);
  float *dst = C + (int64_t)m * ldc + n;
  *dst = accumulate ? *dst + s : s;
}

// ---------------------------------------------------------------------------
// Elementwise kernels
// ---------------------------------------------------------------------------
// a = C + b (stored), h = silu(a) (or a for the last layer) as f32 and bf16
__global__ void k_bias_act(int64_t M, int N, const float *C, const float *b, float *a, float *hf,
                           __nv_bfloat16 *hb, int act) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M * N) return;
  const float v = C[i] + b[i % N];
  if (a) a[i] = v;
  const float h = act ? silu(v) : v;
  if (hf) hf[i] = h;
  if (hb) hb[i] = __float2bfloat16(h);
}

// gather rows of a [R][d] set: dst[r] = src[rows[r]]; an index outside
// [0, R) gives a zero row
__global__ void k_gather_rows(int64_t M, int d, const float *src, int64_t R,
                              const int32_t *rows, float *dst) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M * d) return;
  const int64_t r = i / d;
  const int c = (int)(i % d);
  const int32_t s = rows[r];
  dst[i] = (s >= 0 && (int64_t)s < R) ? src[(int64_t)s * d + c] : 0.0f;
}

// pad/convert an input block [M][din] f32 -> [M][ld] (f32 and bf16), zero pad
__global__ void k_pack_input(int64_t M, int din, int ld, const float *X, float *xf,
                             __nv_bfloat16 *xb) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M * ld) return;
  const int64_t r = i / ld;
  const int c = (int)(i % ld);
  const float v = c < din ? X[r * din + c] : 0.0f;
  if (xf) xf[i] = v;
  if (xb) xb[i] = __float2bfloat16(v);
}

// loss gradient g = 2 (y - t) / (M dout) on the first dout columns, loss sum
__global__ void k_mse_grad(int64_t M, int dout, int ld, const float *y, const float *tgt, float *g,
                           __nv_bfloat16 *gb, float *loss) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float l = 0.0f;
  if (i < M * ld) {
    const int64_t r = i / ld;
    const int c = (int)(i % ld);
    float v = 0.0f;
    if (c < dout) {
      const float d = y[i] - tgt[r * dout + c];
      v = 2.0f * d / (float)(M * dout);
      l = d * d / (float)(M * dout);
    }
    g[i] = v;
    if (gb) gb[i] = __float2bfloat16(v);
  }
  if (loss) {
    for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
    if ((threadIdx.x & 31) == 0 && l != 0.0f) atomicAdd(loss, l);
  }
}

// g = dH * silu'(a)
__global__ void k_silu_back(int64_t n, const float *dH, const float *a, float *g,
                            __nv_bfloat16 *gb) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float v = dH[i] * silu_grad(a[i]);
  g[i] = v;
  if (gb) gb[i] = __float2bfloat16(v);
}

// column sums: out[c] = sum_r g[r][c]; a cluster of eight CTAs per 32 columns,
// its partial sums added through distributed shared memory in a fixed order
// (a thread per column alone walked 4096 rows in sequence)
constexpr int CS_CTAS = 8, CS_THREADS = 512;

__global__ void __cluster_dims__(CS_CTAS, 1, 1) __launch_bounds__(CS_THREADS)
    k_colsum(int64_t M, int N, const float *g, float *out) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ float part[CS_THREADS / 32][32], mine[32];
  const int lane = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int c = (int)(blockIdx.x / CS_CTAS) * 32 + lane;
  const int64_t step = (int64_t)CS_CTAS * (CS_THREADS / 32);
  float s = 0.0f;
  if (c < N) {
#pragma unroll 16
    for (int64_t r = (int64_t)cl.block_rank() * (CS_THREADS / 32) + y; r < M; r += step)
      s += g[r * N + c];
  }
  part[y][lane] = s;
  __syncthreads();
  if (y == 0) {
    float t = 0.0f;
    for (int w = 0; w < CS_THREADS / 32; ++w) t += part[w][lane];
    mine[lane] = t;
  }
  cl.sync();
  if (cl.block_rank() == 0 && y == 0 && c < N) {
    float t = 0.0f;
    for (int k = 0; k < CS_CTAS; ++k) t += cl.map_shared_rank(&mine[0], k)[lane];
    out[c] = t;
  }
  cl.sync();
}

// weight blocks of the network: offset, K, N per layer
struct LayerShapes {
  int64_t woff[4];
  int K[4], N[4];
};

// Adam, then the BF16 copies of the weight (as it lies and transposed)
__global__ void k_adam_refresh(int64_t n, float *p, const float *grad, float *m, float *v,
                               const unsigned char *mask, float lr, float b1, float b2, float eps,
                               float c1, float c2, LayerShapes L, __nv_bfloat16 *wb,
                               __nv_bfloat16 *wbt) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float pi = p[i];
  if (mask[i]) {
    const float gi = grad[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    pi -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
  }
  const __nv_bfloat16 b = __float2bfloat16(pi);
  wb[i] = b;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const int64_t e = i - L.woff[l];
    if (e >= 0 && e < (int64_t)L.K[l] * L.N[l]) {
      const int k = (int)(e / L.N[l]), c = (int)(e % L.N[l]);
      wbt[L.woff[l] + (int64_t)c * L.K[l] + k] = b;
    }
  }
}

// input rows [M][din] (gathered through rows when given; an index outside
// [0, R) gives a zero row) -> BF16 [M][ld], zero padded
__global__ void k_gather_pack(int64_t M, int din, int ld, const float *X, int64_t R,
                              const int32_t *rows, __nv_bfloat16 *xb) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M * ld) return;
  const int64_t r = i / ld;
  const int c = (int)(i % ld);
  int64_t s = r;
  if (rows) {
    const int32_t q = rows[r];
    s = (q >= 0 && (int64_t)q < R) ? (int64_t)q : -1;
  }
  xb[i] = __float2bfloat16(s >= 0 && c < din ? X[s * din + c] : 0.0f);
}

__global__ void k_to_bf16(int64_t n, const float *x, __nv_bfloat16 *y) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = __float2bfloat16(x[i]);
}

// y [N][K] = bf16(x [K][N])^T: a weight block with K contiguous, so the
// forward GEMMs stage their B operand 16 bytes at a time
__global__ void k_to_bf16_t(int K, int N, const float *x, __nv_bfloat16 *y) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)K * N) return;
  const int k = (int)(i / N), n = (int)(i % N);
  y[(int64_t)n * K + k] = __float2bfloat16(x[i]);
}

// C[m][n] (+)= sum over the S partial tiles ws[s][m][n] (split-K GEMMs; a
// fixed summation order, so results do not depend on scheduling)
__global__ void k_splitk_reduce(int M, int N, int S, const float *ws, float *C, int64_t ldc,
                                int accumulate) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)M * N) return;
  const int m = (int)(i / N), n = (int)(i % N);
  float v = 0.0f;
#pragma unroll 16
  for (int q = 0; q < S; ++q) v += ws[(int64_t)q * M * N + i];
  float *dst = C + (int64_t)m * ldc + n;
  *dst = accumulate ? *dst + v : v;
}

// column mean and standard deviation of X [M][d] (two-pass, FP64 sums).  A
// cluster of eight CTAs owns eight columns (one 32-byte sector per row) and
// sums them through distributed shared memory: two passes in one launch
// without a workspace.  Bound by FP64 additions; a thread per column walked
// the rows in sequence (65536 x 160: 14 ms).  The FP32 values are widened on
// the integer pipe.
// Up to MOM_FEW rows a thread per column it is: launching clusters and meeting
// in them takes longer (8 x 16: 12.6 us against 7.7, 8 x 160: 17.6 against 7.7;
// 64 x 16: 13.1 against 15.1).
constexpr int64_t MOM_FEW = 32;

__global__ void k_moments_few(int64_t M, int d, const float *X, float *mean, float *stdv) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d) return;
  double s = 0.0, q = 0.0;
  for (int64_t r = 0; r < M; ++r) s += X[r * d + c];
  const double mu = s / (double)M;
  for (int64_t r = 0; r < M; ++r) {
    const double e = X[r * d + c] - mu;
    q += e * e;
  }
  mean[c] = (float)mu;
  stdv[c] = (float)fmax(sqrt(q / (double)M), 1e-12);
}

constexpr int MOM_CTAS = 8, MOM_COLS = 8, MOM_THREADS = 512;

__global__ void __cluster_dims__(MOM_CTAS, 1, 1) __launch_bounds__(MOM_THREADS)
    k_moments(int64_t M, int d, const float *X, float *mean, float *stdv) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ double part[2][MOM_COLS];  // this CTA's sums, per pass
  __shared__ double warp_part[MOM_THREADS / 32][MOM_COLS];
  const int tid = threadIdx.x, cx = tid % MOM_COLS, warp = tid / 32;
  const int c = (int)(blockIdx.x / MOM_CTAS) * MOM_COLS + cx;
  const int64_t step = (int64_t)MOM_CTAS * (MOM_THREADS / MOM_COLS);
  const int64_t r0 = (int64_t)cl.block_rank() * (MOM_THREADS / MOM_COLS) + tid / MOM_COLS;
  double mu = 0.0, q = 0.0;
  for (int pass = 0; pass < 2; ++pass) {
    double s = 0.0;
    if (c < d) {
      int64_t r = r0;
      for (; r + 3 * step < M; r += 4 * step) {  // four rows' loads in flight
        const float a0 = X[r * d + c], a1 = X[(r + step) * d + c], a2 = X[(r + 2 * step) * d + c],
                    a3 = X[(r + 3 * step) * d + c];
        if (pass == 0) {
          s += (widen(a0) + widen(a1)) + (widen(a2) + widen(a3));
        } else {
          const double e0 = widen(a0) - mu, e1 = widen(a1) - mu, e2 = widen(a2) - mu,
                       e3 = widen(a3) - mu;
          s = fma(e0, e0, fma(e1, e1, fma(e2, e2, fma(e3, e3, s))));
        }
      }
      for (; r < M; r += step) {
        const double e = widen(X[r * d + c]) - mu;
        s += pass == 0 ? e : e * e;
      }
    }
    for (int o = 16; o >= MOM_COLS; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((tid & 31) < MOM_COLS) warp_part[warp][cx] = s;
    __syncthreads();
    if (tid < MOM_COLS) {
      double t = 0.0;
      for (int w = 0; w < MOM_THREADS / 32; ++w) t += warp_part[w][tid];
      part[pass][tid] = t;
    }
    cl.sync();
    double t = 0.0;
    for (int k = 0; k < MOM_CTAS; ++k) t += cl.map_shared_rank(&part[pass][0], k)[cx];
    if (pass == 0)
      mu = t / (double)M;
    else
      q = t;
  }
  if (c < d && cl.block_rank() == 0 && tid < MOM_COLS) {
    mean[c] = (float)mu;
    stdv[c] = (float)fmax(sqrt(q / (double)M), 1e-12);
  }
  cl.sync();  // the peers' sums stay readable until all are done
}

// ---------------------------------------------------------------------------
// Natural logarithm by table (Tang, ACM TOMS 16, 1990): x = 2^e m, an entry
// c near 1/m for each 1/128 of [1, 2), r = m c - 1 (|r| < 2^-7), log x = e ln2
// - log c + log1p(r), the last by its series to r^8 (2^-59 of r).  A dozen FP64
// operations against the library's 35; normal positive x only.
// tab[2 j] = c, tab[2 j + 1] = -log c; a block fills its own copy.
// ---------------------------------------------------------------------------
constexpr int LOG_TAB = 128;

__device__ __forceinline__ void log_table(double *tab) {
  for (int j = threadIdx.x; j < LOG_TAB; j += blockDim.x) {
    // nine significant bits, so m c has no more than 62 and r one rounding
    // (1 and 1/2 at the ends keep log x accurate relative to itself near 1)
    const int q = j == 0 ? 512 : j == LOG_TAB - 1 ? 256 : __float2int_rn(65536.0f / (128.5f + j));
    const double c = q / 512.0;
    tab[2 * j] = c;
    tab[2 * j + 1] = -log(c);
  }
}

__device__ __forceinline__ double tab_log(double x, const double *tab) {
  const long long b = __double_as_longlong(x);
  const int hi = (int)(b >> 32);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return log(x);  // 0, < 0, subnormal, inf, NaN
  const int j = (hi >> 13) & (LOG_TAB - 1), e = (hi >> 20) - 1023;
  const double m = __longlong_as_double((b & 0x000fffffffffffffll) | 0x3ff0000000000000ll);
  const double r = fma(m, tab[2 * j], -1.0);
  // e as a double without the conversion unit: 2^52 + 2^51 + e, less that
  const double ed = __longlong_as_double(0x4338000000000000ll + e) - 6755399441055744.0;
  double p = fma(r, -1.0 / 8.0, 1.0 / 7.0);
  p = fma(p, r, -1.0 / 6.0);
  p = fma(p, r, 1.0 / 5.0);
  p = fma(p, r, -1.0 / 4.0);
  p = fma(p, r, 1.0 / 3.0);
  p = fma(p, r, -0.5);
  p = fma(p * r, r, r);
  return fma(ed, 0.693147180559945309417, tab[2 * j + 1] + p);
}

// features of the integrator's states: [log T, log P, log dt, log10 Y_k],
// standardised with mean / stdv when given, as FP32 rows X [n][3 + ns] or as
// BF16 rows xb [n][ld] with zero padding.  A block stages FEAT_ROWS states in
// shared memory: the species-major reads and the row-major writes are both
// coalesced.  Bound by the FP64 work of the logarithms.
constexpr int FEAT_ROWS = 32, FEAT_COLS = 256, FEAT_THREADS = 256;

__global__ void __launch_bounds__(FEAT_THREADS)
    k_features(int64_t n, int ns, const double *Y, const double *T, const double *P, double logdt,
               const float *mean, const float *stdv, float *X, __nv_bfloat16 *xb, int ld) {
  __shared__ double tab[2 * LOG_TAB];
  __shared__ float tile[FEAT_ROWS][FEAT_COLS + 1];
  const int din = 3 + ns, tid = threadIdx.x;
  log_table(tab);
  __syncthreads();
  for (int64_t i0 = (int64_t)blockIdx.x * FEAT_ROWS; i0 < n; i0 += (int64_t)gridDim.x * FEAT_ROWS) {
    const int rows = (int)(n - i0 < FEAT_ROWS ? n - i0 : FEAT_ROWS);
    for (int c0 = 0; c0 < din; c0 += FEAT_COLS) {
      const int nc = din - c0 < FEAT_COLS ? din - c0 : FEAT_COLS;
      for (int q = tid; q < FEAT_ROWS * nc; q += FEAT_THREADS) {
        const int row = q % FEAT_ROWS, c = c0 + q / FEAT_ROWS;
        const int64_t i = i0 + row;
        if (row >= rows) continue;
        float x;
        if (c == 2) {
          x = (float)logdt;
        } else if (c < 2) {
          x = (float)tab_log((c == 0 ? T : P)[i], tab);
        } else {
          const double y = Y[(int64_t)(c - 3) * n + i];
          // max(y, 1e-12) on the bit pattern: negative values and NaN give the floor
          const long long yb = __double_as_longlong(y), fl = __double_as_longlong(1e-12);
          const double z = (yb > fl && yb <= 0x7ff0000000000000ll) ? y : 1e-12;
          x = (float)(tab_log(z, tab) * 0.434294481903251827651);
        }
        if (mean) x = (x - mean[c]) / stdv[c];
        tile[row][c - c0] = x;
      }
      __syncthreads();
      if (X)
        for (int q = tid; q < rows * nc; q += FEAT_THREADS)
          X[(i0 + q / nc) * din + c0 + q % nc] = tile[q / nc][q % nc];
      if (xb)
        for (int q = tid; q < rows * nc; q += FEAT_THREADS)
          xb[(i0 + q / nc) * ld + c0 + q % nc] = __float2bfloat16(tile[q / nc][q % nc]);
      __syncthreads();
    }
    if (xb)
      for (int q = tid; q < rows * (ld - din); q += FEAT_THREADS)
        xb[(i0 + q / (ld - din)) * ld + din + q % (ld - din)] = __float2bfloat16(0.0f);
  }
}

// network outputs -> h0 (clipped to [1e-14, dt]) and stage guesses [3N][n]
__global__ void k_unpack_prediction(int64_t n, int dout, int ld, const float *y, const float *mean,
                                    const float *stdv, double dt, double *h0, double *z0) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float *r = y + i * ld;
  if (h0) {
    double lh = (double)r[0] * stdv[0] + mean[0];
    double h = exp(lh);
    h0[i] = fmin(fmax(h, 1e-14), dt);
  }
  if (z0)
    for (int c = 1; c < dout; ++c) z0[(int64_t)(c - 1) * n + i] = (double)r[c] * stdv[c] + mean[c];
}

// training targets: [log h, z_1..z_3N] from the integrator's first-step
// outputs, standardised when mean is given; staged like the features
__global__ void __launch_bounds__(FEAT_THREADS)
    k_targets(int64_t n, int nz, const double *h, const double *z, const float *mean,
              const float *stdv, float *tgt) {
  __shared__ float tile[FEAT_ROWS][FEAT_COLS + 1];
  const int d = 1 + nz, tid = threadIdx.x;
  for (int64_t i0 = (int64_t)blockIdx.x * FEAT_ROWS; i0 < n; i0 += (int64_t)gridDim.x * FEAT_ROWS) {
    const int rows = (int)(n - i0 < FEAT_ROWS ? n - i0 : FEAT_ROWS);
    for (int c0 = 0; c0 < d; c0 += FEAT_COLS) {
      const int nc = d - c0 < FEAT_COLS ? d - c0 : FEAT_COLS;
      for (int q = tid; q < FEAT_ROWS * nc; q += FEAT_THREADS) {
        const int row = q % FEAT_ROWS, c = c0 + q / FEAT_ROWS;
        const int64_t i = i0 + row;
        if (row >= rows) continue;
        float x = c == 0 ? (float)log(h[i]) : (float)z[(int64_t)(c - 1) * n + i];
        if (mean) x = (x - mean[c]) / stdv[c];
        tile[row][c - c0] = x;
      }
      __syncthreads();
      for (int q = tid; q < rows * nc; q += FEAT_THREADS)
        tgt[(i0 + q / nc) * d + c0 + q % nc] = tile[q / nc][q % nc];
      __syncthreads();
    }
  }
}

// the same for many narrow rows: a row per thread, whose scattered writes share
// sectors in L2, where a tile leaves its threads few elements between barriers.
// us with tiles / rows: 10^6 x 3 89 / 66, x 14 153 / 90, x 18 188 / 99, x 28 223
// / 215; 2 10^5 x 14 27 / 24; but 3 10^4 x 16 8.3 / 10.
constexpr int TARGET_NARROW = 28;
constexpr int64_t TARGET_MANY = 100000;

__global__ void k_targets_rows(int64_t n, int nz, const double *h, const double *z,
                               const float *mean, const float *stdv, float *tgt) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float *t = tgt + i * (1 + nz);
  for (int c = 0; c <= nz; ++c) {
    float x = c == 0 ? (float)log(h[i]) : (float)z[(int64_t)(c - 1) * n + i];
    if (mean) x = (x - mean[c]) / stdv[c];
    t[c] = x;
  }
}

inline unsigned blocks(int64_t n, int b = 256) { return (unsigned)((n + b - 1) / b); }

}  // namespace

struct kin_mlp {
  int din, dinp, width, dout, doutp, precision;
  int K[LAYERS], N[LAYERS];
  int64_t woff[LAYERS], boff[LAYERS], np;
  float *p = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
  unsigned char *mask = nullptr;
  __nv_bfloat16 *wb = nullptr;  // bf16 copy of the weight blocks (same offsets)
  __nv_bfloat16 *wbt = nullptr; // the same blocks transposed ([N][K] at the same offsets)
  float *ws = nullptr;          // split-K partial tiles
  int64_t ws_floats = 0;
  int64_t step = 0;
  // activations (capacity rows)
  int64_t cap = 0;
  float *xf = nullptr, *a[LAYERS] = {}, *hf[LAYERS] = {}, *C = nullptr, *g = nullptr,
        *dH = nullptr, *y = nullptr, *loss = nullptr;
  float *xg = nullptr, *tg = nullptr;  // gathered minibatch rows (train_step_rows)
  int *err = nullptr;                  // set by a tensor-core GEMM whose wait expired
  __nv_bfloat16 *xb = nullptr, *hb[LAYERS] = {}, *gb = nullptr, *gb2 = nullptr;
  // Tensor maps of the fused path's operands, built with the buffers they
  // describe: encoding two per GEMM took as long as launching it.  Activations
  // and gradients span the buffers' capacity; rows past a batch give
  // accumulator rows that are never stored.
  CUtensorMap mx, mh[LAYERS], mg[2][2];  // mg: buffer gb / gb2, width doutp / width
  CUtensorMap mw[LAYERS], mwt[LAYERS];   // weight blocks [K][N] and transposed [N][K]
  bool maps = false;
};

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library); null when unavailable
static PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    (void)cudaGetLastError();
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

// tensor map of a rows x cols BF16 matrix with row stride ld (elements),
// boxes of 8 columns x 128 rows (swizzle: 64 columns in the 128-byte swizzle),
// zero fill outside; false when the layout
// does not allow the TMA (16-byte base and rows)
static bool make_tmap(CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int64_t ld,
                      bool swizzle = false) {
  std::memset(m, 0, sizeof *m);
  auto enc = tmap_encoder();
  if (!enc || (reinterpret_cast<uintptr_t>(base) & 15) || (ld * 2) % 16 || ld < cols ||
      rows < 1 || cols < 1)
    return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {swizzle ? 64u : 8u, 128}, es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box,
             es, CU_TENSOR_MAP_INTERLEAVE_NONE,
             swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

// The fused path: BF16, both operands of the forward and input-gradient GEMMs
// in 16-byte rows.  Other widths keep the unfused kernels.
static bool mlp_fused(const kin_mlp *n) {
  return n->precision == 0 && n->width % 8 == 0 && tmap_encoder() != nullptr;
}

static bool mlp_maps(kin_mlp *n) {
  if (!mlp_fused(n)) return false;
  bool ok = make_tmap(&n->mx, n->xb, n->cap, n->dinp, n->dinp, true);
  for (int l = 0; l < LAYERS; ++l) {
    ok = ok && make_tmap(&n->mh[l], n->hb[l], n->cap, n->N[l], n->N[l], true);
    ok = ok && make_tmap(&n->mw[l], n->wb + n->woff[l], n->K[l], n->N[l], n->N[l], true);
    ok = ok && make_tmap(&n->mwt[l], n->wbt + n->woff[l], n->N[l], n->K[l], n->K[l], true);
  }
  for (int q = 0; q < 2; ++q)
    for (int w = 0; w < 2; ++w) {
      const int ld = w ? n->width : n->doutp;
      ok = ok && make_tmap(&n->mg[q][w], q ? n->gb2 : n->gb, n->cap, ld, ld, true);
    }
  return ok;
}

template <typename X>
static void drop(X *&p) {
  cudaFree(p);
  p = nullptr;
}

// the activations' buffers and what describes them; the pointers are cleared,
// so that a handle whose growth failed is neither read nor freed again
static void mlp_release(kin_mlp *n) {
  drop(n->xg);
  drop(n->tg);
  drop(n->xf);
  drop(n->xb);
  drop(n->C);
  drop(n->g);
  drop(n->dH);
  drop(n->gb);
  drop(n->gb2);
  for (int l = 0; l < LAYERS; ++l) {
    drop(n->a[l]);
    drop(n->hf[l]);
    drop(n->hb[l]);
  }
  n->y = nullptr;
  n->cap = 0;
  n->maps = false;
}

// Buffers for a number of rows, those that the handle's path touches: the
// fused path gathers rows as it packs them, keeps no FP32 activation but the
// pre-activations its backward pass reads, and alternates between two gradient
// pairs (8.1 KB a row at width 256 with 56 inputs and 160 outputs; with the
// unfused path's buffers beside them it was 14.6 KB, 1.9 GB for 131 072 rows,
// and a first prediction waits for their allocation).
static int mlp_reserve(kin_mlp *n, int64_t rows) {
  if (rows <= n->cap) return KIN_OK;
  mlp_release(n);
  const bool fused = mlp_fused(n);
  const int64_t wmax = n->width > n->doutp ? n->width : n->doutp;
  if (!fused) {
    KIN_CUDA_TRY(cudaMalloc(&n->xg, sizeof(float) * rows * n->din));
    KIN_CUDA_TRY(cudaMalloc(&n->tg, sizeof(float) * rows * n->dout));
    KIN_CUDA_TRY(cudaMalloc(&n->xf, sizeof(float) * rows * n->dinp));
    KIN_CUDA_TRY(cudaMalloc(&n->C, sizeof(float) * rows * wmax));
  }
  KIN_CUDA_TRY(cudaMalloc(&n->xb, sizeof(__nv_bfloat16) * rows * n->dinp));
  KIN_CUDA_TRY(cudaMalloc(&n->g, sizeof(float) * rows * wmax));
  KIN_CUDA_TRY(cudaMalloc(&n->dH, sizeof(float) * rows * wmax));
  KIN_CUDA_TRY(cudaMalloc(&n->gb, sizeof(__nv_bfloat16) * rows * wmax));
  if (fused) KIN_CUDA_TRY(cudaMalloc(&n->gb2, sizeof(__nv_bfloat16) * rows * wmax));
  for (int l = 0; l < LAYERS; ++l) {
    if (!fused || l < LAYERS - 1) KIN_CUDA_TRY(cudaMalloc(&n->a[l], sizeof(float) * rows * n->N[l]));
    if (!fused) KIN_CUDA_TRY(cudaMalloc(&n->hf[l], sizeof(float) * rows * n->N[l]));
    KIN_CUDA_TRY(cudaMalloc(&n->hb[l], sizeof(__nv_bfloat16) * rows * n->N[l]));
  }
  n->y = n->hf[LAYERS - 1];
  n->cap = rows;
  n->maps = mlp_maps(n);
  return KIN_OK;
}

// TMA operand loads (1) or the threads' copies only (0): a build-time knob
#ifndef KIN_MLP_TMA
#define KIN_MLP_TMA 1
#endif

static void gemm(const kin_mlp *n, cudaStream_t st, int M, int N, int K, bool bf, const void *A,
                 int64_t sam, int64_t sak, const void *B, int64_t sbk, int64_t sbn, float *C,
                 int64_t ldc, int acc) {
  if (bf) {
    CUtensorMap tmA, tmB;
    int tma = 0;
    if (KIN_MLP_TMA && sak == 1 && make_tmap(&tmA, A, M, K, sam)) tma |= 1;
    if (KIN_MLP_TMA && sbk == 1 && make_tmap(&tmB, B, N, K, sbn)) tma |= 2;
    if (!(tma & 1)) std::memset(&tmA, 0, sizeof tmA);
    if (!(tma & 2)) std::memset(&tmB, 0, sizeof tmB);
    dim3 grid((M + TC_BM - 1) / TC_BM, (N + TC_BN - 1) / TC_BN, 1);
    // few output tiles and a long K (the weight gradients: K = batch rows):
    // split K over up to 2 x 152 CTAs, partial tiles reduced in fixed order
    const int64_t tiles = (int64_t)grid.x * grid.y, kt = (K + TC_BK - 1) / TC_BK;
    int S = 1;
    if (tiles < 2 * 152 && kt >= 8) {
      S = (int)std::min<int64_t>(kt / 2, (2 * 152 + tiles - 1) / tiles);
      while (S > 1 && (int64_t)S * M * N > n->ws_floats) --S;
    }
    if (S > 1) {
      const int kchunk = (int)((kt + S - 1) / S) * TC_BK;
      S = (K + kchunk - 1) / kchunk;  // every split holds at least one K slice
      grid.z = S;
      k_gemm_tc<<<grid, TC_THREADS, TC_SMEM, st>>>(M, N, K, (const __nv_bfloat16 *)A, sam, sak,
                                                   (const __nv_bfloat16 *)B, sbk, sbn, n->ws, N,
                                                   0, n->err, kchunk, (int64_t)M * N, tmA, tmB,
                                                   tma);
      k_splitk_reduce<<<blocks((int64_t)M * N), 256, 0, st>>>(M, N, S, n->ws, C, ldc, acc);
    } else {
      k_gemm_tc<<<grid, TC_THREADS, TC_SMEM, st>>>(M, N, K, (const __nv_bfloat16 *)A, sam, sak,
                                                   (const __nv_bfloat16 *)B, sbk, sbn, C, ldc,
                                                   acc, n->err, (int)kt * TC_BK, 0, tmA, tmB,
                                                   tma);
    }
  } else {
    k_gemm_f32<<<blocks((int64_t)M * N), 256, 0, st>>>(M, N, K, (const float *)A, sam, sak,
                                                       (const float *)B, sbk, sbn, C, ldc, acc);
  }
}

static int gemm_kk(const kin_mlp *n, cudaStream_t st, int64_t M, int N, int K,
                   const CUtensorMap &A, const CUtensorMap &B, const Epilogue &ep) {
  if (!n->maps) return KIN_ERR_CUDA;
  const dim3 grid((unsigned)((M + TC_BM - 1) / TC_BM), (unsigned)((N + TC_BN - 1) / TC_BN), 1);
  k_gemm_kk<<<grid, KK_THREADS, KK_SMEM, st>>>(M, N, K, n->err, A, B, ep);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

// forward pass of the rows in xb; `last` is the output layer's epilogue
static int mlp_forward_fused(kin_mlp *n, int64_t M, cudaStream_t st, bool keep, Epilogue last) {
  for (int l = 0; l < LAYERS; ++l) {
    Epilogue ep{};
    if (l == LAYERS - 1) {
      ep = last;
    } else {
      ep.mode = EP_HIDDEN;
      ep.a = keep ? n->a[l] : nullptr;  // the backward pass's SiLU derivative
      ep.hb = n->hb[l];
    }
    ep.bias = n->p + n->boff[l];
    ep.dout = n->dout;
    const int rc = gemm_kk(n, st, M, n->N[l], n->K[l], l ? n->mh[l - 1] : n->mx, n->mwt[l], ep);
    if (rc) return rc;
  }
  return KIN_OK;
}

// loss and gradients of the rows in xb against targets gathered through rows
static int mlp_grad_fused(kin_mlp *n, int64_t M, const float *T, const int32_t *rows, int64_t R,
                          float *loss, cudaStream_t st) {
  KIN_CUDA_TRY(cudaMemsetAsync(loss, 0, sizeof(float), st));
  Epilogue ep{};
  ep.mode = EP_MSE;
  ep.tgt = T;
  ep.rows = rows;
  ep.nrows = R;
  ep.g = n->g;
  ep.gb = n->gb;
  ep.loss = loss;
  int rc = mlp_forward_fused(n, M, st, true, ep);
  if (rc) return rc;
  // the gradient alternates between two buffer pairs: a layer's input
  // gradient is written while its own gradient is read
  float *g = n->g, *g2 = n->dH;
  __nv_bfloat16 *gb = n->gb, *gb2 = n->gb2;
  int cur = 0;  // the buffer pair holding layer l's gradient
  for (int l = LAYERS - 1; l >= 0; --l) {
    const int K = n->K[l], N = n->N[l];
    gemm(n, st, K, N, (int)M, true, l ? n->hb[l - 1] : n->xb, 1, K, gb, N, 1,
         n->grad + n->woff[l], N, 0);
    k_colsum<<<CS_CTAS * blocks(N, 32), CS_THREADS, 0, st>>>(M, N, g, n->grad + n->boff[l]);
    if (l == 0) break;
    Epilogue e{};
    e.mode = EP_BACK;
    e.a = n->a[l - 1];
    e.g = g2;
    e.gb = gb2;
    if ((rc = gemm_kk(n, st, M, K, N, n->mg[cur][l < LAYERS - 1], n->mw[l], e))) return rc;
    cur ^= 1;
    std::swap(g, g2);
    std::swap(gb, gb2);
  }
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

// forward pass over M rows already packed in xf/xb; leaves y = hf[L-1]
static int mlp_forward_packed(kin_mlp *n, int64_t M, cudaStream_t st) {
  const bool bf = n->precision == 0;
  for (int l = 0; l < LAYERS; ++l) {
    const void *in = bf ? (l ? (const void *)n->hb[l - 1] : (const void *)n->xb)
                        : (l ? (const void *)n->hf[l - 1] : (const void *)n->xf);
    if (bf)  // B(k, n) = W[k][n] from the transposed copy (K contiguous)
      gemm(n, st, (int)M, n->N[l], n->K[l], bf, in, n->K[l], 1, n->wbt + n->woff[l], 1,
           n->K[l], n->C, n->N[l], 0);
    else
      gemm(n, st, (int)M, n->N[l], n->K[l], bf, in, n->K[l], 1, n->p + n->woff[l], n->N[l], 1,
           n->C, n->N[l], 0);
    const int act = l < LAYERS - 1;
    k_bias_act<<<blocks(M * n->N[l]), 256, 0, st>>>(M, n->N[l], n->C, n->p + n->boff[l], n->a[l],
                                                    n->hf[l], bf ? n->hb[l] : nullptr, act);
  }
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

// backward pass (after mlp_forward_packed and k_mse_grad into g/gb): grad
static int mlp_backward(kin_mlp *n, int64_t M, cudaStream_t st) {
  const bool bf = n->precision == 0;
  for (int l = LAYERS - 1; l >= 0; --l) {
    const int K = n->K[l], N = n->N[l];
    const void *hin = bf ? (l ? (const void *)n->hb[l - 1] : (const void *)n->xb)
                         : (l ? (const void *)n->hf[l - 1] : (const void *)n->xf);
    const void *gv = bf ? (const void *)n->gb : (const void *)n->g;
    // dW[i][o] = sum_b h[b][i] g[b][o]
    gemm(n, st, K, N, (int)M, bf, hin, 1, K, gv, N, 1, n->grad + n->woff[l], N, 0);
    k_colsum<<<CS_CTAS * blocks(N, 32), CS_THREADS, 0, st>>>(M, N, n->g, n->grad + n->boff[l]);
    if (l == 0) break;
    // dH[b][i] = sum_o g[b][o] W[i][o]
    const void *W = bf ? (const void *)(n->wb + n->woff[l]) : (const void *)(n->p + n->woff[l]);
    gemm(n, st, (int)M, K, N, bf, gv, N, 1, W, 1, N, n->dH, K, 0);
    k_silu_back<<<blocks(M * K), 256, 0, st>>>(M * K, n->dH, n->a[l - 1], n->g,
                                               bf ? n->gb : nullptr);
  }
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

static int mlp_pack(kin_mlp *n, const float *X, int64_t M, cudaStream_t st) {
  int rc = mlp_reserve(n, M);
  if (rc) return rc;
  k_pack_input<<<blocks(M * n->dinp), 256, 0, st>>>(M, n->din, n->dinp, X, n->xf,
                                                    n->precision == 0 ? n->xb : nullptr);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

// the rows of X (through rows, when given) as the fused path's BF16 input
static int mlp_gather(kin_mlp *n, const float *X, int64_t R, const int32_t *rows, int64_t M,
                      cudaStream_t st) {
  const int rc = mlp_reserve(n, M);
  if (rc) return rc;
  k_gather_pack<<<blocks(M * n->dinp), 256, 0, st>>>(M, n->din, n->dinp, X, R, rows, n->xb);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

static int mlp_refresh_bf16(kin_mlp *n, cudaStream_t st) {
  k_to_bf16<<<blocks(n->np), 256, 0, st>>>(n->np, n->p, n->wb);
  for (int l = 0; l < LAYERS; ++l)
    k_to_bf16_t<<<blocks((int64_t)n->K[l] * n->N[l]), 256, 0, st>>>(
        n->K[l], n->N[l], n->p + n->woff[l], n->wbt + n->woff[l]);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

extern "C" int kin_mlp_create(int32_t din, int32_t width, int32_t dout, int32_t precision,
                              uint64_t seed, kin_mlp **out) {
  if (!out || din < 1 || width < 8 || dout < 1 || din > 4096 || width > 4096 || dout > 4096 ||
      (precision != 0 && precision != 1))
    return KIN_ERR_INVALID_ARG;
  *out = nullptr;
  kin_mlp *n = new kin_mlp();
  n->din = din;
  n->dinp = (din + 15) / 16 * 16;
  n->width = width;
  n->dout = dout;
  n->doutp = (dout + 7) / 8 * 8;
  n->precision = precision;
  int64_t off = 0;
  for (int l = 0; l < LAYERS; ++l) {
    n->K[l] = l == 0 ? n->dinp : width;
    n->N[l] = l == LAYERS - 1 ? n->doutp : width;
    n->woff[l] = off;
    off += (int64_t)n->K[l] * n->N[l];
    n->boff[l] = off;
    off += n->N[l];
  }
  n->np = off;
  {  // split-K workspace: up to 64 partial tiles of the largest weight block, 64 MB at most
    int64_t big = 0;
    for (int l = 0; l < LAYERS; ++l) big = std::max<int64_t>(big, (int64_t)n->K[l] * n->N[l]);
    n->ws_floats = std::max<int64_t>(big, std::min<int64_t>(64 * big, 16ll << 20));
  }
  // He-style uniform initialisation, zero biases; padding stays zero
  std::vector<float> p(off, 0.0f);
  std::vector<unsigned char> mask(off, 0);
  std::mt19937_64 rng(seed);
  for (int l = 0; l < LAYERS; ++l) {
    const int kin_ = l == 0 ? din : width, nout = l == LAYERS - 1 ? dout : width;
    const float lim = std::sqrt(6.0f / (float)kin_);
    std::uniform_real_distribution<float> U(-lim, lim);
    for (int i = 0; i < kin_; ++i)
      for (int o = 0; o < nout; ++o) {
        p[n->woff[l] + (int64_t)i * n->N[l] + o] = U(rng);
        mask[n->woff[l] + (int64_t)i * n->N[l] + o] = 1;
      }
    for (int o = 0; o < nout; ++o) mask[n->boff[l] + o] = 1;
  }
  if (cudaMalloc(&n->p, sizeof(float) * off) != cudaSuccess ||
      cudaMalloc(&n->grad, sizeof(float) * off) != cudaSuccess ||
      cudaMalloc(&n->m, sizeof(float) * off) != cudaSuccess ||
      cudaMalloc(&n->v, sizeof(float) * off) != cudaSuccess ||
      cudaMalloc(&n->mask, off) != cudaSuccess ||
      cudaMalloc(&n->wb, sizeof(__nv_bfloat16) * off) != cudaSuccess ||
      cudaMalloc(&n->wbt, sizeof(__nv_bfloat16) * off) != cudaSuccess ||
      cudaMalloc(&n->ws, sizeof(float) * n->ws_floats) != cudaSuccess ||
      cudaMalloc(&n->loss, sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->err, sizeof(int)) != cudaSuccess) {
    (void)cudaGetLastError();
    kin_mlp_destroy(n);
    return KIN_ERR_NOMEM;
  }
  if (cudaMemcpy(n->p, p.data(), sizeof(float) * off, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(n->mask, mask.data(), off, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(n->m, 0, sizeof(float) * off) != cudaSuccess ||
      cudaMemset(n->v, 0, sizeof(float) * off) != cudaSuccess ||
      cudaMemset(n->grad, 0, sizeof(float) * off) != cudaSuccess ||
      cudaMemset(n->err, 0, sizeof(int)) != cudaSuccess ||
      cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)TC_SMEM) != cudaSuccess ||
      cudaFuncSetAttribute(k_gemm_kk, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)KK_SMEM) != cudaSuccess ||
      mlp_refresh_bf16(n, nullptr) != KIN_OK || cudaDeviceSynchronize() != cudaSuccess) {
    (void)cudaGetLastError();
    kin_mlp_destroy(n);
    return KIN_ERR_CUDA;
  }
  *out = n;
  return KIN_OK;
}

extern "C" void kin_mlp_destroy(kin_mlp *n) {
  if (!n) return;
  cudaFree(n->p);
  cudaFree(n->grad);
  cudaFree(n->m);
  cudaFree(n->v);
  cudaFree(n->mask);
  cudaFree(n->wb);
  cudaFree(n->wbt);
  cudaFree(n->ws);
  cudaFree(n->loss);
  cudaFree(n->err);
  mlp_release(n);
  delete n;
}

// parameter exchange in the unpadded layout W0 [din][w], b0, W1, b1, W2, b2, W3 [w][dout], b3
extern "C" int64_t kin_mlp_num_params(const kin_mlp *n) {
  if (!n) return -1;
  return (int64_t)n->din * n->width + n->width + 2 * ((int64_t)n->width * n->width + n->width) +
         (int64_t)n->width * n->dout + n->dout;
}

static int mlp_copy_params(kin_mlp *n, float *host, const float *dev_src, bool to_host) {
  std::vector<float> full(n->np);
  if (to_host) {
    KIN_CUDA_TRY(cudaMemcpy(full.data(), dev_src, sizeof(float) * n->np, cudaMemcpyDeviceToHost));
  } else {
    KIN_CUDA_TRY(cudaMemcpy(full.data(), n->p, sizeof(float) * n->np, cudaMemcpyDeviceToHost));
  }
  int64_t q = 0;
  for (int l = 0; l < LAYERS; ++l) {
    const int kin_ = l == 0 ? n->din : n->width, nout = l == LAYERS - 1 ? n->dout : n->width;
    for (int i = 0; i < kin_; ++i)
      for (int o = 0; o < nout; ++o) {
        float &f = full[n->woff[l] + (int64_t)i * n->N[l] + o];
        if (to_host) host[q++] = f; else f = host[q++];
      }
    for (int o = 0; o < nout; ++o) {
      float &f = full[n->boff[l] + o];
      if (to_host) host[q++] = f; else f = host[q++];
    }
  }
  if (!to_host) {
    KIN_CUDA_TRY(cudaMemcpy(n->p, full.data(), sizeof(float) * n->np, cudaMemcpyHostToDevice));
    int rc = mlp_refresh_bf16(n, nullptr);
    if (rc) return rc;
    KIN_CUDA_TRY(cudaDeviceSynchronize());
  }
  return KIN_OK;
}

extern "C" int kin_mlp_get_params(kin_mlp *n, float *host, int64_t len) {
  if (!n || !host || len != kin_mlp_num_params(n)) return KIN_ERR_INVALID_ARG;
  return mlp_copy_params(n, host, n->p, true);
}

extern "C" int kin_mlp_set_params(kin_mlp *n, const float *host, int64_t len) {
  if (!n || !host || len != kin_mlp_num_params(n)) return KIN_ERR_INVALID_ARG;
  n->step = 0;
  KIN_CUDA_TRY(cudaMemset(n->m, 0, sizeof(float) * n->np));
  KIN_CUDA_TRY(cudaMemset(n->v, 0, sizeof(float) * n->np));
  return mlp_copy_params(n, const_cast<float *>(host), nullptr, false);
}

extern "C" int kin_mlp_forward(kin_mlp *n, const float *X, float *Y, int64_t M, void *stream) {
  if (!n || M < 0 || (M > 0 && (!X || !Y))) return KIN_ERR_INVALID_ARG;
  if (M == 0) return KIN_OK;
  cudaStream_t st = (cudaStream_t)stream;
  if (mlp_fused(n)) {
    const int rc = mlp_gather(n, X, 0, nullptr, M, st);
    if (rc) return rc;
    Epilogue ep{};
    ep.mode = EP_OUT;
    ep.out = Y;
    return mlp_forward_fused(n, M, st, false, ep);
  }
  int rc = mlp_pack(n, X, M, st);
  if (rc || (rc = mlp_forward_packed(n, M, st))) return rc;
  KIN_CUDA_TRY(cudaMemcpy2DAsync(Y, sizeof(float) * n->dout, n->y, sizeof(float) * n->doutp,
                                 sizeof(float) * n->dout, M, cudaMemcpyDeviceToDevice, st));
  return KIN_OK;
}

// loss and gradients (into n->grad) of M rows, gathered through rows [M] out
// of R when given
static int mlp_loss_and_grad(kin_mlp *n, const float *X, const float *T, int64_t R,
                             const int32_t *rows, int64_t M, float *loss_out, cudaStream_t st) {
  int rc;
  if (mlp_fused(n)) {
    if ((rc = mlp_gather(n, X, R, rows, M, st))) return rc;
    return mlp_grad_fused(n, M, T, rows, R, loss_out ? loss_out : n->loss, st);
  }
  if (rows) {
    if ((rc = mlp_reserve(n, M))) return rc;
    k_gather_rows<<<blocks(M * n->din), 256, 0, st>>>(M, n->din, X, R, rows, n->xg);
    k_gather_rows<<<blocks(M * n->dout), 256, 0, st>>>(M, n->dout, T, R, rows, n->tg);
    KIN_CUDA_TRY(cudaGetLastError());
    X = n->xg;
    T = n->tg;
  }
  rc = mlp_pack(n, X, M, st);
  if (rc || (rc = mlp_forward_packed(n, M, st))) return rc;
  KIN_CUDA_TRY(cudaMemsetAsync(n->loss, 0, sizeof(float), st));
  k_mse_grad<<<blocks(M * n->doutp), 256, 0, st>>>(M, n->dout, n->doutp, n->y, T, n->g,
                                                   n->precision == 0 ? n->gb : nullptr, n->loss);
  if ((rc = mlp_backward(n, M, st))) return rc;
  if (loss_out)
    KIN_CUDA_TRY(cudaMemcpyAsync(loss_out, n->loss, sizeof(float), cudaMemcpyDeviceToDevice, st));
  return KIN_OK;
}

// gradients (unpadded layout, dev [num_params]) of the MSE loss on (X, T)
extern "C" int kin_mlp_grad(kin_mlp *n, const float *X, const float *T, int64_t M, float *grad_out,
                            float *loss_out, void *stream) {
  if (!n || M < 1 || !X || !T) return KIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = mlp_loss_and_grad(n, X, T, 0, nullptr, M, loss_out, st);
  if (rc) return rc;
  if (grad_out) {
    // gather the unpadded layout on the host side of the stream
    KIN_CUDA_TRY(cudaStreamSynchronize(st));
    int e = 0;
    KIN_CUDA_TRY(cudaMemcpy(&e, n->err, sizeof e, cudaMemcpyDeviceToHost));
    if (e) return KIN_ERR_CUDA;  // a tensor-core wait expired
    std::vector<float> full(n->np), packed(kin_mlp_num_params(n));
    KIN_CUDA_TRY(cudaMemcpy(full.data(), n->grad, sizeof(float) * n->np, cudaMemcpyDeviceToHost));
    int64_t q = 0;
    for (int l = 0; l < LAYERS; ++l) {
      const int kin_ = l == 0 ? n->din : n->width, nout = l == LAYERS - 1 ? n->dout : n->width;
      for (int i = 0; i < kin_; ++i)
        for (int o = 0; o < nout; ++o) packed[q++] = full[n->woff[l] + (int64_t)i * n->N[l] + o];
      for (int o = 0; o < nout; ++o) packed[q++] = full[n->boff[l] + o];
    }
    KIN_CUDA_TRY(cudaMemcpy(grad_out, packed.data(), sizeof(float) * q, cudaMemcpyHostToDevice));
  }
  return KIN_OK;
}

static int mlp_adam(kin_mlp *n, float lr, cudaStream_t st) {
  n->step++;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - std::pow(b1, (float)n->step), c2 = 1.0f - std::pow(b2, (float)n->step);
  LayerShapes L;
  for (int l = 0; l < LAYERS; ++l) {
    L.woff[l] = n->woff[l];
    L.K[l] = n->K[l];
    L.N[l] = n->N[l];
  }
  k_adam_refresh<<<blocks(n->np), 256, 0, st>>>(n->np, n->p, n->grad, n->m, n->v, n->mask, lr, b1,
                                                b2, 1e-8f, c1, c2, L, n->wb, n->wbt);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

// one Adam step on a minibatch (X dev [M][din], T dev [M][dout]); loss_out dev scalar or NULL
extern "C" int kin_mlp_train_step(kin_mlp *n, const float *X, const float *T, int64_t M, float lr,
                                  float *loss_out, void *stream) {
  if (!n || M < 1 || !X || !T || !(lr > 0.0f)) return KIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = mlp_loss_and_grad(n, X, T, 0, nullptr, M, loss_out, st);
  return rc ? rc : mlp_adam(n, lr, st);
}

extern "C" int kin_mlp_train_step_rows(kin_mlp *n, const float *X, const float *T, int64_t R,
                                       const int32_t *rows, int64_t M, float lr, float *loss_out,
                                       void *stream) {
  if (!n || M < 1 || R < 1 || !X || !T || !rows || !(lr > 0.0f)) return KIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = mlp_loss_and_grad(n, X, T, R, rows, M, loss_out, st);
  return rc ? rc : mlp_adam(n, lr, st);
}

extern "C" int kin_moments(const float *X, int64_t M, int32_t d, float *mean, float *stdv,
                           void *stream) {
  if (!X || M < 1 || d < 1 || !mean || !stdv) return KIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (M <= MOM_FEW)
    k_moments_few<<<blocks(d, 64), 64, 0, st>>>(M, d, X, mean, stdv);
  else
    k_moments<<<MOM_CTAS * blocks(d, MOM_COLS), MOM_THREADS, 0, st>>>(M, d, X, mean, stdv);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

static unsigned row_blocks(int64_t n) {
  return (unsigned)std::min<int64_t>((n + FEAT_ROWS - 1) / FEAT_ROWS, 152 * 8);
}

static int launch_features(int ns, const double *Y, const double *T, const double *P, int64_t n,
                           double dt, const float *mean, const float *stdv, float *X,
                           __nv_bfloat16 *xb, int ld, cudaStream_t st) {
  k_features<<<row_blocks(n), FEAT_THREADS, 0, st>>>(n, ns, Y, T, P, std::log(dt), mean, stdv, X,
                                                     xb, ld);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

extern "C" int kin_mlp_features(int32_t ns, const double *Y, const double *T, const double *P,
                                int64_t n, double dt, const float *mean, const float *stdv,
                                float *X, void *stream) {
  if (ns < 2 || n < 0 || (n > 0 && (!Y || !T || !P || !X)) || !(dt > 0.0) ||
      ((mean == nullptr) != (stdv == nullptr)))
    return KIN_ERR_INVALID_ARG;
  if (n == 0) return KIN_OK;
  return launch_features(ns, Y, T, P, n, dt, mean, stdv, X, nullptr, 0, (cudaStream_t)stream);
}

extern "C" int kin_mlp_targets(int32_t nz, const double *h, const double *z, int64_t n,
                               const float *mean, const float *stdv, float *tgt, void *stream) {
  if (nz < 1 || n < 1 || !h || !z || !tgt || ((mean == nullptr) != (stdv == nullptr)))
    return KIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (1 + nz <= TARGET_NARROW && n >= TARGET_MANY)
    k_targets_rows<<<blocks(n), 256, 0, st>>>(n, nz, h, z, mean, stdv, tgt);
  else
    k_targets<<<row_blocks(n), FEAT_THREADS, 0, st>>>(n, nz, h, z, mean, stdv, tgt);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}

extern "C" int kin_mlp_predict(kin_mlp *net, int32_t ns, const double *Y, const double *T,
                               const double *P, int64_t n, double dt, const float *in_mean,
                               const float *in_std, const float *out_mean, const float *out_std,
                               double *h0, double *z0, void *stream) {
  if (!net || n < 0 || !in_mean || !in_std || !out_mean || !out_std || net->din != 3 + ns ||
      net->din > (net->width > net->doutp ? net->width : net->doutp) ||
      net->dout != 1 + 3 * ns || (!h0 && !z0))
    return KIN_ERR_INVALID_ARG;
  if (n == 0) return KIN_OK;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = mlp_reserve(net, n);
  if (rc) return rc;
  if (mlp_fused(net)) {  // features straight into the BF16 input
    if ((rc = launch_features(ns, Y, T, P, n, dt, in_mean, in_std, nullptr, net->xb, net->dinp, st)))
      return rc;
    Epilogue ep{};
    ep.mode = EP_UNPACK;
    ep.mean = out_mean;
    ep.stdv = out_std;
    ep.dt = dt;
    ep.h0 = h0;
    ep.z0 = z0;
    return mlp_forward_fused(net, n, st, false, ep);
  }
  // features straight into the f32 input block (din <= dinp), then pack in place
  if ((rc = launch_features(ns, Y, T, P, n, dt, in_mean, in_std, net->dH, nullptr, 0, st)) ||
      (rc = mlp_pack(net, net->dH, n, st)) || (rc = mlp_forward_packed(net, n, st)))
    return rc;
  k_unpack_prediction<<<blocks(n), 256, 0, st>>>(n, net->dout, net->doutp, net->y, out_mean,
                                                 out_std, dt, h0, z0);
  KIN_CUDA_TRY(cudaGetLastError());
  return KIN_OK;
}
