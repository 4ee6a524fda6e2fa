// surrogate.cu -- kernels of the crack-map surrogate (a U-Net that maps a
// notched-plate run's inputs to its cracked-element map; see
// include/cem_surrogate.h).
//
// Activations are BF16 in NHWC layout, accumulation is FP32, weights are
// kept in FP32 (master copy, Adam state) and mirrored in BF16 for the
// tensor-core GEMMs.  The 3x3 convolution is an implicit GEMM
//   y[p, n] = sum_k A[p, k] W[n, k],  p = pixel, k = (ky, kx, c)
// on the 5th-generation tensor cores: k_conv3x3_halo keeps a tile's input in
// shared memory and reads the nine taps as shifted views; k_conv3x3_tc gathers
// its A rows from the input on the fly (the deepest layers, odd channel
// counts); k_conv3x3 does so for mma.sync m16n8k16 (cem_sg_set_gemm_path 0).
// The data gradient is the same kernel applied to the output gradient with the weights transposed and
// flipped (written by the Adam kernel); the weight gradient is a second
// implicit GEMM over pixels, split along the pixels into fixed chunks whose
// FP32 partial sums are added in chunk order (deterministic).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/cem_surrogate.h"
#include "per_device.h"

namespace {

typedef uint16_t bf16_t;  // BF16 storage

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src),
               "r"(bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

__device__ __forceinline__ void ldsm_x4(uint32_t r[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t r[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float bf2f(bf16_t v) { return __uint_as_float((uint32_t)v << 16); }
__device__ __forceinline__ bf16_t f2bf(float f) {
  __nv_bfloat16 h = __float2bfloat16_rn(f);
  return *reinterpret_cast<bf16_t *>(&h);
}

// ------------------------------------------------------------ conv 3x3
constexpr int FBM = 128, FBN = 64, FBK = 32, FST = 3, FPAD = FBK + 8;

struct ConvArgs {
  const bf16_t *x;   // [P, ldx] input pixels (channels 0..Cin-1 used)
  const bf16_t *w;   // [N, K] weights, K = 9 * Cin, k = (ky * 3 + kx) * Cin + c
  const float *bias; // [N] or null
  bf16_t *y;         // [P, ldy] output, channels yoff .. yoff + N - 1
  const bf16_t *mask;  // [P, ldm] or null: outputs where mask <= 0 are set to 0
  int B, H, W, Cin, ldx, N, K, relu, ldy, yoff, P, ldm;
};

__global__ void __launch_bounds__(256) k_conv3x3(ConvArgs a) {
  __shared__ __align__(128) bf16_t As[FST][FBM][FPAD];
  __shared__ __align__(128) bf16_t Bs[FST][FBN][FPAD];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp >> 1, wn = warp & 1;
  const int p0 = blockIdx.x * FBM, n0 = blockIdx.y * FBN;
  const int HW = a.H * a.W, cpt = a.Cin >> 3;
  const int KT = (a.K + FBK - 1) / FBK;
  // this thread's two A rows and its 8-wide k chunk
  const int kc = tid & 3;
  int rb[2], rh[2], rw[2];
  bool rok[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int p = p0 + (tid >> 2) + r * 64;
    rok[r] = p < a.P;
    const int pp = rok[r] ? p : 0;
    rb[r] = pp / HW;
    const int rem = pp - rb[r] * HW;
    rh[r] = rem / a.W;
    rw[r] = rem - rh[r] * a.W;
  }
  auto load_tile = [&](int kt, int s) {
    const int q = kt * (FBK / 8) + kc;  // 8-wide chunk of k
    const int tap = q / cpt, c0 = (q - tap * cpt) * 8;
    const int ky = tap / 3, kx = tap - ky * 3;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int hh = rh[r] + ky - 1, ww = rw[r] + kx - 1;
      const bool ok = rok[r] && tap < 9 && hh >= 0 && hh < a.H && ww >= 0 && ww < a.W;
      const bf16_t *src = ok ? a.x + ((size_t)(rb[r] * a.H + hh) * a.W + ww) * a.ldx + c0 : a.x;
      cp_async16(&As[s][(tid >> 2) + r * 64][kc * 8], src, ok ? 16 : 0);
    }
    const int n = n0 + (tid >> 2), k = kt * FBK + kc * 8;
    const bool okb = n < a.N && k < a.K;
    const bf16_t *srcb = okb ? a.w + (size_t)n * a.K + k : a.w;
    cp_async16(&Bs[s][tid >> 2][kc * 8], srcb, okb ? 16 : 0);
  };

  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;

#pragma unroll
  for (int s = 0; s < FST - 1; ++s) {
    if (s < KT) load_tile(s, s);
    cp_async_commit();
  }
  for (int kt = 0; kt < KT; ++kt) {
    cp_async_wait<FST - 2>();
    __syncthreads();
    const int nk = kt + FST - 1;
    if (nk < KT) load_tile(nk, nk % FST);
    cp_async_commit();
    const int s = kt % FST;
#pragma unroll
    for (int kk = 0; kk < FBK; kk += 16) {
      uint32_t af[2][4], bfr[2][4];
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
        ldsm_x4(af[mi], &As[s][wm * 32 + mi * 16 + (lane & 15)][kk + (lane >> 4) * 8]);
#pragma unroll
      for (int nj = 0; nj < 2; ++nj) {
        const int mat = lane >> 3, r = lane & 7;
        ldsm_x4(bfr[nj], &Bs[s][wn * 32 + nj * 16 + (mat >> 1) * 8 + r][kk + (mat & 1) * 8]);
      }
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
          mma_bf16(acc[mi][ni], af[mi], bfr[ni >> 1][(ni & 1) * 2], bfr[ni >> 1][(ni & 1) * 2 + 1]);
    }
  }
  cp_async_wait<0>();
  // epilogue: bias, ReLU, BF16 pairs
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni) {
      const int n = n0 + wn * 32 + ni * 8 + (lane & 3) * 2;
      if (n >= a.N) continue;
      const float b0 = a.bias ? a.bias[n] : 0.f, b1 = a.bias ? a.bias[n + 1] : 0.f;
#pragma unroll
      for (int hr = 0; hr < 2; ++hr) {
        const int p = p0 + wm * 32 + mi * 16 + (lane >> 2) + hr * 8;
        if (p >= a.P) continue;
        float v0 = acc[mi][ni][hr * 2] + b0, v1 = acc[mi][ni][hr * 2 + 1] + b1;
        if (a.relu) {
          v0 = fmaxf(v0, 0.f);
          v1 = fmaxf(v1, 0.f);
        }
        if (a.mask) {
          const uint32_t mk = *reinterpret_cast<const uint32_t *>(a.mask + (size_t)p * a.ldm + n);
          if (!(bf2f((bf16_t)(mk & 0xffff)) > 0.f)) v0 = 0.f;
          if (!(bf2f((bf16_t)(mk >> 16)) > 0.f)) v1 = 0.f;
        }
        const uint32_t pk = (uint32_t)f2bf(v0) | ((uint32_t)f2bf(v1) << 16);
        *reinterpret_cast<uint32_t *>(a.y + (size_t)p * a.ldy + a.yoff + n) = pk;
      }
    }
}

// ------------------------------------------------ conv 3x3 on tcgen05
// The same implicit GEMM on the 5th-generation tensor cores: a CTA of four
// warps owns 128 pixels x BN channels; K advances 64 at a time (one 128-byte
// swizzle atom of BF16).  Operands are gathered with 16-byte cp.async copies
// straight into the K-major 128-byte-swizzled layout the MMA descriptors
// describe (row r of a tile at r * 128 bytes, its 16-byte chunk c at
// chunk position c ^ (r & 7)), in a 2-stage ring: one stage is copied
// while the MMAs read the other, and the small ring lets two to five CTAs
// share an SM (by BN), which hides the gathers better than a deeper ring
// (4 stages: 29.7 ms per training step, 3: 23.5 ms, 2: 21.3 ms).  One thread issues
// tcgen05.mma (M = 128, N = BN, K = 16 each) into a TMEM accumulator of BN
// FP32 columns; tcgen05.commit arrives on the stage's mbarrier when the MMAs
// reading it are done, which frees the stage for the next copies.  The
// epilogue reads TMEM with tcgen05.ld (warp w: rows 32w .. 32w+31).  Every
// mbarrier wait is bounded; a wait that gives up records a timeout
// (cem_sg_timeouts), and the CTA stops issuing work, waits (bounded) for the
// MMAs already issued, and frees its TMEM only once they are done.
constexpr int TCM = 128, TCK = 64, TCS = 2;
constexpr long TC_SPIN = 1L << 24;  // mbarrier polls (with a short sleep) before a wait gives up

__device__ int g_tc_timeouts;  // waits that gave up (device-wide, cumulative)

__device__ __forceinline__ void mbar_init(uint64_t *bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count));
}
// true when the barrier's phase with the given parity has completed
// (non-blocking test)
__device__ __forceinline__ bool mbar_test(uint64_t *bar, int parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity));
  return ok != 0;
}
// bounded wait: about a second at most, then false
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, int parity) {
  for (long i = 0; i < TC_SPIN; ++i) {
    if (mbar_test(bar, parity)) return true;
    if (i > 64) __nanosleep(32);
  }
  return false;
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);       // start address
  d |= (uint64_t)1 << 16;                          // leading byte offset (unused here)
  d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset
  d |= (uint64_t)1 << 46;                          // descriptor version
  d |= (uint64_t)2 << 61;                          // 128-byte swizzle
  return d;
}

// instruction descriptor: D FP32, A and B BF16, both K-major, M x N
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

template <int BN>
struct TcSmem {
  uint8_t A[TCS][TCM * 128];
  uint8_t B[TCS][BN * 128];
  uint64_t mma_bar[TCS];
  uint32_t tmem;
  int fail;
};
// the epilogue stages a 128 x (BN + 8) BF16 tile over the operand ring
static_assert(TCM * (32 + 8) * 2 <= TCS * TCM * 128 + TCS * 32 * 128, "staging");
static_assert(TCM * (256 + 8) * 2 <= TCS * TCM * 128 + TCS * 256 * 128, "staging");

template <int BN>
__global__ void __launch_bounds__(128, 1) k_conv3x3_tc(ConvArgs a) {
  extern __shared__ uint8_t tc_raw[];
  TcSmem<BN> &T = *reinterpret_cast<TcSmem<BN> *>(
      (reinterpret_cast<uintptr_t>(tc_raw) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p0 = blockIdx.x * TCM, n0 = blockIdx.y * BN;
  const int HW = a.H * a.W, cpt = a.Cin >> 3;
  const int KB = (a.K + TCK - 1) / TCK;
  const int c = tid & 7;  // this thread's 16-byte chunk column in every tile row

  if (tid == 0) {
    for (int s = 0; s < TCS; ++s) mbar_init(&T.mma_bar[s], 1);
    T.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&T.tmem)),
                 "r"(BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  const uint32_t tmem = T.tmem;

  // rows of A this thread copies: (tid >> 3) + 16 i, i < 8
  int rh[8], rw[8], rb[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int p = p0 + (tid >> 3) + 16 * i;
    if (p < a.P) {
      rb[i] = p / HW;
      const int rem = p - rb[i] * HW;
      rh[i] = rem / a.W;
      rw[i] = rem - rh[i] * a.W;
    } else {
      rb[i] = -1; rh[i] = 0; rw[i] = 0;
    }
  }
  auto load_stage = [&](int kb, int s) {
    const int q = kb * (TCK / 8) + c;  // 8-wide k chunk
    const int tap = q / cpt, c0 = (q - tap * cpt) * 8;
    const int ky = tap / 3, kx = tap - ky * 3;
    const uint32_t abase = smem_u32(T.A[s]), bbase = smem_u32(T.B[s]);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = (tid >> 3) + 16 * i;
      const int hh = rh[i] + ky - 1, ww = rw[i] + kx - 1;
      const bool ok = rb[i] >= 0 && tap < 9 && hh >= 0 && hh < a.H && ww >= 0 && ww < a.W;
      const bf16_t *src = ok ? a.x + ((size_t)(rb[i] * a.H + hh) * a.W + ww) * a.ldx + c0 : a.x;
      const uint32_t dst = abase + row * 128 + ((c ^ (row & 7)) << 4);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                   "r"(ok ? 16 : 0));
    }
    const int k = kb * TCK + c * 8;
#pragma unroll
    for (int i = 0; i < BN / 16; ++i) {
      const int row = (tid >> 3) + 16 * i;
      const int n = n0 + row;
      const bool ok = n < a.N && k < a.K;
      const bf16_t *src = ok ? a.w + (size_t)n * a.K + k : a.w;
      const uint32_t dst = bbase + row * 128 + ((c ^ (row & 7)) << 4);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                   "r"(ok ? 16 : 0));
    }
  };

  constexpr uint32_t idesc = tc_idesc(TCM, BN);
  bool failed = false;
  int last_kb = -1;  // the last stage whose MMAs were issued
#pragma unroll
  for (int s = 0; s < TCS - 1; ++s) {
    if (s < KB) load_stage(s, s);
    cp_async_commit();
  }
  for (int kb = 0; kb < KB && !failed; ++kb) {
    const int s = kb % TCS;
    cp_async_wait<TCS - 2>();
    asm volatile("fence.proxy.async.shared::cta;\n" ::);
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
      const uint64_t ad = sw128_desc(smem_u32(T.A[s])), bd = sw128_desc(smem_u32(T.B[s]));
#pragma unroll
      for (int k = 0; k < TCK / 16; ++k) {
        const uint32_t acc = (kb > 0 || k > 0) ? 1u : 0u;
        // +32 bytes (encoded +2) per K = 16 slice inside the swizzle atom
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(ad + 2 * k), "l"(bd + 2 * k), "r"(idesc), "r"(acc));
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
          smem_u32(&T.mma_bar[s])));
    }
    last_kb = kb;
    const int nk = kb + TCS - 1;
    if (nk < KB) {
      if (kb >= 1 && !mbar_wait(&T.mma_bar[(kb - 1) % TCS], ((kb - 1) / TCS) & 1)) {
        failed = true;
        T.fail = 1;
      }
      if (!failed) load_stage(nk, nk % TCS);
    }
    cp_async_commit();
    failed = __syncthreads_or(failed) != 0;
  }
  cp_async_wait<0>();
  // all MMAs done: the last commit tracks every earlier one
  if (!failed && !mbar_wait(&T.mma_bar[(KB - 1) % TCS], ((KB - 1) / TCS) & 1)) failed = true;
  failed = __syncthreads_or(failed) != 0;
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);

  if (!failed) {
    // TMEM -> (bias, ReLU) -> BF16 tile in shared memory (the operand ring is
    // free now), then coalesced 16-byte stores with the mask applied
    constexpr int LDS = BN + 8;  // padded row of the staged tile (bf16)
    bf16_t *stile = reinterpret_cast<bf16_t *>(T.A[0]);
    const int m = warp * 32 + lane;  // TMEM lane = tile row
#pragma unroll 1
    for (int cb = 0; cb < BN; cb += 32) {
      uint32_t r[32];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
          "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
            "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
            "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
            "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
            "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
            "=r"(r[31])
          : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)cb));
      asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::);
#pragma unroll
      for (int j = 0; j < 32; j += 2) {
        const int n = n0 + cb + j;
        float v0 = __uint_as_float(r[j]), v1 = __uint_as_float(r[j + 1]);
        if (a.bias && n < a.N) {
          v0 += a.bias[n];
          v1 += a.bias[n + 1];
        }
        if (a.relu) {
          v0 = fmaxf(v0, 0.f);
          v1 = fmaxf(v1, 0.f);
        }
        *reinterpret_cast<uint32_t *>(stile + m * LDS + cb + j) =
            (uint32_t)f2bf(v0) | ((uint32_t)f2bf(v1) << 16);
      }
    }
    __syncthreads();
    const bool vec = (a.N & 7) == 0 && (a.ldy & 7) == 0 && (a.yoff & 7) == 0 &&
                     (!a.mask || (a.ldm & 7) == 0);
    for (int idx = tid; idx < TCM * (BN / 8); idx += 128) {
      const int row = idx / (BN / 8), ch = (idx - row * (BN / 8)) * 8;
      const int p = p0 + row, n = n0 + ch;
      if (p >= a.P || n >= a.N) continue;
      uint4 v = *reinterpret_cast<const uint4 *>(stile + row * LDS + ch);
      if (vec) {
        if (a.mask) {
          const uint4 mk = *reinterpret_cast<const uint4 *>(a.mask + (size_t)p * a.ldm + n);
          uint32_t *vw = reinterpret_cast<uint32_t *>(&v);
          const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (!(bf2f((bf16_t)(mw[q] & 0xffff)) > 0.f)) vw[q] &= 0xffff0000u;
            if (!(bf2f((bf16_t)(mw[q] >> 16)) > 0.f)) vw[q] &= 0x0000ffffu;
          }
        }
        *reinterpret_cast<uint4 *>(a.y + (size_t)p * a.ldy + a.yoff + n) = v;
      } else {
        const uint32_t vw[4] = {v.x, v.y, v.z, v.w};
        for (int q = 0; q < 4 && n + 2 * q < a.N; ++q) {
          uint32_t w2 = vw[q];
          if (a.mask) {
            const uint32_t mk =
                *reinterpret_cast<const uint32_t *>(a.mask + (size_t)p * a.ldm + n + 2 * q);
            if (!(bf2f((bf16_t)(mk & 0xffff)) > 0.f)) w2 &= 0xffff0000u;
            if (!(bf2f((bf16_t)(mk >> 16)) > 0.f)) w2 &= 0x0000ffffu;
          }
          *reinterpret_cast<uint32_t *>(a.y + (size_t)p * a.ldy + a.yoff + n + 2 * q) = w2;
        }
      }
    }
  } else if (tid == 0) {
    atomicAdd(&g_tc_timeouts, 1);
  }
  // After a wait gave up, MMAs may still be in flight: wait (bounded) for the
  // last issued commit, which tracks every earlier MMA, before the TMEM is
  // freed; if that wait gives up too, the CTA exits without freeing it (the
  // results of the call are invalid in either case; cem_sg_timeouts says so).
  bool drained = true;
  if (failed && last_kb >= 0)
    drained = __syncthreads_and(mbar_wait(&T.mma_bar[last_kb % TCS], (last_kb / TCS) & 1)) != 0;
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  if (warp == 0 && drained)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(BN));
}

// raises a kernel's dynamic shared-memory limit, once per device
template <class K>
cudaError_t allow_smem(K *kernel, size_t bytes, PerDevice &attrs) {
  return attrs.once([=] {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  });
}

template <int BN>
size_t tc_smem_bytes() {
  return sizeof(TcSmem<BN>) + 1024;
}

template <int BN>
cudaError_t launch_conv_tc(const ConvArgs &a, cudaStream_t st) {
  static PerDevice attrs;
  const cudaError_t ae = allow_smem(k_conv3x3_tc<BN>, tc_smem_bytes<BN>(), attrs);
  if (ae != cudaSuccess) return ae;
  dim3 grid((a.P + TCM - 1) / TCM, (a.N + BN - 1) / BN);
  k_conv3x3_tc<BN><<<grid, 128, tc_smem_bytes<BN>(), st>>>(a);
  return cudaGetLastError();
}

// ------------------------------------------- conv 3x3, resident input tile
// The implicit GEMM again, with each input pixel fetched about 1.4 times
// instead of nine: a CTA fetches the halo of an output tile once and forms the
// nine taps' A operands as shifted views of it.  The gathers of k_conv3x3_tc
// (a 16-byte copy per pixel, tap and 8 channels) bound the layers of few
// channels: 32 -> 32 channels on 64 images of 160 x 400 took 467 us there.
//
// Layout.  A stage holds the tile's input as planes of 64 (32, 16; 8 when
// there are 8) channels, one 128- (64-, 32-, 16-) byte row per pixel slot,
// swizzled by shared-memory address as TMA writes it and the MMA reads it.  A tap is a start address
// shifted by whole slots, the next 8 rows of the tile are one slot row
// further (SBO).  Three tilings:
//   whole  tiles 8 wide x 16 tall inside an image, halo 10 x 18 slots, one TMA box
//          (zero fill outside the image);
//   tall   the same tiles on all images stacked with a row of zeros between
//          two, one TMA box per slot row: images whose height is far from a
//          multiple of 16 leave no ragged rows (20 rows: 1.31 tiles an image
//          instead of 2);
//   flat   narrow images (W <= 30) as one long row with a zero after each
//          image row, 128 consecutive pixels to a tile, one TMA box per image
//          row and plane: 25 x 10 images fill 87% of the rows instead of 71%;
//   box    for more channels than a stage can hold beside a weight ring: tiles
//          bw x bh x bb pixels (wide, tall, images; at most 128, whatever covers the
//          images best), and a stage is the 64 channels of one tap, fetched anew for
//          each tap by one shifted TMA box: nine times the input's bytes, but any
//          number of channels, two tiles to a weight block and no slots beside the
//          tile (25 x 10 images fill 98% of the rows).
// The weights stay in shared memory for the whole (persistent) CTA when they
// fit, else they stream by TMA through a ring, each block serving MT tiles.
//
// Order.  Steps of 16 of k = (ky, kx, c) are accumulated in increasing k, as
// k_conv3x3_tc does: the same sums, bit for bit.
//
// Roles: warps 0-3 and 4-7 the epilogues of the two accumulator sets (TMEM
// lanes 32 (w & 3) ..), warp 8 issues the MMAs, warp 9 fetches weights, warp
// 10 input tiles.  Every wait is bounded; one that gives up raises `fail`,
// which ends the others.
//
// Measured (64 images; before with k_conv3x3_tc):
//   8 -> 32, 160 x 400    318 -> 72 us, 4.6 TB/s
//   32 -> 32, 160 x 400   467 -> 119 us, 4.4 TB/s
//   32 -> 96, 160 x 400   967 -> 192 us, 5.5 TB/s of HBM
//   64 -> 64, 80 x 200    219 -> 66 us
//   128 -> 384, 40 x 100  450 -> 134 us, 1690 TFLOP/s (0.89 of cuBLAS)
//   256 -> 256, 20 x 50   106 -> 52 us, 1460 TFLOP/s
//   768 -> 256, 20 x 50   316 -> 151 us (box)
//   512 -> 512, 10 x 25   94 -> 54 us, 1390 TFLOP/s (box; 113 with whole stages)
//   512 -> 256, 10 x 25   78 -> 33 us (box)
// One image, 256 -> 256, 20 x 50: 47 -> 12 us; 768 -> 256: 105 -> 37 us (box).
// Programmatic dependents: the kernels of a forward pass are short (a single
// image: 4 to 37 us, 30 of them), so each is placed while the one before it
// still runs, sets up its barriers and tensor memory, and waits for that
// kernel's results (dependency_wait) before it touches any global memory.  It
// lets its own successor be placed only when it holds its tensor memory, so
// that no two kernels can wait for each other's columns.  A forward pass of one
// image: 275 -> 225 us.
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void dependency_release() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

constexpr int HB_THREADS = 352, HB_MAXW = 48, HB_MAXA = 8;

enum : int { TILE_WHOLE = 0, TILE_TALL = 1, TILE_FLAT = 2, TILE_BOX = 3 };

struct HaloArgs {
  const float *bias;
  bf16_t *y;
  const bf16_t *mask;
  int B, H, W, N, relu, ldy, yoff, ldm;
  int mode;             // TILE_*
  int planes;           // of a stage (box: of the input)
  int cps;              // stages of a tile (box: one for each 64 of k)
  int bw, bh, bb;       // box: pixels of a tile
  uint32_t inv_bw, inv_bp;  // ceil(2^32 / bw), / (bw bh)
  int ky_st, ps, sbo;   // strides of a tap row, a plane and 8 tile rows (bytes)
  int a_bytes, a_tx;    // a stage's size; the bytes its copies bring in
  int nrows;            // flat: image rows a stage holds
  int tiles_x, tiles_y, tiles;  // sub-tiles of 128 pixels (whole: tiles_y per image)
  uint32_t inv_h, inv_w, inv_x, inv_y;  // ceil(2^32 / (H+1), / (W+1), / tiles_x, / tiles_y)
  int nblk, nb, nbp;    // output-channel blocks, channels of one (its TMEM columns)
  int kblocks;          // 64-wide steps of k
  int na, nw;           // input stages, weight stages
  int nacc;             // accumulator sets
  int cols;             // TMEM columns allocated
  int vec;              // bytes of a row access to y and mask: 32, 16 or 4
  int off_ctl;          // shared-memory offset of HaloCtl
};

struct HaloCtl {
  float bias[256];
  uint64_t a_full[HB_MAXA], a_empty[HB_MAXA], w_full[HB_MAXW], w_empty[HB_MAXW], acc_full[2], acc_empty[2];
  uint64_t drain;
  uint32_t tmem;
  int fail;
};

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
// one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
// Bounded wait (about a second) that also ends when another role has failed;
// the waiting warp is suspended between tries, so that it takes no issue slots
// from the others.
constexpr int ROLE_TRIES = 1 << 20;
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n"
      " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(1000u)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool thread_wait(uint64_t *bar, uint32_t parity, int *fail) {
  for (int i = 0; i < ROLE_TRIES; ++i) {
    if (mbar_try(bar, parity)) return true;
    if (*(volatile int *)fail) return false;
  }
  *(volatile int *)fail = 1;
  return false;
}
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, int *fail) {
  for (int i = 0; i < ROLE_TRIES; ++i) {
    if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
    if (__any_sync(0xffffffffu, *(volatile int *)fail)) return false;
  }
  *(volatile int *)fail = 1;
  return false;
}
// one MMA of 128 x N x 16 (a single thread issues it); acc = 0 overwrites
__device__ __forceinline__ void tc_mma(uint32_t tmem, uint32_t alo, uint32_t ahi, uint32_t blo,
                                       uint32_t bhi, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %6, 0;\n"
      " mov.b64 da, {%1, %2};\n mov.b64 db, {%3, %4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(tmem),
      "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                   smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t r[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
}
__device__ __forceinline__ void ld_row32(const void *p, uint32_t r[8]) {
  asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "l"(p));
}
__device__ __forceinline__ void st_row32(void *p, const uint32_t r[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(p), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// a pair of BF16 outputs set to zero where its mask values are not positive
__device__ __forceinline__ uint32_t mask_pair(uint32_t v, uint32_t mk) {
  if (!(bf2f((bf16_t)(mk & 0xffff)) > 0.f)) v &= 0xffff0000u;
  if (!(bf2f((bf16_t)(mk >> 16)) > 0.f)) v &= 0x0000ffffu;
  return v;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ void tma_load5(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2,
                                          int c3, int c4, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], "
      "[%1, {%2, %3, %4, %5, %6}], [%7];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4),
      "r"(smem_u32(bar))
      : "memory");
}

// n / d by its reciprocal ceil(2^32 / d): exact while n d < 2^32 (the host checks)
__device__ __forceinline__ int div_by(int n, uint32_t inv) { return (int)__umulhi((uint32_t)n, inv); }

// output pixel of row m of a sub-tile, or -1 outside the images
__device__ __forceinline__ int halo_pixel(const HaloArgs &a, int tile, int m) {
  int b, h, c;
  if (a.mode == TILE_BOX) {
    // divisors of 1 have no reciprocal
    const int n = a.bw * a.bh, i = n == 1 ? m : div_by(m, a.inv_bp), k = m - i * n;
    const int r = a.bw == 1 ? k : div_by(k, a.inv_bw);
    const int ty = a.tiles_x == 1 ? tile : div_by(tile, a.inv_x);
    const int tb = a.tiles_y == 1 ? ty : div_by(ty, a.inv_y);
    c = (tile - ty * a.tiles_x) * a.bw + k - r * a.bw;
    h = (ty - tb * a.tiles_y) * a.bh + r;
    b = tb * a.bb + i;
    if (i >= a.bb) return -1;
  } else if (a.mode == TILE_FLAT) {
    const int q = a.W + 1 + tile * 128 + m, T = div_by(q, a.inv_w);
    c = q - T * (a.W + 1);
    b = div_by(T, a.inv_h);
    h = T - b * (a.H + 1) - 1;
  } else {
    const int ty = a.tiles_x == 1 ? tile : div_by(tile, a.inv_x);
    c = (tile - ty * a.tiles_x) * 8 + (m & 7);
    if (a.mode == TILE_WHOLE) {
      b = a.tiles_y == 1 ? ty : div_by(ty, a.inv_y);
      h = (ty - b * a.tiles_y) * 16 + (m >> 3);
    } else {
      const int T = 1 + ty * 16 + (m >> 3);
      b = div_by(T, a.inv_h);
      h = T - b * (a.H + 1) - 1;
    }
  }
  return h >= 0 && h < a.H && b < a.B && c < a.W ? (b * a.H + h) * a.W + c : -1;
}
// flat: position of the halo's first slot in the stage (the stage starts with a whole image row)
__device__ __forceinline__ int flat_first(const HaloArgs &a, int tile, int &row) {
  const int q = tile * 128 - 1;
  row = q < 0 ? -1 : div_by(q, a.inv_w);
  return q - row * (a.W + 1);
}

// RB: bytes of a slot's row in a plane.  PL > 0: the stage's planes, known at
// compile time with the tiling (MODE: WHOLE or TALL), and a tile's steps are
// straight-line code with constant offsets; the issue of a step then costs about
// 30 clocks, less than its MMA, against 65 with the offsets walked (PL = 0).
template <int RB, int MT, bool RES, int PL, int MODE>
__global__ void __launch_bounds__(HB_THREADS, 1)
    k_conv3x3_halo(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap xmap,
                   const HaloArgs a) {
  extern __shared__ uint8_t hb_raw[];
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(hb_raw) + 1023) &
                                              ~(uintptr_t)1023);
  HaloCtl &C = *reinterpret_cast<HaloCtl *>(base + a.off_ctl);
  // weight blocks first, then the input stages (both 1024-byte aligned)
  uint8_t *sw = base, *sa = base + (size_t)a.nw * a.nb * 128;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int nbi = blockIdx.x % a.nblk, n0 = nbi * a.nb;
  const int step = gridDim.x / a.nblk, g0 = blockIdx.x / a.nblk;
  const int groups = (a.tiles + MT - 1) / MT;  // a group: MT sub-tiles

  if (tid == 0) {
    for (int s = 0; s < a.na; ++s) {
      mbar_init(&C.a_full[s], 1);
      mbar_init(&C.a_empty[s], 1);
    }
    for (int s = 0; s < a.nw; ++s) {
      mbar_init(&C.w_full[s], 1);
      mbar_init(&C.w_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&C.acc_full[s], 1);
      mbar_init(&C.acc_empty[s], 128);
    }
    mbar_init(&C.drain, 1);
    C.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&C.tmem)),
                 "r"(a.cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  dependency_wait();
  if (a.bias)
    for (int q = tid; q < a.nb; q += HB_THREADS) C.bias[q] = n0 + q < a.N ? a.bias[n0 + q] : 0.f;
  if (RB == 16) {  // the zero half of the last step: a second plane that no copy writes
    for (int q = tid; q < a.na * MT * 180; q += HB_THREADS)
      *reinterpret_cast<uint4 *>(sa + (size_t)(q / 180) * a.a_bytes + a.ps + (q % 180) * 16) =
          make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  dependency_release();
  const uint32_t tmem = __shfl_sync(0xffffffffu, C.tmem, 0);

  if (warp == 10) {
    // ---- input tiles; the boxes of a tile are issued side by side, one per lane
    int s = 0, ph = 1, it = 0;
    bool ok = true;
    for (int g = g0; g < groups && ok; g += step) {
      int tap = 0, pl = 0;  // of the stage (box)
      for (int cp = 0; cp < a.cps; ++cp, ++it) {
        ok = warp_wait(&C.a_empty[s], ph, &C.fail);
        if (!ok) break;
        if (lane == 0) mbar_expect(&C.a_full[s], (uint32_t)(MT * a.a_tx));
        __syncwarp();
        for (int m = 0; m < MT; ++m) {
          const int tile = g * MT + m;  // one past the last: rows outside the images, all zeros
          const uint32_t dst = smem_u32(sa) + (uint32_t)((s * MT + m) * a.a_bytes);
          if (MODE == TILE_BOX) {
            const int ty = a.tiles_x == 1 ? tile : div_by(tile, a.inv_x);
            const int tb = a.tiles_y == 1 ? ty : div_by(ty, a.inv_y);
            if (lane == 0)
              tma_load5(dst, &xmap, 0, (tile - ty * a.tiles_x) * a.bw + tap % 3 - 1,
                        (ty - tb * a.tiles_y) * a.bh + tap / 3 - 1, tb * a.bb, pl, &C.a_full[s]);
          } else if (a.mode == TILE_FLAT) {
            int row;
            flat_first(a, tile, row);
            for (int q = lane; q < a.nrows * a.planes; q += 32) {
              const int r = q / a.planes, p = q - r * a.planes;
              const int T = row + r, b = T < 0 ? 0 : div_by(T, a.inv_h);
              const int h = T < 0 ? -1 : T - b * (a.H + 1) - 1;
              tma_load5(dst + p * a.ps + r * (a.W + 1) * RB, &xmap, 0, 0, h, b, p, &C.a_full[s]);
            }
          } else {
            const int ty = a.tiles_x == 1 ? tile : div_by(tile, a.inv_x);
            const int c = (tile - ty * a.tiles_x) * 8 - 1;
            if (a.mode == TILE_WHOLE) {
              const int b = a.tiles_y == 1 ? ty : div_by(ty, a.inv_y);
              if (lane == 0)
                tma_load5(dst, &xmap, 0, c, (ty - b * a.tiles_y) * 16 - 1, b, 0, &C.a_full[s]);
            } else if (lane < 18) {
              const int T = ty * 16 + lane, b = div_by(T, a.inv_h);
              tma_load5(dst + lane * a.ky_st, &xmap, 0, c, T - b * (a.H + 1) - 1, b, 0, &C.a_full[s]);
            }
          }
        }
        if (++pl == a.planes) {
          pl = 0;
          ++tap;
        }
        if (++s == a.na) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    // no copy outlives the CTA: wait for those of the last na stages (bounded)
    for (int q = max(0, it - a.na); q < it; ++q) mbar_wait(&C.a_full[q % a.na], (q / a.na) & 1);
  } else if (warp == 9) {
    // ---- weights
    if (elect_one()) {
      const uint32_t bytes = (uint32_t)a.nb * 128;
      const int mine = g0 < groups ? (groups - 1 - g0) / step + 1 : 0;
      const int total = RES ? (mine ? a.kblocks : 0) : mine * a.kblocks;
      int s = 0, ph = 1, kb = 0, q = 0;
      for (; q < total; ++q) {
        if (!RES && !thread_wait(&C.w_empty[s], ph, &C.fail)) break;
        mbar_expect(&C.w_full[s], bytes);
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], "
            "[%1, {%2, %3}], [%4];\n" ::"r"(smem_u32(sw) + (uint32_t)s * bytes),
            "l"(reinterpret_cast<uint64_t>(&wmap)), "r"(kb * 64), "r"(n0), "r"(smem_u32(&C.w_full[s]))
            : "memory");
        if (++kb == a.kblocks) kb = 0;
        if (++s == a.nw) {
          s = 0;
          ph ^= 1;
        }
      }
      for (int p = max(0, q - a.nw); p < q; ++p) mbar_wait(&C.w_full[p % a.nw], (p / a.nw) & 1);
    }
  } else if (warp == 8) {
    // ---- MMAs, issued by one elected lane; a weight block's four steps are
    // straight-line code, or their issue would cost several times the MMA
    if (elect_one()) {
      const uint32_t idesc = tc_idesc(128, a.nb);
      // SBO, descriptor version, swizzle of 128-, 64- or 32-byte rows (none of 16-byte rows)
      const uint32_t ahi = (uint32_t)(a.sbo >> 4) | (1u << 14) |
                           ((RB == 128 ? 2u : RB == 64 ? 4u : RB == 32 ? 6u : 0u) << 29);
      const uint32_t whi = (uint32_t)(sw128_desc(0) >> 32), wlo0 = (uint32_t)sw128_desc(smem_u32(sw));
      const uint32_t sa0 = (smem_u32(sa) >> 4) | (RB == 16 ? 0u : 1u << 16), stage = (uint32_t)a.a_bytes >> 4;
      const uint32_t ps = (uint32_t)a.ps >> 4, wst = (uint32_t)a.nb * 8;  // in units of 16 bytes
      constexpr int ROWS = 128 / RB, PER = RB == 16 ? 1 : RB / 32;  // rows of a weight block, steps of a row
      const uint32_t ky_next = (uint32_t)((a.ky_st - 2 * RB) >> 4);  // from tap kx = 2 to the next row's 0
      int s = 0, sph = 0, ab = 0, abph = 1, ws = 0, wph = 0;
      bool ok = true;
      if (RES && g0 < groups)
        for (int kb = 0; kb < a.kblocks && ok; ++kb) ok = thread_wait(&C.w_full[kb], 0, &C.fail);
      for (int g = g0; g < groups && ok; g += step) {
        if (!thread_wait(&C.acc_empty[ab], abph, &C.fail)) break;
        if constexpr (MODE == TILE_BOX) {
          // a stage and a weight block for each 64 of k
          const uint32_t d0 = tmem + (uint32_t)(ab * MT * a.nbp);
          for (int kb = 0; kb < a.kblocks; ++kb) {
            ok = thread_wait(&C.a_full[s], sph, &C.fail) && thread_wait(&C.w_full[ws], wph, &C.fail);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t wd = wlo0 + (uint32_t)ws * wst, ad = sa0 + (uint32_t)(s * MT) * stage;
#pragma unroll
            for (int i = 0; i < PER; ++i)
#pragma unroll
              for (int m = 0; m < MT; ++m)
                tc_mma(d0 + m * a.nbp, ad + m * stage + 2 * i, ahi, wd + 2 * i, whi, idesc, i ? 1u : (uint32_t)(kb > 0));
            tc_commit(&C.w_empty[ws]);
            tc_commit(&C.a_empty[s]);
            if (++ws == a.nw) {
              ws = 0;
              wph ^= 1;
            }
            if (++s == a.na) {
              s = 0;
              sph ^= 1;
            }
          }
          if (!ok) break;
          tc_commit(&C.acc_full[ab]);
          if (++ab == a.nacc) {
            ab = 0;
            abph ^= 1;
          }
          continue;
        }
        if (!thread_wait(&C.a_full[s], sph, &C.fail)) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        uint32_t tap[MT], row[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          tap[m] = sa0 + (uint32_t)(s * MT + m) * stage;
          if (PL == 0 && a.mode == TILE_FLAT) {
            int r;
            tap[m] += (uint32_t)(flat_first(a, g * MT + m, r) * (RB / 16));
          }
          row[m] = tap[m];
        }
        const uint32_t d0 = tmem + (uint32_t)(ab * MT * a.nbp);
        auto w_next = [&]() {  // the ring's next block
          tc_commit(&C.w_empty[ws]);
          if (++ws == a.nw) {
            ws = 0;
            wph ^= 1;
          }
        };
        if constexpr (RB == 16) {
          // 8 channels: taps 2 q and 2 q + 1 are the halves of step q (LBO apart), the
          // zero plane the second half of the last
#pragma unroll
          for (int q = 0; q < 5; ++q) {
            const int t0 = 2 * q, t1 = t0 + 1;
            const uint32_t o0 = (uint32_t)((t0 / 3) * 10 + t0 % 3);
            const uint32_t o1 = t1 < 9 ? (uint32_t)((t1 / 3) * 10 + t1 % 3) : 180u;
            if (!RES && (q & 3) == 0 && !(ok = thread_wait(&C.w_full[ws], wph, &C.fail))) break;
            const uint32_t wd = wlo0 + (uint32_t)(RES ? q >> 2 : ws) * wst + 2 * (q & 3);
#pragma unroll
            for (int m = 0; m < MT; ++m)
              tc_mma(d0 + m * a.nbp, (tap[m] + o0) | ((o1 - o0) << 16), ahi, wd, whi, idesc, q > 0);
            if (!RES && ((q & 3) == 3 || q == 4)) w_next();
          }
        } else if constexpr (PL > 0) {
          constexpr int PS = (MODE == TILE_TALL ? 10 : 180) * RB / 16, KY = (MODE == TILE_TALL ? PL * 10 : 10) * RB / 16;
          constexpr int STEPS = 9 * PL * PER;
          uint32_t wd = wlo0;
#pragma unroll
          for (int k = 0; k < STEPS; ++k) {
            const int i = k % PER, r = k / PER, p = r % PL, t = r / PL;
            const uint32_t o = (uint32_t)((t / 3) * KY + (t % 3) * (RB / 16) + p * PS + 2 * i);
            if (k % 4 == 0) {
              if (RES) {
                if (k) wd += wst;
              } else {
                if (!(ok = thread_wait(&C.w_full[ws], wph, &C.fail))) break;
                wd = wlo0 + (uint32_t)ws * wst;
              }
            }
#pragma unroll
            for (int m = 0; m < MT; ++m)
              tc_mma(d0 + m * a.nbp, tap[m] + o, ahi, wd + 2 * (k % 4), whi, idesc, k > 0);
            if (!RES && (k % 4 == 3 || k == STEPS - 1)) w_next();
          }
        } else {
          int pl = 0, kx = 0, left = 9 * a.planes;
          for (int kb = 0; kb < a.kblocks; ++kb) {
            if (!RES && !(ok = thread_wait(&C.w_full[ws], wph, &C.fail))) break;
            const uint32_t wd = wlo0 + (uint32_t)(RES ? kb : ws) * wst;
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
              if (ROWS == 1 || left > 0) {
#pragma unroll
                for (int i = 0; i < PER; ++i)
#pragma unroll
                  for (int m = 0; m < MT; ++m)
                    tc_mma(d0 + m * a.nbp, row[m] + 2 * i, ahi, wd + 2 * (r * PER + i), whi, idesc,
                           (r || i) ? 1u : (uint32_t)(kb > 0));
                --left;
                uint32_t adv = ps;
                if (++pl == a.planes) {
                  pl = 0;
                  uint32_t t = RB / 16;
                  if (++kx == 3) {
                    kx = 0;
                    t = ky_next;
                  }
#pragma unroll
                  for (int m = 0; m < MT; ++m) row[m] = tap[m] = tap[m] + t;
                  adv = 0;
                }
#pragma unroll
                for (int m = 0; m < MT; ++m) row[m] += adv;
              }
            }
            if (!RES) w_next();
          }
        }
        if (!ok) break;
        tc_commit(&C.a_empty[s]);
        tc_commit(&C.acc_full[ab]);
        if (++s == a.na) {
          s = 0;
          sph ^= 1;
        }
        if (++ab == a.nacc) {
          ab = 0;
          abph ^= 1;
        }
      }
      // every MMA issued has completed before the CTA's memory is given back
      tc_commit(&C.drain);
      if (!mbar_wait(&C.drain, 0)) *(volatile int *)&C.fail = 2;
    }
  } else {
    // ---- epilogue: bias, ReLU, mask, BF16; each group of four warps has its own
    // accumulator set and takes every second tile group (all, with one set)
    const int e = warp >> 2, w4 = warp & 3;
    const int mrow = w4 * 32 + lane;
    uint32_t ph = 0;
    if (e < a.nacc)
      for (int g = g0 + e * step; g < groups; g += a.nacc * step, ph ^= 1) {
        int pix[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m)
          pix[m] = g * MT + m < a.tiles ? halo_pixel(a, g * MT + m, mrow) : -1;
        if (!warp_wait(&C.acc_full[e], ph, &C.fail)) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          const int p = pix[m];
#pragma unroll 1
          for (int cb = 0; cb < a.nb; cb += 32) {
            uint32_t r[32], o[16];
            __syncwarp();
            tmem_ld32(tmem + ((uint32_t)(w4 * 32) << 16) + (uint32_t)((e * MT + m) * a.nbp + cb), r);
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            if (m == MT - 1 && cb + 32 >= a.nb) {
              asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
              mbar_arrive(&C.acc_empty[e]);
            }
            if (p < 0) continue;
            if (a.bias) {
              const float4 *bp = reinterpret_cast<const float4 *>(C.bias + cb);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float4 b4 = bp[j];
                r[4 * j] = __float_as_uint(__uint_as_float(r[4 * j]) + b4.x);
                r[4 * j + 1] = __float_as_uint(__uint_as_float(r[4 * j + 1]) + b4.y);
                r[4 * j + 2] = __float_as_uint(__uint_as_float(r[4 * j + 2]) + b4.z);
                r[4 * j + 3] = __float_as_uint(__uint_as_float(r[4 * j + 3]) + b4.w);
              }
            }
            if (a.relu) {
#pragma unroll
              for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(fmaxf(__uint_as_float(r[j]), 0.f));
            }
#pragma unroll
            for (int j = 0; j < 16; ++j)
              o[j] = pack_bf16(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
            bf16_t *yp = a.y + (size_t)p * a.ldy + a.yoff + n0 + cb;
            const bf16_t *mp = a.mask + (size_t)p * a.ldm + n0 + cb;
            // channels of this block left from here
            const int left = min(min(a.nb, a.N - n0) - cb, 32);
            if (a.vec == 32) {
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                if (16 * q >= left) continue;
                if (a.mask) {
                  uint32_t mk[8];
                  ld_row32(mp + 16 * q, mk);
#pragma unroll
                  for (int t = 0; t < 8; ++t) o[8 * q + t] = mask_pair(o[8 * q + t], mk[t]);
                }
                st_row32(yp + 16 * q, o + 8 * q);
              }
            } else if (a.vec == 16) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                if (8 * q >= left) continue;
                uint4 v = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
                if (a.mask) {
                  const uint4 mk = *reinterpret_cast<const uint4 *>(mp + 8 * q);
                  v = make_uint4(mask_pair(v.x, mk.x), mask_pair(v.y, mk.y), mask_pair(v.z, mk.z),
                                 mask_pair(v.w, mk.w));
                }
                *reinterpret_cast<uint4 *>(yp + 8 * q) = v;
              }
            } else {
#pragma unroll
              for (int q = 0; q < 16; ++q) {
                if (2 * q >= left) continue;
                uint32_t v = o[q];
                if (a.mask) v = mask_pair(v, *reinterpret_cast<const uint32_t *>(mp + 2 * q));
                *reinterpret_cast<uint32_t *>(yp + 2 * q) = v;
              }
            }
          }
        }
      }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (tid == 0 && C.fail) atomicAdd(&g_tc_timeouts, 1);
  // TMEM is freed unless MMAs may still be in flight (the drain gave up)
  if (warp == 8 && C.fail != 2)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(a.cols));
}

// ---- plan of one call
constexpr int kSms = 152;
constexpr size_t kSmemMax = 232448;  // 227 KB a CTA

struct HaloPlan {
  HaloArgs a;
  int rb, mt, res, grid, box_w, box_h, box_b, box_p;
  size_t smem;
};

// Chooses the tiling, the channel blocks (nblk), the tiles per weight block
// (mt), the input stages (na) and whether the weights stay (res), by an
// estimate in clocks: an MMA of 128 x nb x 16 takes nb / 2 of them, or 58 + nb / 5
// (measured: reading its operands), a tile group 350 besides; an SM draws
// about 45 bytes per clock from L2, a ring no more than it holds in 2000 clocks
// (the latency under load).  Few tiles (a single image's deep levels) come out with
// many narrow channel blocks, so that the K loop runs on more SMs.  False when
// no plan fits (channels that are neither 8 nor a multiple of 16, or more than a
// stage holds and no multiple of 64): k_conv3x3_tc takes those.
bool halo_plan(const ConvArgs &v, HaloPlan &best) {
  if ((v.Cin & 15) && v.Cin != 8) return false;
  const int rb = !(v.Cin & 63) ? 128 : !(v.Cin & 31) ? 64 : !(v.Cin & 15) ? 32 : 16;
  auto up = [](long n, long d) { return (n + d - 1) / d; };
  auto inv = [](long d) { return (uint32_t)(((1ull << 32) + d - 1) / d); };
  const long rows = (long)v.B * (v.H + 1) - 1;  // of the tall image
  const int kblocks = (v.K + 63) / 64;
  const size_t fixed = 1024 + 128 + sizeof(HaloCtl);
  double best_c = 0.0;
  bool found = false;
  for (int mode : {TILE_WHOLE, TILE_TALL, TILE_FLAT, TILE_BOX}) {
    HaloArgs a{};
    a.mode = mode;
    a.planes = v.Cin * 2 / rb;
    a.kblocks = kblocks;
    a.cps = 1;
    a.tiles_x = (int)up(v.W, 8);
    a.tiles_y = (int)up(v.H, 16);
    long tiles;
    if (mode == TILE_BOX) {
      if (rb != 128) continue;
      // the widths' best cover of the images by at most 128 pixels
      tiles = 0;
      for (int bw = 1; bw <= std::min(v.W, 128); ++bw) {
        const int bh = std::min(v.H, 128 / bw), bb = bw == v.W && bh == v.H ? std::min(v.B, 128 / (bw * bh)) : 1;
        const long n = up(v.W, bw) * up(v.H, bh) * up(v.B, bb);
        if (tiles && n >= tiles) continue;
        tiles = n;
        a.bw = bw;
        a.bh = bh;
        a.bb = bb;
      }
      a.tiles_x = (int)up(v.W, a.bw);
      a.tiles_y = (int)up(v.H, a.bh);
      a.inv_bw = inv(a.bw);
      a.inv_bp = inv(a.bw * a.bh);
      a.cps = kblocks;
      a.sbo = 8 * rb;
      a.a_tx = a.bw * a.bh * a.bb * rb;
    } else if (mode == TILE_FLAT) {
      if (v.W > 30 || rb != 128) continue;
      a.tiles_x = 1;
      tiles = up(rows * (v.W + 1), 128);
      a.nrows = (v.W + 128 + 2 * (v.W + 2) - 1) / (v.W + 1) + 1;
      a.ky_st = (v.W + 1) * rb;
      a.ps = a.nrows * a.ky_st;
      a.sbo = 8 * rb;
      a.a_tx = a.planes * a.ps;
    } else {
      if (mode == TILE_TALL && (a.planes * 10 * rb) % 128) continue;  // TMA rows start on 128 bytes
      tiles = (mode == TILE_WHOLE ? (long)v.B * a.tiles_y : up(rows, 16)) * a.tiles_x;
      a.ps = (mode == TILE_WHOLE ? 180 : 10) * rb;
      a.ky_st = a.sbo = mode == TILE_WHOLE ? 10 * rb : a.planes * a.ps;
      a.a_tx = 180 * a.planes * rb;
    }
    a.a_bytes = mode == TILE_BOX ? 128 * rb : ((rb == 16 ? 2 * a.a_tx : a.a_tx) + 1023) & ~1023;
    a.tiles = (int)tiles;
    // limits of the kernel's divisions by reciprocals
    if ((rows + 40) * (v.W + 1) + 256 >= (1L << 32) / (v.W + 1) || (rows + 40) * (v.H + 1) >= (1L << 32) ||
        (tiles + 2) * a.tiles_x >= (1L << 32) || (tiles + 2) * a.tiles_y >= (1L << 32) || tiles > (1L << 30))
      continue;
    a.inv_h = inv(v.H + 1);
    a.inv_w = inv(v.W + 1);
    a.inv_x = inv(a.tiles_x);  // tiles_x, tiles_y of 1 are not divided by
    a.inv_y = inv(a.tiles_y);
    for (int nblk : {1, 2, 3, 4, 6, 8, 12, 16}) {
      const int nb = ((v.N + nblk - 1) / nblk + 15) & ~15;
      if (nb > 256 || (nblk - 1) * nb >= v.N) continue;
      const int nbp = (nb + 31) & ~31;
      const size_t wst = (size_t)nb * 128;
      for (int mt = 1; mt <= 2; ++mt) {
        if (mt * nbp > 512) continue;
        const int nacc = 2 * mt * nbp <= 512 ? 2 : 1;
        const size_t ast = (size_t)mt * a.a_bytes;
        for (int res = mode == TILE_BOX ? 0 : 1; res >= 0; --res) {
          if (res && kblocks > HB_MAXW) continue;
          int na = HB_MAXA;
          while (na && fixed + (res ? kblocks : 2) * wst + na * ast > kSmemMax) --na;
          if (!na) continue;
          const int groups = (a.tiles + mt - 1) / mt;
          int per = kSms / nblk;
          if (per > groups) per = groups;
          const double mma = ((v.K + 15) / 16) * mt * fmax(0.53 * nb, 58.0 + 0.2 * nb) + 350.0;
          // box: a box's start besides, for each stage and its weights
          const double la = a.cps * mt * (double)a.a_tx / 45.0 + (mode == TILE_BOX ? a.cps * (mt + 1) * 75.0 : 0.0);
          const double epi = mt * (nbp / 32) * 300.0;
          if (mode == TILE_BOX) {
            // as many stages as weight blocks
            na = 0;
            while (na < HB_MAXA && fixed + (na + 1) * (wst + ast) <= kSmemMax) ++na;
            if (na < 2) continue;
          }
          // with a ring: one or two input stages, the rest of the memory for the ring
          for (int ns = res || mode == TILE_BOX ? na : na < 2 ? na : 2; ns; ns = res || mode == TILE_BOX ? 0 : ns - 1) {
            int nw = kblocks;
            if (mode == TILE_BOX) {
              nw = ns;
            } else if (!res) {
              nw = 2;
              while (nw < 12 && nw < kblocks && fixed + (nw + 1) * wst + ns * ast <= kSmemMax) ++nw;
            }
            const double fl = nw * (double)wst + (mode == TILE_BOX ? ns * (double)ast : 0.0);  // bytes in flight
            const double lw = kblocks * (double)wst / (res ? 45.0 : fmin(45.0, fl / 2000.0));
            double t = fmax(mma, fmax(la + (res ? 0.0 : lw), epi));
            if (ns == 1) t += la + 1000.0;
            if (nacc == 1) t += epi;
            const double c = ((groups + per - 1) / per) * t + la / a.cps + 2500.0 + (res ? lw : 0.0);
            if (found && c >= best_c) continue;
            found = true;
            best_c = c;
            best.a = a;
            best.a.nblk = nblk;
            best.a.nb = nb;
            best.a.nbp = nbp;
            best.a.nacc = nacc;
            best.a.na = ns;
            best.a.nw = nw;
            best.mt = mt;
            best.res = res;
            best.grid = per * nblk;
            int cols = 32;
            while (cols < nacc * mt * nbp) cols <<= 1;
            best.a.cols = cols;
            best.a.off_ctl = (int)(((size_t)nw * wst + ns * ast + 127) & ~(size_t)127);
            best.smem = 1024 + best.a.off_ctl + sizeof(HaloCtl);
          }
          break;  // resident weights, when they fit, beat the ring of the same blocks
        }
      }
    }
  }
  // k_conv3x3_tc keeps calls it does faster: 256-channel blocks of deep layers
  // (1700 clocks per tile and 64 of k) whose channels are no multiple of 64, where
  // too little memory is left beside the input stage for a weight ring
  const double old_c = (double)up((long)v.B * v.H * v.W, 128) * up(v.N, 256) / kSms * kblocks * 1700.0;
  if (!found || (v.N > 128 && v.B * (long)v.H * v.W >= 128L * kSms / 2 && best_c > old_c)) return false;
  best.rb = rb;
  const int m = best.a.mode;
  best.box_w = m == TILE_BOX ? best.a.bw : m == TILE_FLAT ? v.W + 1 : 10;
  best.box_h = m == TILE_BOX ? best.a.bh : m == TILE_WHOLE ? 18 : 1;
  best.box_b = m == TILE_BOX ? best.a.bb : 1;
  best.box_p = m == TILE_FLAT || m == TILE_BOX ? 1 : best.a.planes;
  return true;
}

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encode_tiled() {
  static const EncodeTiled fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
            cudaSuccess || q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return (EncodeTiled)p;
  }();
  return fn;
}
// BF16 tensor of dims[0] contiguous values; st: byte strides of the others
bool encode_bf16(CUtensorMap *map, int rank, const void *p, const cuuint64_t *dims, const cuuint64_t *st,
                 const cuuint32_t *box, CUtensorMapSwizzle swizzle) {
  const EncodeTiled enc = encode_tiled();
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return enc && enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(p), dims, st,
                    box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// NHWC images as (channel in plane, w, h, image, plane) of planes of rb bytes
bool encode_image(CUtensorMap *map, const void *x, int B, int H, int W, int ld, int planes, int rb,
                  int box_w, int box_h, int box_p, int box_b = 1) {
  const cuuint64_t px = (cuuint64_t)ld * 2;
  const cuuint64_t dims[5] = {(cuuint64_t)rb / 2, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B,
                              (cuuint64_t)planes};
  const cuuint64_t st[4] = {px, px * W, px * W * H, (cuuint64_t)rb};
  const cuuint32_t box[5] = {(cuuint32_t)rb / 2, (cuuint32_t)box_w, (cuuint32_t)box_h, (cuuint32_t)box_b,
                             (cuuint32_t)box_p};
  return encode_bf16(map, 5, x, dims, st, box,
                     rb == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                     : rb == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                     : rb == 32 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_NONE);
}

template <int RB, int MT, bool RES, int PL, int MODE>
cudaError_t launch_halo(const HaloPlan &p, const CUtensorMap &wm, const CUtensorMap &xm, cudaStream_t st) {
  static PerDevice attrs;
  cudaError_t e = allow_smem(k_conv3x3_halo<RB, MT, RES, PL, MODE>, kSmemMax, attrs);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_conv3x3_halo<RB, MT, RES, PL, MODE>, p.grid, HB_THREADS, p.smem, st, wm, xm, p.a);
}
template <int RB, int PL, int MODE>
cudaError_t launch_halo_pl(const HaloPlan &p, const CUtensorMap &wm, const CUtensorMap &xm, cudaStream_t st) {
  if (p.res)
    return p.mt == 2 ? launch_halo<RB, 2, true, PL, MODE>(p, wm, xm, st)
                     : launch_halo<RB, 1, true, PL, MODE>(p, wm, xm, st);
  return p.mt == 2 ? launch_halo<RB, 2, false, PL, MODE>(p, wm, xm, st)
                   : launch_halo<RB, 1, false, PL, MODE>(p, wm, xm, st);
}
cudaError_t launch_halo_plan(const HaloPlan &p, const CUtensorMap &wm, const CUtensorMap &xm, cudaStream_t st) {
  const int m = p.a.mode, n = p.a.planes;
  if (m == TILE_BOX)
    return p.mt == 2 ? launch_halo<128, 2, false, 0, TILE_BOX>(p, wm, xm, st)
                     : launch_halo<128, 1, false, 0, TILE_BOX>(p, wm, xm, st);
  if (p.rb == 16) return launch_halo_pl<16, 0, TILE_WHOLE>(p, wm, xm, st);
  if (p.rb == 32) return launch_halo_pl<32, 0, TILE_WHOLE>(p, wm, xm, st);
  if (p.rb == 64) {
    if (m == TILE_WHOLE && n == 1) return launch_halo_pl<64, 1, TILE_WHOLE>(p, wm, xm, st);
    if (m == TILE_WHOLE && n == 3) return launch_halo_pl<64, 3, TILE_WHOLE>(p, wm, xm, st);
    return launch_halo_pl<64, 0, TILE_WHOLE>(p, wm, xm, st);
  }
  if (m == TILE_WHOLE && n == 1) return launch_halo_pl<128, 1, TILE_WHOLE>(p, wm, xm, st);
  if (m == TILE_WHOLE && n == 3) return launch_halo_pl<128, 3, TILE_WHOLE>(p, wm, xm, st);
  if (m == TILE_TALL && n == 1) return launch_halo_pl<128, 1, TILE_TALL>(p, wm, xm, st);
  if (m == TILE_TALL && n == 2) return launch_halo_pl<128, 2, TILE_TALL>(p, wm, xm, st);
  return launch_halo_pl<128, 0, TILE_WHOLE>(p, wm, xm, st);  // walked: any tiling but box
}

// true when the call was launched here (rc its status); false: not this kernel's
bool conv_halo(const ConvArgs &v, cudaStream_t st, cudaError_t &rc) {
  HaloPlan p;
  if (!halo_plan(v, p)) return false;
  HaloArgs &a = p.a;
  a.bias = v.bias; a.y = v.y; a.mask = v.mask;
  a.B = v.B; a.H = v.H; a.W = v.W; a.N = v.N; a.relu = v.relu;
  a.ldy = v.ldy; a.yoff = v.yoff; a.ldm = v.ldm;
  // widest row access that y, its offset and stride, and the mask allow
  auto fits = [&](int c) {
    const uintptr_t b = (uintptr_t)c * 2 - 1;
    return !(v.N % c) && !(v.ldy % c) && !(v.yoff % c) && !((uintptr_t)v.y & b) &&
           (!v.mask || (!(v.ldm % c) && !((uintptr_t)v.mask & b)));
  };
  a.vec = fits(16) ? 32 : fits(8) ? 16 : 4;
  CUtensorMap wm, xm;
  const cuuint64_t wd[2] = {(cuuint64_t)v.K, (cuuint64_t)v.N}, ws[1] = {(cuuint64_t)v.K * 2};
  const cuuint32_t wb[2] = {64, (cuuint32_t)a.nb};
  if (!encode_bf16(&wm, 2, v.w, wd, ws, wb, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !encode_image(&xm, v.x, v.B, v.H, v.W, v.ldx, a.planes, p.rb, p.box_w, p.box_h, p.box_p, p.box_b))
    return false;
  rc = launch_halo_plan(p, wm, xm, st);
  return true;
}

int g_use_tc = 1;  // cem_sg_set_gemm_path

// ---------------------------------------------------- conv 3x3 weight grad
// dW[n, k] = sum_p dY[p, n] * A[p, k] over the pixels of split z, written
// to ws[z][n][k]; k = (ky * 3 + kx) * Cin + c as in the forward weights.
constexpr int GBM = 64, GBN = 64, GBK = 32, GST = 3, GPAD = 64 + 8;

struct WgradArgs {
  const bf16_t *x;   // [P, ldx] forward input
  const bf16_t *dy;  // [P, lddy] output gradient (channels 0..N-1)
  float *ws;         // [splits][N][K]
  float *wsb;        // [splits][N] bias partials (null: no bias gradient)
  int B, H, W, Cin, ldx, lddy, N, K, P, chunk;  // chunk: pixels per split
};

__global__ void __launch_bounds__(256) k_conv3x3_wgrad(WgradArgs a) {
  __shared__ __align__(128) bf16_t As[GST][GBK][GPAD];  // [pixel][n]
  __shared__ __align__(128) bf16_t Bs[GST][GBK][GPAD];  // [pixel][k]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp >> 2, wn = warp & 3;  // 2 x 4 warps, each 32 (n) x 16 (k)
  const int m0 = blockIdx.x * GBM, k0 = blockIdx.y * GBN, z = blockIdx.z;
  const int pbeg = z * a.chunk, pend = min(a.P, pbeg + a.chunk);
  const int HW = a.H * a.W, cpt = a.Cin >> 3;
  const int KT = (pend - pbeg + GBK - 1) / GBK;
  const int prow = tid >> 3, ch = tid & 7;
  // this thread's k chunk is fixed: tap and channel
  const int kq = (k0 >> 3) + ch;
  const int tap = kq / cpt, c0 = (kq - tap * cpt) * 8;
  const int ky = tap / 3, kx = tap - ky * 3;
  const bool kok = k0 + ch * 8 < a.K;
  const bool nok = m0 + ch * 8 < a.N;
  auto load_tile = [&](int kt, int s) {
    const int p = pbeg + kt * GBK + prow;
    const bool pok = p < pend;
    const bf16_t *srca = (pok && nok) ? a.dy + (size_t)p * a.lddy + m0 + ch * 8 : a.dy;
    cp_async16(&As[s][prow][ch * 8], srca, (pok && nok) ? 16 : 0);
    bool ok = pok && kok;
    const bf16_t *srcb = a.x;
    if (ok) {
      const int b = p / HW, rem = p - b * HW, h = rem / a.W, w = rem - h * a.W;
      const int hh = h + ky - 1, ww = w + kx - 1;
      ok = hh >= 0 && hh < a.H && ww >= 0 && ww < a.W;
      if (ok) srcb = a.x + ((size_t)(b * a.H + hh) * a.W + ww) * a.ldx + c0;
    }
    cp_async16(&Bs[s][prow][ch * 8], srcb, ok ? 16 : 0);
  };
  float acc[2][2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
  // bias: the k-tile-0 blocks also sum dY over their pixels, channel
  // n = tid & 63 over pixel rows (tid >> 6) + 4 r of each staged tile
  const bool do_bias = a.wsb && blockIdx.y == 0;
  float bsum = 0.f;
#pragma unroll
  for (int s = 0; s < GST - 1; ++s) {
    if (s < KT) load_tile(s, s);
    cp_async_commit();
  }
  for (int kt = 0; kt < KT; ++kt) {
    cp_async_wait<GST - 2>();
    __syncthreads();
    const int nk = kt + GST - 1;
    if (nk < KT) load_tile(nk, nk % GST);
    cp_async_commit();
    const int s = kt % GST;
    if (do_bias) {
#pragma unroll
      for (int r = 0; r < GBK / 4; ++r) bsum += bf2f(As[s][(tid >> 6) + 4 * r][tid & 63]);
    }
#pragma unroll
    for (int kk = 0; kk < GBK; kk += 16) {
      const int mat = lane >> 3, r = lane & 7;
      uint32_t af[2][4], bq[4];
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
        ldsm_x4_t(af[mi], &As[s][kk + (mat >> 1) * 8 + r][wm * 32 + mi * 16 + (mat & 1) * 8]);
      ldsm_x4_t(bq, &Bs[s][kk + (mat & 1) * 8 + r][wn * 16 + (mat >> 1) * 8]);
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
        mma_bf16(acc[mi][0], af[mi], bq[0], bq[1]);
        mma_bf16(acc[mi][1], af[mi], bq[2], bq[3]);
      }
    }
  }
  cp_async_wait<0>();
  if (do_bias) {
    __shared__ float red[4][64];
    red[tid >> 6][tid & 63] = bsum;
    __syncthreads();
    if (tid < 64 && m0 + tid < a.N)
      a.wsb[(size_t)z * a.N + m0 + tid] = (red[0][tid] + red[1][tid]) + (red[2][tid] + red[3][tid]);
  }
  float *out = a.ws + (size_t)z * a.N * a.K;
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 2; ++ni) {
      const int k = k0 + wn * 16 + ni * 8 + (lane & 3) * 2;
      if (k >= a.K) continue;
#pragma unroll
      for (int hr = 0; hr < 2; ++hr) {
        const int n = m0 + wm * 32 + mi * 16 + (lane >> 2) + hr * 8;
        if (n >= a.N) continue;
        *reinterpret_cast<float2 *>(out + (size_t)n * a.K + k) =
            make_float2(acc[mi][ni][hr * 2], acc[mi][ni][hr * 2 + 1]);
      }
    }
}

// ------------------------------------------- weight gradient on tcgen05
// dW^T[k'][o] = sum_p A[p][k'] dY[p][o] with k' = (ky * 3 + kx) * Cin + c and
// A the shifted input (zero outside the image): M = k' (128 per CTA), N = o
// (BN), K = pixels, split into fixed pixel chunks (grid z) whose FP32 tiles
// go to a workspace and are added in chunk order.  Both operands are read in
// their natural NHWC layout, i.e. MN-major for the MMA: in shared memory
// each pixel is a 128-byte row of 64 k' (or o) values, 8 pixels form a
// 1024-byte swizzle atom (16-byte chunk c of row r at c ^ (r & 7)), atoms
// along K are 1024 bytes apart (SBO) and 64-wide atoms along M or N are
// 8192 bytes apart (LBO).  One thread issues the MMAs (K = 16 = two atoms
// each), tcgen05.commit frees the stage, the epilogue writes the transposed
// tile (coalesced along k') with tcgen05.ld.
constexpr int WTM = 128, WTK = 64;

// MN-major, 128-byte swizzle
__device__ __forceinline__ uint64_t mn_desc(uint32_t saddr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__host__ __device__ constexpr uint32_t tc_idesc_mn(int M, int N) {
  return tc_idesc(M, N) | (1u << 15) | (1u << 16);
}

template <int BN>
struct TwSmem {
  uint8_t A[TCS][WTM * WTK * 2];  // 16 KB: 2 atoms along k' of 64 pixels x 128 B
  uint8_t B[TCS][BN * WTK * 2];   // BN / 64 atoms along o
  uint64_t mma_bar[TCS];
  uint32_t tmem;
};

template <int BN>
__global__ void __launch_bounds__(128, 1) k_conv3x3_wgrad_tc(WgradArgs a) {
  extern __shared__ uint8_t tw_raw[];
  TwSmem<BN> &T = *reinterpret_cast<TwSmem<BN> *>(
      (reinterpret_cast<uintptr_t>(tw_raw) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * WTM, n0 = blockIdx.y * BN, z = blockIdx.z;
  const int pbeg = z * a.chunk, pend = min(a.P, pbeg + a.chunk);
  const int KB = (pend - pbeg + WTK - 1) / WTK;
  const int HW = a.H * a.W;

  if (tid == 0) {
    for (int s = 0; s < TCS; ++s) mbar_init(&T.mma_bar[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&T.tmem)),
                 "r"(BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  const uint32_t tmem = T.tmem;

  // A: this thread's k' chunk (8 values) is fixed; its pixel rows are
  // (tid >> 4) + 8 i of each stage
  const int ck = tid & 15;
  const int kq = m0 + ck * 8;
  const bool kok = kq < a.K;
  const int tap = kok ? kq / a.Cin : 0, c0 = kok ? kq - tap * a.Cin : 0;
  const int ky = tap / 3, kx = tap - ky * 3;
  const uint32_t aoff_c = (uint32_t)((ck >> 3) * 8192);
  // (b, h, w) of this thread's first pixel row, advanced by 8 pixels per
  // row and 64 per stage without divisions (W >= 8 keeps each carry single)
  int pb0, ph0, pw0;
  {
    const int p = pbeg + (tid >> 4);
    pb0 = p / HW;
    const int rem = p - pb0 * HW;
    ph0 = rem / a.W;
    pw0 = rem - ph0 * a.W;
  }
  auto advance = [&](int &b, int &h, int &w, int n) {
    w += n;
    while (w >= a.W) {
      w -= a.W;
      if (++h == a.H) { h = 0; ++b; }
    }
  };
  auto load_stage = [&](int kb, int s) {
    const int pst = pbeg + kb * WTK;
    const uint32_t abase = smem_u32(T.A[s]), bbase = smem_u32(T.B[s]);
    int b = pb0, h = ph0, w = pw0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int pr = (tid >> 4) + 8 * i;
      const int p = pst + pr;
      bool ok = kok && p < pend;
      const bf16_t *src = a.x;
      if (ok) {
        const int hh = h + ky - 1, ww = w + kx - 1;
        ok = hh >= 0 && hh < a.H && ww >= 0 && ww < a.W;
        if (ok) src = a.x + ((size_t)(b * a.H + hh) * a.W + ww) * a.ldx + c0;
      }
      if (i < 7) advance(b, h, w, 8);
      const int g = pr >> 3, r = pr & 7;
      const uint32_t dst = abase + aoff_c + g * 1024 + r * 128 + (((ck & 7) ^ r) << 4);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                   "r"(ok ? 16 : 0));
    }
    advance(pb0, ph0, pw0, WTK);  // stages are loaded in increasing order
    constexpr int CPR = BN / 8;            // 16-byte chunks per pixel row
    constexpr int RPP = 128 / CPR;         // pixel rows per pass
#pragma unroll
    for (int i = 0; i < WTK / RPP; ++i) {
      const int pr = tid / CPR + RPP * i, cc = tid % CPR;
      const int p = pst + pr, n = n0 + cc * 8;
      const bool ok = p < pend && n < a.N;
      const bf16_t *src = ok ? a.dy + (size_t)p * a.lddy + n : a.dy;
      const int g = pr >> 3, r = pr & 7;
      const uint32_t dst = bbase + (cc >> 3) * 8192 + g * 1024 + r * 128 + (((cc & 7) ^ r) << 4);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                   "r"(ok ? 16 : 0));
    }
  };

  constexpr uint32_t idesc = tc_idesc_mn(WTM, BN);
  bool failed = false;
  int last_kb = -1;  // the last stage whose MMAs were issued
#pragma unroll
  for (int s = 0; s < TCS - 1; ++s) {
    if (s < KB) load_stage(s, s);
    cp_async_commit();
  }
  for (int kb = 0; kb < KB && !failed; ++kb) {
    const int s = kb % TCS;
    cp_async_wait<TCS - 2>();
    asm volatile("fence.proxy.async.shared::cta;\n" ::);
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
      const uint32_t as = smem_u32(T.A[s]), bs = smem_u32(T.B[s]);
#pragma unroll
      for (int k = 0; k < WTK / 16; ++k) {
        // B: with a single 64-wide atom along o the atom stride is unused
        const uint64_t ad = mn_desc(as + k * 2048, 8192),
                       bd = mn_desc(bs + k * 2048, BN > 64 ? 8192 : 1024);
        const uint32_t acc = (kb > 0 || k > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
          smem_u32(&T.mma_bar[s])));
    }
    last_kb = kb;
    const int nk = kb + TCS - 1;
    if (nk < KB) {
      if (kb >= 1 && !mbar_wait(&T.mma_bar[(kb - 1) % TCS], ((kb - 1) / TCS) & 1)) failed = true;
      if (!failed) load_stage(nk, nk % TCS);
    }
    cp_async_commit();
    failed = __syncthreads_or(failed) != 0;
  }
  cp_async_wait<0>();
  if (!failed && KB > 0 && !mbar_wait(&T.mma_bar[(KB - 1) % TCS], ((KB - 1) / TCS) & 1))
    failed = true;
  failed = __syncthreads_or(failed) != 0;
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);

  float *out = a.ws + (size_t)z * a.N * a.K;
  const int kr = m0 + warp * 32 + lane;  // this lane's k' row of the tile
  if (!failed) {
#pragma unroll 1
    for (int cb = 0; cb < BN; cb += 32) {
      uint32_t r[32];
      if (KB > 0) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
            "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
              "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
              "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
              "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
              "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
              "=r"(r[31])
            : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)cb));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::);
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) r[j] = 0u;
      }
      if (kr < a.K) {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int n = n0 + cb + j;
          if (n < a.N) out[(size_t)n * a.K + kr] = __uint_as_float(r[j]);
        }
      }
    }
  } else if (tid == 0) {
    atomicAdd(&g_tc_timeouts, 1);
  }
  // After a wait gave up, MMAs may still be in flight: wait (bounded) for the
  // last issued commit, which tracks every earlier MMA, before the TMEM is
  // freed; if that wait gives up too, the CTA exits without freeing it (the
  // results of the call are invalid in either case; cem_sg_timeouts says so).
  bool drained = true;
  if (failed && last_kb >= 0)
    drained = __syncthreads_and(mbar_wait(&T.mma_bar[last_kb % TCS], (last_kb / TCS) & 1)) != 0;
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  if (warp == 0 && drained)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(BN));
}

// per-channel sums of dY [P, ld] (channels 0..C-1, C a multiple of 8) over
// fixed pixel chunks: ws[chunk][C]; 16-byte loads, a fixed reduction order
__global__ void __launch_bounds__(256) k_colsum8(const bf16_t *t, int P, int C, int ld,
                                                 int chunk, float *ws) {
  __shared__ float red[256][9];
  const int C8 = C >> 3;
  const int lanes = 256 / C8;  // pixel lanes per block (C <= 2048)
  const int cg = threadIdx.x % C8, pl = threadIdx.x / C8;
  const int z = blockIdx.x;
  const int pend = min(P, (z + 1) * chunk);
  float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (pl < lanes) {
    for (int p = z * chunk + pl; p < pend; p += lanes) {
      const uint4 v = *reinterpret_cast<const uint4 *>(t + (size_t)p * ld + cg * 8);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        s[2 * q] += bf2f((bf16_t)(w[q] & 0xffff));
        s[2 * q + 1] += bf2f((bf16_t)(w[q] >> 16));
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) red[threadIdx.x][q] = s[q];
  __syncthreads();
  if (threadIdx.x < C8) {
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int l = 0; l < lanes; ++l)
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[q] += red[l * C8 + threadIdx.x][q];
#pragma unroll
    for (int q = 0; q < 8; ++q) ws[(size_t)z * C + threadIdx.x * 8 + q] = acc[q];
  }
}

template <int BN>
size_t tw_smem_bytes() {
  return sizeof(TwSmem<BN>) + 1024;
}

template <int BN>
cudaError_t launch_wgrad_tc(const WgradArgs &a, int splits, cudaStream_t st) {
  static PerDevice attrs;
  const cudaError_t ae = allow_smem(k_conv3x3_wgrad_tc<BN>, tw_smem_bytes<BN>(), attrs);
  if (ae != cudaSuccess) return ae;
  dim3 grid((a.K + WTM - 1) / WTM, (a.N + BN - 1) / BN, splits);
  k_conv3x3_wgrad_tc<BN><<<grid, 128, tw_smem_bytes<BN>(), st>>>(a);
  return cudaGetLastError();
}

// Non-finite inputs.  Tiles that reach past an image (or across the zero rows and
// columns between two) multiply the image's border pixels with the zero dY outside it:
// nothing is added unless such a pixel is not finite, when 0 x Inf or 0 x NaN would make
// the weight gradients of the taps that look from outside NaN.  Whatever finishes dw
// (k_reduce_sums, or k_wgrad_halo where a range has all of an entry) forms those again from
// the pixels inside, one warp each; it looks for them at entries that are not finite, so
// finite gradients cost a comparison (64 images, 512 -> 512 channels at 10 x 25: 111 us
// with it as without; one infinity at a corner 0.4 ms, all of x NaN 1.3 ms).
struct DwInputs {
  const bf16_t *x, *dy;
  int B, H, W, Cin, ldx, lddy, K;
};
inline DwInputs dw_inputs(const WgradArgs &v) {
  return DwInputs{v.x, v.dy, v.B, v.H, v.W, v.Cin, v.ldx, v.lddy, v.K};
}
__device__ __forceinline__ bool finite_bf(bf16_t v) { return (v & 0x7f80) != 0x7f80; }

// dw entry i = (o, tap, c), whose sum over the tiles is s; whole warps call it
__device__ __noinline__ float dw_inside(const DwInputs &v, long i, float s) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int o = (int)(i / v.K), k = (int)(i - (long)o * v.K), tap = k / v.Cin;
  const int dh = tap / 3 - 1, dw = tap % 3 - 1;
  const bf16_t *x = v.x + (k - tap * v.Cin), *dy = v.dy + o;
  // is one of the border pixels that this tap would read for a pixel outside not finite?
  bool bad = false;
  for (int side = 0; side < 2 && !bad; ++side) {
    // the image's last row (column) for the taps above (left), its first for those below (right)
    const int d = side ? dw : dh, n = d == 0 ? 0 : v.B * (side ? v.H : v.W);
    for (int q0 = 0, steps = 1; q0 < n && !bad; q0 += 32 * steps, steps = 8) {  // the first 32, 256 at a time then
      bool odd = false;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (j >= steps) break;
        const int q = min(q0 + j * 32 + lane, n - 1), b = q / v.W;
        const size_t p = side ? (size_t)q * v.W + (d < 0 ? v.W - 1 : 0)
                              : ((size_t)b * v.H + (d < 0 ? v.H - 1 : 0)) * v.W + (q - b * v.W);
        odd |= !finite_bf(x[p * v.ldx]);
      }
      bad = __any_sync(FULL, odd);
    }
  }
  if (!bad) return s;
  const int P = v.B * v.H * v.W;
  double sum = 0.0;
  for (int p0 = 0, steps = 1; p0 < P; p0 += 32 * steps, steps = 8) {
    float t = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int p = p0 + q * 32 + lane;
      if (q >= steps || p >= P) continue;
      const int r = p / v.W, w = p - r * v.W + dw, h = r % v.H + dh;
      const bool in = h >= 0 && h < v.H && w >= 0 && w < v.W;
      const float xv = in ? bf2f(x[((long)p + dh * v.W + dw) * v.ldx]) : 0.f;
      t += xv * bf2f(dy[(size_t)p * v.lddy]);
    }
    sum += (double)t;
    if (__any_sync(FULL, isnan(sum))) return __int_as_float(0x7fc00000);  // whatever follows
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(FULL, sum, off);
  return (float)sum;
}

// --------------------------- weight gradient with the input tile resident
// dW[o][tap][c] = sum_p dY[p][o] x[p + tap][c], K = pixels.  As in
// k_conv3x3_halo a stage holds the halo of a 128-pixel tile of x, and beside it
// the tile of dY; both are read MN-major (a pixel is a row of channels, the 8
// pixels of a tile row a swizzle atom's 8 rows), so a tap is again a start
// address shifted by whole slots.  The x side stacks taps: with 64-channel
// planes two (the LBO is the distance of their slots), with 32-channel planes
// the three of a tap row (a fourth atom is read and ignored; of 8 channels, unswizzled,
// sixteen slots are), so that a block (plane, taps) is one M = 128 operand and has
// its own accumulator of nb columns.
// (Swapped sides, M = 64 outputs and N = 96, took 107 clocks a step for 32
// outputs against 85.)  Blocks are dealt to the CTAs of grid x (512 columns of
// TMEM hold 512 / nb of them), output-channel blocks to grid y, ranges of
// tiles to grid z.  Every `flush` tiles (the 4096 to 8192 pixels of one chunk of
// k_conv3x3_wgrad_tc, so that the tensor cores' FP32 sums stay as short) a
// CTA adds its accumulators to its slot of the workspace; k_reduce_sums adds
// the slots in order.  The CTAs of x = 0 also sum dY for the bias gradient
// from the tiles they hold.
// k_conv3x3_wgrad_tc fetches each x pixel nine times, in 16-byte copies, which
// bound it, and needs the bias sums and two slow reductions beside it.  64
// images, all of it, before and now: 8 -> 32 channels at 160 x 400 387 -> 155 us, 32 -> 32
// 782 -> 150 (3.5 TB/s), 96 -> 32 1486 -> 389, 64 -> 64 at 80 x 200 413 -> 86, 128 -> 128 at
// 40 x 100 281 -> 92, 768 -> 256 at 20 x 50 462 -> 198, 512 -> 512 at 10 x 25 255 ->
// 111.  What remains is the MMAs' issue and, from 128 channels on, the tiles'
// re-reading from L2 by the CTAs of grid x and y.
// Roles: warps 0-7 bias sums and workspace (two groups of four, alternate
// blocks), warp 8 MMAs, warp 9 tiles.
constexpr int WH_THREADS = 320, WH_MAXA = 8;

struct WgHaloArgs {
  float *ws, *wsb;      // [slots][N][K], [slots][N] (null: no bias gradient)
  int B, H, W, N, K, Cin;
  int mode;             // TILE_*
  int ky_st, sbo;       // x: strides of a tap row and 8 tile pixels (bytes)
  int xps, yps, ysbo;   // plane strides of a stage's x and dY, 8 pixels of dY
  int nrows;            // flat: image rows a stage holds
  int tiles_x, tiles_y, tiles, range, flush;  // sub-tiles of 128 pixels; of a CTA; per flush
  uint32_t inv_h, inv_w, inv_x, inv_y;
  int blocks;           // x blocks in all
  int xplanes, yplanes; // planes of a stage
  int nb;               // output channels of a block, columns of an accumulator
  int nacc;             // accumulator sets
  int na, stage, y_at, cols, off_ctl;
  int inside;           // the range has all of dw's sums, from tiles that reach past the images
  DwInputs in;
};

struct WgHaloCtl {
  uint64_t full[WH_MAXA], empty[WH_MAXA], acc_full[2], acc_empty[2], drain;
  uint32_t tmem;
  int fail;
  float red[4][8][8][8];
};

// tensor maps of x and dY with boxes of 1, 2, 4 and 8 rows (a whole tile's rows in [0])
struct WgMaps {
  CUtensorMap x[4], y[4];
};

// Rows t0 .. t0 + n - 1 of the tall image in as few boxes as its images allow (a box may
// take the zero rows above and below an image): issue(first row, h, image, log2 rows).
// A box costs TMA about 75 clocks besides its bytes.
template <class F>
__device__ __forceinline__ void tall_rows(const WgHaloArgs &a, int t0, int n, F issue) {
  for (int r = 0; r < n;) {
    const int T = t0 + r, b = T < 0 ? 0 : div_by(T, a.inv_h), h = T < 0 ? -1 : T - b * (a.H + 1) - 1;
    const int m = T < 0 ? 1 : min(n - r, a.H + 1 - h);
    const int k = m >= 8 ? 3 : m >= 4 ? 2 : m >= 2 ? 1 : 0;
    issue(r, h, b, k);
    r += 1 << k;
  }
}

template <int RBX, int RBY, int PER>
__global__ void __launch_bounds__(WH_THREADS, 1)
    k_wgrad_halo(const __grid_constant__ WgMaps maps, const __grid_constant__ WgHaloArgs a) {
  extern __shared__ uint8_t wh_raw[];
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(wh_raw) + 1023) &
                                              ~(uintptr_t)1023);
  WgHaloCtl &C = *reinterpret_cast<WgHaloCtl *>(base + a.off_ctl);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  constexpr int TAPB = RBX == 128 ? 5 : 3;  // blocks of a plane
  const int q0 = blockIdx.x * PER, nq = min(PER, a.blocks - q0), p0 = q0 / TAPB;
  const int n0 = blockIdx.y * a.nb, z = blockIdx.z;
  const int tbeg = z * a.range, tend = min(a.tiles, tbeg + a.range);
  const bool bias = a.wsb && blockIdx.x == 0;

  if (tid == 0) {
    for (int s = 0; s < a.na; ++s) {
      mbar_init(&C.full[s], 1);
      mbar_init(&C.empty[s], bias ? 257 : 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&C.acc_full[s], 1);
      mbar_init(&C.acc_empty[s], 256);
    }
    mbar_init(&C.drain, 1);
    C.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&C.tmem)),
                 "r"(a.cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, C.tmem, 0);
  const uint32_t sx = smem_u32(base), sy = sx + (uint32_t)a.y_at;

  if (warp == 9) {
    // ---- tiles of x (halo) and dY; lane = plane where a box holds one
    const uint32_t bytes =
        (uint32_t)(a.mode == TILE_FLAT ? a.nrows * (a.W + 1) * (a.xplanes * RBX + a.yplanes * RBY)
                                       : a.xplanes * 180 * RBX + a.yplanes * 128 * RBY);
    const int y0 = n0 / (RBY / 2);
    int s = 0, ph = 1, it = 0;
    for (int tile = tbeg; tile < tend; ++tile, ++it) {
      if (!warp_wait(&C.empty[s], ph, &C.fail)) break;
      uint64_t *bar = &C.full[s];
      if (lane == 0) mbar_expect(bar, bytes);
      __syncwarp();
      const uint32_t dx = sx + (uint32_t)(s * a.stage), dy = sy + (uint32_t)(s * a.stage);
      const int ty = a.tiles_x == 1 ? tile : div_by(tile, a.inv_x);
      const int c = (tile - ty * a.tiles_x) * 8;
      if (a.mode == TILE_WHOLE) {
        const int b = a.tiles_y == 1 ? ty : div_by(ty, a.inv_y), h = (ty - b * a.tiles_y) * 16;
        if (lane == 0) tma_load5(dx, &maps.x[0], 0, c - 1, h - 1, b, p0, bar);
        if (lane == 1) tma_load5(dy, &maps.y[0], 0, c, h, b, y0, bar);
      } else if (a.mode == TILE_TALL) {
        tall_rows(a, ty * 16, 18, [&](int r, int h, int b, int k) {
          if (lane < a.xplanes)
            tma_load5(dx + lane * a.xps + r * a.ky_st, &maps.x[k], 0, c - 1, h, b, p0 + lane, bar);
        });
        tall_rows(a, ty * 16 + 1, 16, [&](int r, int h, int b, int k) {
          if (lane < a.yplanes)
            tma_load5(dy + lane * a.yps + r * a.ysbo, &maps.y[k], 0, c, h, b, y0 + lane, bar);
        });
      } else {
        const int q = tile * 128 - 1;
        tall_rows(a, q < 0 ? -1 : div_by(q, a.inv_w), a.nrows, [&](int r, int h, int b, int k) {
          if (lane < a.xplanes)
            tma_load5(dx + lane * a.xps + r * (a.W + 1) * RBX, &maps.x[k], 0, 0, h, b, p0 + lane, bar);
          if (lane < a.yplanes)
            tma_load5(dy + lane * a.yps + r * (a.W + 1) * RBY, &maps.y[k], 0, 0, h, b, y0 + lane, bar);
        });
      }
      if (++s == a.na) {
        s = 0;
        ph ^= 1;
      }
    }
    // no copy outlives the CTA
    for (int q = max(0, it - a.na); q < it; ++q) mbar_wait(&C.full[q % a.na], (q / a.na) & 1);
  } else if (warp == 8) {
    // ---- MMAs
    if (elect_one()) {
      const uint32_t idesc = tc_idesc_mn(128, a.nb);
      // 8 channels: unswizzled, SBO steps through M (a slot), LBO through K (a tile row)
      const uint32_t xhi = RBX == 16 ? 1u | (1u << 14)
                                     : (uint32_t)(a.sbo >> 4) | (1u << 14) | ((RBX == 128 ? 2u : 4u) << 29);
      const uint32_t yhi = (uint32_t)(a.ysbo >> 4) | (1u << 14) | ((RBY == 128 ? 2u : 4u) << 29);
      const uint32_t ylbo = (uint32_t)(a.yps >> 4) << 16;
      const uint32_t xst = (uint32_t)(2 * a.sbo) >> 4, yst = (uint32_t)(2 * a.ysbo) >> 4;
      // x operand of each block, relative to the stage (units of 16 bytes), LBO in the high half
      // (past the last block: the last again, into columns that nobody reads; the
      // steps are straight-line code without tests, or their issue would bound them)
      uint32_t off[PER];
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        const int q = q0 + min(j, nq - 1), pl = q / TAPB - p0, t = q % TAPB;
        auto at = [&](int tap) { return (uint32_t)(((tap / 3) * a.ky_st + (tap % 3) * RBX) >> 4); };
        uint32_t o, lbo;
        if (RBX == 128) {
          o = at(2 * t);
          lbo = t < 4 ? at(2 * t + 1) - o : 0;  // the ninth tap stands alone
        } else {
          o = at(3 * t);
          lbo = RBX == 64 ? RBX >> 4 : (uint32_t)a.sbo >> 4;
        }
        off[j] = (o + (uint32_t)(pl * (a.xps >> 4))) | (lbo << 16);
      }
      int s = 0, ph = 0, ab = 0, abph = 1, left = 0;
      bool ok = true;
      for (int tile = tbeg; tile < tend; ++tile) {
        uint32_t acc = 1;
        if (left == 0) {  // a new set of sums
          if (!(ok = thread_wait(&C.acc_empty[ab], abph, &C.fail))) break;
          left = min(a.flush, tend - tile);
          acc = 0;
        }
        if (!(ok = thread_wait(&C.full[s], ph, &C.fail))) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        uint32_t ax = (sx + (uint32_t)(s * a.stage)) >> 4, by = ((sy + (uint32_t)(s * a.stage)) >> 4) | ylbo;
        if (a.mode == TILE_FLAT) {
          const int q = tile * 128 - 1, row = q < 0 ? -1 : div_by(q, a.inv_w);
          const int f = q - row * (a.W + 1);
          ax += (uint32_t)(f * (RBX >> 4));
          by += (uint32_t)((f + a.W + 2) * (RBY >> 4));
        }
        const uint32_t d0 = tmem + (uint32_t)(ab * PER * a.nb);
#pragma unroll
        for (int i = 0; i < 8; ++i, ax += xst, by += yst) {
#pragma unroll
          for (int j = 0; j < PER; ++j)
            tc_mma(d0 + (uint32_t)(j * a.nb), ax + off[j], xhi, by, yhi, idesc, i ? 1u : acc);
        }
        tc_commit(&C.empty[s]);
        if (++s == a.na) {
          s = 0;
          ph ^= 1;
        }
        if (--left == 0) {
          tc_commit(&C.acc_full[ab]);
          if (++ab == a.nacc) {
            ab = 0;
            abph ^= 1;
          }
        }
      }
      tc_commit(&C.drain);
      if (!mbar_wait(&C.drain, 0)) *(volatile int *)&C.fail = 2;
    }
  } else {
    // ---- bias sums as the tiles pass, accumulators to the workspace as they fill
    constexpr int CH = RBY / 16, RSTEP = 256 / CH;  // 16-byte chunks of a row; rows in a pass
    const int e = warp >> 2, w4 = warp & 3, cc = tid % CH, r0 = tid / CH;
    float sum[4][8];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int k = 0; k < 8; ++k) sum[p][k] = 0.f;
    float *out = a.ws + (size_t)z * a.N * a.K;
    // where this lane's row of a unit's 32 columns goes (null: nowhere)
    const int ncb = a.nb / 32, units = nq * ncb;
    auto dest = [&](int u) -> float * {
      const int j = u / ncb, cb = (u - j * ncb) * 32;
      const int q = q0 + j, pl = q / TAPB, t = q - pl * TAPB;
      const int tap = RBX == 128 ? 2 * t + (w4 >> 1) : RBX == 64 ? 3 * t + w4 : 3 * t + (lane >> 3);
      const int c = RBX == 128 ? pl * 64 + (w4 & 1) * 32 + lane : RBX == 64 ? pl * 32 + lane : lane & 7;
      if (u >= units || (RBX == 128 ? tap >= 9 : RBX == 64 ? w4 >= 3 : w4 > 0 || lane >= 24)) return nullptr;
      return out + (size_t)(n0 + cb) * a.K + tap * a.Cin + c;
    };
    float odd = 0.f;  // NaN once a sum of the range is not finite
    int s = 0, ph = 0, ab = 0, abph = 0;
    bool ok = true;
    for (int tile = tbeg; tile < tend && ok;) {
      const int n = min(a.flush, tend - tile);
      if (bias)
        for (int k = 0; k < n && ok; ++k) {
          if (!(ok = warp_wait(&C.full[s], ph, &C.fail))) break;
          uint32_t yb = sy + (uint32_t)(s * a.stage);
          if (a.mode == TILE_FLAT) {
            const int q = (tile + k) * 128 - 1, row = q < 0 ? -1 : div_by(q, a.inv_w);
            yb += (uint32_t)((q - row * (a.W + 1) + a.W + 2) * RBY);
          }
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            if (p >= a.yplanes) break;
#pragma unroll
            for (int r = 0; r < 128 / RSTEP; ++r) {
              const uint32_t ad = yb + (uint32_t)(p * a.yps + (r0 + r * RSTEP) * RBY);
              const uint32_t x = RBY == 128 ? (ad >> 7) & 7 : (ad >> 7) & 3;  // swizzle, by address
              uint32_t w[4];
              asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];\n"
                           : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                           : "r"(ad + ((cc ^ x) << 4)));
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                sum[p][2 * q] += bf2f((bf16_t)(w[q] & 0xffff));
                sum[p][2 * q + 1] += bf2f((bf16_t)(w[q] >> 16));
              }
            }
          }
          mbar_arrive(&C.empty[s]);
          if (++s == a.na) {
            s = 0;
            ph ^= 1;
          }
        }
      // unit u: 32 columns of a block.  What the slot holds already is read a unit
      // ahead (the first before the sums are in), so that its latency is hidden.
      const bool add = tile > tbeg;
      float old[32];
      float *d = dest(e);
      auto fetch = [&](const float *from) {
#pragma unroll
        for (int k = 0; k < 32; ++k) old[k] = add && from ? from[(size_t)k * a.K] : 0.f;
      };
      fetch(d);
      if (!ok || !(ok = warp_wait(&C.acc_full[ab], abph, &C.fail))) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint32_t t0 = tmem + ((uint32_t)(w4 * 32) << 16) + (uint32_t)(ab * PER * a.nb);
      for (int u = e; u < units; u += 2) {
        uint32_t r[32];
        __syncwarp();
        tmem_ld32(t0 + (uint32_t)(u * 32), r);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        float *now = d;
#pragma unroll
        for (int k = 0; k < 32; ++k) r[k] = __float_as_uint(__uint_as_float(r[k]) + old[k]);
        d = dest(u + 2);
        fetch(d);
        if (now) {
          float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int k = 0; k < 32; ++k) {
            now[(size_t)k * a.K] = __uint_as_float(r[k]);
            z[k & 3] = fmaf(__uint_as_float(r[k]), 0.f, z[k & 3]);
          }
          odd += (z[0] + z[1]) + (z[2] + z[3]);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      mbar_arrive(&C.acc_empty[ab]);
      if (++ab == a.nacc) {
        ab = 0;
        abph ^= 1;
      }
      tile += n;
    }
    if (ok && a.inside && __any_sync(0xffffffffu, isnan(odd))) {
#pragma unroll 1
      for (int u = e; u < units; u += 2) {
        float *d = dest(u);
#pragma unroll 1
        for (int k = 0; k < 32; ++k) {
          const float was = d ? d[(size_t)k * a.K] : 0.f;
          unsigned again = __ballot_sync(0xffffffffu, !isfinite(was));
          while (again) {
            const int q = __ffs(again) - 1;
            again &= again - 1;
            const long at = (long)__shfl_sync(0xffffffffu, (long long)(d - out) + (long long)k * a.K, q);
            const float t = dw_inside(a.in, at, __shfl_sync(0xffffffffu, was, q));
            if (lane == q) d[(size_t)k * a.K] = t;
          }
        }
      }
    }
    if (bias) {
      // over the pixel rows: lanes first, then the warps' sums in order
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        if (p >= a.yplanes) break;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          float v = sum[p][k];
#pragma unroll
          for (int o = CH; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane < CH) C.red[p][warp][lane][k] = v;
        }
      }
      asm volatile("bar.sync 1, 256;\n" ::: "memory");
      for (int n = tid; n < a.yplanes * (RBY / 2); n += 256) {
        const int p = n / (RBY / 2), c = (n % (RBY / 2)) >> 3, k = n & 7;
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += C.red[p][w][c][k];
        a.wsb[(size_t)z * a.N + n0 + n] = v;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (tid == 0 && C.fail) atomicAdd(&g_tc_timeouts, 1);
  if (warp == 8 && C.fail != 2)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(a.cols));
}

// Sums over chunks in a fixed order: out[i] = sum_z ws[z][i] for i < n, and out2[i] =
// sum_z ws2[z][i] for i < n2.  G groups of 256 / G threads take every G-th chunk, and
// their sums are added in order: eight groups of a warp for many chunks (one
// thread per output walking up to 512 chunks left most of the GPU idle, 51 us for 9,216
// outputs), one group for few.  INSIDE: out is a weight gradient from tiles that reach
// past the images (see dw_inside).
template <int G, bool INSIDE>
__global__ void __launch_bounds__(256, 8) k_reduce_sums(const float *ws, long n, float *out, const float *ws2,
                                                        int n2, float *out2, int chunks,
                                                        const __grid_constant__ DwInputs v) {
  constexpr int L = 256 / G;
  __shared__ float red[G][L];
  const int l = threadIdx.x % L, g = threadIdx.x / L;
  const long nb1 = (n + L - 1) / L, nb2 = (n2 + L - 1) / L;
  float odd = 0.f;  // NaN once an entry of out is not finite
  for (long b = blockIdx.x; b < nb1 + nb2; b += gridDim.x) {
    const bool second = b >= nb1;
    const float *src = second ? ws2 : ws;
    const long m = second ? n2 : n, i = (second ? b - nb1 : b) * L + l;
    float s = 0.f;
    if (i < m)
      for (int z = g; z < chunks; z += G) s += src[(size_t)z * m + i];
    if (G > 1) {
      red[g][l] = s;
      __syncthreads();
      if (g == 0) {
#pragma unroll
        for (int k = 1; k < G; ++k) s += red[k][l];
      }
    }
    if (g == 0 && i < m) {
      (second ? out2 : out)[i] = s;
      if (INSIDE && !second) odd = fmaf(s, 0.f, odd);
    }
    if (G > 1) __syncthreads();
  }
  if (INSIDE && g == 0 && __any_sync(0xffffffffu, isnan(odd))) {  // whole warps
    for (long b = blockIdx.x; b < nb1; b += gridDim.x) {
      const long i = b * L + l;
      const float s = i < n ? out[i] : 0.f;
      unsigned again = __ballot_sync(0xffffffffu, !isfinite(s));
      while (again) {
        const int q = __ffs(again) - 1;
        again &= again - 1;
        const float t = dw_inside(v, i - (threadIdx.x & 31) + q, __shfl_sync(0xffffffffu, s, q));
        if ((threadIdx.x & 31) == q) out[i] = t;
      }
    }
  }
}

void reduce_sums(const float *ws, long n, float *out, const float *ws2, int n2, float *out2, int chunks,
                 cudaStream_t st, const DwInputs *v = nullptr) {
  const int per = chunks >= 16 ? 32 : 256;  // outputs of a block
  const long nblk = (n + per - 1) / per + (n2 + per - 1) / per;
  const int g = (int)(nblk < 8 * 1216 ? nblk : 8 * 1216);
  auto launch = [&](auto kernel) {
    kernel<<<g, 256, 0, st>>>(ws, n, out, ws2, n2, out2, chunks, v ? *v : DwInputs{});
  };
  if (chunks >= 16) v ? launch(k_reduce_sums<8, true>) : launch(k_reduce_sums<8, false>);
  else v ? launch(k_reduce_sums<1, true>) : launch(k_reduce_sums<1, false>);
}

struct WgHaloPlan {
  WgHaloArgs a;
  int rbx, rby, per, slots, gx, gy, box_w, box_h, box_p, ybox_w, ybox_h, ybox_p;
  size_t smem;
};

// Chooses the tiling, the output-channel block (nb), the blocks of a CTA (per)
// and the tile ranges, at most `most` of them (the workspace's slots), by an
// estimate in clocks like halo_plan's.
bool wgrad_halo_plan(const WgradArgs &v, int most, WgHaloPlan &best) {
  if (((v.Cin & 31) && v.Cin != 8) || (v.N & 31)) return false;
  const int rbx = v.Cin == 8 ? 16 : v.Cin & 63 ? 64 : 128, rby = v.N & 63 ? 64 : 128;
  auto up = [](long n, long d) { return (n + d - 1) / d; };
  auto inv = [](long d) { return (uint32_t)(((1ull << 32) + d - 1) / d); };
  const long rows = (long)v.B * (v.H + 1) - 1;
  const int tapb = rbx == 128 ? 5 : 3, planes = v.Cin * 2 / rbx;
  double best_c = 0.0;
  bool found = false;
  for (int mode : {TILE_WHOLE, TILE_TALL, TILE_FLAT}) {
    WgHaloArgs a{};
    a.mode = mode;
    a.tiles_x = (int)up(v.W, 8);
    a.tiles_y = (int)up(v.H, 16);
    long tiles;
    double boxes = 0.0;  // TMA boxes of a plane of x and one of dY
    if (mode == TILE_FLAT) {
      if (v.W > 30 || rbx != 128 || rby != 128) continue;
      a.tiles_x = 1;
      tiles = up(rows * (v.W + 1), 128);
      a.nrows = (v.W + 128 + 2 * (v.W + 2) - 1) / (v.W + 1) + 1;
      a.ky_st = (v.W + 1) * rbx;
      a.sbo = 8 * rbx;
      a.xps = a.yps = a.nrows * a.ky_st;
      boxes = v.H >= 8 ? 8.0 : 2.0 * a.nrows;
    } else {
      if (mode == TILE_TALL && rbx == 16) continue;  // its rows do not start on 128 bytes
      tiles = (mode == TILE_WHOLE ? (long)v.B * a.tiles_y : up(rows, 16)) * a.tiles_x;
      a.ky_st = a.sbo = 10 * rbx;
      a.xps = 180 * rbx;
      a.yps = 128 * rby;
      if (mode == TILE_TALL) boxes = v.H >= 8 ? 11.0 : 34.0;
    }
    a.ysbo = 8 * rby;
    a.tiles = (int)tiles;
    if ((rows + 40) * (v.W + 1) + 256 >= (1L << 32) / (v.W + 1) || (rows + 40) * (v.H + 1) >= (1L << 32) ||
        (tiles + 2) * a.tiles_x >= (1L << 32) || (tiles + 2) * a.tiles_y >= (1L << 32) || tiles > (1L << 30))
      continue;
    a.inv_h = inv(v.H + 1);
    a.inv_w = inv(v.W + 1);
    a.inv_x = inv(a.tiles_x);
    a.inv_y = inv(a.tiles_y);
    a.blocks = planes * tapb;
    for (int nb : {32, 64, 128, 256}) {
      if (nb > v.N || v.N % nb || nb % (rby / 2) || nb / (rby / 2) > 4) continue;
      const int ny = v.N / nb;
      for (int per : {9, 5, 4, 3, 2, 1}) {
        if (per * nb > 512 || per > a.blocks || (rbx == 16 && per != 3 && per != 1)) continue;
        const int gx = (int)up(a.blocks, per);
        if (gx * ny > 4 * kSms) continue;
        int xpl = 1;  // planes that a CTA's blocks touch
        for (int q = 0; q < a.blocks; q += per) {
          const int last = q + per < a.blocks ? q + per - 1 : a.blocks - 1;
          if (last / tapb - q / tapb + 1 > xpl) xpl = last / tapb - q / tapb + 1;
        }
        const int ypl = nb / (rby / 2);
        const long y_at = ((long)xpl * a.xps + 1023) & ~1023L;
        const long stage = (y_at + (long)ypl * a.yps + 1023) & ~1023L;
        const int nacc = 2 * per * nb <= 512 ? 2 : 1;
        int cols = 32;
        while (cols < nacc * per * nb) cols <<= 1;
        int na = WH_MAXA;
        while (na && 1024 + 128 + (long)sizeof(WgHaloCtl) + na * stage > (long)kSmemMax) --na;
        if (na < 2) continue;
        long z = kSms / (gx * ny);
        if (z < 1) z = 1;
        if (z > most) z = most;
        if (z > tiles) z = tiles;
        const long range = up(tiles, z);
        z = up(tiles, range);
        const long nf = up(range, up(tiles, most));  // flushes of a range
        const double mma = 8.0 * per * fmax(0.53 * nb, 32.0 + 0.25 * nb) + 300.0;
        const double load = (double)(xpl * a.xps + ypl * a.yps) / 45.0 + 75.0 * boxes * 0.5 * (xpl + ypl);
        const double flush = per * (nb / 32) * 400.0 + 2000.0;
        const double c = (double)up(z * gx * ny, kSms) *
                         (range * fmax(mma, load) + (nacc == 2 ? 1 : nf) * flush + 4000.0);
        if (found && c >= best_c) continue;
        found = true;
        best_c = c;
        best.a = a;
        best.a.range = (int)range;
        best.a.flush = (int)up(range, nf);
        best.a.xplanes = xpl;
        best.a.yplanes = ypl;
        best.a.nb = nb;
        best.a.nacc = nacc;
        best.a.na = na;
        best.a.stage = (int)stage;
        best.a.y_at = (int)y_at;
        best.a.cols = cols;
        best.a.off_ctl = (int)((na * stage + 127) & ~127L);
        best.smem = 1024 + best.a.off_ctl + sizeof(WgHaloCtl);
        best.per = per;
        best.slots = (int)z;
        best.gx = gx;
        best.gy = ny;
      }
    }
  }
  if (!found) return false;
  best.rbx = rbx;
  best.rby = rby;
  const int m = best.a.mode;
  best.box_w = m == TILE_FLAT ? v.W + 1 : 10;
  best.ybox_w = m == TILE_FLAT ? v.W + 1 : 8;
  best.box_h = m == TILE_WHOLE ? 18 : 1;
  best.ybox_h = m == TILE_WHOLE ? 16 : 1;
  best.box_p = m == TILE_WHOLE ? best.a.xplanes : 1;
  best.ybox_p = m == TILE_WHOLE ? best.a.yplanes : 1;
  return true;
}

template <int RBX, int RBY, int PER>
cudaError_t launch_wgrad_per(const WgHaloPlan &p, const WgMaps &m, cudaStream_t st) {
  static PerDevice attrs;
  cudaError_t e = allow_smem(k_wgrad_halo<RBX, RBY, PER>, kSmemMax, attrs);
  if (e != cudaSuccess) return e;
  k_wgrad_halo<RBX, RBY, PER><<<dim3(p.gx, p.gy, p.slots), WH_THREADS, p.smem, st>>>(m, p.a);
  return cudaGetLastError();
}
template <int RBX, int RBY>
cudaError_t launch_wgrad_halo(const WgHaloPlan &p, const WgMaps &m, cudaStream_t st) {
  if constexpr (RBX == 16)
    return p.per == 3 ? launch_wgrad_per<16, RBY, 3>(p, m, st) : launch_wgrad_per<16, RBY, 1>(p, m, st);
  else switch (p.per) {
    case 9: return launch_wgrad_per<RBX, RBY, 9>(p, m, st);
    case 5: return launch_wgrad_per<RBX, RBY, 5>(p, m, st);
    case 4: return launch_wgrad_per<RBX, RBY, 4>(p, m, st);
    case 3: return launch_wgrad_per<RBX, RBY, 3>(p, m, st);
    case 2: return launch_wgrad_per<RBX, RBY, 2>(p, m, st);
    default: return launch_wgrad_per<RBX, RBY, 1>(p, m, st);
  }
}

// weight partials (and, when db, bias partials into wsb) of every tile range;
// slots their number; with one slot the gradients themselves; outside: tiles reach past
// the images, the sums still need dw_inside
bool wgrad_halo(const WgradArgs &v, int most, float *wsb, float *dw, float *db, cudaStream_t st, int &slots,
                bool &outside, cudaError_t &rc) {
  WgHaloPlan p;
  if (!wgrad_halo_plan(v, most, p)) return false;
  WgMaps m;
  for (int k = 0; k < 4; ++k) {
    const int whole = p.a.mode == TILE_WHOLE;
    if (whole && k) {
      m.x[k] = m.x[0];
      m.y[k] = m.y[0];
    } else if (!encode_image(&m.x[k], v.x, v.B, v.H, v.W, v.ldx, v.Cin * 2 / p.rbx, p.rbx, p.box_w,
                             whole ? p.box_h : 1 << k, p.box_p) ||
               !encode_image(&m.y[k], v.dy, v.B, v.H, v.W, v.lddy, v.N * 2 / p.rby, p.rby, p.ybox_w,
                             whole ? p.ybox_h : 1 << k, p.ybox_p)) {
      return false;
    }
  }
  WgHaloArgs &a = p.a;
  a.ws = p.slots == 1 ? dw : v.ws;
  a.wsb = !db ? nullptr : p.slots == 1 ? db : wsb;
  a.B = v.B; a.H = v.H; a.W = v.W; a.N = v.N; a.K = v.K; a.Cin = v.Cin;
  a.in = dw_inputs(v);
  slots = p.slots;
  outside = a.mode != TILE_WHOLE || v.W % 8 || v.H % 16;
  a.inside = outside && slots == 1;
  rc = p.rbx == 128 ? (p.rby == 128 ? launch_wgrad_halo<128, 128>(p, m, st)
                                    : launch_wgrad_halo<128, 64>(p, m, st))
     : p.rbx == 64 ? (p.rby == 128 ? launch_wgrad_halo<64, 128>(p, m, st)
                                   : launch_wgrad_halo<64, 64>(p, m, st))
                   : (p.rby == 128 ? launch_wgrad_halo<16, 128>(p, m, st)
                                   : launch_wgrad_halo<16, 64>(p, m, st));
  return true;
}

// ------------------------------------------------------------- elementwise
// dy[p, c] = 0 where y[p, c] <= 0 (gradient through ReLU, given its output)
__global__ void k_relu_bwd(bf16_t *dy, int lddy, const bf16_t *y, int ldy, long P, int C) {
  const long n = P * C;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const long p = i / C;
    const int c = (int)(i - p * C);
    if (!(bf2f(y[p * ldy + c]) > 0.f)) dy[p * lddy + c] = 0;
  }
}

// Pooling and upsampling move 8 channels (16 bytes) per thread; channel
// counts, strides and offsets are multiples of 8.
__device__ __forceinline__ void unpack8(uint4 v, float f[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    f[2 * q] = bf2f((bf16_t)(w[q] & 0xffff));
    f[2 * q + 1] = bf2f((bf16_t)(w[q] >> 16));
  }
}
__device__ __forceinline__ uint4 pack8(const float f[8]) {
  uint32_t w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) w[q] = (uint32_t)f2bf(f[2 * q]) | ((uint32_t)f2bf(f[2 * q + 1]) << 16);
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ uint4 ld8(const bf16_t *p) { return *reinterpret_cast<const uint4 *>(p); }
__device__ __forceinline__ void st8(bf16_t *p, uint4 v) { *reinterpret_cast<uint4 *>(p) = v; }

// They are bound by HBM, so a thread's index work must stay small: one 32-bit index over
// (image row, pixel, 8 channels) and two divisions.  (A 64-bit index and three 64-bit
// divisions took 286 us for the level-0 pooling gradient of 64 images, this 176, 4.9 TB/s;
// upsampling 94 -> 83.  A block to an image row, with one division, took 197 and 83, and
// left most of its threads idle on narrow images: 4096 of 4 x 4, 8 channels, 90 us
// against 6.)
struct Piece {
  unsigned r, w, c;  // image row, pixel, first channel
  __device__ __forceinline__ Piece(unsigned t, unsigned n, unsigned C8) : r(t / n) {
    const unsigned i = t - r * n;
    w = i / C8;
    c = (i - w * C8) * 8;
  }
};

// 2x2 max pooling: x [B, 2H, 2W] (pixel stride ldx) -> y [B, H, W, C] dense
__global__ void __launch_bounds__(256) k_maxpool2(const bf16_t *x, int ldx, unsigned rows, int W, int C, bf16_t *y) {
  dependency_wait();
  dependency_release();
  const unsigned C8 = C >> 3, n = W * C8, total = rows * n;
  for (unsigned t = blockIdx.x * 256 + threadIdx.x; t < total; t += gridDim.x * 256) {
    const Piece q0(t, n, C8);
    const unsigned r = q0.r, w = q0.w, c = q0.c;
    const bf16_t *p = x + ((size_t)r * 4 * W + 2 * w) * ldx + c;
    const size_t row = (size_t)2 * W * ldx;
    float v[4][8], o[8];
    unpack8(ld8(p), v[0]);
    unpack8(ld8(p + ldx), v[1]);
    unpack8(ld8(p + row), v[2]);
    unpack8(ld8(p + row + ldx), v[3]);
#pragma unroll
    for (int q = 0; q < 8; ++q) o[q] = fmaxf(fmaxf(v[0][q], v[1][q]), fmaxf(v[2][q], v[3][q]));
    st8(y + ((size_t)r * W + w) * C + c, pack8(o));
  }
}

// gradient of 2x2 max pooling to the first maximum of each window, plus an
// optional skip gradient (dskip [.., ldskip] at channel offset skoff), zero
// where x <= 0 when relu_mask (x is a ReLU output): dx [B, 2H, 2W, C] dense
__global__ void __launch_bounds__(256) k_maxpool2_bwd(const bf16_t *x, int ldx, const bf16_t *dy,
                                                      const bf16_t *dskip, int ldskip, int skoff, unsigned rows,
                                                      int W, int C, int relu_mask, bf16_t *dx) {
  const unsigned C8 = C >> 3, n = W * C8, total = rows * n;
  for (unsigned t = blockIdx.x * 256 + threadIdx.x; t < total; t += gridDim.x * 256) {
    const Piece q0(t, n, C8);
    const unsigned r = q0.r, w = q0.w, c = q0.c;
    uint4 raw[4], sk[4];
    size_t pp[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      pp[q] = (size_t)r * 4 * W + (q >> 1) * 2 * W + 2 * w + (q & 1);
      raw[q] = ld8(x + pp[q] * ldx + c);
    }
    const uint4 gr = ld8(dy + ((size_t)r * W + w) * C + c);
    if (dskip)
#pragma unroll
      for (int q = 0; q < 4; ++q) sk[q] = ld8(dskip + pp[q] * ldskip + skoff + c);
    float v[4][8], g[8], m[8];
    bool taken[8];
    unpack8(gr, g);
#pragma unroll
    for (int q = 0; q < 4; ++q) unpack8(raw[q], v[q]);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      m[k] = fmaxf(fmaxf(v[0][k], v[1][k]), fmaxf(v[2][k], v[3][k]));
      taken[k] = false;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float s[8], o[8];
      if (dskip) unpack8(sk[q], s);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        o[k] = 0.f;
        if (!taken[k] && v[q][k] == m[k]) {
          o[k] = g[k];
          taken[k] = true;
        }
        if (dskip) o[k] += s[k];
        if (relu_mask && !(v[q][k] > 0.f)) o[k] = 0.f;
      }
      st8(dx + pp[q] * C + c, pack8(o));
    }
  }
}

// nearest 2x upsampling: x [B, H, W, C] dense -> y [B, 2H, 2W, ldy] at channel offset yoff
__global__ void __launch_bounds__(256) k_upsample2(const bf16_t *x, unsigned rows, int W, int C, bf16_t *y, int ldy,
                                                   int yoff) {
  dependency_wait();
  dependency_release();
  const unsigned C8 = C >> 3, n = W * C8, total = rows * n;
  for (unsigned t = blockIdx.x * 256 + threadIdx.x; t < total; t += gridDim.x * 256) {
    const Piece q0(t, n, C8);
    const unsigned r = q0.r, w = q0.w, c = q0.c;
    const uint4 v = ld8(x + ((size_t)r * W + w) * C + c);
    bf16_t *p = y + ((size_t)r * 4 * W + 2 * w) * ldy + yoff + c;
    const size_t row = (size_t)2 * W * ldy;
    st8(p, v);
    st8(p + ldy, v);
    st8(p + row, v);
    st8(p + row + ldy, v);
  }
}

// gradient of nearest 2x upsampling: dy [B, 2H, 2W, lddy] channels 0..C-1 ->
// dx [B, H, W, C], zero where mask <= 0 (mask [B, H, W, ldm], may be null)
__global__ void __launch_bounds__(256) k_upsample2_bwd(const bf16_t *dy, int lddy, unsigned rows, int W, int C,
                                                       const bf16_t *mask, int ldm, bf16_t *dx) {
  const unsigned C8 = C >> 3, n = W * C8, total = rows * n;
  for (unsigned t = blockIdx.x * 256 + threadIdx.x; t < total; t += gridDim.x * 256) {
    const Piece q0(t, n, C8);
    const unsigned r = q0.r, w = q0.w, c = q0.c;
    const size_t pix = (size_t)r * W + w;
    uint4 raw[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      raw[q] = ld8(dy + ((size_t)r * 4 * W + (q >> 1) * 2 * W + 2 * w + (q & 1)) * lddy + c);
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, d[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      unpack8(raw[q], d);
#pragma unroll
      for (int k = 0; k < 8; ++k) s[k] += d[k];
    }
    if (mask) {
      float mk[8];
      unpack8(ld8(mask + pix * ldm + c), mk);
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (!(mk[k] > 0.f)) s[k] = 0.f;
    }
    st8(dx + pix * C + c, pack8(s));
  }
}

// ------------------------------------------------------------------- head
// z[p] = b + sum_c x[p, c] w[c]   (1x1 convolution to one logit, FP32), channels in
// increasing order.  A pixel's channels are read in 16-byte rows when they
// allow it (64 images, 32 channels: 2-byte reads took 232 us, these 50).
__global__ void __launch_bounds__(256) k_head_fwd(const bf16_t *x, int P, int C, int vec, const float *w,
                                                  const float *b, float *z) {
  dependency_wait();
  dependency_release();
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x) {
    const bf16_t *xp = x + (size_t)p * C;
    float s = b[0];
    if (vec) {
      for (int c0 = 0; c0 < C; c0 += 32) {
        uint4 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (c0 + 8 * q < C) v[q] = ld8(xp + c0 + 8 * q);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (c0 + 8 * q < C) {
            float f[8];
            unpack8(v[q], f);
#pragma unroll
            for (int k = 0; k < 8; ++k) s += f[k] * w[c0 + 8 * q + k];
          }
      }
    } else {
      for (int c = 0; c < C; ++c) s += bf2f(xp[c]) * w[c];
    }
    z[p] = s;
  }
}

// dx[p, c] = dz[p] w[c]; per-chunk partials of dw[c] = sum_p dz[p] x[p, c]
// and db = sum_p dz[p] into ws[chunk][C], wsb[chunk]
__global__ void k_head_bwd(const bf16_t *x, int P, int C, const float *w, const float *dz,
                           bf16_t *dx, int chunk, float *ws, float *wsb) {
  const int z = blockIdx.x;
  const int pend = min(P, (z + 1) * chunk);
  __shared__ float red[33][33];
  const int c = threadIdx.x & 31, lane_p = threadIdx.x >> 5;  // 32 channels x 8 pixel lanes
  float s = 0.f, sb = 0.f;
  for (int p = z * chunk + lane_p; p < pend; p += 8) {
    const float g = dz[p];
    for (int cc = c; cc < C; cc += 32) {
      const float xv = bf2f(x[(size_t)p * C + cc]);
      // x is a ReLU output: its gradient is zero where x <= 0
      dx[(size_t)p * C + cc] = xv > 0.f ? f2bf(g * w[cc]) : (bf16_t)0;
      if (cc == c) s += g * xv;
    }
    sb += g;
  }
  red[lane_p][c] = s;
  if (c == 0) red[lane_p][32] = sb;
  __syncthreads();
  if (lane_p == 0) {
    float t = 0.f, tb = 0.f;
    for (int q = 0; q < 8; ++q) {
      t += red[q][c];
      tb += red[q][32];
    }
    if (c < C) ws[(size_t)z * C + c] = t;
    if (c == 0) wsb[z] = tb;
  }
}

// The same for C = 8, 16 or 32 and aligned rows: a thread holds 8 channels (16 bytes) of
// every (2048 / C)-th pixel of the chunk, four at a time (2-byte accesses took 318 us
// for 64 images of 32 channels, this 84).
template <int C>
__global__ void __launch_bounds__(256) k_head_bwd8(const bf16_t *x, int P, const float *w, const float *dz,
                                                   bf16_t *dx, int chunk, float *ws, float *wsb) {
  constexpr int C8 = C / 8, LANES = 256 / C8;
  __shared__ float red[8][C + 1];
  const int z = blockIdx.x, cg = threadIdx.x % C8, pl = threadIdx.x / C8;
  const int pend = min(P, (z + 1) * chunk);
  float wc[8], s[8], sb = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    wc[k] = w[cg * 8 + k];
    s[k] = 0.f;
  }
  for (int p0 = z * chunk + pl; p0 < pend; p0 += 4 * LANES) {
    uint4 v[4];
    float g[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int p = p0 + q * LANES;
      g[q] = p < pend ? dz[p] : 0.f;
      v[q] = p < pend ? ld8(x + (size_t)p * C + cg * 8) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int p = p0 + q * LANES;
      if (p >= pend) break;
      float f[8], o[8];
      unpack8(v[q], f);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        o[k] = f[k] > 0.f ? g[q] * wc[k] : 0.f;
        s[k] += g[q] * f[k];
      }
      sb += g[q];
      st8(dx + (size_t)p * C + cg * 8, pack8(o));
    }
  }
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
  for (int o = C8; o < 32; o <<= 1) {
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    sb += __shfl_xor_sync(0xffffffffu, sb, o);
  }
  if (lane < C8) {
#pragma unroll
    for (int k = 0; k < 8; ++k) red[wp][lane * 8 + k] = s[k];
    if (lane == 0) red[wp][C] = sb;
  }
  __syncthreads();
  if (threadIdx.x <= C) {
    float t = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
    if (threadIdx.x < C) ws[(size_t)z * C + threadIdx.x] = t;
    else wsb[z] = t;
  }
}

// ------------------------------------------------------------------- loss
// class-weighted binary cross-entropy with logits, mean over n elements:
// dz = (pw t (sigma - 1) + (1 - t) sigma) / n; per-block loss partials
__global__ void k_bce(const float *z, const uint8_t *t, long n, float pw, float *dz, float *ws) {
  __shared__ float red[256];
  float s = 0.f;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const float zi = z[i];
    const float tt = t[i] ? 1.f : 0.f;
    // log(1 + e^-z) and log(1 + e^z) without overflow
    const float sp_neg = fmaxf(-zi, 0.f) + log1pf(expf(-fabsf(zi)));
    const float sp_pos = sp_neg + zi;
    s += pw * tt * sp_neg + (1.f - tt) * sp_pos;
    const float sig = 1.f / (1.f + expf(-zi));
    dz[i] = (pw * tt * (sig - 1.f) + (1.f - tt) * sig) / (float)n;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) ws[blockIdx.x] = red[0];
}

// soft Dice over B samples of n_per logits each: per-(sample, chunk) partial
// sums of p t, p and t (p = sigma(z)), block (c, b) covering elements
// [c * chunk, (c + 1) * chunk) of sample b
constexpr int kDiceChunk = 4096;

__device__ __forceinline__ float block_sum256(float v, float *red) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  const float s = red[0];
  __syncthreads();
  return s;
}

__global__ void __launch_bounds__(256) k_dice_partial(const float *z, const uint8_t *t, long n_per,
                                                      float *ws) {
  __shared__ float red[256];
  const int c = blockIdx.x, b = blockIdx.y, nchunk = gridDim.x;
  const long lo = (long)c * kDiceChunk, hi = min(n_per, lo + kDiceChunk);
  const float *zb = z + (size_t)b * n_per;
  const uint8_t *tb = t + (size_t)b * n_per;
  float spt = 0.f, sp = 0.f, st = 0.f;
  for (long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const float p = 1.f / (1.f + expf(-zb[i]));
    const float tt = tb[i] ? 1.f : 0.f;
    spt += p * tt;
    sp += p;
    st += tt;
  }
  spt = block_sum256(spt, red);
  sp = block_sum256(sp, red);
  st = block_sum256(st, red);
  if (threadIdx.x == 0) {
    float *o = ws + ((size_t)b * nchunk + c) * 3;
    o[0] = spt;
    o[1] = sp;
    o[2] = st;
  }
}

// dz += -(w / B) (2 t (S + eps) - (2 I + eps)) / (S + eps)^2 p (1 - p), the
// sample's sums I = sum p t, S = sum p + sum t added in chunk order
__global__ void __launch_bounds__(256) k_dice_grad(const float *z, const uint8_t *t, long n_per,
                                                   int B, float w, float eps, const float *ws,
                                                   float *dz) {
  const int c = blockIdx.x, b = blockIdx.y, nchunk = gridDim.x;
  float I = 0.f, S = 0.f;
  for (int q = 0; q < nchunk; ++q) {
    const float *o = ws + ((size_t)b * nchunk + q) * 3;
    I += o[0];
    S += o[1] + o[2];
  }
  const float Se = S + eps, num = 2.f * I + eps, scale = -w / ((float)B * Se * Se);
  const long lo = (long)c * kDiceChunk, hi = min(n_per, lo + kDiceChunk);
  const float *zb = z + (size_t)b * n_per;
  const uint8_t *tb = t + (size_t)b * n_per;
  float *db = dz + (size_t)b * n_per;
  for (long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const float p = 1.f / (1.f + expf(-zb[i]));
    const float tt = tb[i] ? 1.f : 0.f;
    db[i] += scale * (2.f * tt * Se - num) * p * (1.f - p);
  }
}

// loss = w (1 - mean_b D_b), D_b = (2 I_b + eps) / (S_b + eps), one block: a
// sample's chunks in order by one thread, the samples' terms one after another by
// thread 0 (the Dice term of 64 images of 64,000 pixels, all three kernels: 84 us
// when a single thread walked all of it, 34 so)
__global__ void __launch_bounds__(256) k_dice_loss(const float *ws, int nchunk, int B, float w, float eps,
                                                   float *loss) {
  __shared__ float term[256];
  float d = 0.f;
  for (int b0 = 0; b0 < B; b0 += 256) {
    const int b = b0 + threadIdx.x;
    if (b < B) {
      float I = 0.f, S = 0.f;
      for (int q = 0; q < nchunk; ++q) {
        const float *o = ws + ((size_t)b * nchunk + q) * 3;
        I += o[0];
        S += o[1] + o[2];
      }
      term[threadIdx.x] = (2.f * I + eps) / (S + eps);
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int q = 0; q < min(256, B - b0); ++q) d += term[q];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss[0] = w * (1.f - d / (float)B);
}
__global__ void __launch_bounds__(256) k_sum_scaled(const float *ws, int m, float scale, float *out) {
  // added one after another in a fixed order, from shared memory (from global
  // memory the two sums of a loss took 230 us, nearly all of it waiting)
  __shared__ __align__(16) float v[4096];
  float s = 0.f;
  for (int i0 = 0; i0 < m; i0 += 4096) {
    const int k = min(4096, m - i0);
    for (int i = threadIdx.x; i < k; i += 256) v[i] = ws[i0 + i];
    __syncthreads();
    if (threadIdx.x == 0) {
      int i = 0;
      for (; i + 16 <= k; i += 16) {
        float4 a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = *reinterpret_cast<const float4 *>(v + i + 4 * q);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          s += a[q].x;
          s += a[q].y;
          s += a[q].z;
          s += a[q].w;
        }
      }
      for (; i < k; ++i) s += v[i];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = s * scale;
}

// ------------------------------------------------------------------- adam
// w -= lr * mhat / (sqrt(vhat) + eps); BF16 copy of w, and for 3x3 weights
// [Cout][3][3][Cin] the transposed, flipped copy wt[Cin][3][3][Cout] with
// wt[c][ky][kx][o] = w[o][2-ky][2-kx][c] used by the data gradient
__global__ void k_adam(float *w, const float *g, float *m, float *v, long n, float lr, float b1,
                       float b2, float eps, float c1, float c2, bf16_t *wb, bf16_t *wt, int Cout,
                       int Cin) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    const bf16_t h = f2bf(wi);
    if (wb) wb[i] = h;
    if (wt) {
      const int c = (int)(i % Cin);
      const long r = i / Cin;
      const int kx = (int)(r % 3), ky = (int)((r / 3) % 3), o = (int)(r / 9);
      wt[(((size_t)c * 3 + (2 - ky)) * 3 + (2 - kx)) * Cout + o] = h;
    }
  }
}

__global__ void k_to_bf16(const float *x, long n, bf16_t *y) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    y[i] = f2bf(x[i]);
}

// Launches of the pooling and upsampling kernels: launch(first image row, rows, blocks), one
// unless the pieces (a pixel's 8 channels) need more than 31 bits
template <class F>
cudaError_t for_pieces(long rows, long per_row, F launch) {
  const long most = per_row < (1L << 31) ? ((1L << 31) - 1) / per_row : 1;
  for (long r = 0; r < rows; r += most) {
    const long k = rows - r < most ? rows - r : most, blocks = (k * per_row + 255) / 256;
    const cudaError_t e = launch(r, (unsigned)k, (unsigned)(blocks < (1 << 22) ? blocks : 1 << 22));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int grid_1d(long n, int block) {
  long b = (n + block - 1) / block;
  return (int)(b < 1 ? 1 : (b > 4 * 1216 ? 4 * 1216 : b));
}

}  // namespace

// ======================================================================= ABI
extern "C" {

int cem_sg_conv3x3(const void *x, int B, int H, int W, int Cin, int ldx, const void *w,
                   const float *bias, int Cout, int relu, const void *mask, int ldmask, void *y,
                   int ldy, int yoff, void *stream) {
  if (!x || !w || !y || B < 1 || H < 1 || W < 1 || Cin < 8 || (Cin & 7) || ldx < Cin ||
      (ldx & 7) || Cout < 2 || (Cout & 1) || ldy < yoff + Cout || (yoff & 1) ||
      (mask && (ldmask < Cout || (ldmask & 1))))
    return CEM_SG_ERR_ARG;
  ConvArgs a;
  a.x = (const bf16_t *)x;
  a.w = (const bf16_t *)w;
  a.bias = bias;
  a.y = (bf16_t *)y;
  a.B = B; a.H = H; a.W = W; a.Cin = Cin; a.ldx = ldx; a.N = Cout; a.K = 9 * Cin;
  a.relu = relu; a.ldy = ldy; a.yoff = yoff; a.P = B * H * W;
  a.mask = (const bf16_t *)mask;
  a.ldm = ldmask;
  cudaStream_t st = (cudaStream_t)stream;
  if (g_use_tc) {
    cudaError_t e;
    if (!conv_halo(a, st, e))
      e = Cout > 128 ? launch_conv_tc<256>(a, st)
                  : Cout > 64 ? launch_conv_tc<128>(a, st)
                  : Cout > 32 ? launch_conv_tc<64>(a, st) : launch_conv_tc<32>(a, st);
    return e == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
  }
  dim3 grid((a.P + FBM - 1) / FBM, (Cout + FBN - 1) / FBN);
  k_conv3x3<<<grid, 256, 0, st>>>(a);
  return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

long cem_sg_wgrad_workspace(int B, int H, int W, int Cin, int Cout) {
  const long P = (long)B * H * W;
  long splits = (P + 4095) / 4096;
  if (splits > 512) splits = 512;
  return splits * (long)Cout * 9 * Cin * 4 + (long)Cout * 4 * 1024;
}

int cem_sg_conv3x3_wgrad(const void *x, int ldx, const void *dy, int lddy, int B, int H, int W,
                         int Cin, int Cout, float *dw, float *db, void *ws, long ws_bytes,
                         void *stream) {
  if (!x || !dy || !dw || !ws || B < 1 || H < 1 || W < 1 || Cin < 8 || (Cin & 7) ||
      (ldx & 7) || ldx < Cin || Cout < 8 || (Cout & 7) || lddy < Cout || (lddy & 7))
    return CEM_SG_ERR_ARG;
  if (ws_bytes < cem_sg_wgrad_workspace(B, H, W, Cin, Cout)) return CEM_SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  WgradArgs a;
  a.x = (const bf16_t *)x;
  a.dy = (const bf16_t *)dy;
  a.ws = (float *)ws;
  a.B = B; a.H = H; a.W = W; a.Cin = Cin; a.ldx = ldx; a.lddy = lddy; a.N = Cout;
  a.K = 9 * Cin; a.P = B * H * W;
  int splits = (a.P + 4095) / 4096;
  if (splits > 512) splits = 512;
  a.chunk = ((a.P + splits - 1) / splits + GBK - 1) / GBK * GBK;
  splits = (a.P + a.chunk - 1) / a.chunk;
  const long nw = (long)Cout * a.K;
  if (g_use_tc) {
    cudaError_t he;
    int hs;
    bool outside;
    // the bias partials lie behind the weight partials of `splits` chunks
    float *wsb = a.ws + (size_t)splits * Cout * a.K;
    if (wgrad_halo(a, splits, wsb, dw, db, st, hs, outside, he)) {
      if (he != cudaSuccess) return CEM_SG_ERR_CUDA;
      if (hs == 1) return CEM_SG_OK;  // the kernel wrote dw and db
      const DwInputs in = dw_inputs(a);
      reduce_sums(a.ws, nw, dw, wsb, db ? Cout : 0, db, hs, st, outside ? &in : nullptr);
      return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
    }
    // tcgen05: dW^T tiles of 128 k' x BN outputs; bias sums by a separate
    // coalesced reduction into the workspace after the weight partials
    a.wsb = nullptr;
    cudaError_t e = Cout > 128 ? launch_wgrad_tc<256>(a, splits, st)
                  : Cout > 64 ? launch_wgrad_tc<128>(a, splits, st)
                              : launch_wgrad_tc<64>(a, splits, st);
    if (e != cudaSuccess) return CEM_SG_ERR_CUDA;
    reduce_sums(a.ws, nw, dw, nullptr, 0, nullptr, splits, st);
    if (db) {
      // more pixel chunks than the weight partials use: the sums are a pure
      // bandwidth pass (at most 608 chunks, four per SM; the workspace holds 1024)
      float *wsb = a.ws + (size_t)splits * Cout * a.K;
      const long bs = (a.P + 2047) / 2048;
      const int bsplits = (int)(bs < 1 ? 1 : (bs > 608 ? 608 : bs));
      const int bch = (a.P + bsplits - 1) / bsplits;
      k_colsum8<<<bsplits, 256, 0, st>>>(a.dy, a.P, Cout, lddy, bch, wsb);
      reduce_sums(wsb, Cout, db, nullptr, 0, nullptr, bsplits, st);
    }
    return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
  }
  a.wsb = db ? a.ws + (size_t)splits * Cout * a.K : nullptr;
  dim3 grid((Cout + GBM - 1) / GBM, (a.K + GBN - 1) / GBN, splits);
  k_conv3x3_wgrad<<<grid, 256, 0, st>>>(a);
  reduce_sums(a.ws, nw, dw, a.wsb, db ? Cout : 0, db, splits, st);
  return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

int cem_sg_relu_bwd(void *dy, int lddy, const void *y, int ldy, long P, int C, void *stream) {
  if (!dy || !y || P < 0 || C < 1 || lddy < C || ldy < C) return CEM_SG_ERR_ARG;
  k_relu_bwd<<<grid_1d(P * C, 256), 256, 0, (cudaStream_t)stream>>>((bf16_t *)dy, lddy,
                                                                    (const bf16_t *)y, ldy, P, C);
  return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

int cem_sg_maxpool2(const void *x, int ldx, int B, int H, int W, int C, void *y, void *stream) {
  if (!x || !y || B < 1 || H < 1 || W < 1 || C < 8 || (C & 7) || ldx < C || (ldx & 7))
    return CEM_SG_ERR_ARG;
  const cudaError_t e = for_pieces((long)B * H, (long)W * (C >> 3), [&](long r, unsigned rows, unsigned blocks) {
    return launch_dependent(k_maxpool2, blocks, 256, 0, (cudaStream_t)stream,
                            (const bf16_t *)x + r * 4 * W * ldx, ldx, rows, W, C, (bf16_t *)y + r * W * C);
  });
  return e == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

int cem_sg_maxpool2_bwd(const void *x, int ldx, const void *dy, const void *dskip, int ldskip,
                        int skoff, int B, int H, int W, int C, int relu_mask, void *dx,
                        void *stream) {
  if (!x || !dy || !dx || B < 1 || H < 1 || W < 1 || C < 8 || (C & 7) || ldx < C || (ldx & 7) ||
      (dskip && (ldskip < skoff + C || (ldskip & 7) || (skoff & 7))))
    return CEM_SG_ERR_ARG;
  const cudaError_t e = for_pieces((long)B * H, (long)W * (C >> 3), [&](long r, unsigned rows, unsigned blocks) {
    k_maxpool2_bwd<<<blocks, 256, 0, (cudaStream_t)stream>>>(
        (const bf16_t *)x + r * 4 * W * ldx, ldx, (const bf16_t *)dy + r * W * C,
        dskip ? (const bf16_t *)dskip + r * 4 * W * ldskip : nullptr, ldskip, skoff, rows, W, C, relu_mask,
        (bf16_t *)dx + r * 4 * W * C);
    return cudaGetLastError();
  });
  return e == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

int cem_sg_upsample2(const void *x, int B, int H, int W, int C, void *y, int ldy, int yoff,
                     void *stream) {
  if (!x || !y || B < 1 || H < 1 || W < 1 || C < 8 || (C & 7) || ldy < yoff + C || (ldy & 7) ||
      (yoff & 7))
    return CEM_SG_ERR_ARG;
  const cudaError_t e = for_pieces((long)B * H, (long)W * (C >> 3), [&](long r, unsigned rows, unsigned blocks) {
    return launch_dependent(k_upsample2, blocks, 256, 0, (cudaStream_t)stream, (const bf16_t *)x + r * W * C, rows,
                            W, C, (bf16_t *)y + r * 4 * W * ldy, ldy, yoff);
  });
  return e == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

int cem_sg_upsample2_bwd(const void *dy, int lddy, int B, int H, int W, int C, const void *mask,
                         int ldmask, void *dx, void *stream) {
  if (!dy || !dx || B < 1 || H < 1 || W < 1 || C < 8 || (C & 7) || lddy < C || (lddy & 7) ||
      (mask && (ldmask < C || (ldmask & 7))))
    return CEM_SG_ERR_ARG;
  const cudaError_t e = for_pieces((long)B * H, (long)W * (C >> 3), [&](long r, unsigned rows, unsigned blocks) {
    k_upsample2_bwd<<<blocks, 256, 0, (cudaStream_t)stream>>>(
        (const bf16_t *)dy + r * 4 * W * lddy, lddy, rows, W, C,
        mask ? (const bf16_t *)mask + r * W * ldmask : nullptr, ldmask, (bf16_t *)dx + r * W * C);
    return cudaGetLastError();
  });
  return e == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

int cem_sg_head_fwd(const void *x, int P, int C, const float *w, const float *b, float *z,
                    void *stream) {
  if (!x || !w || !b || !z || P < 1 || C < 1) return CEM_SG_ERR_ARG;
  const int vec = !(C & 7) && !((uintptr_t)x & 15);
  return launch_dependent(k_head_fwd, grid_1d(P, 256), 256, 0, (cudaStream_t)stream, (const bf16_t *)x, P, C,
                          vec, w, b, z) == cudaSuccess
             ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

long cem_sg_head_workspace(int P, int C) {
  const long nz = (P + 4095) / 4096;
  return nz * (C + 1) * 4;
}

int cem_sg_head_bwd(const void *x, int P, int C, const float *w, const float *dz, void *dx,
                    float *dw, float *db, void *ws, long ws_bytes, void *stream) {
  if (!x || !w || !dz || !dx || !dw || !db || !ws || P < 1 || C < 1 || C > 32)
    return CEM_SG_ERR_ARG;
  if (ws_bytes < cem_sg_head_workspace(P, C)) return CEM_SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int chunk = 4096, nz = (P + chunk - 1) / chunk;
  float *wsf = (float *)ws, *wsb = wsf + (size_t)nz * C;
  const bf16_t *xb = (const bf16_t *)x;
  bf16_t *db16 = (bf16_t *)dx;
  const bool vec = !(((uintptr_t)x | (uintptr_t)dx) & 15);
  if (vec && C == 32) k_head_bwd8<32><<<nz, 256, 0, st>>>(xb, P, w, dz, db16, chunk, wsf, wsb);
  else if (vec && C == 16) k_head_bwd8<16><<<nz, 256, 0, st>>>(xb, P, w, dz, db16, chunk, wsf, wsb);
  else if (vec && C == 8) k_head_bwd8<8><<<nz, 256, 0, st>>>(xb, P, w, dz, db16, chunk, wsf, wsb);
  else k_head_bwd<<<nz, 256, 0, st>>>(xb, P, C, w, dz, db16, chunk, wsf, wsb);
  reduce_sums(wsf, C, dw, wsb, 1, db, nz, st);
  return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

long cem_sg_bce_workspace(long n) { return 4 * 1216 * 4 + 16; }

int cem_sg_bce(const float *z, const unsigned char *t, long n, float pos_weight, float *dz,
               float *loss, void *ws, long ws_bytes, void *stream) {
  if (!z || !t || !dz || !loss || !ws || n < 1) return CEM_SG_ERR_ARG;
  if (ws_bytes < cem_sg_bce_workspace(n)) return CEM_SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int g = grid_1d(n, 256);
  k_bce<<<g, 256, 0, st>>>(z, t, n, pos_weight, dz, (float *)ws);
  k_sum_scaled<<<1, 256, 0, st>>>((const float *)ws, g, 1.f / (float)n, loss);
  return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

long cem_sg_dice_workspace(int B, long n_per) {
  if (B < 1 || n_per < 1) return 0;
  return (long)B * ((n_per + kDiceChunk - 1) / kDiceChunk) * 3 * 4;
}

int cem_sg_dice(const float *z, const unsigned char *t, int B, long n_per, float weight, float eps,
                float *dz, float *loss, void *ws, long ws_bytes, void *stream) {
  if (!z || !t || !dz || !loss || !ws || B < 1 || n_per < 1 || !(eps > 0.f)) return CEM_SG_ERR_ARG;
  if (ws_bytes < cem_sg_dice_workspace(B, n_per)) return CEM_SG_ERR_ARG;
  const long nchunk = (n_per + kDiceChunk - 1) / kDiceChunk;
  if (nchunk > 65535 || B > 65535) return CEM_SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const dim3 grid((unsigned)nchunk, (unsigned)B);
  k_dice_partial<<<grid, 256, 0, st>>>(z, t, n_per, (float *)ws);
  k_dice_grad<<<grid, 256, 0, st>>>(z, t, n_per, B, weight, eps, (const float *)ws, dz);
  k_dice_loss<<<1, 256, 0, st>>>((const float *)ws, (int)nchunk, B, weight, eps, loss);
  return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

int cem_sg_adam(float *w, const float *g, float *m, float *v, long n, float lr, float beta1,
                float beta2, float eps, int step, void *w_bf16, void *wt_bf16, int Cout, int Cin,
                void *stream) {
  if (!w || !g || !m || !v || n < 1 || step < 1 || !(lr >= 0.f)) return CEM_SG_ERR_ARG;
  if (wt_bf16 && (Cout < 1 || Cin < 1 || (long)Cout * 9 * Cin != n)) return CEM_SG_ERR_ARG;
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  k_adam<<<grid_1d(n, 256), 256, 0, (cudaStream_t)stream>>>(
      w, g, m, v, n, lr, beta1, beta2, eps, c1, c2, (bf16_t *)w_bf16, (bf16_t *)wt_bf16, Cout, Cin);
  return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

int cem_sg_set_gemm_path(int use_tcgen05) {
  g_use_tc = use_tcgen05 ? 1 : 0;
  return CEM_SG_OK;
}

int cem_sg_timeouts(int *count) {
  if (!count) return CEM_SG_ERR_ARG;
  return cudaMemcpyFromSymbol(count, g_tc_timeouts, sizeof(int)) == cudaSuccess ? CEM_SG_OK
                                                                             : CEM_SG_ERR_CUDA;
}

int cem_sg_to_bf16(const float *x, long n, void *y, void *stream) {
  if (!x || !y || n < 0) return CEM_SG_ERR_ARG;
  k_to_bf16<<<grid_1d(n, 256), 256, 0, (cudaStream_t)stream>>>(x, n, (bf16_t *)y);
  return cudaGetLastError() == cudaSuccess ? CEM_SG_OK : CEM_SG_ERR_CUDA;
}

}  // extern "C"
