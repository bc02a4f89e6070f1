// Learned heuristic network: crop extraction, BF16 forward and backward
// passes on the tensor cores, and Adam (training and inference kernels).
//
// The paper's multi-heuristic search (Sec. IV-B/C) admits any inadmissible
// heuristic and names learned ones as the next step (Sec. IV-C, Sec. VI); it
// fixes no network. This one predicts y = log(1 + edge cost) of one MSGT
// successor from a 2 x 64 x 64 crop (observed depth, parent z-buffer) centred
// on the projected hypothesis, and a one-hot of (mesh, yaw):
//   conv 3x3 2->32 s1, 32->64 s2, 64->128 s2, 128->128 s2 (pad 1, ReLU)
//   -> flatten (h, w, c) ++ one-hot -> FC 96 (ReLU) -> FC 1; loss 0.5 (pred - y)^2
//
// Data layout: activations NHWC bfloat16. Every convolution is one GEMM over
// rows = output pixels (N x Ho x Wo) and columns = (tap, channel). The 2-channel
// input layer works on mma.sync from strips of the crop (k_conv1, k_wgrad1); the
// others, their data gradients (k_conv_tma) and their weight gradients
// (k_wgrad_tma) run on tcgen05 with operands loaded by TMA. Weight gradients are
// split along the pixel reduction and summed in a fixed order (deterministic).
// The FC layers use k_gemm: mma.sync m16n8k16 (BF16 in, FP32 accumulate) fed by
// a 3-stage cp.async pipeline and ldmatrix (.trans for MN-contiguous operands).
// Gradients between layers are rounded to bfloat16, like the activations;
// weights keep an FP32 master copy updated by Adam and re-rounded to bfloat16
// after each step.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "perch_ctx.h"

using namespace perch;
typedef __nv_bfloat16 bf16;

namespace {

constexpr int kCrop = 64;
constexpr int kHidden = 96;
constexpr int kConvs = 4;
constexpr int kCin[kConvs] = {2, 32, 64, 128};
constexpr int kCout[kConvs] = {32, 64, 128, 128};
constexpr int kStride[kConvs] = {1, 2, 2, 2};
constexpr int kHin[kConvs] = {64, 64, 32, 16};  // input side of each layer
constexpr int kFeat = 128 * 8 * 8;               // flattened last conv output
constexpr float kMissing = -4.0f, kClamp = 3.0f;
constexpr double kScale = 10.0;  // per metre

int round32(int v) { return (v + 31) / 32 * 32; }
int kp_of(int l) { return round32(9 * kCin[l]); }

// ---------------------------------------------------------------- GEMM
constexpr int BM = 128, BK = 32, LDS = BK + 8, STAGES = 3;

struct GemmArgs {
  const bf16* A;  // [M][lda], K-contiguous
  long long lda;
  const bf16* B;  // [N][ldb], K-contiguous
  long long ldb;
  int M, N, K, Ksplit;  // split z covers columns [z Ksplit, min(K, (z + 1) Ksplit))
  float* Cf;  // output (partial z at Cf + z split_stride)
  long long ldc, split_stride;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool pred) {
  const int sz = pred ? 16 : 0;  // src-size 0: the 16 bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(sz));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// C[M x N] = A B^T over K. A is K-contiguous (AK: element (m, k) at
// m lda + k) or M-contiguous (element (m, k) at k lda + m); B likewise
// (BKC: (n, k) at n ldb + k, else k ldb + n). MN-contiguous operands are
// staged as [k][m] tiles and fed to the tensor cores with ldmatrix .trans, so
// weight and data gradients need no transposed copies. 256 threads; CTA tile
// 128 x BN; warp tile (128 / (8 / (BN / 32))) x 32. K and Ksplit multiples of
// 32; an MN-contiguous operand needs its M (or N) to be a multiple of 8.
template <int BN, bool AK, bool BKC>
__global__ void __launch_bounds__(256) k_gemm(GemmArgs p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int A_LD = AK ? LDS : BM + 8, A_STAGE = AK ? BM * LDS : BK * (BM + 8);
  constexpr int B_LD = BKC ? LDS : BN + 8, B_STAGE = BKC ? BN * LDS : BK * (BN + 8);
  bf16* As = reinterpret_cast<bf16*>(smem_raw);  // [STAGES][A_STAGE]
  bf16* Bs = As + STAGES * A_STAGE;               // [STAGES][B_STAGE]
  constexpr int WN = BN / 32, WM = 8 / WN, TM = BM / WM, MI = TM / 16;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wm = warp / WN, wn = warp % WN;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int kbeg = blockIdx.z * p.Ksplit;
  const int kend = min(p.K, kbeg + p.Ksplit);
  const int KT = kend > kbeg ? (kend - kbeg) / BK : 0;
  float acc[MI][4][4];
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.0f;

  auto load = [&](int stage, int kt) {
    const int k0 = kbeg + kt * BK;
    bf16* as = As + stage * A_STAGE;
    bf16* bs = Bs + stage * B_STAGE;
    if (AK) {
      for (int c = tid; c < BM * 4; c += 256) {
        const int r = c >> 2, q = c & 3, gm = m0 + r;
        const bool ok = gm < p.M;
        const bf16* src = ok ? p.A + (long long)gm * p.lda + k0 + q * 8 : p.A;
        cp_async16(smem_addr(as + r * A_LD + q * 8), src, ok);
      }
    } else {
      for (int c = tid; c < BK * (BM / 8); c += 256) {
        const int r = c / (BM / 8), q = c % (BM / 8), gm = m0 + q * 8;
        const bool ok = gm < p.M;
        const bf16* src = ok ? p.A + (long long)(k0 + r) * p.lda + gm : p.A;
        cp_async16(smem_addr(as + r * A_LD + q * 8), src, ok);
      }
    }
    if (BKC) {
      for (int c = tid; c < BN * 4; c += 256) {
        const int r = c >> 2, q = c & 3, gn = n0 + r;
        const bool ok = gn < p.N;
        const bf16* src = ok ? p.B + (long long)gn * p.ldb + k0 + q * 8 : p.B;
        cp_async16(smem_addr(bs + r * B_LD + q * 8), src, ok);
      }
    } else {
      for (int c = tid; c < BK * (BN / 8); c += 256) {
        const int r = c / (BN / 8), q = c % (BN / 8), gn = n0 + q * 8;
        const bool ok = gn < p.N;
        const bf16* src = ok ? p.B + (long long)(k0 + r) * p.ldb + gn : p.B;
        cp_async16(smem_addr(bs + r * B_LD + q * 8), src, ok);
      }
    }
  };
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < KT) load(s, s);
    cp_commit();
  }
  for (int kt = 0; kt < KT; ++kt) {
    cp_wait<STAGES - 2>();
    __syncthreads();  // stage kt landed for every thread; stage kt - 1 is free
    {
      const int nk = kt + STAGES - 1;
      if (nk < KT) load(nk % STAGES, nk);
      cp_commit();
    }
    const bf16* as = As + (kt % STAGES) * A_STAGE;
    const bf16* bs = Bs + (kt % STAGES) * B_STAGE;
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      uint32_t af[MI][4], bfr[4][2];
#pragma unroll
      for (int i = 0; i < MI; ++i) {
        const int mb = wm * TM + i * 16;
        if (AK) {
          const int row = mb + (lane & 15), col = kk * 16 + (lane >> 4) * 8;
          ldsm_x4(smem_addr(as + row * A_LD + col), af[i][0], af[i][1], af[i][2], af[i][3]);
        } else {  // matrices (m, k) blocks: (0, 0), (8, 0), (0, 8), (8, 8)
          const int q = lane >> 3;
          const int mm = mb + 8 * (q & 1), kr = kk * 16 + 8 * (q >> 1) + (lane & 7);
          ldsm_x4_t(smem_addr(as + kr * A_LD + mm), af[i][0], af[i][1], af[i][2], af[i][3]);
        }
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int nb = wn * 32 + j * 16;
        if (BKC) {
          const int row = nb + (lane & 7) + ((lane >> 4) << 3);
          const int col = kk * 16 + ((lane >> 3) & 1) * 8;
          ldsm_x4(smem_addr(bs + row * B_LD + col), bfr[2 * j][0], bfr[2 * j][1], bfr[2 * j + 1][0],
                  bfr[2 * j + 1][1]);
        } else {  // matrices (n, k) blocks: (0, 0), (0, 8), (8, 0), (8, 8)
          const int q = lane >> 3;
          const int nn = nb + 8 * (q >> 1), kr = kk * 16 + 8 * (q & 1) + (lane & 7);
          ldsm_x4_t(smem_addr(bs + kr * B_LD + nn), bfr[2 * j][0], bfr[2 * j][1], bfr[2 * j + 1][0],
                    bfr[2 * j + 1][1]);
        }
      }
#pragma unroll
      for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bfr[j][0], bfr[j][1]);
    }
  }
  cp_wait<0>();
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = m0 + wm * TM + i * 16 + g + h * 8;
        const int col = n0 + wn * 32 + j * 8 + 2 * t;
        if (row >= p.M || col >= p.N) continue;
        *reinterpret_cast<float2*>(p.Cf + (long long)blockIdx.z * p.split_stride + (long long)row * p.ldc + col) =
            make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
      }
}

template <int BN, bool AK, bool BKC>
cudaError_t gemm_bn(const GemmArgs& p, int splits, cudaStream_t s) {
  constexpr int A_STAGE = AK ? BM * LDS : BK * (BM + 8), B_STAGE = BKC ? BN * LDS : BK * (BN + 8);
  const int smem = STAGES * (A_STAGE + B_STAGE) * (int)sizeof(bf16);
  cudaError_t e =
      cudaFuncSetAttribute(k_gemm<BN, AK, BKC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  dim3 grid((p.N + BN - 1) / BN, (p.M + BM - 1) / BM, splits);
  k_gemm<BN, AK, BKC><<<grid, 256, smem, s>>>(p);
  return cudaGetLastError();
}

// C = A B^T (layouts as k_gemm); `splits` CTAs along K, each writing its
// partial at Cf + z split_stride.
template <bool AK = true, bool BKC = true>
cudaError_t gemm(const GemmArgs& p, int splits, cudaStream_t s) {
  if ((!AK && p.M % 8) || (!BKC && p.N % 8) || p.K % 32 || p.Ksplit % 32) return cudaErrorInvalidValue;
  if (p.N <= 32) return gemm_bn<32, AK, BKC>(p, splits, s);
  if (p.N <= 64) return gemm_bn<64, AK, BKC>(p, splits, s);
  return gemm_bn<128, AK, BKC>(p, splits, s);
}

// --------------------------------------- tcgen05 convolutions fed by TMA
// The 3x3, stride-2, pad-1 convolutions of layers 2-4 and their data gradients,
// as one persistent warp-specialised kernel on the fifth-generation tensor
// cores. Both are sums over taps of 128-row GEMMs whose rows are consecutive
// pixels of a regular grid, so a k-block's A operand (KC channels of one tap) is
// one box of a 4D tensor map (channel, x, y, image), zero-filled outside the
// image, and there is no gather:
// - forward: the input pixels of one tap have one parity in y and in x, so
//   each layer has four maps of its input, one per parity, with strides of
//   two pixels (row 2i - 1 + kh is row i - [kh = 0] of parity [kh != 1]);
// - data gradient: the input pixels of parity class (py, px) take 1, 2, 2 or 4
//   taps of dz at (y + dy, x + dx), dy, dx in {0, 1}. A tile is 128 pixels of
//   dz's grid with all four classes: each of the four boxes of dz is loaded
//   once and multiplied with the taps of all classes that take it, side by side
//   in one MMA (k_dgrad_weights lays them out so).
// With 32 channels two horizontal neighbours are one 128-byte row of the box, taps
// kw = 1 and 2 together. K runs over (tap, channel) in order in steps of 16 for
// each output, as the mma.sync kernels run it, and the results are the same bit for bit.
//
// One CTA per SM: warp 0 fills a ring of stages (A 128 x KC, swizzled K-major
// rows), warp 1 issues the MMAs into one of two tensor-memory accumulators,
// warps 4-7 and 8-11 take turns in reading the other one back (bias + ReLU, or
// the ReLU mask of the layer input) and storing bfloat16 rows. The weights stay in
// shared memory, loaded with the first tile (layer 4's 295 KB do not fit and
// are staged with A). Warps 0 and 1 run their loops as whole warps and issue
// from one elected lane: from a branch on a lane number an MMA took 62 clocks to
// issue, not 23, and a k-block 800, not 510. Every wait is bounded; a wait that
// gives up raises s_abort, which ends the other roles' waits, the copies and MMAs in
// flight are waited for, the tensor memory is freed and *err is set.
//
// Bound by that issue chain per k-block (the MMAs of one take 256 clocks of the
// tensor pipe) and, in the data gradient of layer 2, by reading the mask and
// storing (134 MB). 256 crops, cp.async gathers of the same GEMMs on mma.sync -> first
// tcgen05 version (one thread a role, weights staged, a class per tile, 4
// epilogue warps) -> now: conv2 64 -> 48 -> 20 us, conv3 52 -> 22 -> 16, conv4
// 52 -> 14 -> 11, data gradients 341 -> 139 -> 35 + 19 + 19.
constexpr int kTcRows = 128, kTcThreads = 384;

struct ConvMaps {
  CUtensorMap a[4];  // forward: the input's parities 2 py + px (KC = 96: 2 py + {tap 0, taps 1 and 2});
                     // data gradient: a[0] = dz
  CUtensorMap b[2];  // weights (KC = 96: the columns of taps 1 and 2, of tap 0)
};

struct ConvArgs {
  int M, tiles;          // output rows (data gradient: pixels of one parity class), 128-row tiles of them
  int lg_wo, lg_ho;      // the row space: images of Ho x Wo pixels
  int lg_c;              // log2 channels per tap of A
  int k_blocks;          // forward: k-blocks of a tile
  const float* bias;     // forward
  bf16* out;
  long long ldc, ldg;    // forward: row m at (m / grp) ldg + (m % grp) ldc
  int grp;
  const bf16* mask;      // data gradient: the layer input (ReLU mask), NHWC with C channels, side H
  int H, C, parts;       // its N-channel parts
};

// barriers are given by their shared-memory address
__device__ __forceinline__ void tc_mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool tc_try(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
// wait for the phase of the given parity: bounded by polls and by 4e9 clocks
// (about 2 s), and ended by `stop` (nullptr: not)
__device__ __noinline__ bool tc_poll(uint32_t bar, uint32_t parity, volatile int* stop) {
  const long long t0 = clock64();
  for (int i = 0; i < (1 << 22); ++i) {
    if (tc_try(bar, parity)) return true;
    if ((i & 63) == 63 && ((stop && *stop) || clock64() - t0 > 4000000000ll)) break;
  }
  if (stop) *stop = 1;
  return false;
}
// by whole warps: all lanes or none see it end
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity, volatile int* stop) {
  if (__all_sync(0xffffffffu, tc_try(bar, parity))) return true;
  return __all_sync(0xffffffffu, tc_poll(bar, parity, stop));
}
__device__ __forceinline__ bool tc_elect() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void tc_load4(uint32_t dst, const CUtensorMap* map, int c, int x, int y, int n, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(map), "r"(c), "r"(x), "r"(y), "r"(n), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tc_load2(uint32_t dst, const CUtensorMap* map, int k, int row, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(map), "r"(k), "r"(row), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tc_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// arrives at the barrier when the MMAs issued so far have finished
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// shared-memory matrix descriptor of a K-major operand with rows of 2 KC bytes
// in the 128-byte (KC = 64) or 64-byte (KC = 32) swizzle: start address, stride
// between groups of eight rows, descriptor version 1, swizzle mode
template <int KC>
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)(8 * 2 * KC >> 4) << 32) | (1ull << 46) |
         ((uint64_t)(KC == 64 ? 2 : 4) << 61);
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tc_expect(uint32_t bar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, M = 128, N
__device__ __forceinline__ uint32_t tc_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTcRows >> 4) << 24);
}

// four lanes exchange 16-byte pieces: lane q of a quad gets piece q of the
// rows of its lanes 0 .. 3
__device__ __forceinline__ void quad_exchange(uint4 (&o)[4], int lane) {
  auto swap = [&](uint4& x, uint4& y, int bit) {
    const bool up = lane & bit;
    uint4 s = up ? x : y;
    s.x = __shfl_xor_sync(0xffffffffu, s.x, bit);
    s.y = __shfl_xor_sync(0xffffffffu, s.y, bit);
    s.z = __shfl_xor_sync(0xffffffffu, s.z, bit);
    s.w = __shfl_xor_sync(0xffffffffu, s.w, bit);
    if (up) x = s;
    else y = s;
  };
  swap(o[0], o[1], 1);
  swap(o[2], o[3], 1);
  swap(o[0], o[2], 2);
  swap(o[1], o[3], 2);
}

template <int KC, int N, bool DGRAD, bool RES, int STAGES>
__global__ void __launch_bounds__(kTcThreads, 1) k_conv_tma(const __grid_constant__ ConvMaps maps, ConvArgs p,
                                                            int* err) {
  static_assert((KC == 64 || (KC == 96 && !DGRAD && RES)) && (N == 32 || N == 64 || N == 128), "operand shapes");
  constexpr int A_BYTES = kTcRows * KC * 2, B_BYTES = N * KC * 2, STAGE = A_BYTES + (RES ? 0 : B_BYTES);
  constexpr int NC = DGRAD ? 4 : 1;  // accumulators of a tile
  constexpr int A0 = kTcRows * 64 * 2, B0 = N * 64 * 2;  // KC = 96: tap 0 lies after taps 1 and 2
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[2 * STAGES + 5];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // warp: uniform
  const uint32_t sbase = (smem_addr(smem) + 1023u) & ~1023u;  // the swizzle's period
  const uint32_t full = smem_addr(s_bar), empty = full + 8 * STAGES, acc_full = empty + 8 * STAGES;
  const uint32_t acc_empty = acc_full + 16, drain = acc_full + 32;
  if (tid == 0) {
    for (int s = 0; s < 2 * STAGES; ++s) tc_mbar_init(full + 8 * s, 1);
    for (int k = 0; k < 2; ++k) {
      tc_mbar_init(acc_full + 8 * k, 1);
      tc_mbar_init(acc_empty + 8 * k, 4);
    }
    tc_mbar_init(drain, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {  // two sets of accumulators
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                 "r"(2 * NC * N)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
  volatile int* stop = &s_abort;
  const int part = DGRAD ? blockIdx.x % p.parts : 0;  // of the layer input's channels
  const int t0 = DGRAD ? blockIdx.x / p.parts : blockIdx.x, dt = DGRAD ? gridDim.x / p.parts : gridDim.x;
  const int sub = DGRAD ? p.lg_c - 6 : 0, nb = DGRAD ? 4 << sub : p.k_blocks;  // k-blocks of a tile
  // resident weights of k-block kb; the data gradient's box b has 1, 2, 2, 4 classes
  const uint32_t wbase = sbase + STAGES * STAGE;
  auto n_cls = [](int b) { return b == 0 ? 1 : b == 3 ? 4 : 2; };
  auto w_at = [&](int kb) -> uint32_t {
    if (!DGRAD) return wbase + kb * B_BYTES;
    const int b = kb >> sub, j = kb & ((1 << sub) - 1);
    return wbase + (((2 * b - (b > 0)) << sub) + n_cls(b) * j) * B_BYTES;
  };

  if (warp == 0) {  // producer: the warp runs the loop, its elected lane issues the copies
    const bool lead = tc_elect();
    int s = 0, used = 0;  // the next stage, stages filled so far (up to STAGES)
    uint32_t ph = 0;      // phase of the round over the ring
    bool ok = true;
    for (int t = t0; ok && t < p.tiles; t += dt) {
      const int m0 = t * kTcRows;
      const int y0 = (m0 >> p.lg_wo) & ((1 << p.lg_ho) - 1), n0 = m0 >> (p.lg_wo + p.lg_ho);
      for (int kb = 0; kb < nb; ++kb) {
        if (used == STAGES && !(ok = tc_wait(empty + 8 * s, ph ^ 1u, stop))) break;
        if (lead) {
          const uint32_t a = sbase + s * STAGE, bar = full + 8 * s;
          const int box = kb >> sub, cnt = DGRAD ? n_cls(box) : 1;
          if (RES && t == t0) {  // with the first tile its block of the weights, which stays
            tc_expect(bar, STAGE + cnt * B_BYTES);
            const uint32_t b = w_at(kb);
            if (DGRAD) {
              const int r9 = part * 9 + 2 * box - (box > 0);
              for (int k = 0; k < cnt; ++k)
                tc_load2(b + k * B_BYTES, &maps.b[0], (kb & ((1 << sub) - 1)) * KC, (r9 + k) * N, bar);
            } else {
              tc_load2(b, &maps.b[0], kb * KC + (KC == 96 ? 32 : 0), 0, bar);
              if (KC == 96) tc_load2(b + B0, &maps.b[1], kb * KC, 0, bar);
            }
          } else {
            tc_expect(bar, STAGE);
          }
          const int k0 = kb * KC, tap = k0 >> p.lg_c, ch = k0 & ((1 << p.lg_c) - 1);
          if (DGRAD) {
            tc_load4(a, &maps.a[0], ch, !(tap & 1), y0 + !(tap >> 1), n0, bar);
          } else if (KC == 96) {  // row kb of the window
            tc_load4(a, &maps.a[2 * (kb != 1) + 1], 0, 0, y0 - (kb == 0), n0, bar);
            tc_load4(a + A0, &maps.a[2 * (kb != 1)], 32, -1, y0 - (kb == 0), n0, bar);
          } else {
            const int kh = tap / 3, kw = tap % 3;
            tc_load4(a, &maps.a[2 * (kh != 1) + (kw != 1)], ch, kw == 0 ? -1 : 0, y0 - (kh == 0), n0, bar);
          }
          if (!RES) tc_load2(a + A_BYTES, &maps.b[0], k0, 0, bar);
        }
        __syncwarp();
        if (used < STAGES) ++used;
        if (++s == STAGES) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    // after a failure wait for the copies in flight (each stage's last one)
    if (!ok || *stop)
      for (int k = 0; k < used; ++k) tc_wait(full + 8 * k, k < s ? ph : ph ^ 1u, nullptr);
  } else if (warp == 1) {  // MMA issuer, likewise
    const bool lead = tc_elect();
    int s = 0, i = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = t0; ok && t < p.tiles; t += dt, ++i) {
      const int buf = i & 1;
      const uint32_t d = tmem + (uint32_t)(buf * NC * N);
      if (i >= 2 && !tc_wait(acc_empty + 8 * buf, (uint32_t)((i >> 1) - 1) & 1u, stop)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int kb = 0; kb < nb; ++kb) {
        if (!(ok = tc_wait(full + 8 * s, ph, stop))) break;
        const uint32_t a = sbase + (uint32_t)(s * STAGE), b = RES ? w_at(kb) : a + A_BYTES, acc = kb != 0;
        if (lead) {
          if (DGRAD) {
            // the box's classes lie side by side in the accumulator (2, 3, 1, 0) and in the
            // weights: one MMA for all, but for the class that starts with this box
            const int box = kb >> sub, p0 = box & 1 ? 0 : 1 - (box == 3), cnt = n_cls(box);
            const int fresh = (kb & ((1 << sub) - 1)) == 0 ? (box == 0 ? 1 : box == 1 ? 0 : box) : -1;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint64_t ad = tc_desc<64>(a + 32 * j);
              int lo = p0, hi = p0 + cnt;
              if (j == 0 && fresh >= 0) {
                tc_mma(d + fresh * N, ad, tc_desc<64>(b + (fresh - p0) * B_BYTES), tc_idesc(N), 0);
                if (fresh == lo) ++lo;
                else --hi;
              }
              if (lo < hi)
                tc_mma(d + lo * N, ad, tc_desc<64>(b + (lo - p0) * B_BYTES + 32 * j), tc_idesc((hi - lo) * N), 1);
            }
          } else {
            if (KC == 96)
#pragma unroll
              for (int j = 0; j < 2; ++j)
                tc_mma(d, tc_desc<32>(a + A0 + 32 * j), tc_desc<32>(b + B0 + 32 * j), tc_idesc(N), j ? 1u : acc);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              tc_mma(d, tc_desc<64>(a + 32 * j), tc_desc<64>(b + 32 * j), tc_idesc(N), j || KC == 96 ? 1u : acc);
          }
          tc_commit(empty + 8 * s);
          if (kb == nb - 1) tc_commit(acc_full + 8 * buf);
        }
        __syncwarp();
        if (++s == STAGES) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    // every MMA issued has finished before the tensor memory is freed
    if (lead) tc_commit(drain);
    __syncwarp();
    tc_wait(drain, 0, nullptr);
  } else if (warp >= 4) {  // epilogue: warps 4-7 the even tiles, 8-11 the odd ones; rows 32 (warp % 4) .. + 31
    const int qd = warp & 3, buf = (warp - 4) >> 2;
    // after the exchange below a lane stores 16 bytes of rows r4 .. r4 + 3
    const int r4 = 32 * qd + (lane & ~3), q8 = 8 * (lane & 3);
    const long long rs = DGRAD ? 2LL * p.C : p.ldc;
    int i = buf;
    for (int t = t0 + buf * dt; t < p.tiles; t += 2 * dt, i += 2) {
      const int row = t * kTcRows + r4;
      const bool in = row < p.M;
      long long base;
      if (DGRAD) {  // class pixel -> NHWC input pixel
        const int x = row & ((1 << p.lg_wo) - 1), y = (row >> p.lg_wo) & ((1 << p.lg_ho) - 1);
        const int n = row >> (p.lg_wo + p.lg_ho);
        base = (((long long)n * p.H + 2 * y) * p.H + 2 * x) * p.C + part * N + q8;
      } else {
        base = (long long)(row / p.grp) * p.ldg + (long long)(row % p.grp) * p.ldc + q8;
      }
      // columns c0 .. c0 + 31 of the accumulators: classes 2, 3, 1, 0 (2 py + px)
      auto offset = [&](int c0) {
        if (!DGRAD) return base + c0;
        const int k = c0 / N, py = k < 2, px = k == 1 || k == 2;
        return base + (py * p.H + px) * (long long)p.C + c0 % N;
      };
      uint4 mk[4];  // the mask of the next 32 columns, the first ones read before the accumulator is ready
      if (DGRAD)
#pragma unroll
        for (int g = 0; g < 4; ++g)
          mk[g] = in ? __ldg(reinterpret_cast<const uint4*>(p.mask + offset(0) + g * rs)) : make_uint4(0u, 0u, 0u, 0u);
      if (!tc_wait(acc_full + 8 * buf, (uint32_t)(i >> 1) & 1u, stop)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int c0 = 0; c0 < NC * N; c0 += 32) {
        uint32_t v[32];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
            "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
              "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]),
              "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
              "=r"(v[30]), "=r"(v[31])
            : "r"(tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(buf * NC * N + c0)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        uint4 o[4];  // this lane's row: 4 x 8 channels
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint32_t h[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float v0 = __uint_as_float(v[8 * g + 2 * e]), v1 = __uint_as_float(v[8 * g + 2 * e + 1]);
            if (!DGRAD) {
              const float2 b = __ldg(reinterpret_cast<const float2*>(p.bias + c0 + 8 * g + 2 * e));
              v0 = fmaxf(v0 + b.x, 0.0f);
              v1 = fmaxf(v1 + b.y, 0.0f);
            }
            const __nv_bfloat162 w = __floats2bfloat162_rn(v0, v1);
            h[e] = *reinterpret_cast<const uint32_t*>(&w);
          }
          o[g] = make_uint4(h[0], h[1], h[2], h[3]);
        }
        quad_exchange(o, lane);  // a store instruction writes eight rows of 64 bytes instead of 32 of 16
        if (in) {
          bf16* dst = p.out + offset(c0);
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            if (DGRAD) {  // zero where the layer input is not above zero
              const uint32_t m[4] = {mk[g].x, mk[g].y, mk[g].z, mk[g].w};
              uint32_t w[4] = {o[g].x, o[g].y, o[g].z, o[g].w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const __nv_bfloat162 m2 = *reinterpret_cast<const __nv_bfloat162*>(&m[e]);
                if (!(__low2float(m2) > 0.0f)) w[e] &= 0xffff0000u;
                if (!(__high2float(m2) > 0.0f)) w[e] &= 0x0000ffffu;
              }
              o[g] = make_uint4(w[0], w[1], w[2], w[3]);
              if (c0 + 32 < NC * N) mk[g] = __ldg(reinterpret_cast<const uint4*>(p.mask + offset(c0 + 32) + g * rs));
            }
            *reinterpret_cast<uint4*>(dst + g * rs) = o[g];
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc_arrive(acc_empty + 8 * buf);
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (tid == 0 && s_abort) atomicOr(err, 1);
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * NC * N) : "memory");
}

// Weight gradients of layers 2-4: D[co][tap, ci] = sum over output pixels of
// dz[pixel][co] x[pixel at tap][ci], both operands pixel-major (MN-major for
// the tensor core). A CTA takes one row kh of the window (N = 3 Cin columns in
// tensor memory, one MMA per 16 pixels, two with N = 384) and one split of the pixels;
// its boxes are 32 output pixels of dz and, from the parity maps, of x at each tap: TMA
// loads them with the padding, PB boxes a stage. Roles and waits as in
// k_conv_tma; at the end warps 0-3 write the partial sums, which
// k_sums adds in order. Splits and the order of pixels are those of the mma.sync
// GEMM that it replaces (implicit im2col by cp.async gathers, which bound
// it), and so are the results, bit for bit. 256 crops: layers 2, 3, 4
// 56 us each (mean) -> 23, 16, 12.
struct WgradArgs {
  int blocks, split;  // 32-pixel blocks in all and of one split
  int lg_wo;          // output side
  float* part;        // partial z at part + z split_stride: [co][Kp]
  long long split_stride;
  int Kp;
};

// shared-memory matrix descriptor of an MN-major operand: rows (K) of W
// channels in the swizzle of their length, groups of eight rows back to back,
// `step` bytes between blocks of W channels
template <int W>
__device__ __forceinline__ uint64_t tc_desc_mn(uint32_t saddr, int step) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(step >> 4) << 16) | ((uint64_t)(8 * 2 * W >> 4) << 32) |
         (1ull << 46) | ((uint64_t)(W == 64 ? 2 : 4) << 61);
}

// W: channels of an x box, NB of them; MB boxes of 64 channels of dz
template <int W, int NB, int MB, int PB, int STAGES>
__global__ void __launch_bounds__(128) k_wgrad_tma(const __grid_constant__ ConvMaps maps, WgradArgs p, int* err) {
  constexpr int ABOX = 32 * 64 * 2, XBOX = 32 * W * 2, N = NB * W, COLS = N <= 128 ? 128 : N <= 256 ? 256 : 512;
  constexpr int X0 = MB * PB * ABOX, STAGE = X0 + NB * PB * XBOX, N1 = N <= 256 ? N : N / 2;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[2 * STAGES + 1];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const uint32_t sbase = (smem_addr(smem) + 1023u) & ~1023u;
  const uint32_t full = smem_addr(s_bar), empty = full + 8 * STAGES, acc_full = empty + 8 * STAGES;
  if (tid == 0) {
    for (int s = 0; s < 2 * STAGES + 1; ++s) tc_mbar_init(full + 8 * s, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                 "r"(COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
  volatile int* stop = &s_abort;
  const int kh = blockIdx.x, b0 = blockIdx.y * p.split, nblk = min(p.blocks - b0, p.split);
  const int rounds = (nblk + PB - 1) / PB;

  if (warp == 0) {  // producer
    const bool lead = tc_elect();
    int s = 0, used = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int r = 0; r < rounds; ++r) {
      if (used == STAGES && !(ok = tc_wait(empty + 8 * s, ph ^ 1u, stop))) break;
      if (lead) {
        const int cnt = min(PB, nblk - r * PB);
        const uint32_t a = sbase + s * STAGE, bar = full + 8 * s;
        tc_expect(bar, cnt * (STAGE / PB));
        for (int h = 0; h < cnt; ++h) {
          const int m = (b0 + r * PB + h) * 32, y = (m >> p.lg_wo) & ((1 << p.lg_wo) - 1), n = m >> (2 * p.lg_wo);
#pragma unroll
          for (int k = 0; k < MB; ++k) tc_load4(a + (k * PB + h) * ABOX, &maps.b[0], 64 * k, 0, y, n, bar);
#pragma unroll
          for (int k = 0; k < NB; ++k) {
            const int kw = k / (NB / 3), ch = k % (NB / 3) * W;
            tc_load4(a + X0 + (k * PB + h) * XBOX, &maps.a[2 * (kh != 1) + (kw != 1)], ch, kw == 0 ? -1 : 0,
                     y - (kh == 0), n, bar);
          }
        }
      }
      __syncwarp();
      if (used < STAGES) ++used;
      if (++s == STAGES) {
        s = 0;
        ph ^= 1u;
      }
    }
    if (!ok || *stop)  // after a failure wait for the copies in flight
      for (int k = 0; k < used; ++k) tc_wait(full + 8 * k, k < s ? ph : ph ^ 1u, nullptr);
  } else if (warp == 1) {  // MMA issuer
    const bool lead = tc_elect();
    // M = 64 MB, both operands MN-major
    const uint32_t idesc =
        (1u << 4) | (1u << 7) | (1u << 10) | (3u << 15) | ((uint32_t)(N1 >> 3) << 17) | ((uint32_t)(4 * MB) << 24);
    int s = 0;
    uint32_t ph = 0;
    for (int r = 0; r < rounds; ++r) {
      if (!tc_wait(full + 8 * s, ph, stop)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (lead) {
        const uint32_t a = sbase + s * STAGE, x = a + X0;
        const int steps = 2 * min(PB, nblk - r * PB);
#pragma unroll
        for (int j = 0; j < 2 * PB; ++j)
          if (j < steps)
#pragma unroll
            for (int h = 0; h < N / N1; ++h)
              tc_mma(tmem + h * N1, tc_desc_mn<64>(a + j * 2048, PB * ABOX),
                     tc_desc_mn<W>(x + j * 32 * W + h * (NB / 2) * PB * XBOX, PB * XBOX), idesc, r > 0 || j > 0);
        tc_commit(empty + 8 * s);
      }
      __syncwarp();
      if (++s == STAGES) {
        s = 0;
        ph ^= 1u;
      }
    }
    if (lead) tc_commit(acc_full);  // also after a failure: every MMA issued ends before the memory is freed
    __syncwarp();
    tc_wait(acc_full, 0, nullptr);
  }
  __syncwarp();
  if (tc_wait(acc_full, 0, stop)) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // with M = 64 a warp's first 16 lanes hold its rows
    const int row = (MB == 2 ? 32 : 16) * warp + (lane & ~3);
    float* out = p.part + blockIdx.y * p.split_stride + (long long)row * p.Kp + kh * N + 4 * (lane & 3);
    for (int c0 = 0; c0 < N; c0 += 32) {
      uint32_t v[32];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
          "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
            "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
            "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
            "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
          : "r"(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint4 o[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const uint32_t* w = v + 16 * h + 4 * g;
          o[g] = make_uint4(w[0], w[1], w[2], w[3]);
        }
        quad_exchange(o, lane);
        if (MB == 2 || lane < 16)
#pragma unroll
          for (int g = 0; g < 4; ++g) *reinterpret_cast<uint4*>(out + g * (long long)p.Kp + c0 + 16 * h) = o[g];
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (tid == 0 && s_abort) atomicOr(err, 1);
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
}

template <int W, int NB, int MB, int PB, int STAGES>
cudaError_t wgrad_tma_t(const ConvMaps& maps, const WgradArgs& p, int splits, int* err, cudaStream_t s) {
  constexpr int smem = STAGES * PB * 64 * (64 * MB + NB * W) + 1024;
  auto kern = k_wgrad_tma<W, NB, MB, PB, STAGES>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  kern<<<dim3(3, (unsigned)splits), 128, smem, s>>>(maps, p, err);
  return cudaGetLastError();
}

// Weights of the data gradients, in the order of the boxes (dy, dx) = (1, 1),
// (1, 0), (0, 1), (0, 0) of dz and of the parity classes 2 py + px that take
// them: 3; 2, 3; 3, 1; 2, 3, 1, 0. Row (9 part + box's class) N + c is input
// channel part N + c, column o is W[o][kh][kw][channel]; an even coordinate
// takes the middle tap, an odd one taps 0 (offset 1) and 2.
__global__ void k_dgrad_weights(const bf16* __restrict__ w, int Kp, int cin, int cout, int N, bf16* __restrict__ out) {
  const int n = 9 * cin * cout;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int o = e % cout, row = e / cout, c = row / (9 * N) * N + row % N, r9 = row / N % 9;
    const int box = (r9 > 0) + (r9 > 2) + (r9 > 4), k = r9 - (2 * box - (box > 0));
    const int cls = box == 0 ? 3 : box == 1 ? 2 + k : box == 2 ? 3 - 2 * k : k < 2 ? 2 + k : 3 - k;
    const int kh = cls >> 1 ? (box < 2 ? 0 : 2) : 1, kw = cls & 1 ? (box & 1 ? 2 : 0) : 1;
    out[e] = w[(long long)o * Kp + (kh * 3 + kw) * cin + c];
  }
}

typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// a tensor map of bfloat16 values with rows (dimension 0) of 64 or 32 channels in a box
cudaError_t encode_map(CUtensorMap* map, const void* base, int rank, const long long* dims, const long long* strides,
                       const int* box) {
  static const EncodeTiled fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &r) != cudaSuccess ||
        r != cudaDriverEntryPointSuccess)
      f = nullptr;
    return (EncodeTiled)f;
  }();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t d[5], st[4];
  cuuint32_t b[5], one[5] = {1, 1, 1, 1, 1};
  for (int k = 0; k < rank; ++k) {
    d[k] = (cuuint64_t)dims[k];
    b[k] = (cuuint32_t)box[k];
    if (k) st[k - 1] = (cuuint64_t)strides[k - 1];
  }
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), d, st, b, one,
                        CU_TENSOR_MAP_INTERLEAVE_NONE,
                        box[0] == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// K: the columns of the resident weights (0: staged with A)
template <int KC, int N, bool DGRAD, int K>
cudaError_t conv_tma_t(const ConvMaps& maps, const ConvArgs& p, int* err, int sm_count, cudaStream_t s) {
  constexpr int stage = (kTcRows + (K ? 0 : N)) * KC * 2, wres = N * K * 2;
  constexpr int stages = std::min(12, (224 * 1024 - wres) / stage), smem = stages * stage + wres + 1024;
  static_assert(stages >= 3, "ring");
  auto kern = k_conv_tma<KC, N, DGRAD, K != 0, stages>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int parts = DGRAD ? p.parts : 1;
  kern<<<(unsigned)(std::min(p.tiles, sm_count / parts) * parts), kTcThreads, smem, s>>>(maps, p, err);
  return cudaGetLastError();
}

int ilog2(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return l;
}

// splits along K so that the grid has about two CTAs per SM (each split a
// multiple of 32 long, at least 256)
int choose_splits(int M, int N, int K, int* ksplit) {
  const int bn = N <= 32 ? 32 : N <= 64 ? 64 : 128;
  const int tiles = ((M + BM - 1) / BM) * ((N + bn - 1) / bn);
  int S = std::max(1, std::min((2 * 152 + tiles - 1) / tiles, K / 256));
  int ks = (K / S + 31) / 32 * 32;
  S = (K + ks - 1) / ks;
  *ksplit = ks;
  return S;
}

// ------------------------------------------------ input layer (2 -> 32 channels)
// Direct 3x3 convolution of the 2-channel crops with bias and ReLU, on mma.sync
// m16n8k16: K = (tap, channel) padded to 32, so one register of an A fragment
// is one pixel's two channels at one tap, read from a strip of the crop in
// shared memory: no im2col matrix is written and read back (67 + 67 MB per 256
// crops), and the kernel is bound by storing its output (67 MB). A CTA takes
// eight rows of a crop, a warp one row. The output channels are dealt to the
// four n-tiles so that a thread ends up with eight consecutive ones: one
// 16-byte store per pixel. 256 crops: 18 us instead of 76 (im2col 20,
// GEMM 56). Accumulation order and results are the GEMM's.
__global__ void __launch_bounds__(256) k_conv1(const uint32_t* __restrict__ x, const bf16* __restrict__ w,
                                               const float* __restrict__ bias, bf16* __restrict__ out,
                                               const int32_t* __restrict__ onehot, int n_onehot_pad, long long ldf,
                                               bf16* __restrict__ feat) {
  constexpr int P = kCrop + 2;
  __shared__ uint32_t px[10 * P];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int r0 = 8 * (blockIdx.x & 7);
  const uint32_t* img = x + (long long)(blockIdx.x >> 3) * kCrop * kCrop;
  if (r0 == 0) {  // the crop's one-hot columns of the FC input
    const int hot = __ldg(&onehot[blockIdx.x >> 3]);
    bf16* dst = feat + (blockIdx.x >> 3) * ldf + kFeat;
    for (int j = tid; j < n_onehot_pad; j += 256) dst[j] = __float2bfloat16_rn(j == hot ? 1.0f : 0.0f);
  }
  for (int i = tid; i < 10 * P; i += 256) {
    const int r = r0 - 1 + i / P, c = i % P - 1;
    px[i] = r >= 0 && r < kCrop && c >= 0 && c < kCrop ? __ldg(&img[r * kCrop + c]) : 0u;
  }
  uint32_t bf[4][2][2];  // weights: n-tile j, k-step, register
  float bs[4][2];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int ch = 8 * (g >> 1) + 2 * j + (g & 1);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      bf[j][k][0] = *reinterpret_cast<const uint32_t*>(w + ch * 32 + 16 * k + 2 * t);
      bf[j][k][1] = *reinterpret_cast<const uint32_t*>(w + ch * 32 + 16 * k + 2 * t + 8);
    }
    bs[j][0] = bias[8 * t + 2 * j];
    bs[j][1] = bias[8 * t + 2 * j + 1];
  }
  __syncthreads();
  const uint32_t* row = px + warp * P;
  const int o0 = t / 3 * P + t % 3, o4 = (t + 4) / 3 * P + (t + 4) % 3, o8 = 2 * P + 2;
  bf16* dst = out + ((long long)(blockIdx.x >> 3) * kCrop * kCrop + (r0 + warp) * kCrop) * 32 + 8 * t;
#pragma unroll
  for (int m = 0; m < kCrop; m += 16) {
    const uint32_t* a = row + m + g;
    const uint32_t a0[4] = {a[o0], a[o0 + 8], a[o4], a[o4 + 8]};
    const uint32_t a1[4] = {t == 0 ? a[o8] : 0u, t == 0 ? a[o8 + 8] : 0u, 0u, 0u};
    uint32_t lo[4], hi[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      mma_bf16(acc, a0, bf[j][0][0], bf[j][0][1]);
      mma_bf16(acc, a1, bf[j][1][0], bf[j][1][1]);
      const __nv_bfloat162 l = __floats2bfloat162_rn(fmaxf(acc[0] + bs[j][0], 0.0f), fmaxf(acc[1] + bs[j][1], 0.0f));
      const __nv_bfloat162 h = __floats2bfloat162_rn(fmaxf(acc[2] + bs[j][0], 0.0f), fmaxf(acc[3] + bs[j][1], 0.0f));
      lo[j] = *reinterpret_cast<const uint32_t*>(&l);
      hi[j] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(dst + (m + g) * 32) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    *reinterpret_cast<uint4*>(dst + (m + g + 8) * 32) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  }
}

// Weight gradient of the input layer: D[co][tap, channel] = sum over pixels of
// dz[pixel][co] x[pixel at tap][channel], one split of the pixels a CTA. dz rows
// pass once through a cp.async ring; a B fragment of mma.sync is two
// neighbouring pixels of the crop at a tap, put together from the CTA's strip of
// crop rows in shared memory (rows outside the image: a row of zeros). Warps
// 0-5 hold 16 x 8 outputs each (18 of 32 columns exist). Bound by
// reading dz (67 MB per 256 crops); splits and order of pixels are
// those of the GEMM over an im2col matrix that it replaces, and so are the
// results, bit for bit. 256 crops: 31 us instead of 81 (im2col 20, GEMM 61).
constexpr int kW1Px = 128, kW1Ld = 80, kW1Stages = 7, kW1Row = kCrop + 2;
__global__ void __launch_bounds__(256) k_wgrad1(const uint32_t* __restrict__ x, const bf16* __restrict__ dz, int M,
                                                int ksplit, float* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* strip = reinterpret_cast<uint32_t*>(smem_raw + kW1Stages * kW1Px * kW1Ld);  // row 0: zeros
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int kbeg = blockIdx.x * ksplit, kend = min(M, kbeg + ksplit);
  const int R0 = kbeg / kCrop - 1, nrows = (kend - 1) / kCrop + 1 - R0 + 1, rounds = (kend - kbeg + kW1Px - 1) / kW1Px;
  auto load = [&](int st) {
    const int m0 = kbeg + st * kW1Px;
    const uint32_t dst = smem_addr(smem_raw + (st % kW1Stages) * kW1Px * kW1Ld);
    for (int c = tid; c < kW1Px * 4; c += 256) {
      const int m = m0 + (c >> 2);
      cp_async16(dst + (c >> 2) * kW1Ld + (c & 3) * 16, dz + (long long)min(m, kend - 1) * 32 + (c & 3) * 8, m < kend);
    }
  };
#pragma unroll
  for (int st = 0; st < kW1Stages - 1; ++st) {
    if (st < rounds) load(st);
    cp_commit();
  }
  for (int i = tid; i < (nrows + 1) * kW1Row; i += 256) {
    const int r = R0 + i / kW1Row - 1, c = i % kW1Row - 1;
    const bool in = i >= kW1Row && r >= 0 && r < M / kCrop && c >= 0 && c < kCrop;
    strip[i] = in ? __ldg(&x[(long long)r * kCrop + c]) : 0u;
  }
  const int mt = warp < 6 ? warp / 3 : warp - 6, nt = warp < 6 ? warp % 3 : 3;
  const int col = 8 * nt + g, tap = col >> 1, kh = tap / 3, kw = tap % 3;
  const uint32_t sel = col & 1 ? 0x7632u : 0x5410u;
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  for (int st = 0; st < rounds; ++st) {
    cp_wait<kW1Stages - 2>();
    __syncthreads();  // stage st landed for every thread; stage st - 1 is free
    if (st + kW1Stages - 1 < rounds) load(st + kW1Stages - 1);
    cp_commit();
    if (warp >= 6) continue;
    const int m0 = kbeg + st * kW1Px;
    const uint32_t a0 = smem_addr(smem_raw + (st % kW1Stages) * kW1Px * kW1Ld) +
                        (8 * (lane >> 4) + (lane & 7)) * kW1Ld + (16 * mt + 8 * ((lane >> 3) & 1)) * 2;
    auto step = [&](int h) {  // 32 pixels of one row
      const int m = m0 + 32 * h, R = m / kCrop, i = R % kCrop - 1 + kh;
      const bool in = col < 18 && i >= 0 && i < kCrop;
      const uint32_t* row = strip + (in ? (R - 1 + kh - R0 + 1) * kW1Row + m % kCrop + kw : 0) + 2 * t;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        uint32_t af[4];
        ldsm_x4_t(a0 + (32 * h + 16 * k) * kW1Ld, af[0], af[1], af[2], af[3]);
        mma_bf16(acc, af, __byte_perm(row[16 * k], row[16 * k + 1], sel),
                 __byte_perm(row[16 * k + 8], row[16 * k + 9], sel));
      }
    };
    if (m0 + kW1Px <= kend) {
#pragma unroll
      for (int h = 0; h < kW1Px / 32; ++h) step(h);
    } else {
      for (int h = 0; m0 + 32 * h < kend; ++h) step(h);
    }
  }
  cp_wait<0>();
  float* out = part + (long long)blockIdx.x * 32 * 32 + (16 * mt + g) * 32 + 8 * nt + 2 * t;
  *reinterpret_cast<float2*>(out) = make_float2(acc[0], acc[1]);
  *reinterpret_cast<float2*>(out + 8 * 32) = make_float2(acc[2], acc[3]);
}

// ---------------------------------------------------------------- small kernels
// part[b][c] = sum of column c over rows [b R, (b + 1) R) of a bfloat16
// [M][C] matrix (bias gradients), 128 threads a block b: a thread adds two
// columns of every G-th row in order, then the G = 256 / C row groups are added
// in order. Bound by reading the matrix: 16 rows in flight a thread.
// 256 crops, five layers: 58 -> 45 us.
__global__ void __launch_bounds__(128) k_col_sum(const bf16* __restrict__ in, long long M, int C, int R,
                                                 float* __restrict__ part) {
  __shared__ float red[256];
  const int G = 256 / C, L = C / 2, c = threadIdx.x % L, grp = threadIdx.x / L;
  const long long r0 = (long long)blockIdx.x * R, r1 = min(M, r0 + R);
  float a0 = 0.0f, a1 = 0.0f;
  if (grp < G) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(in) + c;
    for (long long r = r0 + grp; r < r1; r += 16 * G) {
      uint32_t v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = r + k * G < r1 ? __ldg(src + (r + k * G) * L) : 0u;
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (r + k * G < r1) {
          const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&v[k]);
          a0 += __low2float(h);
          a1 += __high2float(h);
        }
    }
    red[grp * C + 2 * c] = a0;
    red[grp * C + 2 * c + 1] = a1;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < C; k += 128) {
    float v = 0.0f;
    for (int g = 0; g < G; ++g) v += red[g * C + k];
    part[(long long)blockIdx.x * C + k] = v;
  }
}

// Sums of partials in a fixed order (deterministic), both reductions of a
// layer in one launch: out[e] = sum over z of part[z][e], 32 outputs to G
// groups of 32 threads, group g adding z = g, g + G, ..., then the groups in
// order. The first blocks add nb bias partials (G = 32), the others the
// weight partials (four sets of outputs a block, G = 8). Bound by the latency of
// reading: 16 partials in flight a thread. 256 crops, nine sums: 79 us in nine
// launches -> 59 in five.
struct Sums {
  const float *bias_part, *part;
  float *bias_out, *out;
  int nb, C;         // bias partials and columns
  int splits;        // weight partials
  long long n;       // weights (0: none)
};
__global__ void __launch_bounds__(1024) k_sums(Sums p) {
  __shared__ float red[32][33];
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31, bias_blocks = (p.C + 31) / 32;
  const bool bias = (int)blockIdx.x < bias_blocks;
  const int G = bias ? 32 : 8, cnt = bias ? p.nb : p.splits;
  const long long n = bias ? p.C : p.n;
  const long long e = bias ? blockIdx.x * 32 + lane : ((blockIdx.x - bias_blocks) * 4 + (q >> 3)) * 32ll + lane;
  const float* part = (bias ? p.bias_part : p.part) + e;
  float a = 0.0f;
  if (e < n)
    for (int z = q % G; z < cnt; z += 16 * G) {
      float v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = z + k * G < cnt ? __ldg(part + (z + k * G) * n) : 0.0f;
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (z + k * G < cnt) a += v[k];
    }
  red[q][lane] = a;
  __syncthreads();
  if (q % G == 0 && e < n) {
    float v = 0.0f;
    for (int k = 0; k < G; ++k) v += red[q + k][lane];
    (bias ? p.bias_out : p.out)[e] = v;
  }
}

// The rest of the FC layers after FC1's split-K partial sums, one warp a
// crop: h1 = bf16(relu(sum over z of part[z] + b1)), kept for the backward pass,
// pred = h1 . bf16(w2) + b2 and, with a target, err = pred - y. One launch instead
// of two (256 crops: 5.7 + 3.7 -> 5.6 us).
__global__ void __launch_bounds__(128) k_fc_tail(const float* __restrict__ part, int splits,
                                                 const float* __restrict__ b1, const float* __restrict__ w2,
                                                 const float* __restrict__ b2, int n, bf16* __restrict__ h1,
                                                 float* __restrict__ pred, const float* __restrict__ target,
                                                 float* __restrict__ err) {
  constexpr int J = kHidden / 32;
  const int row = (blockIdx.x * 128 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= n) return;
  const float* src = part + (long long)row * kHidden + lane;
  const long long stride = (long long)n * kHidden;
  float s[J];
#pragma unroll
  for (int j = 0; j < J; ++j) s[j] = 0.0f;
  for (int z = 0; z < splits; z += 8) {  // eight partials read at a time, added in order
    float v[8][J];
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int j = 0; j < J; ++j) v[k][j] = z + k < splits ? __ldg(src + (z + k) * stride + 32 * j) : 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (z + k < splits) s[j] += v[k][j];
  }
  float a = 0.0f;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const bf16 h = __float2bfloat16_rn(fmaxf(s[j] + b1[lane + 32 * j], 0.0f));
    h1[(long long)row * kHidden + lane + 32 * j] = h;
    a += __bfloat162float(h) * __bfloat162float(__float2bfloat16_rn(w2[lane + 32 * j]));
  }
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (lane == 0) {
    const float pr = a + b2[0];
    if (pred) pred[row] = pr;
    if (target) err[row] = pr - target[row];
  }
}

// loss = mean 0.5 err^2 and the gradient of b2 (one block)
__global__ void k_fc2_loss(const float* __restrict__ err, int n, float* __restrict__ g_b2, float* __restrict__ loss) {
  __shared__ float red[2][32];
  const float inv = 1.0f / (float)n;
  float l = 0.0f, gb = 0.0f;
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    l += 0.5f * err[r] * err[r];
    gb += err[r] * inv;
  }
  for (int o = 16; o > 0; o >>= 1) {
    l += __shfl_xor_sync(0xffffffffu, l, o);
    gb += __shfl_xor_sync(0xffffffffu, gb, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = l;
    red[1][threadIdx.x >> 5] = gb;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.0f, b = 0.0f;
    for (int k = 0; k < (int)blockDim.x / 32; ++k) {
      a += red[0][k];
      b += red[1][k];
    }
    if (loss) *loss = a * inv;
    g_b2[0] = b;
  }
}

// gradient of w2: one block per hidden unit j, sum over the batch
__global__ void k_fc2_wgrad(const bf16* __restrict__ h1, const float* __restrict__ err, int n, float* __restrict__ g_w2) {
  __shared__ float red[32];
  const int j = blockIdx.x;
  const float inv = 1.0f / (float)n;
  float a = 0.0f;
  for (int r = threadIdx.x; r < n; r += blockDim.x) a += err[r] * inv * __bfloat162float(h1[(long long)r * kHidden + j]);
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    float v = 0.0f;
    for (int k = 0; k < (int)blockDim.x / 32; ++k) v += red[k];
    g_w2[j] = v;
  }
}

// dz1 = (err / n) bf16(w2) [h1 > 0]
__global__ void k_fc2_dz1(const bf16* __restrict__ h1, const float* __restrict__ w2, const float* __restrict__ err,
                          int n, bf16* __restrict__ dz1) {
  const float inv = 1.0f / (float)n;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)n * kHidden;
       e += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(e / kHidden), j = (int)(e % kHidden);
    float v = 0.0f;
    if (__bfloat162float(h1[e]) > 0.0f) v = err[r] * inv * __bfloat162float(__float2bfloat16_rn(w2[j]));
    dz1[e] = __float2bfloat16_rn(v);
  }
}

// dz of the last convolution: dfeat (fp32, [n][kFeat]) times [x4 > 0], where
// x4 is read back from the FC input rows
__global__ void k_feat_relu_grad(const float* __restrict__ dfeat, const bf16* __restrict__ feat, long long ldf,
                                 int n, bf16* __restrict__ dz) {
  const int total = n * (kFeat / 8);  // eight columns a thread
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int r = e / (kFeat / 8), k = e % (kFeat / 8) * 8;
    const uint4 x4 = __ldg(reinterpret_cast<const uint4*>(feat + r * ldf + k));
    const float4* d4 = reinterpret_cast<const float4*>(dfeat) + 2 * (long long)e;
    const float4 p = __ldg(d4), q = __ldg(d4 + 1);
    const float d[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
    const uint32_t x[4] = {x4.x, x4.y, x4.z, x4.w};
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&x[i]);
      const __nv_bfloat162 v = __floats2bfloat162_rn(__low2float(h) > 0.0f ? d[2 * i] : 0.0f,
                                                     __high2float(h) > 0.0f ? d[2 * i + 1] : 0.0f);
      o[i] = *reinterpret_cast<const uint32_t*>(&v);
    }
    reinterpret_cast<uint4*>(dz)[e] = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// Adam on four parameters a thread (n and n16 multiples of 4), and the bfloat16 weights
// (the first n16) rounded from the result: 10.9 + 5.4 -> 10.2 us for a million parameters
__global__ void k_adam(float4* __restrict__ p, const float4* __restrict__ g, float4* __restrict__ m,
                       float4* __restrict__ v, int n4, float lr, float b1, float b2, float c1, float c2, float eps,
                       int n16_4, uint2* __restrict__ w16) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n4; e += gridDim.x * blockDim.x) {
    float4 P = p[e], M = m[e], V = v[e];
    const float4 G = __ldg(&g[e]);
    auto one = [&](float& pi, float gi, float& mo, float& vo) {
      const float mi = b1 * mo + (1.0f - b1) * gi;
      const float vi = b2 * vo + (1.0f - b2) * gi * gi;
      mo = mi;
      vo = vi;
      pi -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    };
    one(P.x, G.x, M.x, V.x);
    one(P.y, G.y, M.y, V.y);
    one(P.z, G.z, M.z, V.z);
    one(P.w, G.w, M.w, V.w);
    m[e] = M;
    v[e] = V;
    p[e] = P;
    if (e < n16_4) {
      const __nv_bfloat162 a = __floats2bfloat162_rn(P.x, P.y), b = __floats2bfloat162_rn(P.z, P.w);
      w16[e] = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    }
  }
}

__global__ void k_to_bf16(const float* __restrict__ in, long long n, bf16* __restrict__ out) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    out[e] = __float2bfloat16_rn(in[e]);
}

// The value of a depth d against the centre's depth zr, before it is rounded to
// bfloat16: clamp(RN32(RN64(RN64(zr - d) scale))). The double operations run at a small
// fraction of the binary32 rate and bound the kernel, so the value is first taken
// in binary32, zr as zh + zl and the difference as a sum and its exact error:
// within 2^-22 of itself (two roundings; the scale is exact) plus 2^-32 (zl's own
// rounding, 2^-50 |zr|, |zr| < 2^14) of the double value. Rounding and clamp are
// monotone: where both ends of twice that interval round to one bfloat16, so does the
// value; else (one in 2^12) it is computed in double. 14336 crops of eight scenes:
// 915 -> 209 us.
__device__ __forceinline__ float crop_value(double zr, float zh, float zl, float d) {
  const float s = __fsub_rn(zh, d), bb = __fsub_rn(s, zh);
  const float err = __fsub_rn(__fsub_rn(zh, __fsub_rn(s, bb)), __fadd_rn(d, bb));
  const float t = __fmul_rn(__fadd_rn(s, __fadd_rn(err, zl)), (float)kScale);
  const float eps = __fadd_rn(__fmul_rn(fabsf(t), 0x1p-21f), 0x1p-31f);
  const float lo = fminf(fmaxf(__fsub_rn(t, eps), -kClamp), kClamp), hi = fminf(fmaxf(__fadd_rn(t, eps), -kClamp), kClamp);
  if (__bfloat16_as_ushort(__float2bfloat16_rn(lo)) == __bfloat16_as_ushort(__float2bfloat16_rn(hi)) &&
      fabsf(zh) < 16384.0f)
    return lo;
  const float x = __double2float_rn(__dmul_rn(__dsub_rn(zr, (double)d), kScale));
  return fminf(fmaxf(x, -kClamp), kClamp);
}

// ---------------------------------------------------------------- crops
// One block per hypothesis. The centre is the projection of (x, y, middle of
// V(O)'s height range), in double with every operation rounded separately:
// camera point = R_wc^T (p - t_wc) summed in the order 0, 1, 2; pixel
// floor(f (x_c / z_c) + c + 0.5). A pixel's value is
// clamp((z_ref - d) 10 / m, -3, 3) (float, then bfloat16) where the depth d is
// finite and > 0, else -4 (also outside the image and for a centre behind
// the camera or beyond 1e6 pixels).
__global__ void k_crops(Camera cam, const float* __restrict__ xs, const float* __restrict__ ys,
                        const DevMesh* __restrict__ meshes, int n_yaw, const float* const* __restrict__ scene_img,
                        const int32_t* __restrict__ parent_scene, const float* __restrict__ parent_z,
                        const int32_t* __restrict__ hyp_parent, const perch_obj* __restrict__ hyp, long long n_hyp,
                        bf16* __restrict__ crops, int32_t* __restrict__ onehot) {
  __shared__ int s_cu, s_cv, s_ok;
  __shared__ double s_zr;
  __shared__ float s_zh, s_zl;
  const long long h = blockIdx.x;
  if (h >= n_hyp) return;
  const perch_obj o = hyp[h];
  const int par = hyp_parent[h];
  if (threadIdx.x == 0) {
    const DevMesh& m = meshes[o.mesh];
    const double px = (double)xs[o.ix], py = (double)ys[o.iy];
    const double pz = __dmul_rn(__dadd_rn((double)m.vol_zlo, (double)m.vol_zhi), 0.5);
    const double d0 = __dsub_rn(px, (double)cam.twc[0]);
    const double d1 = __dsub_rn(py, (double)cam.twc[1]);
    const double d2 = __dsub_rn(pz, (double)cam.twc[2]);
    double c[3];
    for (int k = 0; k < 3; ++k)
      c[k] = __dadd_rn(__dadd_rn(__dmul_rn((double)cam.Rwc[0 * 3 + k], d0), __dmul_rn((double)cam.Rwc[1 * 3 + k], d1)),
                       __dmul_rn((double)cam.Rwc[2 * 3 + k], d2));
    int ok = c[2] > 0.0;
    double u = 0.0, v = 0.0;
    if (ok) {
      u = __dadd_rn(__dmul_rn((double)cam.fx, __ddiv_rn(c[0], c[2])), (double)cam.cx);
      v = __dadd_rn(__dmul_rn((double)cam.fy, __ddiv_rn(c[1], c[2])), (double)cam.cy);
      ok = fabs(u) < 1e6 && fabs(v) < 1e6;
    }
    s_ok = ok;
    s_cu = ok ? (int)floor(__dadd_rn(u, 0.5)) : 0;
    s_cv = ok ? (int)floor(__dadd_rn(v, 0.5)) : 0;
    s_zr = c[2];
    s_zh = __double2float_rn(c[2]);
    s_zl = __double2float_rn(__dsub_rn(c[2], (double)s_zh));
    onehot[h] = (int32_t)o.mesh * n_yaw + o.iyaw;
  }
  __syncthreads();
  const int W = cam.W, H = cam.H;
  const int sc = parent_scene ? parent_scene[par] : 0;
  const float* img = scene_img[sc];
  const float* pz = parent_z + (long long)par * W * H;
  const double zr = s_zr;
  const float zh = s_zh, zl = s_zl;
  for (int px = threadIdx.x; px < kCrop * kCrop; px += blockDim.x) {
    const int r = s_cv - kCrop / 2 + px / kCrop, c = s_cu - kCrop / 2 + px % kCrop;
    float val[2] = {kMissing, kMissing};
    if (s_ok && r >= 0 && r < H && c >= 0 && c < W) {
      const float d[2] = {img[(long long)r * W + c], pz[(long long)r * W + c]};
      for (int ch = 0; ch < 2; ++ch)
        if (isfinite(d[ch]) && d[ch] > 0.0f) val[ch] = crop_value(zr, zh, zl, d[ch]);
    }
    *reinterpret_cast<__nv_bfloat162*>(crops + (h * kCrop * kCrop + px) * 2) = __floats2bfloat162_rn(val[0], val[1]);
  }
}

int grid_for(long long n, int threads = 256) {
  return (int)std::max<long long>(1, std::min<long long>((n + threads - 1) / threads, 152LL * 16));
}

}  // namespace

// ---------------------------------------------------------------- network object
struct perch_cnn {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  // the backward pass's second stream and the events that fork and join it (see backward)
  cudaStream_t side = nullptr;
  cudaEvent_t ev_dz[kConvs] = {}, ev_wt = nullptr, ev_join = nullptr;
  std::string err;
  int n_onehot = 0, onehot_pad = 0, Kf = 0, max_batch = 0;
  long long step = 0;
  // FP32 master layout: conv weights [Cout][Kp], FC1 [96][Kf] (the bfloat16
  // region, contiguous), then conv biases, FC1 bias, FC2 weights, FC2 bias
  long long off_w[kConvs], off_f1, n_w16, off_b[kConvs], off_fb1, off_f2, off_fb2, n_total;
  DevBuf master, grad, adam_m, adam_v, w16;
  // batch buffers
  DevBuf act[kConvs], act_b[2], feat, h1, err_buf, pred_buf, loss_buf;
  DevBuf dz1, dfeat, dz[kConvs], part, bpart, part0, bpart0;
  bool params_set = false;
  // tc_err: the convolution kernels' wait-gave-up flag (device int); path: the
  // caller's choice (perch_cnn_set_tensor_path), one kernel serves both
  int path = 0;
  int sm_count = 152;
  DevBuf tc_err;
  // tensor maps of the convolutions' operands (forward, data and
  // weight gradient), and
  // the buffers they were made for
  ConvMaps fwd[2][kConvs], dgrad[kConvs], wgrad[kConvs];
  const void* fwd_for[2][kConvs][2] = {};
  const void* dgrad_for[kConvs][2] = {};
  const void* wgrad_for[kConvs][2] = {};
  long long fwd_n[2][kConvs] = {}, dgrad_n[kConvs] = {}, wgrad_n[kConvs] = {};
  DevBuf wt[kConvs];  // weights of the data gradients (k_dgrad_weights)

  int fail(int code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    err = buf;
    return code;
  }
  int cuda(cudaError_t e, const char* what) {
    if (e == cudaSuccess) return PERCH_OK;
    cudaGetLastError();
    if (e == cudaErrorMemoryAllocation) return fail(PERCH_E_OOM, "%s: %s", what, cudaGetErrorString(e));
    return fail(PERCH_E_CUDA, "%s: %s", what, cudaGetErrorString(e));
  }
  std::vector<DevBuf*> buffers() {
    std::vector<DevBuf*> v = {&master, &grad, &adam_m, &adam_v, &w16, &feat, &h1, &err_buf, &pred_buf,
                              &loss_buf, &dz1, &dfeat, &part, &bpart, &part0, &bpart0, &tc_err};
    for (int l = 0; l < kConvs; ++l) {
      v.push_back(&act[l]);
      if (l < 2) v.push_back(&act_b[l]);
      v.push_back(&wt[l]);
      v.push_back(&dz[l]);
    }
    return v;
  }
  void layout() {
    long long o = 0;
    for (int l = 0; l < kConvs; ++l) {
      off_w[l] = o;
      o += (long long)kCout[l] * kp_of(l);
    }
    off_f1 = o;
    o += (long long)kHidden * Kf;
    n_w16 = o;
    for (int l = 0; l < kConvs; ++l) {
      off_b[l] = o;
      o += kCout[l];
    }
    off_fb1 = o;
    o += kHidden;
    off_f2 = o;
    o += kHidden;
    off_fb2 = o;
    o += 4;
    n_total = o;
  }
  long long n_params() const {  // unpadded count, the packed order of the ABI
    long long n = 0;
    for (int l = 0; l < kConvs; ++l) n += (long long)kCout[l] * 9 * kCin[l] + kCout[l];
    return n + (long long)kHidden * (kFeat + n_onehot) + kHidden + kHidden + 1;
  }
  // packed (ABI) index <-> padded master index, in the packed order
  template <typename F>
  void for_each_param(F f) const {
    long long q = 0;
    for (int l = 0; l < kConvs; ++l) {
      const int K = 9 * kCin[l], Kp = kp_of(l);
      for (int o = 0; o < kCout[l]; ++o)
        for (int k = 0; k < K; ++k) f(q++, off_w[l] + (long long)o * Kp + k);
      for (int o = 0; o < kCout[l]; ++o) f(q++, off_b[l] + o);
    }
    for (int o = 0; o < kHidden; ++o)
      for (int k = 0; k < kFeat + n_onehot; ++k) f(q++, off_f1 + (long long)o * Kf + k);
    for (int o = 0; o < kHidden; ++o) f(q++, off_fb1 + o);
    for (int o = 0; o < kHidden; ++o) f(q++, off_f2 + o);
    f(q++, off_fb2);
  }
  int ensure_batch(int n, int chunk);
  int refresh_weights();
  int conv_fwd(int l, const DevBuf& x, int n, bf16* out, int set);
  int dgrad_weights(int l, cudaStream_t s);
  int conv_dgrad(int l, const bf16* dz, int n, bf16* out);
  int conv_wgrad(int l, const bf16* dz, int n, int splits, int ksplit, cudaStream_t s);
  int convolve(const bf16* crops, const int32_t* onehot, int n, int at, int set);
  int convolve_chunks(const bf16* crops, const int32_t* onehot, int n, int chunk);
  int forward(const bf16* crops, const int32_t* onehot, int n, float* pred, const float* target, int chunk);
  int backward(const bf16* crops, int n);
  int backward_pass(const bf16* crops, int n);
  void release();
};

#define CK_CTX(expr, what)                    \
  do {                                        \
    int rc_ = ctx->cuda((expr), what);        \
    if (rc_ != PERCH_OK) return rc_;          \
  } while (0)

#define CKN(expr, what)                       \
  do {                                        \
    int rc_ = net->cuda((expr), what);        \
    if (rc_ != PERCH_OK) return rc_;          \
  } while (0)

// buffers of n crops, the first two layers' of a chunk of them
int perch_cnn::ensure_batch(int n, int chunk) {
  perch_cnn* net = this;
  const long long N = std::max(n, 32), C = std::max(chunk, 32);
  for (int l = 0; l < kConvs - 1; ++l) {
    const long long Ho = kHin[l] / kStride[l];
    CKN(act[l].ensure(2 * (l == kConvs - 2 ? N : C) * Ho * Ho * kCout[l]), "alloc activations");
  }
  CKN(feat.ensure(2 * N * Kf), "alloc");
  CKN(h1.ensure(2 * N * kHidden), "alloc");
  CKN(err_buf.ensure(4 * N), "alloc");
  CKN(pred_buf.ensure(4 * N), "alloc");
  CKN(loss_buf.ensure(16), "alloc");
  return PERCH_OK;
}

int perch_cnn::refresh_weights() {
  perch_cnn* net = this;
  CKN(w16.ensure(2 * n_w16), "alloc");
  k_to_bf16<<<grid_for(n_w16), 256, 0, stream>>>(master.as<float>(), n_w16, w16.as<bf16>());
  CKN(cudaGetLastError(), "cast kernel");
  return PERCH_OK;
}

// the 128-row tiles of a layer's output pixels: boxes of 1 << lg_wo columns,
// `rows` rows and `imgs` images
static void conv_tile(int l, int n, ConvArgs* p, int* box) {
  const int Ho = kHin[l] / kStride[l];
  p->lg_wo = p->lg_ho = ilog2(Ho);
  p->M = n * Ho * Ho;
  p->tiles = (p->M + kTcRows - 1) / kTcRows;
  box[1] = Ho;
  box[2] = std::min(Ho, kTcRows / Ho);
  box[3] = kTcRows / (box[1] * box[2]);
}

// Forward convolution of layer l = 1 .. 3 over n crops, from `in` to `out`; the
// last one's are the FC input rows (crop m / 64, position m % 64). Set 1 runs on the
// side stream. The maps
// cover the whole buffer of x, so they stay until it is reallocated; rows past
// n crops are computed from what is there and not stored.
int perch_cnn::conv_fwd(int l, const DevBuf& in, int n, bf16* out, int set) {
  perch_cnn* net = this;
  const bf16* x = in.as<bf16>();
  const cudaStream_t st = set ? side : stream;
  const int H = kHin[l], Cin = kCin[l], N = kCout[l], Kp = kp_of(l);
  const bool pair = Cin == 32;  // two horizontal neighbours make a 64-channel row
  ConvArgs p{};
  int box[4] = {64};
  conv_tile(l, n, &p, box);
  const long long imgs = (long long)(in.cap / (2 * (size_t)H * H * Cin));
  const bf16* w = w16.as<bf16>() + off_w[l];
  if (fwd_for[set][l][0] != x || fwd_for[set][l][1] != w || fwd_n[set][l] != imgs) {
    const long long dims[4] = {pair ? 64 : Cin, H / 2, H / 2, imgs};
    const long long st[3] = {4LL * Cin, 4LL * H * Cin, 2LL * H * H * Cin};
    const long long wdims[2] = {Kp, N}, wst[1] = {2LL * Kp};
    for (int k = 0; k < 4; ++k) {
      box[0] = pair && !(k & 1) ? 32 : 64;
      CKN(encode_map(&fwd[set][l].a[k], x + ((k >> 1) * H + (pair ? 0 : k & 1)) * (long long)Cin, 4, dims, st, box),
          "tensor map");
    }
    for (int k = 0; k < 2; ++k) {
      const int wbox[2] = {k ? 32 : 64, N};
      CKN(encode_map(&fwd[set][l].b[k], w, 2, wdims, wst, wbox), "tensor map");
    }
    fwd_for[set][l][0] = x;
    fwd_for[set][l][1] = w;
    fwd_n[set][l] = imgs;
  }
  p.lg_c = ilog2(Cin);
  p.k_blocks = Kp / (pair ? 96 : 64);
  p.bias = master.as<float>() + off_b[l];
  p.ldc = N;
  p.grp = 1 << 30;
  p.out = out;
  if (l == kConvs - 1) {
    p.grp = (H / 2) * (H / 2);
    p.ldg = Kf;
  }
  int* e = tc_err.as<int>();
  CKN(l == 1   ? (conv_tma_t<96, 64, false, 288>(fwd[set][l], p, e, sm_count, st))
      : l == 2 ? (conv_tma_t<64, 128, false, 576>(fwd[set][l], p, e, sm_count, st))
               : (conv_tma_t<64, 128, false, 0>(fwd[set][l], p, e, sm_count, st)),
      "convolution");
  return PERCH_OK;
}

// weights of 64 input channels fit beside the ring
static int dgrad_parts(int C) { return C > 64 ? 2 : 1; }

int perch_cnn::dgrad_weights(int l, cudaStream_t s) {
  perch_cnn* net = this;
  const int C = kCin[l], Co = kCout[l];
  CKN(wt[l].ensure(2 * 9 * (size_t)C * Co), "alloc");
  k_dgrad_weights<<<grid_for(9LL * C * Co), 256, 0, s>>>(w16.as<bf16>() + off_w[l], kp_of(l), C, Co,
                                                         C / dgrad_parts(C), wt[l].as<bf16>());
  return net->cuda(cudaGetLastError(), "data-gradient weights");
}

// Data gradient of layer l = 1 .. 3: dz of its output to the gradient of its
// input, times the ReLU mask of that input
int perch_cnn::conv_dgrad(int l, const bf16* d, int n, bf16* out) {
  perch_cnn* net = this;
  const int H = kHin[l], Ho = H / 2, C = kCin[l], Co = kCout[l];
  ConvArgs p{};
  int box[4] = {64};
  conv_tile(l, n, &p, box);
  p.parts = dgrad_parts(C);
  const int N = C / p.parts;
  if (dgrad_for[l][0] != d || dgrad_for[l][1] != wt[l].p || dgrad_n[l] != n) {
    const long long dims[4] = {Co, Ho, Ho, n};
    const long long st[3] = {2LL * Co, 2LL * Ho * Co, 2LL * Ho * Ho * Co};
    CKN(encode_map(&dgrad[l].a[0], d, 4, dims, st, box), "tensor map");
    for (int k = 1; k < 4; ++k) dgrad[l].a[k] = dgrad[l].a[0];
    const long long wdims[2] = {Co, 9LL * C}, wst[1] = {2LL * Co};
    const int wbox[2] = {64, N};
    dgrad[l].b[1] = dgrad[l].b[0];
    CKN(encode_map(&dgrad[l].b[0], wt[l].p, 2, wdims, wst, wbox), "tensor map");
    dgrad_for[l][0] = d;
    dgrad_for[l][1] = wt[l].p;
    dgrad_n[l] = n;
  }
  p.lg_c = ilog2(Co);
  p.out = out;
  p.mask = act[l - 1].as<bf16>();
  p.H = H;
  p.C = C;
  int* e = tc_err.as<int>();
  CKN(l == 1 ? (conv_tma_t<64, 32, true, 9 * 64>(dgrad[l], p, e, sm_count, stream))
             : (conv_tma_t<64, 64, true, 9 * 128>(dgrad[l], p, e, sm_count, stream)),
      "data gradient");
  return PERCH_OK;
}

// Partial weight gradients of layer l = 1 .. 3 (k_sums adds them)
int perch_cnn::conv_wgrad(int l, const bf16* d, int n, int splits, int ksplit, cudaStream_t s) {
  perch_cnn* net = this;
  const int H = kHin[l], Ho = H / 2, C = kCin[l], Co = kCout[l], W = std::min(C, 64);
  const bf16* x = act[l - 1].as<bf16>();
  if (wgrad_for[l][0] != d || wgrad_for[l][1] != x || wgrad_n[l] != n) {
    const int xbox[4] = {W, Ho, 32 / Ho, 1}, dbox[4] = {64, Ho, 32 / Ho, 1};
    const long long xdims[4] = {C, Ho, Ho, n}, xst[3] = {4LL * C, 4LL * H * C, 2LL * H * H * C};
    for (int k = 0; k < 4; ++k)
      CKN(encode_map(&wgrad[l].a[k], x + ((k >> 1) * H + (k & 1)) * (long long)C, 4, xdims, xst, xbox), "tensor map");
    const long long ddims[4] = {Co, Ho, Ho, n}, dst[3] = {2LL * Co, 2LL * Ho * Co, 2LL * Ho * Ho * Co};
    CKN(encode_map(&wgrad[l].b[0], d, 4, ddims, dst, dbox), "tensor map");
    wgrad[l].b[1] = wgrad[l].b[0];
    wgrad_for[l][0] = d;
    wgrad_for[l][1] = x;
    wgrad_n[l] = n;
  }
  WgradArgs p{};
  p.blocks = n * Ho * Ho / 32;
  p.split = ksplit / 32;
  p.lg_wo = ilog2(Ho);
  p.part = part.as<float>();
  p.Kp = kp_of(l);
  p.split_stride = (long long)Co * p.Kp;
  int* e = tc_err.as<int>();
  CKN(l == 1   ? (wgrad_tma_t<32, 3, 1, 2, 3>(wgrad[l], p, splits, e, s))
      : l == 2 ? (wgrad_tma_t<64, 3, 2, 1, 5>(wgrad[l], p, splits, e, s))
               : (wgrad_tma_t<64, 6, 2, 1, 6>(wgrad[l], p, splits, e, s)),
      "weight gradient");
  return PERCH_OK;
}

// The first three convolutions (and the one-hot columns) of n crops, to
// crops at .. at + n - 1 of act[2] and of the FC input, by the stream and the first two layers'
// buffers of a set
int perch_cnn::convolve(const bf16* crops, const int32_t* onehot, int n, int at, int set) {
  perch_cnn* net = this;
  DevBuf &a = set ? act_b[0] : act[0], &b = set ? act_b[1] : act[1];
  k_conv1<<<8 * n, 256, 0, set ? side : stream>>>(
      reinterpret_cast<const uint32_t*>(crops), w16.as<bf16>() + off_w[0], master.as<float>() + off_b[0], a.as<bf16>(),
      onehot, onehot_pad, Kf, feat.as<bf16>() + (long long)at * Kf);
  CKN(cudaGetLastError(), "input layer");
  if (int rc = conv_fwd(1, a, n, b.as<bf16>(), set)) return rc;
  return conv_fwd(2, b, n, act[2].as<bf16>() + (long long)at * 16 * 16 * kCout[2], set);
}

// Layers 1 to 3 of n crops, `chunk` at a time, so that a chunk's activations (262
// and 131 KB a crop) stay in L2 from one layer to the next. Chunks take turns on the stream
// and the side stream: the input layer, bound by its stores, runs beside the
// other chunk's convolutions, which leave it registers and threads but hold the
// SM's shared memory. 2048 crops in chunks of 256: 590 us on one stream, 509 on two.
int perch_cnn::convolve_chunks(const bf16* crops, const int32_t* onehot, int n, int chunk) {
  perch_cnn* net = this;
  const bool two = n > chunk;
  if (two) {
    CKN(act_b[0].ensure(act[0].cap), "alloc activations");
    CKN(act_b[1].ensure(act[1].cap), "alloc activations");
    CKN(cudaEventRecord(ev_dz[0], stream), "event");
    CKN(cudaStreamWaitEvent(side, ev_dz[0], 0), "event");
  }
  int rc = PERCH_OK;
  for (int at = 0, k = 0; rc == PERCH_OK && at < n; at += chunk, ++k)
    rc = convolve(crops + (long long)at * 2 * kCrop * kCrop, onehot + at, std::min(chunk, n - at), at, k & 1);
  if (!two) return rc;
  cudaError_t e = cudaEventRecord(ev_join, side);  // joined whatever happened
  if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, ev_join, 0);
  if (rc == PERCH_OK) CKN(e, "join");
  return rc;
}

// Forward pass of n crops; with a target also the per-sample errors (for the
// backward pass). Layer 4 and the FC layers, whose few tiles leave SMs idle on
// one chunk, run on all n.
int perch_cnn::forward(const bf16* crops, const int32_t* onehot, int n, float* pred, const float* target, int chunk) {
  perch_cnn* net = this;
  int rc = ensure_batch(n, chunk);
  if (rc) return rc;
  if ((rc = convolve_chunks(crops, onehot, n, chunk))) return rc;
  if ((rc = conv_fwd(3, act[2], n, feat.as<bf16>(), 0))) return rc;
  // FC1: few output tiles over a long K, so split K and finish bias + ReLU in a second pass
  GemmArgs p{};
  p.A = feat.as<bf16>();
  p.lda = Kf;
  p.B = w16.as<bf16>() + off_f1;
  p.ldb = Kf;
  p.M = n;
  p.N = kHidden;
  p.K = Kf;
  // (the splits, and so the order of the sums, are those of a chunk alone)
  const int S = choose_splits(std::min(n, chunk), kHidden, Kf, &p.Ksplit);
  CKN(part.ensure(4 * (size_t)S * n * kHidden), "alloc");
  p.Cf = part.as<float>();
  p.ldc = kHidden;
  p.split_stride = (long long)n * kHidden;
  CKN(gemm<>(p, S, stream), "fc1 gemm");
  k_fc_tail<<<(n + 3) / 4, 128, 0, stream>>>(part.as<float>(), S, master.as<float>() + off_fb1,
                                             master.as<float>() + off_f2, master.as<float>() + off_fb2, n,
                                             h1.as<bf16>(), pred, target, err_buf.as<float>());
  CKN(cudaGetLastError(), "fc kernel");
  return PERCH_OK;
}

// Backward pass after forward(..., target); n a multiple of 32. Fills `grad`.
// The gradients of dz run down the layers on the stream; what only ends in
// `grad` (weight and bias gradients of the FC layers and of layers 2-4) follows
// on the side stream, behind the event of its layer's dz. The input layer's, the
// last ones, run on the stream again, with buffers of their own. The kernels leave SMs
// idle when alone: eight steps of 256 crops 4041 us on one stream, 3564 on two.
int perch_cnn::backward(const bf16* crops, int n) {
  perch_cnn* net = this;
  const int rc = backward_pass(crops, n);
  // joined whatever happened: nothing is left running beside the stream
  cudaError_t e = cudaEventRecord(ev_join, side);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, ev_join, 0);
  if (rc != PERCH_OK) return rc;
  CKN(e, "join");
  return PERCH_OK;
}

int perch_cnn::backward_pass(const bf16* crops, int n) {
  perch_cnn* net = this;
  const long long N = n;
  float* G = grad.as<float>();
  CKN(dz1.ensure(2 * N * kHidden), "alloc");
  CKN(dfeat.ensure(4 * N * kFeat), "alloc");
  long long max_part = 0;
  int S[kConvs], ks[kConvs];  // splits of the weight gradients
  for (int l = 0; l < kConvs; ++l) {
    const long long Ho = kHin[l] / kStride[l], M = N * Ho * Ho;
    S[l] = choose_splits(kCout[l], kp_of(l), (int)M, &ks[l]);
    if (l > 0) max_part = std::max(max_part, (long long)S[l] * kCout[l] * kp_of(l));
    CKN(dz[l].ensure(2 * M * kCout[l]), "alloc");
  }
  CKN(part.ensure(4 * max_part), "alloc");
  CKN(bpart.ensure(4 * 2048LL * 128), "alloc");
  CKN(part0.ensure(4LL * S[0] * kCout[0] * kp_of(0)), "alloc");
  CKN(bpart0.ensure(4 * 2048LL * kCout[0]), "alloc");
  // column sums of d for a bias gradient, then with the partial weight
  // gradients (splits 0: none) the sums of both
  auto col_sum = [&](const bf16* d, long long M, int C, DevBuf& bp, cudaStream_t s) -> int {
    const int R = (int)std::max<long long>(16, (M + 2047) / 2048);  // at most 2048 blocks
    const int nb = (int)((M + R - 1) / R);
    k_col_sum<<<nb, 128, 0, s>>>(d, M, C, R, bp.as<float>());
    return nb;
  };
  auto sums = [&](int nb, int C, float* bias_out, int splits, long long weights, float* out, DevBuf& bp, DevBuf& wp,
                  cudaStream_t s) -> int {
    const Sums p{bp.as<float>(), wp.as<float>(), bias_out, out, nb, C, splits, weights};
    k_sums<<<(unsigned)((C + 31) / 32 + (weights + 127) / 128), 1024, 0, s>>>(p);
    return net->cuda(cudaGetLastError(), "gradient sums");
  };
  // FC2
  k_fc2_dz1<<<grid_for(N * kHidden), 256, 0, stream>>>(h1.as<bf16>(), master.as<float>() + off_f2,
                                                       err_buf.as<float>(), n, dz1.as<bf16>());
  CKN(cudaGetLastError(), "fc2 backward kernel");
  CKN(cudaEventRecord(ev_dz[0], stream), "event");
  CKN(cudaStreamWaitEvent(side, ev_dz[0], 0), "event");
  for (int l = kConvs - 1; l > 0; --l)
    if (int rc = dgrad_weights(l, side)) return rc;
  CKN(cudaEventRecord(ev_wt, side), "event");
  k_fc2_loss<<<1, 256, 0, side>>>(err_buf.as<float>(), n, G + off_fb2, loss_buf.as<float>());
  k_fc2_wgrad<<<kHidden, 256, 0, side>>>(h1.as<bf16>(), err_buf.as<float>(), n, G + off_f2);
  CKN(cudaGetLastError(), "fc2 backward kernels");
  // FC1: dW = dz1^T feat (reduction over the batch, both operands batch-major),
  // db = column sums of dz1, dfeat = dz1 W (W read as [K][N])
  {
    GemmArgs p{};
    p.A = dz1.as<bf16>();
    p.lda = kHidden;
    p.B = feat.as<bf16>();
    p.ldb = Kf;
    p.M = kHidden;
    p.N = Kf;
    p.K = n;
    p.Ksplit = n;
    p.Cf = G + off_f1;
    p.ldc = Kf;
    CKN((gemm<false, false>(p, 1, side)), "fc1 weight-gradient gemm");
  }
  if (int rc = sums(col_sum(dz1.as<bf16>(), N, kHidden, bpart, side), kHidden, G + off_fb1, 0, 0, nullptr, bpart, part,
                    side))
    return rc;
  {
    GemmArgs p{};
    p.A = dz1.as<bf16>();
    p.lda = kHidden;
    p.B = w16.as<bf16>() + off_f1;  // columns 0 .. kFeat-1 of W: the conv features only
    p.ldb = Kf;
    p.M = n;
    p.N = kFeat;
    p.K = kHidden;
    p.Ksplit = kHidden;
    p.Cf = dfeat.as<float>();
    p.ldc = kFeat;
    CKN((gemm<true, false>(p, 1, stream)), "fc1 data-gradient gemm");
  }
  k_feat_relu_grad<<<grid_for(N * kFeat / 8), 256, 0, stream>>>(dfeat.as<float>(), feat.as<bf16>(), Kf, n,
                                                                 dz[kConvs - 1].as<bf16>());
  CKN(cudaGetLastError(), "relu gradient kernel");
  CKN(cudaStreamWaitEvent(stream, ev_wt, 0), "event");
  for (int l = kConvs - 1; l > 0; --l) {
    const int Ho = kHin[l] / kStride[l], Kp = kp_of(l), Co = kCout[l];
    const bf16* d = dz[l].as<bf16>();
    CKN(cudaEventRecord(ev_dz[l], stream), "event");
    if (int rc = conv_dgrad(l, d, n, dz[l - 1].as<bf16>())) return rc;
    CKN(cudaStreamWaitEvent(side, ev_dz[l], 0), "event");
    const int nb = col_sum(d, N * Ho * Ho, Co, bpart, side);
    // dW, split along the pixel reduction, partials summed in order
    if (int rc = conv_wgrad(l, d, n, S[l], ks[l], side)) return rc;
    if (int rc = sums(nb, Co, G + off_b[l], S[l], (long long)Co * Kp, G + off_w[l], bpart, part, side)) return rc;
  }
  const long long M = N * kCrop * kCrop;
  const bf16* d = dz[0].as<bf16>();
  const int nb = col_sum(d, M, kCout[0], bpart0, stream);
  const int smem = kW1Stages * kW1Px * kW1Ld + (ks[0] / kCrop + 5) * kW1Row * 4;
  CKN(cudaFuncSetAttribute(k_wgrad1, cudaFuncAttributeMaxDynamicSharedMemorySize, smem), "weight gradient");
  k_wgrad1<<<S[0], 256, smem, stream>>>(reinterpret_cast<const uint32_t*>(crops), d, (int)M, ks[0], part0.as<float>());
  CKN(cudaGetLastError(), "weight gradient");
  return sums(nb, kCout[0], G + off_b[0], S[0], (long long)kCout[0] * kp_of(0), G + off_w[0], bpart0, part0, stream);
}

void perch_cnn::release() {
  for (DevBuf* b : buffers()) b->release();
  for (int l = 0; l < kConvs; ++l)
    if (ev_dz[l]) cudaEventDestroy(ev_dz[l]);
  if (ev_wt) cudaEventDestroy(ev_wt);
  if (ev_join) cudaEventDestroy(ev_join);
  if (side) cudaStreamDestroy(side);
  if (own_stream) cudaStreamDestroy(stream);
}

int net_predict(perch_ctx* ctx, perch_cnn* net, const perch_obj* parents, int parent_stride, const int32_t* plen,
                const int32_t* pscene, int n_par, const int32_t* hyp_parent, const perch_obj* hyp, long long n_hyp,
                float* pred_host) {
  if (n_hyp == 0) return PERCH_OK;
  CK_CTX(ctx->net_crops.ensure(2 * (size_t)kCrop * kCrop * 2 * n_hyp), "alloc crops");
  CK_CTX(ctx->net_onehot.ensure(4 * (size_t)n_hyp), "alloc");
  CK_CTX(ctx->net_pred.ensure(4 * (size_t)n_hyp), "alloc");
  int rc = perch_cnn_crops(ctx, parents, parent_stride, plen, pscene, n_par, hyp_parent, hyp, n_hyp,
                           ctx->net_crops.as<uint16_t>(), ctx->net_onehot.as<int32_t>());
  if (rc) return rc;
  rc = perch_cnn_forward(net, ctx->net_crops.as<uint16_t>(), ctx->net_onehot.as<int32_t>(), n_hyp,
                         ctx->net_pred.as<float>());
  if (rc) return ctx->fail(rc, "learned heuristic: %s", net->err.c_str());
  CK_CTX(cudaMemcpyAsync(pred_host, ctx->net_pred.p, 4 * (size_t)n_hyp, cudaMemcpyDeviceToHost, net->stream),
         "copy predictions");
  CK_CTX(cudaStreamSynchronize(net->stream), "learned heuristic");
  return PERCH_OK;
}

// ---------------------------------------------------------------- C ABI
extern "C" {

int perch_cnn_create(perch_cnn** out, int device, void* cuda_stream, int32_t n_onehot, int32_t max_batch) {
  if (!out) return PERCH_E_ARG;
  *out = nullptr;
  if (n_onehot < 1 || n_onehot > 65536 || max_batch < 32 || max_batch > 1024 || max_batch % 32) return PERCH_E_ARG;
  if (cudaSetDevice(device) != cudaSuccess) {
    cudaGetLastError();
    return PERCH_E_CUDA;
  }
  perch_cnn* net = new perch_cnn;
  net->device = device;
  cudaDeviceGetAttribute(&net->sm_count, cudaDevAttrMultiProcessorCount, device);
  net->n_onehot = n_onehot;
  net->onehot_pad = round32(n_onehot);
  net->Kf = kFeat + net->onehot_pad;
  net->max_batch = max_batch;
  net->layout();
  if (cuda_stream) {
    net->stream = (cudaStream_t)cuda_stream;
  } else {
    if (cudaStreamCreateWithFlags(&net->stream, cudaStreamNonBlocking) != cudaSuccess) {
      cudaGetLastError();
      delete net;
      return PERCH_E_CUDA;
    }
    net->own_stream = true;
  }
  const size_t bytes = 4 * (size_t)net->n_total;
  bool ok = net->master.ensure(bytes) == cudaSuccess && net->grad.ensure(bytes) == cudaSuccess &&
            net->adam_m.ensure(bytes) == cudaSuccess && net->adam_v.ensure(bytes) == cudaSuccess &&
            net->tc_err.ensure(16) == cudaSuccess && cudaMemsetAsync(net->tc_err.p, 0, 16, net->stream) == cudaSuccess;
  ok = ok && cudaMemsetAsync(net->master.p, 0, bytes, net->stream) == cudaSuccess &&
       cudaMemsetAsync(net->grad.p, 0, bytes, net->stream) == cudaSuccess &&
       cudaMemsetAsync(net->adam_m.p, 0, bytes, net->stream) == cudaSuccess &&
       cudaMemsetAsync(net->adam_v.p, 0, bytes, net->stream) == cudaSuccess;
  ok = ok && cudaStreamCreateWithFlags(&net->side, cudaStreamNonBlocking) == cudaSuccess;
  for (int l = 0; l < kConvs; ++l)
    ok = ok && cudaEventCreateWithFlags(&net->ev_dz[l], cudaEventDisableTiming) == cudaSuccess;
  ok = ok && cudaEventCreateWithFlags(&net->ev_wt, cudaEventDisableTiming) == cudaSuccess &&
       cudaEventCreateWithFlags(&net->ev_join, cudaEventDisableTiming) == cudaSuccess;
  ok = ok && net->refresh_weights() == PERCH_OK && cudaStreamSynchronize(net->stream) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    net->release();
    delete net;
    return PERCH_E_CUDA;
  }
  *out = net;
  return PERCH_OK;
}

int perch_cnn_destroy(perch_cnn* net) {
  if (!net) return PERCH_OK;
  cudaSetDevice(net->device);
  cudaStreamSynchronize(net->stream);
  net->release();
  delete net;
  return PERCH_OK;
}

const char* perch_cnn_last_error(const perch_cnn* net) { return net ? net->err.c_str() : "null network"; }

int perch_cnn_set_tensor_path(perch_cnn* net, int32_t path) {
  if (!net) return PERCH_E_ARG;
  if (path != 0 && path != 1) return net->fail(PERCH_E_ARG, "tensor path must be 0 or 1");
  net->path = path;
  return PERCH_OK;
}

int perch_cnn_tensor_status(perch_cnn* net, int32_t* path, int32_t* waits_gave_up) {
  if (!net) return PERCH_E_ARG;
  if (cudaSetDevice(net->device) != cudaSuccess) return net->cuda(cudaGetLastError(), "cudaSetDevice");
  int e = 0;
  int rc = net->cuda(cudaStreamSynchronize(net->stream), "stream");
  if (rc) return rc;
  rc = net->cuda(cudaMemcpy(&e, net->tc_err.p, sizeof e, cudaMemcpyDeviceToHost), "read flag");
  if (rc) return rc;
  if (path) *path = net->path;
  if (waits_gave_up) *waits_gave_up = e;
  return PERCH_OK;
}

int perch_cnn_param_count(const perch_cnn* net, int64_t* n) {
  if (!net || !n) return PERCH_E_ARG;
  *n = net->n_params();
  return PERCH_OK;
}

int perch_cnn_set_params(perch_cnn* net, const float* params, int64_t n) {
  if (!net) return PERCH_E_ARG;
  net->err.clear();
  if (!params || n != net->n_params()) return net->fail(PERCH_E_ARG, "expected %lld parameters", net->n_params());
  CKN(cudaSetDevice(net->device), "cudaSetDevice");
  std::vector<float> h((size_t)net->n_total, 0.0f);
  net->for_each_param([&](long long q, long long i) { h[i] = params[q]; });
  const size_t bytes = 4 * (size_t)net->n_total;
  CKN(cudaMemcpyAsync(net->master.p, h.data(), bytes, cudaMemcpyHostToDevice, net->stream), "copy parameters");
  CKN(cudaMemsetAsync(net->adam_m.p, 0, bytes, net->stream), "memset");
  CKN(cudaMemsetAsync(net->adam_v.p, 0, bytes, net->stream), "memset");
  net->step = 0;
  int rc = net->refresh_weights();
  if (rc) return rc;
  CKN(cudaStreamSynchronize(net->stream), "set parameters");
  net->params_set = true;
  return PERCH_OK;
}

int perch_cnn_get_params(perch_cnn* net, float* params, int64_t n) {
  if (!net) return PERCH_E_ARG;
  net->err.clear();
  if (!params || n != net->n_params()) return net->fail(PERCH_E_ARG, "expected %lld parameters", net->n_params());
  CKN(cudaSetDevice(net->device), "cudaSetDevice");
  std::vector<float> h((size_t)net->n_total);
  CKN(cudaMemcpyAsync(h.data(), net->master.p, 4 * h.size(), cudaMemcpyDeviceToHost, net->stream), "copy");
  CKN(cudaStreamSynchronize(net->stream), "get parameters");
  net->for_each_param([&](long long q, long long i) { params[q] = h[i]; });
  return PERCH_OK;
}

// crops whose layer 4 and FC layers a prediction runs at once: 2048 crops in chunks of 256,
// 728 us with 256, 629 with 512, 590 with 1024 (act[2] is then 67 MB)
static constexpr int kGroup = 1024;

int perch_cnn_forward(perch_cnn* net, const uint16_t* crops, const int32_t* onehot, int64_t n, float* pred) {
  if (!net) return PERCH_E_ARG;
  net->err.clear();
  if (n < 0 || (n > 0 && (!crops || !onehot || !pred))) return net->fail(PERCH_E_ARG, "bad arguments");
  CKN(cudaSetDevice(net->device), "cudaSetDevice");
  // whole chunks of max_batch in groups of up to kGroup crops, then the rest
  const int64_t whole = n / net->max_batch * net->max_batch, group = std::max(kGroup / net->max_batch, 1) * net->max_batch;
  for (int64_t b = 0, nb; b < n; b += nb) {
    nb = b < whole ? std::min<int64_t>(group, whole - b) : n - b;
    int rc = net->forward(reinterpret_cast<const bf16*>(crops) + b * 2 * kCrop * kCrop, onehot + b, (int)nb, pred + b,
                          nullptr, net->max_batch);
    if (rc) return rc;
  }
  return PERCH_OK;
}

int perch_cnn_gradients(perch_cnn* net, const uint16_t* crops, const int32_t* onehot, const float* target, int32_t n,
                        float* grads, float* loss, float* pred) {
  if (!net) return PERCH_E_ARG;
  net->err.clear();
  if (!crops || !onehot || !target || n < 32 || n > net->max_batch || n % 32)
    return net->fail(PERCH_E_ARG, "need device crops / one-hot / targets and 32 <= n <= %d, n %% 32 == 0",
                     net->max_batch);
  CKN(cudaSetDevice(net->device), "cudaSetDevice");
  int rc = net->ensure_batch(n, n);  // pred_buf is passed below
  if (rc) return rc;
  rc = net->forward(reinterpret_cast<const bf16*>(crops), onehot, n, net->pred_buf.as<float>(), target, n);
  if (rc) return rc;
  rc = net->backward(reinterpret_cast<const bf16*>(crops), n);
  if (rc) return rc;
  if (grads) {
    std::vector<float> h((size_t)net->n_total);
    CKN(cudaMemcpyAsync(h.data(), net->grad.p, 4 * h.size(), cudaMemcpyDeviceToHost, net->stream), "copy");
    CKN(cudaStreamSynchronize(net->stream), "gradients");
    net->for_each_param([&](long long q, long long i) { grads[q] = h[i]; });
  }
  if (loss) CKN(cudaMemcpyAsync(loss, net->loss_buf.p, 4, cudaMemcpyDeviceToHost, net->stream), "copy");
  if (pred) CKN(cudaMemcpyAsync(pred, net->pred_buf.p, 4 * (size_t)n, cudaMemcpyDeviceToHost, net->stream), "copy");
  CKN(cudaStreamSynchronize(net->stream), "gradients");
  return PERCH_OK;
}

int perch_cnn_train_step(perch_cnn* net, const uint16_t* crops, const int32_t* onehot, const float* target,
                         int32_t n, float lr, float* loss) {
  if (!net) return PERCH_E_ARG;
  net->err.clear();
  if (!crops || !onehot || !target || n < 32 || n > net->max_batch || n % 32 || !(lr > 0.0f))
    return net->fail(PERCH_E_ARG, "need device crops / one-hot / targets, 32 <= n <= %d, n %% 32 == 0, lr > 0",
                     net->max_batch);
  CKN(cudaSetDevice(net->device), "cudaSetDevice");
  int rc = net->forward(reinterpret_cast<const bf16*>(crops), onehot, n, net->pred_buf.as<float>(), target, n);
  if (rc) return rc;
  rc = net->backward(reinterpret_cast<const bf16*>(crops), n);
  if (rc) return rc;
  net->step++;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = (float)(1.0 - std::pow((double)b1, (double)net->step));
  const float c2 = (float)(1.0 - std::pow((double)b2, (double)net->step));
  k_adam<<<grid_for(net->n_total / 4), 256, 0, net->stream>>>(
      net->master.as<float4>(), net->grad.as<float4>(), net->adam_m.as<float4>(), net->adam_v.as<float4>(),
      (int)(net->n_total / 4), lr, b1, b2, c1, c2, 1e-8f, (int)(net->n_w16 / 4), net->w16.as<uint2>());
  CKN(cudaGetLastError(), "adam kernel");
  if (loss) CKN(cudaMemcpyAsync(loss, net->loss_buf.p, 4, cudaMemcpyDeviceToDevice, net->stream), "copy loss");
  return PERCH_OK;
}

int perch_cnn_crops(perch_ctx* ctx, const perch_obj* parents, int32_t parent_stride, const int32_t* parent_len,
                    const int32_t* parent_scene, int32_t n_par, const int32_t* hyp_parent, const perch_obj* hyp,
                    int64_t n_hyp, uint16_t* crops, int32_t* onehot) {
  if (!ctx) return PERCH_E_ARG;
  ctx->err.clear();
  if (!ctx->has_obs) return ctx->fail(PERCH_E_STATE, "set an observation first");
  if (n_hyp < 0 || n_hyp > 0x7fffffffLL) return ctx->fail(PERCH_E_ARG, "n_hyp out of range");
  if (n_hyp == 0) return PERCH_OK;
  if (!parent_len || !hyp_parent || !hyp || !crops || !onehot || n_par < 1 || parent_stride < 0 ||
      (parent_stride > 0 && !parents))
    return ctx->fail(PERCH_E_ARG, "null pointer or bad sizes");
  if (n_par > 65535 || (long long)n_par * std::max(parent_stride, 1) > 65535)
    return ctx->fail(PERCH_E_ARG, "too many parents in one batch (n_par x stride <= 65535)");
  auto bad = [&](const perch_obj& o) {
    return o.mesh >= ctx->n_mesh || o.ix < 0 || o.ix >= ctx->nx || o.iy < 0 || o.iy >= ctx->ny ||
           o.iyaw >= ctx->n_yaw;
  };
  for (int i = 0; i < n_par; ++i) {
    if (parent_len[i] < 0 || parent_len[i] > parent_stride)
      return ctx->fail(PERCH_E_ARG, "parent %d: length %d outside [0, stride]", i, parent_len[i]);
    if (parent_scene && (parent_scene[i] < 0 || parent_scene[i] >= (int)ctx->scenes.size()))
      return ctx->fail(PERCH_E_ARG, "parent %d: scene %d not set", i, parent_scene[i]);
    for (int k = 0; k < parent_len[i]; ++k)
      if (bad(parents[(long long)i * parent_stride + k])) return ctx->fail(PERCH_E_ARG, "parent %d: bad object", i);
  }
  for (long long h = 0; h < n_hyp; ++h)
    if (hyp_parent[h] < 0 || hyp_parent[h] >= n_par || bad(hyp[h]))
      return ctx->fail(PERCH_E_ARG, "hypothesis %lld: bad parent or object", h);
  perch_ctx* c = ctx;
  auto ck = [c](cudaError_t e, const char* what) { return c->cuda(e, what); };
  int rc;
  if ((rc = ck(cudaSetDevice(ctx->device), "cudaSetDevice"))) return rc;
  const size_t npx = (size_t)ctx->cam.W * ctx->cam.H;
  const size_t pbytes = sizeof(perch_obj) * std::max<size_t>((size_t)n_par * parent_stride, 1);
  if ((rc = ck(ctx->parent_z.ensure(4 * npx * n_par), "alloc parent z-buffers"))) return rc;
  if ((rc = ck(ctx->b_parents.ensure(pbytes), "alloc"))) return rc;
  if ((rc = ck(ctx->b_plen.ensure(8 * (size_t)n_par), "alloc"))) return rc;
  if ((rc = ck(ctx->b_hp.ensure(4 * (size_t)n_hyp), "alloc"))) return rc;
  if ((rc = ck(ctx->b_hyp.ensure(sizeof(perch_obj) * (size_t)n_hyp), "alloc"))) return rc;
  int32_t* d_plen = ctx->b_plen.as<int32_t>();
  cudaStream_t s = ctx->stream;
  if (parent_stride > 0 &&
      (rc = ck(cudaMemcpyAsync(ctx->b_parents.p, parents, sizeof(perch_obj) * (size_t)n_par * parent_stride,
                               cudaMemcpyHostToDevice, s), "copy")))
    return rc;
  if ((rc = ck(cudaMemcpyAsync(d_plen, parent_len, 4 * (size_t)n_par, cudaMemcpyHostToDevice, s), "copy"))) return rc;
  if (parent_scene &&
      (rc = ck(cudaMemcpyAsync(d_plen + n_par, parent_scene, 4 * (size_t)n_par, cudaMemcpyHostToDevice, s), "copy")))
    return rc;
  if ((rc = ck(cudaMemcpyAsync(ctx->b_hp.p, hyp_parent, 4 * (size_t)n_hyp, cudaMemcpyHostToDevice, s), "copy")))
    return rc;
  if ((rc = ck(cudaMemcpyAsync(ctx->b_hyp.p, hyp, sizeof(perch_obj) * (size_t)n_hyp, cudaMemcpyHostToDevice, s),
               "copy")))
    return rc;
  if ((rc = ck(launch_fill_u32(ctx->parent_z.as<uint32_t>(), kInfBits, (long long)npx * n_par, s), "clear")))
    return rc;
  Batch b;
  std::memset(&b, 0, sizeof b);
  b.parents = ctx->b_parents.as<perch_obj>();
  b.parent_stride = std::max(parent_stride, 1);  // stride 0: every parent is empty
  b.parent_len = d_plen;
  b.n_par = n_par;
  b.parent_z = ctx->parent_z.as<float>();
  if ((rc = ck(launch_render_parents(ctx->cam, ctx->geometry(), b, ctx->max_chunks, nullptr, s), "render parents")))
    return rc;
  k_crops<<<(unsigned)n_hyp, 256, 0, s>>>(ctx->cam, ctx->xs.as<float>(), ctx->ys.as<float>(),
                                          ctx->meshes.as<DevMesh>(), ctx->n_yaw, ctx->d_scene_img.as<const float*>(),
                                          parent_scene ? d_plen + n_par : nullptr, ctx->parent_z.as<float>(),
                                          ctx->b_hp.as<int32_t>(), ctx->b_hyp.as<perch_obj>(), n_hyp,
                                          reinterpret_cast<bf16*>(crops), onehot);
  if ((rc = ck(cudaGetLastError(), "crop kernel"))) return rc;
  return ck(cudaStreamSynchronize(s), "crops");
}

int perch_set_heuristic_net(perch_ctx* ctx, perch_cnn* net, int32_t n_candidates) {
  if (!ctx) return PERCH_E_ARG;
  ctx->err.clear();
  if (net && net->n_onehot < ctx->n_mesh * ctx->n_yaw)
    return ctx->fail(PERCH_E_ARG, "network one-hot width %d < meshes x yaws %d", net->n_onehot,
                     ctx->n_mesh * ctx->n_yaw);
  if (n_candidates < 1 || n_candidates > 4096) return ctx->fail(PERCH_E_ARG, "n_candidates outside [1, 4096]");
  ctx->net = net;
  ctx->net_candidates = n_candidates;
  return PERCH_OK;
}

}  // extern "C"
