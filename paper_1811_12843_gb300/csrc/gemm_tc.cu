// Grouped GEMM on the tensor cores for bf16 networks of any size: the shapes that the chained MLP
// kernels (hidden width 256, rows of whole 16-byte units) do not take. One 128 x BN output tile of
// one problem per CTA, fp32 accumulation in tensor memory, the epilogues of the CUDA-core GEMM.
//
// Operands are staged by every thread with cp.async, in copies of the widest size that their rows'
// starts allow (TMA wants 16-byte row strides, which widths such as 500 or 50 do not give), straight
// into the 128-byte swizzle: K-major or MN-major as they lie in memory, so that the backward's
// transposed products need no transposition. Three chunks of 64 k: two in flight while one is
// multiplied.
// Bound: the launch and the latency of a tile's chunks on small grids (11 us a launch), the staging's
// L2 reads and instructions on large ones (270 TFLOP/s at 100 problems of 768 x 512 x 1000).
// Measured per phase against the CUDA-core kernel, 3x4 cells, 37 rows, 50 -> 200 -> 200 -> 500:
// generators 82 -> 35 us, discriminators 210 -> 45, backward 157 -> 67 (52 with the generator's weight
// gradients, over 37 rows, here too).
#include <type_traits>

#include "common.cuh"
#include "engine.h"
#include "tc_ptx.cuh"

namespace lipz {

namespace {

using namespace tc;

constexpr int BM = 128, BK = 64;
constexpr int STAGES = 3;
constexpr int NT = 256;
constexpr int BOX = 64 * BK * 2;          // one {64 MN, 64 K} box of an MN-major operand
constexpr int EPI_LD = 33;                // floats per row of a warp's 32 x 32 staging block
constexpr int CTRL = 128;

constexpr int gemm_tc_smem(int bn) { return 1024 + STAGES * (BM + bn) * BK * 2 + CTRL; }

template <int N>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, int bytes) {
  if (N == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(N),
                 "r"(bytes)
                 : "memory");
}

// Eight elements (one 16-byte unit of a tile), the first n of them from src, the rest zero, in
// copies of A bytes.
template <int A>
__device__ __forceinline__ void copy_unit(uint32_t dst, const bf16* src, int n) {
  if (A >= 4) {
#pragma unroll
    for (int i = 0; i < 16 / A; ++i) {
      const int left = min(A, max(0, 2 * n - i * A));
      cp_async<(A >= 4 ? A : 4)>(dst + i * A, left ? src + i * (A / 2) : src, left);
    }
  } else {
    const unsigned short* s = reinterpret_cast<const unsigned short*>(src);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t lo = 2 * i < n ? __ldg(s + 2 * i) : 0u;
      const uint32_t hi = 2 * i + 1 < n ? __ldg(s + 2 * i + 1) : 0u;
      w[i] = lo | hi << 16;
    }
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w[0]), "r"(w[1]),
                 "r"(w[2]), "r"(w[3])
                 : "memory");
  }
}

// This thread's share of an operand tile [ROWS][64 k]: ROWS / 32 units, in the 128-byte swizzle,
// K-major when k is the unit stride and MN-major otherwise. Rows past the operand's last are left
// as they are (they meet only results that are not stored); k past K up to the MMA's last step of
// 16 reads as zero.
template <int ROWS>
struct TileLoader {
  static constexpr int U = ROWS / 32;
  static constexpr int PER_K = ROWS / 8;  // units of one k row, MN-major
  const bf16* src;
  int64_t ustep, kstep;  // elements from unit to unit and from chunk to chunk
  uint32_t dst, dstep;
  int k, kinc;           // k of unit 0 and from unit to unit (K-major: 0)
  int n0, uinc;          // K-major: rows left from unit 0's on; MN-major: elements of a unit
  bool kmaj;

  __device__ __forceinline__ void init(const bf16* p, int64_t sr, int64_t sk, int r0, int rows) {
    const int t = threadIdx.x;
    kmaj = sk == 1;
    if (kmaj) {
      const int r = t >> 3, c = t & 7;
      src = p + (int64_t)(r0 + r) * sr + c * 8;
      ustep = 32 * sr;
      kstep = BK;
      dst = (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4));
      dstep = 32 * 128;
      k = c * 8;
      kinc = 0;
      n0 = rows - r0 - r;
      uinc = 32;
    } else {
      const int kr = t / PER_K, c = t % PER_K;
      src = p + r0 + c * 8 + (int64_t)kr * sk;
      ustep = (int64_t)(NT / PER_K) * sk;
      kstep = BK * sk;
      dst = (uint32_t)((c >> 3) * BOX + kr * 128 + (((c & 7) ^ (kr & 7)) << 4));
      dstep = (uint32_t)(NT / PER_K) * 128;
      k = kr;
      kinc = NT / PER_K;
      n0 = min(8, rows - r0 - c * 8);
      uinc = 0;
    }
  }
  template <int A>
  __device__ __forceinline__ void load(uint32_t tile, int kc, int K) const {
    const bf16* s = src + kc * kstep;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int kk = kc * BK + k + u * kinc, left = n0 - u * uinc;
      if (left <= 0 || kk >= ((K + 15) & ~15)) continue;
      const int n = kmaj ? min(8, K - kk) : (kk < K ? left : 0);
      copy_unit<A>(tile + dst + u * dstep, n > 0 ? s + u * ustep : src, max(n, 0));
    }
  }
  __device__ __forceinline__ void load(uint32_t tile, int kc, int K, int align) const {
    if (align == 3) load<16>(tile, kc, K);
    else if (align == 2) load<8>(tile, kc, K);
    else if (align == 1) load<4>(tile, kc, K);
    else load<2>(tile, kc, K);
  }
};

template <int BN>
__global__ void __launch_bounds__(NT, 2)
    k_gemm_tc(const GemmDesc* __restrict__ descs, const int2* __restrict__ tiles, float slope,
              int* err) {
  constexpr int STAGE = (BM + BN) * BK * 2;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + STAGES * STAGE);  // [2]: a sum's MMAs done
  const uint32_t bar = smem_u32(bars);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gbase + STAGES * STAGE + 64);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + STAGES * STAGE + 68);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 8, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32((const void*)tmem_slot)),
                 "n"(2 * BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int2 tl = __ldg(&tiles[blockIdx.x]);
  const GemmDesc& d = descs[tl.x];
  const int m0 = (tl.y >> 16) * BM, n0 = (tl.y & 0xFFFF) * BN;
  const int M = d.M, N = d.N, K = d.K;
  const int al_a = d.vec & 3, al_b = d.vec >> 2;
  // (the problem list is the host's; only the operands are the previous kernel's results)
  pdl_wait();
  const bf16* A = (const bf16*)d.A;
  const bf16* Bm = (const bf16*)d.B;
  const float* bias = d.bias;
  if (d.wsel) {
    const int64_t off = (int64_t)d.wsel[d.cell] * d.wsel_stride;
    if (d.wsel_op == 1) A += off; else Bm += off;
    if (bias) bias += off;
  }
  TileLoader<BM> la;
  TileLoader<BN> lb;
  la.init(A, d.sam, d.sak, m0, M);
  lb.init(Bm, d.sbn, d.sbk, n0, N);
  const int nk = (K + BK - 1) / BK;
  auto load = [&](int kc) {
    if (kc < nk) {
      const uint32_t s = base + (uint32_t)(kc % STAGES) * STAGE;
      la.load(s, kc, K, al_a);
      lb.load(s + BM * BK * 2, kc, K, al_b);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // two chunks in flight ahead of the one that is multiplied
  load(0);
  load(1);
  const int n = (min(BN, N - n0) + 63) & ~63;
  const uint32_t idesc = idesc_bf16_major(BM, n, la.kmaj ? 0 : 1, lb.kmaj ? 0 : 1);
  // A chunk's sums stand in tensor memory (even and odd ones apart) and are added to fp32 sums in
  // registers, rounded to nearest: the tensor cores' own additions truncate. That costs 7 to 20 % of
  // the kernel's time with chunks of 64 k; where fewer additions follow, K below GEMM_TC_CHUNK_K, every
  // MMA step of 16 k is a sum of its own. Error against 64 bits, in 2^-24 of the result's root mean
  // square, as one sum in tensor memory, by chunks of 64, of 16, and of an fp32 FMA chain (in brackets
  // for operands that are half zeros, as a weight gradient's are): 784 k 12.3, 1.56, 2.11 and 3.19;
  // 160 k by 64 1.19 (0.657), chain 1.37 (0.667); 144 k by 16 1.00 (0.595), chain 1.28 (0.638); 64 k
  // 0.97, 0.97, 0.74 (0.396) and 0.87 (0.398). 48 k by 16 0.66 (0.332), chain 0.73 (0.324): weight
  // gradients over fewer than GEMM_TC_MIN_K_STORE rows go to k_gemm, and so do other products over
  // fewer than GEMM_TC_MIN_K (16 k 0.43 and 0.38).
  constexpr int CW = BN / 2;  // columns of a thread: half of the tile's
  const int q = warp & 3, half = warp >> 2;
  const bool elected = elect_one();
  bool ok = true;
  float acc[CW];
#pragma unroll
  for (int e = 0; e < CW; ++e) acc[e] = 0.f;
  auto add_sum = [&](int i) {
    tc_fence_after();
    const uint32_t t = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)((i & 1) * BN + half * CW);
#pragma unroll
    for (int c = 0; c < CW; c += 32) {
      uint32_t r[32];
      LIPZ_TMEM_LD32(t + c, r);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 32; ++e) acc[c + e] += __uint_as_float(r[e]);
    }
  };
  // the sums of `per` MMA steps
  auto product = [&](auto per_c) {
    constexpr int per = decltype(per_c)::value;
    const int steps = (K + 15) / 16, sums = (steps + per - 1) / per;
    for (int i = 0; i < sums; ++i) {
      const int s0 = i * per, kc = s0 / (BK / 16), k0 = s0 % (BK / 16);  // first step; in its chunk
      if (k0 == 0) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      // (and every warp has read the sum before the last, whose place this one takes)
      tc_fence_before();
      __syncthreads();
      if (warp == 0) {
        tc_fence_after();
        const uint32_t sA = base + (uint32_t)(kc % STAGES) * STAGE, sB = sA + BM * BK * 2;
        // (a step of 16 k further on: 32 bytes K-major, 2048 MN-major; 16-byte units)
        const uint32_t iA = la.kmaj ? 2 : 128, iB = lb.kmaj ? 2 : 128;
        const uint64_t dA = (la.kmaj ? sw128_desc(sA) : sw128_mn_desc(sA, BOX)) + k0 * iA;
        const uint64_t dB = (lb.kmaj ? sw128_desc(sB) : sw128_mn_desc(sB, BOX)) + k0 * iB;
        const uint32_t dt = tmem + (uint32_t)(i & 1) * BN;
        const int n_mma = min(per, steps - s0);
        if (elected) {
          tc_mma(dt, dA, dB, idesc, 0u);
#pragma unroll
          for (int kk = 1; kk < BK / 16; ++kk)
            if (kk < n_mma) tc_mma_acc(dt, dA + kk * iA, dB + kk * iB, idesc);
          tc_commit(bar + 8 * (i & 1));
        }
      }
      __syncwarp();
      if (i > 0)
        ok = mbar_wait_warp(bar + 8 * ((i - 1) & 1), (uint32_t)(((i - 1) >> 1) & 1), abort_flag, err,
                            1) && ok;
      // chunk kc + 2 goes where chunk kc - 1 was, whose MMAs have read it
      if (k0 == 0) load(kc + 2);
      if (i > 0) add_sum(i - 1);
    }
    // the last commit covers every MMA of the tile
    ok = mbar_wait_warp(bar + 8 * ((sums - 1) & 1), (uint32_t)(((sums - 1) >> 1) & 1), abort_flag, err,
                        2) && ok;
    add_sum(sums - 1);
  };
  if (K < GEMM_TC_CHUNK_K) product(std::integral_constant<int, 1>{});
  else product(std::integral_constant<int, BK / 16>{});
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  ok = __syncthreads_and(ok);
  // 32 x 32 blocks of a warp's lane quarter, turned in shared memory so that a warp's global
  // accesses run along the rows
  float* st = reinterpret_cast<float*>(gbase) + warp * 32 * EPI_LD;
  const int rows = min(32, M - m0 - q * 32);
#pragma unroll
  for (int c = 0; c < CW; c += 32) {
    const int c0 = n0 + half * CW + c, col = c0 + lane;
    if (!ok || rows <= 0 || c0 >= N) break;
#pragma unroll
    for (int e = 0; e < 32; ++e) st[lane * EPI_LD + e] = acc[c + e];
    __syncwarp();
    if (col < N) {
      const int64_t row0 = m0 + q * 32;
      const int64_t o0 = row0 * d.scm + (int64_t)col * d.scn;
      if (d.epi == EPI_STORE) {
        float* out = (float*)d.C + o0;
#pragma unroll 8
        for (int i = 0; i < rows; ++i) out[i * d.scm] = st[i * EPI_LD + lane];
      } else if (d.epi == EPI_BIAS_ACT) {
        bf16* out = (bf16*)d.C + o0;
        const float b = bias ? bias[col] : 0.f;
#pragma unroll 4
        for (int i = 0; i < rows; ++i)
          out[i * d.scm] = __float2bfloat16(act_fwd(d.act, st[i * EPI_LD + lane] + b, slope));
      } else {
        bf16* out = (bf16*)d.C + o0;
        const bf16* aux = (const bf16*)d.aux + row0 * d.sxm + (int64_t)col * d.sxn;
        for (int i0 = 0; i0 < rows; i0 += 8) {
          float a[8];
#pragma unroll
          for (int i = 0; i < 8; ++i)
            a[i] = i0 + i < rows ? __bfloat162float(aux[(i0 + i) * d.sxm]) : 0.f;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (i0 + i < rows)
              out[(i0 + i) * d.scm] = __float2bfloat16(st[(i0 + i) * EPI_LD + lane] *
                                                       act_bwd(d.act, a[i], slope));
        }
      }
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "n"(2 * BN));
}

template <int BN>
cudaError_t launch_bn(const GemmDesc* descs, const int2* tiles, int n, float slope, int* err,
                      cudaStream_t st) {
  static_assert(8 * 32 * EPI_LD * 4 <= STAGES * (BM + BN) * BK * 2, "epilogue staging");
  const cudaError_t e = cudaFuncSetAttribute(
      k_gemm_tc<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_tc_smem(BN));
  if (e != cudaSuccess) return e;
  return launch_pdl(k_gemm_tc<BN>, dim3(n), dim3(NT), gemm_tc_smem(BN), st, descs, tiles, slope,
                    err);
}

}  // namespace

// Alignment class of an operand's unit-stride rows for GemmDesc::vec: log2 of the bytes (up to 16)
// that divide every row's start, less one.
static int align_class(const void* p, int64_t stride, int64_t wstride) {
  const uint64_t bits = (uint64_t)(uintptr_t)p | (uint64_t)stride * 2 | (uint64_t)wstride * 2 | 16;
  int c = 0;
  while (c < 3 && !(bits >> (c + 1) & 1)) ++c;
  return c;
}

void gemm_tc_align(GemmDesc* d) {
  const int a = align_class(d->A, d->sak == 1 ? d->sam : d->sak,
                            d->wsel && d->wsel_op == 1 ? d->wsel_stride : 0);
  const int b = align_class(d->B, d->sbk == 1 ? d->sbn : d->sbk,
                            d->wsel && d->wsel_op == 2 ? d->wsel_stride : 0);
  d->vec = a | b << 2;
}

void launch_gemm_tc(const GemmDesc* descs, const int2* tiles, int n, int shape, float slope,
                    int* err, cudaStream_t st) {
  if (n <= 0) return;
  if (shape == 0) launch_bn<128>(descs, tiles, n, slope, err, st);
  else launch_bn<64>(descs, tiles, n, slope, err, st);
}

}  // namespace lipz
