// Tensor-core backward of the training step (Section 3, step 3: the gradient update of every
// cell's selected generator and discriminator), bf16 operands and fp32 accumulation in TMEM.
//
// One persistent grouped-GEMM kernel runs every product of the backward of every cell: 128 x BN
// output tiles of C = A * B over K, A read by TMA K-major (rows of K) or MN-major (K in the outer
// dimension; used for the transposed products dW = delta^T X), B always MN-major, so no transposed
// copy is ever written. The z coordinate of a weight operand is the cell's selected individual.
// Epilogues: bf16 delta times the activation derivative of the stored forward output; Adam on the
// spot for a weight gradient (it never leaves the accumulator), or its fp32 store. What an
// epilogue reads besides the accumulator (the old weights and moments, the forward output)
// streams through shared memory in chunks that one warp loads and another stores by TMA.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstring>
#include <vector>

#include "bwd_tc.h"
#include "common.cuh"
#include "tc_ptx.cuh"

namespace lipz {
namespace tcb {

using namespace lipz::tc;

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int A_BYTES = BM * BK * 2;        // 16 KB
constexpr int MN_BOX_BYTES = 64 * BK * 2;   // one {64 MN, 64 K} box
constexpr int NUM_EPI_WARPS = 8;
constexpr int EPI_THREADS = 32 * NUM_EPI_WARPS;
// Chunk stream. A chunk is 64 rows (one half of a tile) of what the epilogue reads besides the
// accumulator, updated in place in shared memory; chunks alternate between the two row halves, so
// each half of the epilogue works through its own two of the four buffers (an even number: a half
// that met the other's buffers could run a phase ahead of their barriers).
//   Adam: 32 fp32 columns of each of w, m, v (one 128-byte row each, 128-byte swizzle), plus the
//   new bf16 copy (64-byte rows, no swizzle). w, m and v lie a fixed distance apart in memory, so
//   that one TMA box {32, 64, 1, 3} of a 4-D map moves the chunk's three arrays: a tiled TMA
//   operation holds its issuing thread for about 0.2 us whatever its size up to 16 KB, so one box
//   per array made the issuing thread, not the bytes, bound the stream.
//   Delta: up to 128 bf16 columns of the stored forward output in boxes {64, 64} (128-byte rows,
//   128-byte swizzle), replaced by the deltas.
constexpr int CHUNK_ROWS = 64;
constexpr int ADAM_COLS = 32;
constexpr int ADAM_ARRAY_BYTES = CHUNK_ROWS * ADAM_COLS * 4;           // 8 KB
constexpr int ADAM_WB_BYTES = CHUNK_ROWS * ADAM_COLS * 2;              // 4 KB
constexpr int DELTA_COLS = 128;
constexpr int DELTA_BOX_BYTES = CHUNK_ROWS * 64 * 2;                   // 8 KB
constexpr int CHUNK_BYTES = 3 * ADAM_ARRAY_BYTES + ADAM_WB_BYTES;      // 28 KB
// barriers, the ring of claimed tiles and the TMEM slot
constexpr int MISC_BYTES = 512;
// Claimed tiles a CTA holds: the one in its epilogue and the next, whose operands load meanwhile.
// (Four: the tiles claimed early by busy CTAs lengthen the tail, 1 % at 12x12.)
constexpr int RING = 2;
constexpr int CHUNK_BUFS = 4;
// Operand ring: 96 KB in stages of 16 KB of A and BN x 128 bytes of B, BN the grid's tile width
// (128: three stages, 64: four).
constexpr int RING_BYTES = 3 * (A_BYTES + 128 * BK * 2);
constexpr int MAX_OPS = 4;
constexpr int SMEM = 1024 + RING_BYTES + CHUNK_BUFS * CHUNK_BYTES + MISC_BYTES;
static_assert(SMEM <= 232448, "backward: shared memory");
// producer, MMA issuer, epilogue, chunk loader, chunk storer
constexpr int THREADS = 64 + EPI_THREADS + 64;

enum { EPI_F32 = 0, EPI_DACT = 1, EPI_ADAM = 2 };  // fp32 store; deltas; Adam step

// Adam of one weight tensor fused into the tile that computes its gradient (Section 3, step 3:
// the selected individual of the cell takes one Adam step and becomes the cell's new centre).
// The old snapshot is read and the new one written through the stage's tensor maps.
struct AdamRef {
  const int* src;                  // individual each cell trains
  const float4* coef;              // per cell: lr, 1 / (1 - beta1^t), 1 / (1 - beta2^t), t
  float beta1, beta2, eps;
};

struct GParams {
  int M, N, K, BN;
  int mtiles, ntiles, kchunks;
  int a_mn;             // A's layout: 1 = MN-major (B always is)
  int a_row0;           // first row of a K-major A
  const int* a_sel;     // z coordinate of A: a_sel[cell] (weights of the selected individual)
  const int* b_sel;     //   or the cell itself when null
  int epi, act;
  float slope;
  float* C;             // EPI_F32: C[cell * c_cell + m * N + n]
  int64_t c_cell;
  // EPI_DACT: the stored forward output of row m is row x_row0 + m of the stage's aux map; with
  // x_slot (non-null) a 4-D map {n, rows, slots, cells}, slot 1 + x_slot[cell]
  int x_row0;
  const int* x_slot;
  // split K (ksplit > 0): chunks [0, ksplit) read K rows kc * 64 of A's part 0 and of B's slot 0;
  // chunks [ksplit, kchunks) read K rows (kc - ksplit) * 64 of A's part 1 and of B's slot
  // 1 + b_slot_sel[cell]. Both maps are 4-D, {m or n, K rows, parts or slots, cells}, so that rows
  // past a part read as zero in both (A's next part belongs to a stage that may still be writing)
  int ksplit;
  const int* b_slot_sel;
  // EPI_DACT: column sums of the fp32 deltas over the 32 rows q of row tile i go to
  // bias_part[cell * bias_cell + (4 i + q) * N + n] (together a bias gradient); null = none
  float* bias_part;
  int64_t bias_cell;
  AdamRef adam;
};

// ---------------------------------------------------------------------------------------------
// The backward of every cell as one list of tiles. A cell's ten products are stages; a stage's
// tiles are entries of a list that orders the whole grid's work so that every tile comes after
// the tiles it reads: level by level along the chain, cell by cell within a level, so that the
// tiles a tile reads lie a whole level (every cell's Adam tiles of that level among it) earlier.
// Persistent CTAs claim entries in list order from a counter in global memory: each runs what it
// claimed in that order, so the oldest unfinished tile never waits for a tile that nobody runs,
// however few CTAs are resident. A delta tile that others read is counted in global memory once
// its stores are written; the producer of a tile that reads it acquires the count before its loads.
//
// Bound: HBM on large grids (26 B per parameter through the chunk stream; 2.32 GB in all at 12x12,
// B = 100: 373 us, 0.92 of the measured copy rate), the chain of five dependent tiles
// on small ones (about 7 us each). One CTA per cell walking its own tiles took 422 us at 12x12
// (its delta tiles stopped its stream), and left most SMs idle on small grids: 307 us at 1x1
// (now 38), 421 at 5x5, B = 256 (99). Cells 4 to 40 apart per level instead of all of them (a
// smaller window of activations) were slower: 400 to 535 us at 12x12.
// ---------------------------------------------------------------------------------------------
constexpr int MAX_STAGES = 10;
constexpr int RANGES_STAGE = MAX_STAGES;  // + 0, 1: list entries of G's and D's ranges of a cell
constexpr int SYNC_WORDS = TCB_SYNC_WORDS;  // counters per cell in TcbBuffers::sync

struct Stage {
  GParams p;
  int dep;       // stage whose output this one reads (-1: none)
  int dep_need;  // tiles of that stage per cell
};

// A cell's ranges entry of one population: the gradients of its biases from their partial sums,
// then the Adam step of the ranges (biases, D's output layer), or the gradients stored.
constexpr int MAX_RANGES = 4;
constexpr int RANGE_REPS = 6;  // elements per epilogue thread and pass
struct RangeTask {
  AdamRanges r;
  float* grad;                     // gradient vectors (r.grad), written without fused Adam
  const float* part[MAX_RANGES];   // first cell's partials [4 tiles][len]; null: r.grad holds it
  int tiles[MAX_RANGES];           // row tiles of the partials
  int64_t part_cell;
  int total;                       // elements of all ranges
  int n_dep, dep[MAX_RANGES], need[MAX_RANGES];  // stages that write the partials
};

struct CellPlan {
  Stage st[MAX_STAGES];
  const int2* list;  // {cell, stage << 16 | tile}
  int n_list;
  int n_ops, op_bytes;  // operand ring: stages and bytes per stage
  // [SYNC_WORDS] per cell: finished tiles by stage; after the last cell's, the claim counter
  int* sync;
  int cells;
  int* err;
  RangeTask rt[2];  // G, D
  int adam;         // the weight matrices' tiles and the ranges take their Adam step
  float beta1, beta2, eps;
};

struct StageMaps {
  CUtensorMap a[MAX_STAGES];
  CUtensorMap b[MAX_STAGES];
  // EPI_ADAM: old w, m, v {in, out, individual, array}, new w, m, v {in, out, cell, array}, new
  // bf16 copy; EPI_DACT: the stored forward output, the deltas (clipped to the stage's rows)
  CUtensorMap in[MAX_STAGES];
  CUtensorMap out[MAX_STAGES];
  CUtensorMap nb[MAX_STAGES];
};

__device__ __forceinline__ void stage_tile(const GParams& p, int t, int& m0, int& n0, int& n) {
  m0 = (t / p.ntiles) * BM;
  n0 = (t % p.ntiles) * p.BN;
  n = min(p.BN, p.N - n0);
  n = (n + 63) & ~63;  // B is MN-major: boxes of 64 columns
}

// Weight-gradient tile kept for the caller: fp32 store, a row per thread.
__device__ __forceinline__ void store_tile(const GParams& p, int cell, int m0, int n0, int n,
                                           uint32_t tbase, int hf, int row) {
  const int m = m0 + row, ng = n / 16, half = (ng + 1) / 2;
  float* C = p.C + (int64_t)cell * p.c_cell + (int64_t)m * p.N + n0;
  for (int g = hf ? half : 0; g < (hf ? ng : half); ++g) {
    uint32_t r[16];
    LIPZ_TMEM_LD16(tbase + g * 16, r);
    tmem_wait_ld();
    if (m >= p.M) continue;
    // (the tensors' rows are multiples of 16 columns: a group lies inside or outside)
    if (n0 + g * 16 >= p.N) continue;
    float4* o = reinterpret_cast<float4*>(C + g * 16);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      o[u] = make_float4(__uint_as_float(r[4 * u]), __uint_as_float(r[4 * u + 1]),
                         __uint_as_float(r[4 * u + 2]), __uint_as_float(r[4 * u + 3]));
  }
}

// Sum of v over the 32 lanes of a warp for 16 columns, reduce-scattered: lanes 2j and 2j + 1
// return the sum of column j. Each partial sum is formed by one lane, in a fixed order.
__device__ __forceinline__ float warp_colsum16(const float (&v)[16], int lane) {
  float a8[8], a4[4], a2[2];
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    a8[i] = (b4 ? v[8 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, b4 ? v[i] : v[8 + i], 16);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    a4[i] = (b3 ? a8[4 + i] : a8[i]) + __shfl_xor_sync(0xffffffffu, b3 ? a8[i] : a8[4 + i], 8);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    a2[i] = (b2 ? a4[2 + i] : a4[i]) + __shfl_xor_sync(0xffffffffu, b2 ? a4[i] : a4[2 + i], 4);
  const float a1 = (b1 ? a2[1] : a2[0]) + __shfl_xor_sync(0xffffffffu, b1 ? a2[0] : a2[1], 2);
  return a1 + __shfl_xor_sync(0xffffffffu, a1, 1);
}

// Delta epilogue of one tile: warp (q, hf) owns TMEM lane quarter q (rows 32q .. 32q + 31) and
// column half hf of each chunk. A chunk's stored forward outputs wait in its buffer (chunk number
// cj of a row half, as in adam_tile) as boxes of 64 columns, 16-byte unit u of box row r at unit
// u ^ (r & 7); the bf16 deltas go back to the same places and the storer warp writes the boxes
// out. With a bias output, the column sums of the warp's 32 rows of fp32 deltas go to global
// memory as partials (before the chunk's arrival, so that the storer's count of the tile covers
// them). Through per-thread global loads and stores (a row per lane) a 128 x 256 tile took 7 us.
__device__ __forceinline__ bool delta_tile(const GParams& p, int cell, int m0, int n0, int n,
                                           uint32_t tbase, int hf, int row, int q, int lane,
                                           uint32_t sChunk, uint32_t cFull, uint32_t cDone, int& cj,
                                           volatile int* abort_flag, int* err) {
  const bool row_ok = m0 + row < p.M;
  const bool is_tanh = p.act == ACT_TANH;
  const float dlo = p.act == ACT_RELU ? 0.f : p.slope;
  const int h = row / CHUNK_ROWS, rr = row % CHUNK_ROWS;
  float* bp = p.bias_part ? p.bias_part + (int64_t)cell * p.bias_cell +
                                (int64_t)(m0 / BM * 4 + q) * p.N + n0
                          : nullptr;
  for (int c0 = 0; c0 < n; c0 += DELTA_COLS, ++cj) {
    const int bi = (2 * cj + h) % CHUNK_BUFS, use = (2 * cj + h) / CHUNK_BUFS;
    const int cw = min(DELTA_COLS, n - c0) / 2;  // 64 or 32 columns of this thread
    if (!mbar_wait_warp(cFull + 8 * bi, (uint32_t)(use & 1), abort_flag, err, 18))
      return false;
    const uint32_t rb = sChunk + (uint32_t)(bi * CHUNK_BYTES) + (uint32_t)rr * 128u;
#pragma unroll 1
    for (int g = 0; g < cw; g += 32) {
      const int cl = hf * cw + g;  // first column, within the chunk
      // the TMEM load is warp-collective: every lane takes part, live row or not
      uint32_t r[32];
      LIPZ_TMEM_LD32(tbase + c0 + cl, r);
      const uint32_t bx = rb + (uint32_t)((cl >> 6) * DELTA_BOX_BYTES);
      const uint32_t u0 = (uint32_t)(cl & 63) >> 3;
      uint32_t x[16];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(x[4 * u]), "=r"(x[4 * u + 1]), "=r"(x[4 * u + 2]), "=r"(x[4 * u + 3])
                     : "r"(bx + (((u0 + u) ^ (uint32_t)(rr & 7)) << 4))
                     : "memory");
      tmem_wait_ld();
      float v[32];
#pragma unroll
      for (int e = 0; e < 32; e += 2) {
        const __nv_bfloat162 y2 = *reinterpret_cast<const __nv_bfloat162*>(&x[e >> 1]);
        const float y0 = __low2float(y2), y1 = __high2float(y2);
        const float d0 = is_tanh ? 1.f - y0 * y0 : (y0 > 0.f ? 1.f : dlo);
        const float d1 = is_tanh ? 1.f - y1 * y1 : (y1 > 0.f ? 1.f : dlo);
        v[e] = __uint_as_float(r[e]) * d0;
        v[e + 1] = __uint_as_float(r[e + 1]) * d1;
        x[e >> 1] = pack_bf16(v[e], v[e + 1]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                         bx + (((u0 + u) ^ (uint32_t)(rr & 7)) << 4)),
                     "r"(x[4 * u]), "r"(x[4 * u + 1]), "r"(x[4 * u + 2]), "r"(x[4 * u + 3])
                     : "memory");
      if (bp) {
        // rows past the stage's M are not counted
        const float(&va)[16] = *reinterpret_cast<const float(*)[16]>(&v[0]);
        const float(&vb)[16] = *reinterpret_cast<const float(*)[16]>(&v[16]);
        if (!row_ok) {
#pragma unroll
          for (int e = 0; e < 32; ++e) v[e] = 0.f;
        }
        const float s0 = warp_colsum16(va, lane), s1 = warp_colsum16(vb, lane);
        // (even lanes hold the first 16 columns' sums, odd lanes store the others')
        const int col = c0 + cl + (lane >> 1) + (lane & 1) * 16;
        if (n0 + col < p.N) bp[col] = lane & 1 ? s1 : s0;
      }
    }
    // make the deltas visible to the TMA store, then hand the chunk to the storer warp
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive(cDone + 8 * bi);
  }
  return true;
}

// Adam epilogue of one weight-gradient tile: for each 32-column chunk of the thread's row half
// h, the warp's 16 columns of its row. Chunk number cj of a half, the CTA's chunk 2 cj + h, sits
// in buffer (2 cj + h) mod CHUNK_BUFS as three 64 x 128-byte boxes of old w, m, v in the 128-byte swizzle
// (16-byte unit u of box row r at unit u ^ (r & 7)); the new values go back to the same places,
// the bf16 copy to the buffer's 64-byte-row box, and the storer warp stores the four boxes once
// the half's 128 threads have arrived on cDone. Returns false on a timeout.
__device__ __forceinline__ bool adam_tile(const GParams& p, int cell, int m0, int n0,
                                          uint32_t tbase, int hf, int row, uint32_t sChunk,
                                          uint32_t cFull, uint32_t cDone, int& cj,
                                          volatile int* abort_flag, int* err) {
  const AdamRef& a = p.adam;
  const float4 cf = __ldg(&a.coef[cell]);
  const bool row_ok = m0 + row < p.M;
  const int h = row / CHUNK_ROWS, rr = row % CHUNK_ROWS;
  const int nch = (min(p.BN, p.N - n0) + ADAM_COLS - 1) / ADAM_COLS;
  for (int k = 0; k < nch; ++k, ++cj) {
    const int bi = (2 * cj + h) % CHUNK_BUFS, use = (2 * cj + h) / CHUNK_BUFS;
    if (!mbar_wait_warp(cFull + 8 * bi, (uint32_t)(use & 1), abort_flag, err, 18))
      return false;
    const int cl = k * ADAM_COLS + 16 * hf;  // first column of this thread, within the tile
    const uint32_t bb = sChunk + (uint32_t)(bi * CHUNK_BYTES);
    const uint32_t rb = bb + (uint32_t)rr * 128u;
    // the TMEM load is warp-collective: every lane takes part, live row or not
    uint32_t r[16];
    LIPZ_TMEM_LD16(tbase + cl, r);
    tmem_wait_ld();
    if (row_ok && n0 + cl < p.N) {
      float w[16], mm[16], v[16];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t off = (uint32_t)(((4 * hf + u) ^ (rr & 7)) << 4);
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(w[4 * u]), "=f"(w[4 * u + 1]), "=f"(w[4 * u + 2]), "=f"(w[4 * u + 3])
                     : "r"(rb + off)
                     : "memory");
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(mm[4 * u]), "=f"(mm[4 * u + 1]), "=f"(mm[4 * u + 2]),
                       "=f"(mm[4 * u + 3])
                     : "r"(rb + ADAM_ARRAY_BYTES + off)
                     : "memory");
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[4 * u]), "=f"(v[4 * u + 1]), "=f"(v[4 * u + 2]), "=f"(v[4 * u + 3])
                     : "r"(rb + 2 * ADAM_ARRAY_BYTES + off)
                     : "memory");
      }
#pragma unroll
      for (int e = 0; e < 16; ++e)
        adam_elem(w[e], mm[e], v[e], __uint_as_float(r[e]), a.beta1, a.beta2, cf.x, cf.y, cf.z,
                  a.eps);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t off = (uint32_t)(((4 * hf + u) ^ (rr & 7)) << 4);
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(rb + off), "f"(w[4 * u]),
                     "f"(w[4 * u + 1]), "f"(w[4 * u + 2]), "f"(w[4 * u + 3])
                     : "memory");
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(rb + ADAM_ARRAY_BYTES + off),
                     "f"(mm[4 * u]), "f"(mm[4 * u + 1]), "f"(mm[4 * u + 2]), "f"(mm[4 * u + 3])
                     : "memory");
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(rb + 2 * ADAM_ARRAY_BYTES +
                                                                      off),
                     "f"(v[4 * u]), "f"(v[4 * u + 1]), "f"(v[4 * u + 2]), "f"(v[4 * u + 3])
                     : "memory");
      }
      const uint32_t wbr = bb + 3 * ADAM_ARRAY_BYTES + (uint32_t)rr * 64u + (uint32_t)hf * 32u;
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(wbr),
                   "r"(pack_bf16(w[0], w[1])), "r"(pack_bf16(w[2], w[3])),
                   "r"(pack_bf16(w[4], w[5])), "r"(pack_bf16(w[6], w[7]))
                   : "memory");
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(wbr + 16),
                   "r"(pack_bf16(w[8], w[9])), "r"(pack_bf16(w[10], w[11])),
                   "r"(pack_bf16(w[12], w[13])), "r"(pack_bf16(w[14], w[15]))
                   : "memory");
    }
    // make the new values visible to the TMA store, then hand the chunk to the storer warp
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive(cDone + 8 * bi);
  }
  return true;
}

// Bounded wait until *cnt (counted by other CTAs) reaches `need`.
__device__ __forceinline__ bool count_wait(const int* cnt, int need, volatile int* abort_flag,
                                           int* err, int code) {
  const unsigned long long t0 = globaltimer();
  for (uint32_t it = 1;; ++it) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
    if (v >= need) return true;
    if ((it & 63u) == 0) {
      if (*abort_flag) return false;
      if (globaltimer() - t0 > WAIT_NS) {
        *abort_flag = 1;
        atomicExch(err, code);
        return false;
      }
    }
  }
}

// Form for warps whose lanes all poll and go on together.
__device__ __forceinline__ bool count_wait_warp(const int* cnt, int need, volatile int* abort_flag,
                                                int* err, int code) {
  return __all_sync(0xffffffffu, count_wait(cnt, need, abort_flag, err, code));
}

// A cell's ranges entry: epilogue thread et takes elements et, et + 256, ... of the population's
// ranges laid end to end. A pass's loads are issued before any is used (one memory latency per
// row tile of partials; element by element, an entry took 14 us). A bias gradient is the sum of
// its partials: the four lane quarters of a row tile in order, then the row tiles in order.
__device__ __forceinline__ bool ranges_entry(const CellPlan& cp, const RangeTask& t, int cell,
                                             int et, int lane, volatile int* abort_flag) {
  int good = 1;
  if (lane < t.n_dep)
    good = count_wait(cp.sync + (int64_t)cell * SYNC_WORDS + t.dep[lane], t.need[lane], abort_flag,
                      cp.err, 24);
  if (!__all_sync(0xffffffffu, good)) return false;
  __syncwarp();
  const AdamRanges& r = t.r;
  const int src = __ldg(&r.src[cell]);
  const float4 cf = __ldg(&r.coef[cell]);
  if (cp.adam && et == 0) {
    r.new_p.step[cell] = (int)cf.w;
    r.new_p.lr[cell] = cf.x;
  }
  const int64_t so = (int64_t)src * r.Ps, co = (int64_t)cell * r.Ps;
  for (int j0 = et; j0 < t.total; j0 += RANGE_REPS * EPI_THREADS) {
    int64_t k[RANGE_REPS];          // the element's place in the parameter vector
    const float* part[RANGE_REPS];  // its partials' column, null: none
    int len[RANGE_REPS], tiles[RANGE_REPS], most = 0;
    float w[RANGE_REPS], m[RANGE_REPS], v[RANGE_REPS], g[RANGE_REPS];
#pragma unroll
    for (int u = 0; u < RANGE_REPS; ++u) {
      int j = j0 + u * EPI_THREADS;
      k[u] = -1;
      part[u] = nullptr;
      tiles[u] = len[u] = 0;
      w[u] = m[u] = v[u] = g[u] = 0.f;
      if (j >= t.total) continue;
      int q = 0;
      while (j >= r.len[q]) j -= r.len[q++];
      k[u] = r.off[q] + j;
      len[u] = r.len[q];
      if (t.part[q]) {
        part[u] = t.part[q] + cell * t.part_cell + j;
        tiles[u] = t.tiles[q];
        most = max(most, tiles[u]);
      } else if (cp.adam) {
        g[u] = t.grad[co + k[u]];
      }
      if (cp.adam) {
        w[u] = r.old_p.w[so + k[u]];
        m[u] = r.old_p.m[so + k[u]];
        v[u] = r.old_p.v[so + k[u]];
      }
    }
    for (int i = 0; i < most; ++i) {
      float a[RANGE_REPS][4];
#pragma unroll
      for (int u = 0; u < RANGE_REPS; ++u)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          a[u][q] = i < tiles[u] ? __ldcg(part[u] + (int64_t)(4 * i + q) * len[u]) : 0.f;
#pragma unroll
      for (int u = 0; u < RANGE_REPS; ++u) {
        const float s = ((a[u][0] + a[u][1]) + a[u][2]) + a[u][3];
        if (i < tiles[u]) g[u] = i ? g[u] + s : s;
      }
    }
#pragma unroll
    for (int u = 0; u < RANGE_REPS; ++u) {
      if (k[u] < 0) continue;
      if (!cp.adam) {
        if (part[u]) t.grad[co + k[u]] = g[u];
        continue;
      }
      adam_elem(w[u], m[u], v[u], g[u], cp.beta1, cp.beta2, cf.x, cf.y, cf.z, cp.eps);
      r.new_p.w[co + k[u]] = w[u];
      r.new_p.m[co + k[u]] = m[u];
      r.new_p.v[co + k[u]] = v[u];
      if (r.new_p.wb) r.new_p.wb[co + k[u]] = __float2bfloat16_rn(w[u]);
    }
  }
  return true;
}

__global__ void __launch_bounds__(THREADS, 1)
    k_bwd(const __grid_constant__ StageMaps maps, const __grid_constant__ CellPlan cp) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t sChunk = base + RING_BYTES;
  uint8_t* misc = gbase + RING_BYTES + CHUNK_BUFS * CHUNK_BYTES;
  const uint32_t bFull = smem_u32(misc), bEmpty = bFull + 8 * MAX_OPS;
  const uint32_t bAcc = bEmpty + 8 * MAX_OPS, bReg = bAcc + 16, bFinal = bReg + 16;
  const uint32_t cFull = bFinal + 8;          // [CHUNK_BUFS] the chunk's old values landed
  const uint32_t cDone = cFull + 8 * CHUNK_BUFS;  // new values written by the epilogue half
  const uint32_t cFree = cDone + 8 * CHUNK_BUFS;  // the stores have read the buffer
  const uint32_t tFull = cFree + 8 * CHUNK_BUFS;  // [RING] a claimed tile is in the ring slot
  const uint32_t tEmpty = tFull + 8 * RING;  // [RING] every role has read the slot
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc + 384);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 388);
  volatile int2* ring = reinterpret_cast<volatile int2*>(misc + 400);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_OPS; ++s) {
      mbar_init(bFull + 8 * s, 1);
      mbar_init(bEmpty + 8 * s, 1);
    }
    for (int r = 0; r < 2; ++r) {
      mbar_init(bAcc + 8 * r, 1);
      mbar_init(bReg + 8 * r, EPI_THREADS);
    }
    mbar_init(bFinal, 1);
    for (int b = 0; b < CHUNK_BUFS; ++b) {
      mbar_init(cFull + 8 * b, 1);
      mbar_init(cDone + 8 * b, EPI_THREADS / 2);
      mbar_init(cFree + 8 * b, 1);
    }
    for (int b = 0; b < RING; ++b) {
      mbar_init(tFull + 8 * b, 1);
      // readers: one lane of the MMA warp, of each epilogue warp, of the chunk loader and storer
      mbar_init(tEmpty + 8 * b, 1 + NUM_EPI_WARPS + 2);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
        smem_u32((const void*)tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  int* err = cp.err;
  int* const claim = cp.sync + (int64_t)cp.cells * SYNC_WORDS;
  const int n_ops = cp.n_ops, op_bytes = cp.op_bytes;  // operand ring: stages, bytes of each
  // the set-up above touched no global memory: from here on the previous kernel's results
  // are needed (programmatic dependent launch)
  pdl_wait();

  // The next claimed tile for a role of a warp: waits for ring slot i, returns its entry
  // {cell, stage << 16 | tile} and releases the slot. False: the list is done or the CTA gave up.
  auto next_tile = [&](int i, int2& e) -> bool {
    const int s = i % RING;
    if (!mbar_wait_all(tFull + 8 * s, (uint32_t)((i / RING) & 1), abort_flag, err, 22)) return false;
    e.x = ring[s].x;
    e.y = ring[s].y;
    __syncwarp();
    if (lane == 0) mbar_arrive(tEmpty + 8 * s);
    return e.x >= 0;
  };

  if (warp == 0) {
    {
      const bool elected = elect_one();
      int issued[MAX_OPS] = {};
      bool ok = true;
      int stage = 0;
      uint32_t phase = 0;
      for (int i = 0; ok; ++i) {
        int idx = lane == 0 ? atomicAdd(claim, 1) : 0;
        idx = __shfl_sync(0xffffffffu, idx, 0);
        const int2 e = idx < cp.n_list ? __ldg(&cp.list[idx]) : make_int2(-1, 0);
        const int s = i % RING;
        if (i >= RING && !mbar_wait_all(tEmpty + 8 * s, (uint32_t)((i / RING - 1) & 1), abort_flag,
                                        err, 23)) {
          ok = false;
          break;
        }
        if (lane == 0) {
          ring[s].x = e.x;
          ring[s].y = e.y;
          mbar_arrive(tFull + 8 * s);
        }
        if (e.x < 0) break;
        const int cell = e.x, si = e.y >> 16, t = e.y & 0xFFFF;
        if (si >= RANGES_STAGE) continue;
        const GParams& p = cp.st[si].p;
        const int dep = cp.st[si].dep;
        const CUtensorMap* mA = &maps.a[si];
        const CUtensorMap* mB = &maps.b[si];
        const int za = p.a_sel ? __ldg(&p.a_sel[cell]) : cell;
        const int zb = p.b_sel ? __ldg(&p.b_sel[cell]) : cell;
        const int fake_slot = p.ksplit > 0 ? 1 + __ldg(&p.b_slot_sel[cell]) : 0;
        const uint32_t bytes = (uint32_t)(A_BYTES + p.BN * 128);
        int m0, n0, n;
        stage_tile(p, t, m0, n0, n);
        auto load_a = [&](int kc, int st) {
          const int ka = kc * BK;
          const uint32_t sA = base + st * op_bytes, full = bFull + 8 * st;
          if (!elected) {
          } else if (p.ksplit > 0) {
            const int part = kc >= p.ksplit, kp = ka - part * p.ksplit * BK;
            tma_load_4d(sA, mA, full, m0, kp, part, za);
            tma_load_4d(sA + MN_BOX_BYTES, mA, full, m0 + 64, kp, part, za);
          } else if (p.a_mn) {
            tma_load_3d(sA, mA, full, m0, ka, za);
            tma_load_3d(sA + MN_BOX_BYTES, mA, full, m0 + 64, ka, za);
          } else {
            tma_load_3d(sA, mA, full, ka, p.a_row0 + m0, za);
          }
        };
        auto load_b = [&](int kc, int st) {
          const uint32_t sB = base + st * op_bytes + A_BYTES, full = bFull + 8 * st;
          issued[st]++;
          if (!elected) return;
          mbar_expect_tx(full, bytes);
          if (p.ksplit > 0) {
            const bool part1 = kc >= p.ksplit;
            const int kb = (part1 ? kc - p.ksplit : kc) * BK, slot = part1 ? fake_slot : 0;
            for (int u = 0; u < p.BN / 64; ++u)
              tma_load_4d(sB + u * MN_BOX_BYTES, mB, full, n0 + 64 * u, kb, slot, cell);
          } else {
            for (int u = 0; u < p.BN / 64; ++u)
              tma_load_3d(sB + u * MN_BOX_BYTES, mB, full, n0 + 64 * u, kc * BK, zb);
          }
        };
        // a tile that reads the output of the cell's stage `dep` (its A, written by any CTA)
        // loads its first chunks' B, which does not depend on it, before it waits
        const int ahead = dep >= 0 ? min(p.kchunks, n_ops) : 0;
        const int stage0 = stage;
        for (int kc = 0; kc < p.kchunks && ok; ++kc) {
          if (kc == ahead && ahead > 0) {
            if (!count_wait_warp(cp.sync + (int64_t)cell * SYNC_WORDS + dep, cp.st[si].dep_need,
                                 abort_flag, err, 16)) {
              ok = false;
              break;
            }
            asm volatile("fence.proxy.async;" ::: "memory");
            for (int u = 0; u < ahead; ++u) load_a(u, (stage0 + u) % n_ops);
          }
          if (!mbar_wait_all(bEmpty + 8 * stage, phase ^ 1u, abort_flag, err, 11)) {
            ok = false;
            break;
          }
          load_b(kc, stage);
          if (kc >= ahead) load_a(kc, stage);
          if (++stage == n_ops) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (ok && ahead == p.kchunks) {
          if (!count_wait_warp(cp.sync + (int64_t)cell * SYNC_WORDS + dep, cp.st[si].dep_need,
                               abort_flag, err, 16)) {
            ok = false;
            break;
          }
          asm volatile("fence.proxy.async;" ::: "memory");
          for (int u = 0; u < ahead; ++u) load_a(u, (stage0 + u) % n_ops);
        }
      }
      if (!ok) {
        for (int s = 0; s < MAX_OPS; ++s)
          if (issued[s] > 0) {
            volatile int never = 0;
            mbar_wait(bFull + 8 * s, (uint32_t)((issued[s] - 1) & 1), &never, err, 11);
          }
      }
    }
  } else if (warp == 1) {
    {
      const bool elected = elect_one();
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int lt = 0;
      int2 e;
      for (int i = 0; ok && next_tile(i, e); ++i) {
        const int si = e.y >> 16;
        if (si >= RANGES_STAGE) continue;
        const GParams& p = cp.st[si].p;
        int m0, n0, n;
        stage_tile(p, e.y & 0xFFFF, m0, n0, n);
        const int R = lt & 1, use = lt >> 1;
        if (use > 0 && !mbar_wait_all(bReg + 8 * R, (uint32_t)((use - 1) & 1), abort_flag, err, 15)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(R * 256);
        const uint32_t idesc = idesc_bf16_major(BM, n, p.a_mn, 1);
        for (int kc = 0; kc < p.kchunks; ++kc) {
          if (!mbar_wait_all(bFull + 8 * stage, phase, abort_flag, err, 12)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sA = base + stage * op_bytes, sB = sA + A_BYTES;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t ad = p.a_mn ? sw128_mn_desc(sA + kk * 2048, MN_BOX_BYTES)
                                       : sw128_desc(sA + kk * 32);
            const uint64_t bd = sw128_mn_desc(sB + kk * 2048, MN_BOX_BYTES);
            if (elected) tc_mma(d, ad, bd, idesc, (kc | kk) != 0 ? 1u : 0u);
          }
          if (elected) tc_commit(bEmpty + 8 * stage);
          if (++stage == n_ops) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        if (elected) tc_commit(bAcc + 8 * R);
        ++lt;
      }
      if (elected) tc_commit(bFinal);
      volatile int never = 0;
      mbar_wait(bFinal, 0u, &never, err, 14);
    }
  } else if (warp >= 2 + NUM_EPI_WARPS) {
    // ===== chunk stream: the epilogue's inputs of every chunk of every EPI_ADAM and EPI_DACT
    // tile, in tile order, into the four buffers in turn, and its results back out. A tiled TMA
    // operation holds its issuing warp for a time (0.2 us in a loop of one lane; all lanes and an
    // elected issuer: 381 -> 373 us at 12x12), so two warps share the work:
    //   loader: a chunk's load, once the storer has released the chunk's buffer;
    //   storer: a chunk's stores once its epilogue half is done, then, when the stores have read
    //           the buffer, its release to the loader (releasing it one chunk later, to keep a
    //           store group in flight, was slower: the stream is bound by the latency of each
    //           buffer's round trip); after a delta tile's last chunk, once its stores are
    //           written, it counts the tile for the tiles that read it. =====
    const bool storer = warp == 3 + NUM_EPI_WARPS;
    {
      const bool elected = elect_one();
      int buf = 0, uses[CHUNK_BUFS] = {};
      bool ok = true;
      int2 e;
      for (int i = 0; ok && next_tile(i, e); ++i) {
        const int cell = e.x, si = e.y >> 16;
        if (si >= RANGES_STAGE) continue;
        const GParams& p = cp.st[si].p;
        if (p.epi == EPI_F32) continue;
        const bool adam = p.epi == EPI_ADAM;
        int m0, n0, n;
        stage_tile(p, e.y & 0xFFFF, m0, n0, n);
        const int cols = adam ? ADAM_COLS : DELTA_COLS;
        const int nch = ((adam ? min(p.BN, p.N - n0) : n) + cols - 1) / cols;
        const int zi = adam ? __ldg(&p.adam.src[cell]) : cell;
        const int slot = !adam && p.x_slot ? 1 + __ldg(&p.x_slot[cell]) : -1;
        for (int k = 0; k < 2 * nch; ++k) {
          const int x0 = n0 + (k >> 1) * cols, y0 = m0 + (k & 1) * CHUNK_ROWS;
          const int boxes = adam ? 1 : min(2, (n - (k >> 1) * cols) / 64);
          const uint32_t bb = sChunk + (uint32_t)(buf * CHUNK_BYTES);
          if (storer) {
            // the (uses[buf] + 1)-th chunk of this buffer is written back
            if (!mbar_wait_all(cDone + 8 * buf, (uint32_t)(uses[buf] & 1), abort_flag, err, 19)) {
              ok = false;
              break;
            }
            if (!elected) {
            } else if (adam) {
              tma_store_4d(&maps.out[si], bb, x0, y0, cell, 0);
              tma_store_3d(&maps.nb[si], bb + 3 * ADAM_ARRAY_BYTES, x0, y0, cell);
            } else {
              for (int u = 0; u < boxes; ++u)
                tma_store_3d(&maps.out[si], bb + u * DELTA_BOX_BYTES, x0 + 64 * u, y0, cell);
            }
            if (elected) {
              bulk_commit();
              bulk_wait_read<0>();  // the stores have read the buffer: it may be refilled
              mbar_arrive(cFree + 8 * buf);
            }
          } else {
            if (uses[buf] > 0 && !mbar_wait_all(cFree + 8 * buf, (uint32_t)((uses[buf] - 1) & 1),
                                            abort_flag, err, 21)) {
              ok = false;
              break;
            }
            const uint32_t full = cFull + 8 * buf;
            if (!elected) {
            } else if (adam) {
              mbar_expect_tx(full, (uint32_t)(3 * ADAM_ARRAY_BYTES));
              tma_load_4d(bb, &maps.in[si], full, x0, y0, zi, 0);
            } else {
              mbar_expect_tx(full, (uint32_t)(boxes * DELTA_BOX_BYTES));
              for (int u = 0; u < boxes; ++u) {
                const uint32_t d = bb + u * DELTA_BOX_BYTES;
                if (slot >= 0)
                  tma_load_4d(d, &maps.in[si], full, x0 + 64 * u, p.x_row0 + y0, slot, cell);
                else
                  tma_load_3d(d, &maps.in[si], full, x0 + 64 * u, p.x_row0 + y0, cell);
              }
            }
          }
          uses[buf]++;
          if (++buf == CHUNK_BUFS) buf = 0;
        }
        if (storer && !adam && ok && elected) {
          bulk_wait_all();
          __threadfence();
          asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(
                           cp.sync + (int64_t)cell * SYNC_WORDS + si)
                       : "memory");
        }
      }
      if (storer) {
        if (elected) bulk_wait_all();
      } else if (*abort_flag) {
        // loads issued here land on this CTA's barriers: wait for them before it leaves
        for (int b = 0; b < CHUNK_BUFS; ++b)
          if (uses[b] > 0) {
            volatile int never = 0;
            mbar_wait(cFull + 8 * b, (uint32_t)((uses[b] - 1) & 1), &never, err, 19);
          }
      }
    }
  } else {
    const int ew = warp - 2, q = warp & 3, hf = ew >> 2;
    const int row = q * 32 + lane;
    int lt = 0;
    int cj = 0;  // chunks of this thread's row half so far
    for (int i = 0;; ++i) {
      const int s = i % RING;
      if (!mbar_wait_warp(tFull + 8 * s, (uint32_t)((i / RING) & 1), abort_flag, err, 22)) break;
      __syncwarp();
      const int cell = ring[s].x, w = ring[s].y;
      __syncwarp();
      if (lane == 0) mbar_arrive(tEmpty + 8 * s);
      if (cell < 0) break;
      const int si = w >> 16;
      if (si >= RANGES_STAGE) {
        if (!ranges_entry(cp, cp.rt[si - RANGES_STAGE], cell, threadIdx.x - 64, lane, abort_flag))
          break;
        continue;
      }
      const GParams& p = cp.st[si].p;
      int m0, n0, n;
      stage_tile(p, w & 0xFFFF, m0, n0, n);
      const int R = lt & 1, use = lt >> 1;
      if (!mbar_wait_warp(bAcc + 8 * R, (uint32_t)(use & 1), abort_flag, err, 13)) break;
      tc_fence_after();
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(R * 256);
      if (p.epi == EPI_ADAM) {
        if (!adam_tile(p, cell, m0, n0, tbase, hf, row, sChunk, cFull, cDone, cj, abort_flag, err))
          break;
      } else if (p.epi == EPI_DACT) {
        if (!delta_tile(p, cell, m0, n0, n, tbase, hf, row, q, lane, sChunk, cFull, cDone, cj,
                        abort_flag, err))
          break;
      } else {
        store_tile(p, cell, m0, n0, n, tbase, hf, row);
      }
      tc_fence_before();
      mbar_arrive(bReg + 8 * R);
      ++lt;
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

}  // namespace tcb

// ---- host side -----------------------------------------------------------------------------
namespace {

PFN_cuTensorMapEncodeTiled_v12000 g_enc = nullptr;

bool encoder(std::string* msg) {
  if (g_enc) return true;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                   cudaEnableDefault, &q);
  if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) {
    cudaGetLastError();
    if (msg) *msg = "cuTensorMapEncodeTiled is unavailable";
    return false;
  }
  g_enc = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  return true;
}

// bf16 3-D map {inner, rows, depth}; box {64, box_rows, 1}, 128-byte swizzle.
bool map3(CUtensorMap* m, const void* base, uint64_t inner, uint64_t rows, uint64_t depth,
          uint64_t depth_elems, uint32_t box_rows, std::string* msg) {
  cuuint64_t dims[3] = {inner, rows, depth};
  cuuint64_t strides[2] = {inner * 2, depth_elems * 2};
  cuuint32_t box[3] = {64, box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = g_enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides,
                     box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (msg) *msg = "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")";
    return false;
  }
  return true;
}

// fp32 4-D map over one weight tensor [out][in] of w, m and v of every individual: {in, out,
// individuals, array}, the arrays `part` floats apart; box {32, 64, 1, 3} (the three arrays'
// 64 x 128-byte boxes one after another in shared memory), 128-byte swizzle.
bool map4f(CUtensorMap* m, const float* base, uint64_t inner, uint64_t rows, uint64_t depth,
           uint64_t depth_elems, uint64_t part, std::string* msg) {
  cuuint64_t dims[4] = {inner, rows, depth, 3};
  cuuint64_t strides[3] = {inner * 4, depth_elems * 4, part * 4};
  cuuint32_t box[4] = {(cuuint32_t)tcb::ADAM_COLS, (cuuint32_t)tcb::CHUNK_ROWS, 1, 3};
  cuuint32_t es[4] = {1, 1, 1, 1};
  CUresult r = g_enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(base), dims,
                     strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (msg) *msg = "cuTensorMapEncodeTiled (fp32, 4-D) failed (" + std::to_string((int)r) + ")";
    return false;
  }
  return true;
}

// bf16 3-D map over one tensor's bf16 copy of every cell: {in, out, cells}, box {32, 64, 1},
// no swizzle (64-byte rows).
bool map3b_rows(CUtensorMap* m, const bf16* base, uint64_t inner, uint64_t rows, uint64_t depth,
                uint64_t depth_elems, std::string* msg) {
  cuuint64_t dims[3] = {inner, rows, depth};
  cuuint64_t strides[2] = {inner * 2, depth_elems * 2};
  cuuint32_t box[3] = {(cuuint32_t)tcb::ADAM_COLS, (cuuint32_t)tcb::CHUNK_ROWS, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = g_enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(base), dims,
                     strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (msg) *msg = "cuTensorMapEncodeTiled (bf16 rows) failed (" + std::to_string((int)r) + ")";
    return false;
  }
  return true;
}

// bf16 4-D map {inner, rows, slots, depth} (E seen as [cells][6][B][x], the D-loss rows of D1 as
// [cells][2][B][h]); box {64, 64, 1, 1},
// 128-byte swizzle: rows past `rows` within a slot read as zero.
bool map4(CUtensorMap* m, const void* base, uint64_t inner, uint64_t rows, uint64_t slots,
          uint64_t depth, uint64_t slot_elems, uint64_t depth_elems, std::string* msg) {
  cuuint64_t dims[4] = {inner, rows, slots, depth};
  cuuint64_t strides[3] = {inner * 2, slot_elems * 2, depth_elems * 2};
  cuuint32_t box[4] = {64, 64, 1, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  CUresult r = g_enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims,
                     strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (msg) *msg = "cuTensorMapEncodeTiled (4-D) failed (" + std::to_string((int)r) + ")";
    return false;
  }
  return true;
}

}  // namespace

struct TcbPlan {
  int* err;
  int2* list;     // the grid's tiles in claim order
  float* bpart;   // bias-gradient partial sums per cell, stage and row tile
  tcb::StageMaps maps;
  tcb::CellPlan cells;
  int grid;
};

namespace {
void free_plan(TcbPlan* P) {
  if (P->err) cudaFree(P->err);
  if (P->list) cudaFree(P->list);
  if (P->bpart) cudaFree(P->bpart);
  delete P;
}

// Stages: the chain D1 (rows of G's loss, then of D's) -> A3 -> A2 -> A1, then the weight
// gradients. S_DEP: the stage whose output a stage reads; S_LEVEL: its place along the chain.
enum { S_D1G = 0, S_D1D, S_A3, S_A2, S_A1, S_DW2D, S_DW1D, S_DW3G, S_DW2G, S_DW1G };
constexpr int S_DEP[tcb::MAX_STAGES] = {-1, -1, S_D1G, S_A3, S_A2, -1, S_D1D, S_A3, S_A2, S_A1};
constexpr int S_LEVEL[tcb::MAX_STAGES + 2] = {0, 0, 1, 2, 3, 0, 1, 2, 3, 4, 4, 1};  // + ranges

// The grid's tiles in claim order (CellPlan::list): by level, then by cell; a cell's chain tiles
// first. `tiles`: tiles per cell of each stage.
std::vector<int2> tile_list(int cells, const int* tiles) {
  static const int order[] = {S_A1, S_A2, S_A3, S_D1G, S_D1D, S_DW1G, S_DW2G, S_DW3G, S_DW1D,
                              S_DW2D, tcb::RANGES_STAGE, tcb::RANGES_STAGE + 1};
  std::vector<int2> out;
  for (int level = 0; level < 5; ++level)
    for (int c = 0; c < cells; ++c)
      for (int k : order) {
        if (S_LEVEL[k] != level) continue;
        const int n = k >= tcb::RANGES_STAGE ? 1 : tiles[k];
        for (int t = 0; t < n; ++t) out.push_back(int2{c, k << 16 | t});
      }
  return out;
}
}  // namespace

bool tcb_supported(int z, int h, int x, int B) {
  return h == 256 && z == 64 && x % 16 == 0 && x >= 64 && B >= 1 && B <= 256;
}

TcbPlan* tcb_plan_create(const TcbShape& s, const TcbBuffers& b, std::string* msg) {
  if (!tcb_supported(s.z, s.h, s.x, s.B)) {
    if (msg) *msg = "shape not supported by the tensor-core backward";
    return nullptr;
  }
  if (!encoder(msg)) return nullptr;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  TcbPlan* P = new TcbPlan();
  memset(P, 0, sizeof *P);
  if (cudaMalloc(&P->err, 4) != cudaSuccess || cudaMemset(P->err, 0, 4) != cudaSuccess) {
    cudaGetLastError();
    if (msg) *msg = "cudaMalloc for the error flag failed";
    free_plan(P);
    return nullptr;
  }
  const int C = s.cells, B = s.B, h = s.h, x = s.x, z = s.z;
  const uint64_t NI = s.n_indiv;
  const bf16* Gw = b.Gwb;
  const bf16* Dw = b.Dwb;
  // Tiles of 128 columns: their operands leave three ring stages (256: two, and coarser tiles at
  // the end of the list; 1 % slower at 12x12, 6 % at 5x5). Where a cell's 42 or
  // so weight tiles of 128 columns would leave SMs idle, 64 (10 % faster at 1x1; 17 %
  // slower at 12x12, four loads of A's 128 rows where 128 columns need two).
  const int bn = C * ((h / 128) * (2 * (h / 128) + (x + 127) / 128 + 1) + (x + 127) / 128 * 2) < sms
                     ? 64
                     : 128;
  bool ok = true;
  // bias-gradient partials [4 x row tiles][column] of D1's D-loss rows and of A3, A2, A1
  const int mt2 = (2 * B + 127) / 128, mt = (B + 127) / 128;
  const int64_t bp_cell = 4 * ((int64_t)mt2 * h + (int64_t)mt * (x + 2 * h));
  if (cudaMalloc(&P->bpart, (size_t)C * bp_cell * 4) != cudaSuccess) {
    cudaGetLastError();
    if (msg) *msg = "cudaMalloc for the bias partial sums failed";
    free_plan(P);
    return nullptr;
  }
  int64_t bp_off = 0;
  P->cells.adam = b.fuse_adam;
  P->cells.beta1 = b.beta1;
  P->cells.beta2 = b.beta2;
  P->cells.eps = b.eps;
  for (int pop = 0; pop < 2; ++pop) {
    tcb::RangeTask& t = P->cells.rt[pop];
    t.r = b.ranges[pop];
    t.grad = pop ? b.gD : b.gG;
    t.part_cell = bp_cell;
    for (int q = 0; q < t.r.n; ++q) t.total += t.r.len[q];
  }
  // C = A * B^T: M rows, N columns in tiles of BN, over K
  auto stage = [&](int si, int M, int N, int K, int BN) -> tcb::GParams& {
    tcb::GParams& q = P->cells.st[si].p;
    q.M = M;
    q.N = N;
    q.K = K;
    q.BN = BN;
    q.mtiles = (M + 127) / 128;
    q.ntiles = (N + BN - 1) / BN;
    q.kchunks = (K + 63) / 64;
    q.slope = s.slope;
    return q;
  };
  // delta product: A's rows from a_row0 of `amap` {k, rows}, B the selected individual's weight
  // tensor [k][n]; times act' of the stored output (aux map), into `out` [cells][rows][N] at
  // out_cell elements per cell. bias_pop >= 0: the column sums are the gradient of that
  // population's range at bias_off
  auto delta = [&](int si, int act, const void* A, int a_rows, int64_t a_cell, int a_row0,
                   const bf16* W, int64_t Ps, const int* sel, void* out, int64_t out_cell,
                   int bias_pop, int64_t bias_off) {
    tcb::GParams& q = P->cells.st[si].p;
    q.epi = tcb::EPI_DACT;
    q.act = act;
    q.a_row0 = a_row0;
    q.b_sel = sel;
    ok = ok && map3(&P->maps.a[si], A, q.K, a_rows, C, a_cell, 128, msg) &&
         map3(&P->maps.b[si], W, q.N, q.K, NI, Ps, 64, msg) &&
         map3(&P->maps.out[si], out, q.N, q.M, C, out_cell, 64, msg);
    if (bias_pop < 0) return;
    q.bias_part = P->bpart + bp_off;
    q.bias_cell = bp_cell;
    bp_off += 4 * (int64_t)q.mtiles * q.N;
    tcb::RangeTask& t = P->cells.rt[bias_pop];
    for (int k = 0; k < t.r.n; ++k)
      if (t.r.off[k] == bias_off && t.r.len[k] == q.N) {
        t.part[k] = q.bias_part;
        t.tiles[k] = q.mtiles;
        t.dep[t.n_dep] = si;
        t.need[t.n_dep++] = q.mtiles * q.ntiles;
      }
  };
  auto aux3 = [&](int si, const void* X, int rows, int64_t cell, int row0) {
    P->cells.st[si].p.x_row0 = row0;
    ok = ok && map3(&P->maps.in[si], X, P->cells.st[si].p.N, rows, C, cell, 64, msg);
  };
  // weight gradient dW[o][i] = sum_r A[r][o] Bm[r][i] (both read MN-major) of the tensor at `off`
  // of a population: the Adam step in the epilogue, or the gradient stored. A's rows: a_rows per
  // cell, with split K a_rows per part
  auto weight = [&](int si, const void* A, int a_rows, int64_t a_cell, const TcbBuffers::AdamPop& ap,
                    const int* src, int64_t off, int64_t Ps, float* grad) {
    tcb::GParams& q = P->cells.st[si].p;
    q.a_mn = 1;
    q.epi = tcb::EPI_F32;
    q.C = grad + off;
    q.c_cell = Ps;
    ok = ok && (q.ksplit > 0 ? map4(&P->maps.a[si], A, q.M, a_rows, 2, C, (int64_t)a_rows * q.M,
                                    a_cell, msg)
                             : map3(&P->maps.a[si], A, q.M, a_rows, C, a_cell, 64, msg));
    if (!b.fuse_adam) return;
    // w, m, v are one allocation in three equal parts: the part size is the 4th dimension's
    // stride, the same for the old and the new snapshot
    const int64_t part = ap.m - ap.w;
    if (q.N % 16 != 0 || off % 8 != 0 || Ps % 8 != 0 || part <= 0 || ap.v - ap.m != part ||
        ap.m_new - ap.w_new != part || ap.v_new - ap.m_new != part) {
      if (msg) *msg = "fused Adam needs 16-column tensors at 8-element offsets and w, m, v at "
                      "equal distances";
      ok = false;
      return;
    }
    q.epi = tcb::EPI_ADAM;
    q.adam.src = src;
    q.adam.coef = ap.coef;
    q.adam.beta1 = b.beta1;
    q.adam.beta2 = b.beta2;
    q.adam.eps = b.eps;
    ok = ok && map4f(&P->maps.in[si], ap.w + off, q.N, q.M, NI, Ps, part, msg) &&
         map4f(&P->maps.out[si], ap.w_new + off, q.N, q.M, C, Ps, part, msg) &&
         map3b_rows(&P->maps.nb[si], ap.wb_new + off, q.N, q.M, C, Ps, msg);
  };
  auto act3 = [&](int si, const void* X, int rows, int64_t cell) {
    ok = ok && map3(&P->maps.b[si], X, P->cells.st[si].p.N, rows, C, cell, 64, msg);
  };
  const int64_t Bh = (int64_t)B * h, Bx = (int64_t)B * x;
  // D1 = (J2 @ W2d) * lrelu'(TG1): J2's rows [0, 2B) (D's loss; with D's b1) and [2B, 3B) (G's
  // loss, on TG1's fake rows)
  stage(S_D1G, B, h, h, bn);
  delta(S_D1G, ACT_LRELU, b.J2, 3 * B, 3 * Bh, 2 * B, Dw + b.doff[2], b.PDs, b.src_d,
        (bf16*)b.D1 + 2 * Bh, 3 * Bh, -1, 0);
  aux3(S_D1G, b.TG1, 2 * B, 2 * Bh, B);
  stage(S_D1D, 2 * B, h, h, bn);
  delta(S_D1D, ACT_LRELU, b.J2, 3 * B, 3 * Bh, 0, Dw + b.doff[2], b.PDs, b.src_d, b.D1, 3 * Bh,
        1, b.doff[1]);
  aux3(S_D1D, b.TG1, 2 * B, 2 * Bh, 0);
  // A3 = (D1[2B + r] @ W1d) * (1 - F^2), F the selected generator's fakes: E[c] slot 1 + sel_g[c]
  // (with G's b3)
  stage(S_A3, B, x, h, bn).x_slot = b.sel_g;
  delta(S_A3, ACT_TANH, b.D1, 3 * B, 3 * Bh, 2 * B, Dw + b.doff[0], b.PDs, b.src_d, b.A3, Bx, 0,
        b.goff[5]);
  ok = ok && map4(&P->maps.in[S_A3], b.E, x, B, 6, C, Bx, b.e_cell, msg);
  // A2 = (A3 @ W3g) * relu'(TH2) (with G's b2), A1 = (A2 @ W2g) * relu'(TH1) (with G's b1)
  stage(S_A2, B, h, x, bn);
  delta(S_A2, ACT_RELU, b.A3, B, Bx, 0, Gw + b.goff[4], b.PGs, b.src_g, b.A2, Bh, 0,
        b.goff[3]);
  aux3(S_A2, b.TH2, B, Bh, 0);
  stage(S_A1, B, h, h, bn);
  delta(S_A1, ACT_RELU, b.A2, B, Bh, 0, Gw + b.goff[2], b.PGs, b.src_g, b.A1, Bh, 0,
        b.goff[1]);
  aux3(S_A1, b.TH1, B, Bh, 0);
  // dW2d = J2^T TG1 and dW1d = D1^T X over the 2B D-loss rows. X = [E[c] rows 0..B-1 (real); E[c]
  // fake rows of slot sel_g[c]] is read in place: K splits into the two B-row parts of X and of D1
  stage(S_DW2D, h, h, 2 * B, bn);
  weight(S_DW2D, b.J2, 3 * B, 3 * Bh, b.adam_d, b.src_d, b.doff[2], b.PDs, b.gD);
  act3(S_DW2D, b.TG1, 2 * B, 2 * Bh);
  {
    tcb::GParams& q = stage(S_DW1D, h, x, 2 * B, bn);
    q.ksplit = (B + 63) / 64;
    q.kchunks = 2 * q.ksplit;
    q.b_slot_sel = b.sel_g;
  }
  weight(S_DW1D, b.D1, B, 3 * Bh, b.adam_d, b.src_d, b.doff[0], b.PDs, b.gD);
  ok = ok && map4(&P->maps.b[S_DW1D], b.E, x, B, 6, C, Bx, b.e_cell, msg);
  // dW3g = A3^T TH2, dW2g = A2^T TH1, dW1g = A1^T Z
  stage(S_DW3G, x, h, B, bn);
  weight(S_DW3G, b.A3, B, Bx, b.adam_g, b.src_g, b.goff[4], b.PGs, b.gG);
  act3(S_DW3G, b.TH2, B, Bh);
  stage(S_DW2G, h, h, B, bn);
  weight(S_DW2G, b.A2, B, Bh, b.adam_g, b.src_g, b.goff[2], b.PGs, b.gG);
  act3(S_DW2G, b.TH1, B, Bh);
  stage(S_DW1G, h, z, B, z);
  weight(S_DW1G, b.A1, B, Bh, b.adam_g, b.src_g, b.goff[0], b.PGs, b.gG);
  act3(S_DW1G, b.Z, B, (int64_t)B * z);
  if (ok) {
    int tiles[tcb::MAX_STAGES];
    for (int k = 0; k < tcb::MAX_STAGES; ++k) {
      const tcb::GParams& q = P->cells.st[k].p;
      tiles[k] = q.mtiles * q.ntiles;
    }
    for (int k = 0; k < tcb::MAX_STAGES; ++k) {
      P->cells.st[k].dep = S_DEP[k];
      P->cells.st[k].dep_need = S_DEP[k] >= 0 ? tiles[S_DEP[k]] : 0;
    }
    P->cells.op_bytes = tcb::A_BYTES + bn * tcb::BK * 2;
    P->cells.n_ops = tcb::RING_BYTES / P->cells.op_bytes;
    if (P->cells.n_ops > tcb::MAX_OPS) P->cells.n_ops = tcb::MAX_OPS;
    const std::vector<int2> list = tile_list(C, tiles);
    P->cells.n_list = (int)list.size();
    if (cudaMalloc(&P->list, list.size() * sizeof(int2)) != cudaSuccess ||
        cudaMemcpy(P->list, list.data(), list.size() * sizeof(int2), cudaMemcpyHostToDevice) !=
            cudaSuccess) {
      cudaGetLastError();
      if (msg) *msg = "cudaMalloc for the backward's tile list failed";
      ok = false;
    }
    P->cells.list = P->list;
    P->cells.sync = b.sync;
    P->cells.cells = C;
    P->cells.err = P->err;
    P->grid = P->cells.n_list < sms ? P->cells.n_list : sms;
    if (cudaFuncSetAttribute(tcb::k_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, tcb::SMEM) !=
        cudaSuccess) {
      cudaGetLastError();
      if (msg) *msg = "cannot reserve shared memory for the backward";
      ok = false;
    }
  }
  if (!ok) {
    free_plan(P);
    return nullptr;
  }
  return P;
}

int tcb_run(TcbPlan* P, cudaStream_t st, std::string* msg) {
  launch_pdl(tcb::k_bwd, dim3(P->grid), dim3(tcb::THREADS), tcb::SMEM, st, P->maps, P->cells);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    if (msg) *msg = std::string("backward launch: ") + cudaGetErrorString(e);
    return 1;
  }
  return 0;
}

int* tcb_error_flag(TcbPlan* P) { return P ? P->err : nullptr; }

void tcb_plan_destroy(TcbPlan* P) {
  if (P) free_plan(P);
}

}  // namespace lipz
