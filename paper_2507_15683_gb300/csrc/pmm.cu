// Probabilistic mutual matching (PMM) of a query and a rendered feature map,
// coarse to fine: Hi^2-GSLoc Sec. 3.4, Eq. 11.
//
// Coarse level. Each 8 x 8 block of the fine maps becomes one coarse cell: its
// mean, L2-normalised in binary32 (k_pmm_codes) and split into two bfloat16
// vectors, hi = bf16(u) and lo = bf16(u - hi), which carry u to about 2^-17.
// The cosine matrix M of all query cells against all rendered cells is the
// 32-deep contraction hi_q . hi_r + lo_q . hi_r + hi_q . lo_r (the lo . lo term
// is below 2^-17), computed tile by tile on the 5th generation tensor cores
// (tcgen05.mma, bf16 operands in shared memory, fp32 accumulator in tensor
// memory) and never stored: M is the fp32-accurate cosine of the unrounded
// cell means, not that of bf16-rounded ones (which would move the dual-softmax
// decisions whose margins are below about 1e-2). Two passes over the tiles:
//   1. row and column sums of exp((M - 1) / tau), hence the row and column
//      log-sum-exps r_i, c_j of M / tau (|M| <= 1 makes 1 / tau a fixed
//      shift, so one exponential serves the row and the column);
//   2. per row i the first argmax over j of log P_M + r_i = 2 M / tau - c_j,
//      per column j the first argmax over i of 2 M / tau - r_i.
// Partial results per tile row / column are reduced in a fixed order, and a
// query cell i matches rendered cell j when each is the other's argmax (MNN).
//
// Fine level. For every coarse match the 64 fine query vectors of cell i and
// the 64 rendered vectors of cell j (normalised in fp32) give a 64 x 64 cosine
// matrix; the same dual softmax and MNN inside the window pair give the fine
// matches (one CTA per coarse match).
#include <cudaTypedefs.h>  // CUtensorMap; its encoder comes through the runtime
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <type_traits>

#include "gsr_launch.h"
#include "gsr_pmm.h"

namespace gsr {
void set_last_error(const std::string& msg);
}

namespace {

constexpr int kC = 32;         // channels
constexpr int kRatio = 8;      // H_f / H_c
constexpr int kTile = 128;     // cells per tile side (MMA M = N = 128)
constexpr uint32_t kTmemCols = 128;
constexpr int kWaitLimit = GS_PMM_DEFAULT_WAIT_POLLS;  // polls of an mbarrier before giving up (far beyond a 2-MMA tile)
constexpr int kMaxCells = 1 << 18;
constexpr int kScanThreads = 1024;
constexpr int kWin = kRatio * kRatio;  // fine vectors per window
constexpr int kCode = 2 * kC;          // bf16 per coarse code: hi[32], then lo[32]
static_assert(kWin == 64, "k_pmm_fine tiles the window over 8 x 8 threads");

// Tensor-core operand layout of a block of kTile codes (no swizzle, K-major):
// the byte offset of the 16-byte chunk (row r, k-chunk c) is that of core
// matrix (r / 8, c), 128 bytes each, with the 8 k-chunks of a row group (hi
// 0..3, lo 0..3) adjacent, so row groups are kChunks x 128 = 1024 bytes apart.
// The codes kernel also writes every block of kTile cells in this layout, so
// that a tile's operand is one contiguous kTileBytes bulk copy, and, for the
// rows of pass 1, every pair of blocks with bit 3 of the row moved up: block
// 2 s + u of that copy holds the rows of super-block s whose bit 3 is u.
constexpr int kChunks = kCode * 2 / 16;         // 16-byte k-chunks per code
constexpr int kTileBytes = kTile * kCode * 2;   // one operand block (16 KB)
__host__ __device__ __forceinline__ int core_off(int r, int c) {
  return ((r >> 3) * kChunks + c) * 128 + (r & 7) * 16;
}

constexpr int kPair = 2 * kTile;  // rows of a super-block
__host__ __device__ __forceinline__ size_t paired_off(int cell, int c) {
  const int r = cell % kPair;
  return (size_t)(2 * (cell / kPair) + ((r >> 3) & 1)) * kTileBytes + core_off(((r >> 4) << 3) | (r & 7), c);
}

// ---------------------------------------------------------------------------
// coarse codes: a CTA takes 32 horizontally adjacent cells; warp c sums channel c
// of each cell (lane = cell: the 32 lanes read one contiguous row of 256
// pixels), warp 0 forms the norms, and the codes leave as one contiguous block
// ---------------------------------------------------------------------------
struct CodeMap {  // one feature map and its codes; paired is NULL for the rendered map
  const float* F;
  unsigned short* codes;
  unsigned char *tiled, *paired;
};

// blockIdx.z: the map (both in one launch, so that one's last blocks overlap the other's first)
__global__ void __launch_bounds__(1024) k_pmm_codes(CodeMap query, CodeMap render, int H, int W, int Wc) {
  const CodeMap& map = blockIdx.z ? render : query;
  const float* __restrict__ F = map.F;
  unsigned short* __restrict__ codes = map.codes;
  unsigned char *__restrict__ tiled = map.tiled, *__restrict__ paired = map.paired;
  __shared__ float m_s[kC][32];
  __shared__ float inv_s[32];
  __shared__ unsigned short u_s[32][kCode + 2];  // padded rows: the per-channel stores hit distinct banks
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cy = blockIdx.y, cx = blockIdx.x * 32 + lane;
  const bool ok = cx < Wc;
  float m = 0.0f;
  if (ok) {
    const float* base = F + (size_t)c * H * W + (size_t)(cy * kRatio) * W + cx * kRatio;
    float s = 0.0f;  // block sum in row-major order
#pragma unroll
    for (int dy = 0; dy < kRatio; ++dy) {
      const float4 a = *reinterpret_cast<const float4*>(base + (size_t)dy * W);
      const float4 b = *reinterpret_cast<const float4*>(base + (size_t)dy * W + 4);
      s = __fadd_rn(s, a.x);
      s = __fadd_rn(s, a.y);
      s = __fadd_rn(s, a.z);
      s = __fadd_rn(s, a.w);
      s = __fadd_rn(s, b.x);
      s = __fadd_rn(s, b.y);
      s = __fadd_rn(s, b.z);
      s = __fadd_rn(s, b.w);
    }
    m = __fmul_rn(s, 1.0f / (kRatio * kRatio));  // exact scaling
  }
  m_s[c][lane] = m;
  __syncthreads();
  if (c == 0) {  // squares summed over channels in channel order
    float ss = 0.0f;
#pragma unroll
    for (int k = 0; k < kC; ++k) ss = __fadd_rn(ss, __fmul_rn(m_s[k][lane], m_s[k][lane]));
    inv_s[lane] = __fsqrt_rn(ss);
  }
  __syncthreads();
  const float n = inv_s[lane];
  const float u = n > 0.0f ? __fdiv_rn(m, n) : 0.0f;
  const __nv_bfloat16 hi = __float2bfloat16_rn(u);
  const __nv_bfloat16 lo = __float2bfloat16_rn(__fsub_rn(u, __bfloat162float(hi)));  // exact difference
  u_s[lane][c] = __bfloat16_as_ushort(hi);
  u_s[lane][kC + c] = __bfloat16_as_ushort(lo);
  __syncthreads();
  const int cell0 = cy * Wc + blockIdx.x * 32;
  const int ncell = min(32, Wc - blockIdx.x * 32);
  // 32 cells x 64 bf16, contiguous in the output: two 16-bit values per thread
  const int t = threadIdx.x;
  if (t < ncell * kC) {
    const int e = 2 * t;
    const uint32_t v = (uint32_t)u_s[e / kCode][e % kCode] | ((uint32_t)u_s[e / kCode][e % kCode + 1] << 16);
    reinterpret_cast<uint32_t*>(codes + (size_t)cell0 * kCode)[t] = v;
    const int cell = cell0 + e / kCode, el = e % kCode;  // the same two values in the tiled copy
    const size_t off = (size_t)(cell / kTile) * kTileBytes + core_off(cell % kTile, el / 8) + (el % 8) * 2;
    *reinterpret_cast<uint32_t*>(tiled + off) = v;
    if (paired) *reinterpret_cast<uint32_t*>(paired + paired_off(cell, el / 8) + (el % 8) * 2) = v;
  }
}

// ---------------------------------------------------------------------------
// tcgen05 helpers (inline PTX)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major, no swizzle. The operand is stored
// as 8 x 16-byte core matrices; adjacent core matrices along K are `lbo` bytes
// apart and adjacent 8-row groups `sbo` bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version field (0b001)
  return d;                 // base offset 0, relative LBO, no swizzle
}

// Instruction descriptor of tcgen05.mma kind::f16: fp32 accumulator, bf16 A and
// B, both K-major, N = M = 128.
constexpr uint32_t kIdesc = (1u << 4)                         // D format: f32
                            | (1u << 7)                       // A format: bf16
                            | (1u << 10)                      // B format: bf16
                            | ((uint32_t)(kTile >> 3) << 17)  // N >> 3
                            | ((uint32_t)(kTile >> 4) << 24);  // M >> 4

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// bounded wait for the phase `parity` of an mbarrier: at most `limit` polls,
// false when they run out (limit 0 gives up at once)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int limit) {
  for (int it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive fp32 accumulator columns of this thread's lane, without the wait
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// 32 consecutive columns, without the wait
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}

// wait for the loads of r, tied to them so that no use moves above it
template <int N>
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < N; ++k) asm volatile("" : "+r"(r[k]));
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// mbar_wait that also gives up once *stop is set; a poll may suspend the warp
// for up to a microsecond, so that waiting warps leave the issue slots alone
__device__ __forceinline__ bool mbar_wait_or(uint32_t bar, uint32_t parity, int limit, const volatile int* stop) {
  for (int it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (*stop) return false;
  }
  return false;
}

// contiguous bulk copy global -> shared, completing on an mbarrier
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// the six MMAs of a tile: hi . hi, lo . hi, hi . lo, each K = 32 as two K = 16
// steps (k-chunks (0, 1) then (2, 3) at +256 bytes); the lo half starts 512 bytes in
__device__ __forceinline__ void mma_tile(uint32_t tmem, uint32_t sa, uint32_t sb) {
  constexpr uint32_t kSbo = kChunks * 128;
  mma_bf16(tmem, smem_desc(sa, 128, kSbo), smem_desc(sb, 128, kSbo), 0u);
  mma_bf16(tmem, smem_desc(sa + 256, 128, kSbo), smem_desc(sb + 256, 128, kSbo), 1u);
  mma_bf16(tmem, smem_desc(sa + 512, 128, kSbo), smem_desc(sb, 128, kSbo), 1u);
  mma_bf16(tmem, smem_desc(sa + 768, 128, kSbo), smem_desc(sb + 256, 128, kSbo), 1u);
  mma_bf16(tmem, smem_desc(sa, 128, kSbo), smem_desc(sb + 512, 128, kSbo), 1u);
  mma_bf16(tmem, smem_desc(sa + 256, 128, kSbo), smem_desc(sb + 768, 128, kSbo), 1u);
}

// ---------------------------------------------------------------------------
// similarity tiles
// ---------------------------------------------------------------------------
constexpr int kTileThreads = 256;  // warp w: tensor-memory lanes 32 (w % 4) .. +31, columns 64 (w / 4) .. +63

// Sums over the 16 lanes of a half warp of v[0..15], one column each: the lane
// ends with the sum of column (bit 2, bit 1, bit 0, bit 3 of the lane, high to
// low). The adding order is fixed: lanes l ^ 4, l ^ 2, l ^ 1, l ^ 8.
template <int S>
__device__ __forceinline__ void scatter_step(float (&v)[16], int lane, int o) {
  const bool up = (lane & o) != 0;
#pragma unroll
  for (int i = 0; i < S; ++i) {
    const float send = up ? v[i] : v[i + S];
    const float keep = up ? v[i + S] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
}
__device__ __forceinline__ float half_scatter16(float (&v)[16], int lane) {
  scatter_step<8>(v, lane, 4);
  scatter_step<4>(v, lane, 2);
  scatter_step<2>(v, lane, 1);
  scatter_step<1>(v, lane, 8);
  return v[0];
}

// 2^x for x in [-120, 1]: the results stay normal binary32 numbers, so the
// flush-to-zero form of the hardware approximation is exact enough here
__device__ __forceinline__ float ex2_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// argmax order: larger value wins, equal values go to the smaller index
__device__ __forceinline__ bool better(float v, int i, float bv, int bi) { return v > bv || (v == bv && i < bi); }

// ---------------------------------------------------------------------------
// Pass 1 over M = A B^T (A, B: n x 32 split bf16 codes), with e = exp((M - 1) /
// tau): prow_v[c n + i] = sum of e over row i and the 128 columns of block c,
// pcol_v[b n + j] = the same over column j and the 128 rows of block b.
//
// A row sum stays in its thread (tensor-memory lane = row). A column sum runs
// over the lanes, and its shuffles and selects cost more than the exponential,
// so the rows are paired: the two accumulators of a super-block (256 rows x 128
// columns) hold the rows whose bit 3 is 0 and 1, which puts rows r and r ^ 8
// into one thread. Their sum is one addition, and the 15 exchange steps of 16
// columns serve two rows. The adding order of a column is r ^ 8, ^ 4, ^ 2, ^ 1,
// ^ 16, then the four 32-row groups in order; of a row, its two 64-column
// halves each in ascending order.
//
// Roles: warp 8 copies operands and issues the MMAs; an accumulator is handed
// back as soon as it is read, so that its next MMAs run beside the sums.
//
// 282 us at 32,400 cells (371 us with one row per thread, 16 exchange steps per
// 16 columns of it and block barriers around the MMAs): 4 warps per scheduler
// at 96 registers, issue 65 %, ex2 unit 40 %, tensor pipe 30 %.
// ---------------------------------------------------------------------------
constexpr int kSumThreads = kTileThreads + 32;
constexpr int kSumStages = 3;
struct SumSmem {
  uint4 a[2][kTileBytes / 16];  // the super-block's operands, by row parity
  uint4 b[kSumStages][kTileBytes / 16];
  float colv[2][2][4][kTile];  // [buffer][128-row block][32-row group][column]
  float rowv[2][2][2][kTile];  // [buffer][128-row block][column half][row]
  unsigned long long a_full, a_free, b_full[kSumStages], b_free[kSumStages], acc_full[2], acc_free[2];
  unsigned long long part[2];  // both partial arrays of a 128-row block are written
  uint32_t tmem;
  int stop;
};
constexpr size_t kSumSmemBytes = 96 * 1024;  // keeps at most 2 CTAs (of 256 tensor-memory columns) on an SM
static_assert(sizeof(SumSmem) <= kSumSmemBytes && 3 * kSumSmemBytes > 228 * 1024, "super-tile shared memory");

__global__ void __launch_bounds__(kSumThreads, 2) k_pmm_sums(const unsigned char* __restrict__ ca,
                                                             const unsigned char* __restrict__ cb, int n, int nb,
                                                             int per, float s_exp, float* __restrict__ prow_v,
                                                             float* __restrict__ pcol_v, int* __restrict__ err,
                                                             int wait_limit) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  SumSmem& S = *reinterpret_cast<SumSmem*>(smem_raw);
  const int t0 = (int)blockIdx.x * per, nt = min(per, (nb + 1) / 2 * nb - t0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)),
                 "r"(2 * kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    bar_init(smem_u32(&S.a_full), 1);
    bar_init(smem_u32(&S.a_free), 1);
    for (int i = 0; i < kSumStages; ++i) {
      bar_init(smem_u32(&S.b_full[i]), 1);
      bar_init(smem_u32(&S.b_free[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      bar_init(smem_u32(&S.acc_full[i]), 1);
      bar_init(smem_u32(&S.acc_free[i]), kTileThreads / 32);
      bar_init(smem_u32(&S.part[i]), 4);
    }
    S.stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;
  const volatile int* stop = &S.stop;
  // as in pass 2: a wait that runs out sets the error flag and `stop`, which
  // ends all roles, and each waits for what it has in flight
  auto give_up = [&]() {
    atomicExch(err, 1);
    *(volatile int*)&S.stop = 1;
  };
  int sr = t0 / nb, c = t0 - sr * nb;  // super-block of rows and column block at hand
  if (warp == 8) {
    if (lane == 0) {
      auto load_a = [&](int r) {
        bar_expect(smem_u32(&S.a_full), 2 * kTileBytes);
        for (int u = 0; u < 2; ++u)
          bulk_copy(smem_u32(S.a[u]), ca + (size_t)(2 * r + u) * kTileBytes, kTileBytes, smem_u32(&S.a_full));
      };
      int next_c = c;
      auto load_b = [&](int k) {  // the CTA's k-th column block, in order
        const int s = k % kSumStages;
        bar_expect(smem_u32(&S.b_full[s]), kTileBytes);
        bulk_copy(smem_u32(S.b[s]), cb + (size_t)next_c * kTileBytes, kTileBytes, smem_u32(&S.b_full[s]));
        if (++next_c == nb) next_c = 0;
      };
      load_a(sr);
      int issued = 0;
      for (; issued < min(nt, kSumStages); ++issued) load_b(issued);
      uint32_t a_fill = 0;
      int k = 0, s = 0;
      int done[2] = {0, 0}, freed = 0;  // accumulators committed, super-blocks released
      uint32_t lap = 0;
      bool ok = true;
      for (; k < nt && ok; ++k) {
        if (k > 0 && c == 0) {  // a new super-block: its operands take the place of the last one's
          ok = mbar_wait_or(smem_u32(&S.a_free), a_fill, kWaitLimit, stop);
          if (!ok) break;
          a_fill ^= 1u;
          load_a(sr);
        }
        if (k == 0 || c == 0) ok = mbar_wait_or(smem_u32(&S.a_full), a_fill, kWaitLimit, stop);
        ok = ok && mbar_wait_or(smem_u32(&S.b_full[s]), lap, kWaitLimit, stop);
        for (int u = 0; u < 2 && ok; ++u) {
          if (k > 0) ok = mbar_wait_or(smem_u32(&S.acc_free[u]), (uint32_t)(k - 1) & 1u, kWaitLimit, stop);
          if (!ok) break;
          tc_fence_after();
          mma_tile(tmem + (uint32_t)u * kTmemCols, smem_u32(S.a[u]), smem_u32(S.b[s]));
          if (u == 1) {
            mma_commit(smem_u32(&S.b_free[s]));
            if (c == nb - 1) {
              mma_commit(smem_u32(&S.a_free));
              ++freed;
            }
          }
          mma_commit(smem_u32(&S.acc_full[u]));
          ++done[u];
        }
        if (!ok) break;
        // the stage before this one is read once its MMAs, which these follow, are done
        if (k > 0 && issued < nt) {
          ok = mbar_wait_or(smem_u32(&S.b_free[(k - 1) % kSumStages]), (uint32_t)((k - 1) / kSumStages) & 1u, kWaitLimit,
                            stop);
          if (ok) load_b(issued++);
        }
        if (++s == kSumStages) {
          s = 0;
          lap ^= 1u;
        }
        if (++c == nb) {
          c = 0;
          ++sr;
        }
      }
      if (!ok && !*stop) give_up();
      // copies and MMAs in flight end before the memory they use is released
      mbar_wait(smem_u32(&S.a_full), a_fill, kWaitLimit);
      for (int j = max(0, issued - kSumStages); j < issued; ++j)
        mbar_wait(smem_u32(&S.b_full[j % kSumStages]), (uint32_t)(j / kSumStages) & 1u, kWaitLimit);
      for (int u = 0; u < 2; ++u)
        if (done[u] > 0) mbar_wait(smem_u32(&S.acc_full[u]), (uint32_t)(done[u] - 1) & 1u, kWaitLimit);
      if (done[1] > 0)
        mbar_wait(smem_u32(&S.b_free[(done[1] - 1) % kSumStages]), (uint32_t)((done[1] - 1) / kSumStages) & 1u, kWaitLimit);
      if (freed > 0) mbar_wait(smem_u32(&S.a_free), (uint32_t)(freed - 1) & 1u, kWaitLimit);
    }
  } else {
    const int quarter = warp & 3, half = warp >> 2;
    const int blk = quarter >> 1;                                  // 128-row block of the super-block
    const int row = (quarter & 1) * 64 + (lane >> 3) * 16 + (lane & 7);  // of the block, parity 0; parity 1: + 8
    const int grp = (quarter & 1) * 2 + (lane >> 4);               // 32-row group of the block
    const int col = ((lane >> 2 & 1) << 3) | ((lane >> 1 & 1) << 2) | ((lane & 1) << 1) | (lane >> 3 & 1);
    const int out = (half * 2 + (quarter & 1)) * 32 + lane;        // the row and column of the block this thread writes
    const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 64);
    for (int k = 0; k < nt; ++k) {
      const uint32_t par = (uint32_t)k & 1u;
      const int row0 = sr * kPair + blk * kTile + row, col0 = c * kTile + half * 64;
      // a row past n gives exponentials of -inf, i.e. zeros, without a mask
      const bool ok0 = row0 < n, ok1 = row0 + 8 < n;
      const float2 sa = ok0 ? make_float2(s_exp, s_exp) : make_float2(0.0f, 0.0f);
      const float2 ba = ok0 ? make_float2(-s_exp, -s_exp) : make_float2(-INFINITY, -INFINITY);
      const float2 sb = ok1 ? make_float2(s_exp, s_exp) : make_float2(0.0f, 0.0f);
      const float2 bb = ok1 ? make_float2(-s_exp, -s_exp) : make_float2(-INFINITY, -INFINITY);
      bool ok = mbar_wait_or(smem_u32(&S.acc_full[0]), par, wait_limit, stop);
      ok = ok && mbar_wait_or(smem_u32(&S.acc_full[1]), par, wait_limit, stop);
      if (!__all_sync(0xffffffffu, ok)) {
        if (!*stop) give_up();
        break;
      }
      tc_fence_after();
      float2 sum = make_float2(0.0f, 0.0f);  // row sums of the two parities
      auto tile = [&](auto masked) {  // two copies: only the ragged last column block masks
        constexpr bool kMasked = decltype(masked)::value;
        uint32_t r[2][16], q[2][16];  // 16 columns of each parity, and the next 16
        tmem_ld16(tbase, r[0]);
        tmem_ld16(tbase + kTmemCols, q[0]);
        tmem_wait(r[0]);
        tmem_wait(q[0]);
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          if (ch < 3) {
            tmem_ld16(tbase + (uint32_t)(ch * 16 + 16), r[(ch + 1) & 1]);
            tmem_ld16(tbase + kTmemCols + (uint32_t)(ch * 16 + 16), q[(ch + 1) & 1]);
          }
          if (ch == 2) {  // everything is in registers half way through the sums
            tmem_wait(r[1]);
            tmem_wait(q[1]);
            tc_fence_before();
            if (lane == 0) {
              bar_arrive(smem_u32(&S.acc_free[0]));
              bar_arrive(smem_u32(&S.acc_free[1]));
            }
          }
          float v[16];
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const uint32_t *ra = r[ch & 1] + i, *qa = q[ch & 1] + i;
            const float2 x = __ffma2_rn(make_float2(__uint_as_float(ra[0]), __uint_as_float(ra[1])), sa, ba);
            const float2 y = __ffma2_rn(make_float2(__uint_as_float(qa[0]), __uint_as_float(qa[1])), sb, bb);
            float2 e0 = make_float2(ex2_ftz(x.x), ex2_ftz(y.x)), e1 = make_float2(ex2_ftz(x.y), ex2_ftz(y.y));
            if (kMasked && col0 + ch * 16 + i >= n) e0 = make_float2(0.0f, 0.0f);
            if (kMasked && col0 + ch * 16 + i + 1 >= n) e1 = make_float2(0.0f, 0.0f);
            sum = __fadd2_rn(sum, e0);
            sum = __fadd2_rn(sum, e1);
            v[i] = e0.x + e0.y;
            v[i + 1] = e1.x + e1.y;
          }
          S.colv[par][blk][grp][half * 64 + ch * 16 + col] = half_scatter16(v, lane);
          if (ch < 2) {
            tmem_wait(r[(ch + 1) & 1]);
            tmem_wait(q[(ch + 1) & 1]);
          }
        }
      };
      if ((c + 1) * kTile <= n) tile(std::false_type{});
      else tile(std::true_type{});
      S.rowv[par][blk][half][row] = sum.x;
      S.rowv[par][blk][half][row + 8] = sum.y;
      __syncwarp();
      if (lane == 0) bar_arrive(smem_u32(&S.part[blk]));
      // the four warps of the block; their next partials go to the other buffer
      ok = mbar_wait_or(smem_u32(&S.part[blk]), par, kWaitLimit, stop);
      if (!__all_sync(0xffffffffu, ok)) {
        if (!*stop) give_up();
        break;
      }
      const int b = 2 * sr + blk, rr = b * kTile + out, cc = c * kTile + out;
      if (rr < n) prow_v[(size_t)c * n + rr] = S.rowv[par][blk][0][out] + S.rowv[par][blk][1][out];
      if (cc < n && b < nb) {
        const float(*v)[kTile] = S.colv[par][blk];
        pcol_v[(size_t)b * n + cc] = ((v[0][out] + v[1][out]) + v[2][out]) + v[3][out];
      }
      if (++c == nb) {
        c = 0;
        ++sr;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------
// Pass 2: for every row i of M = A B^T the first argmax over the columns j of
// 2 M_ij / tau - lse_j. With A = query, B = rendered and the column
// log-sum-exps this is the row argmax of log P_M; with the operands swapped and
// the row log-sum-exps, its column argmax.
//
// A CTA takes `per` consecutive tiles in row-block order, so a thread keeps the
// running best of its row (over its 64 of the 128 columns) in registers across
// the column blocks and writes it once per row block. Roles: warp 9 copies the
// operands (row block: two buffers; column blocks: kBestStages), warp 8 issues
// the MMAs into two accumulators, warps 0-7 read them: a warp loads its 64
// columns, hands the accumulator back and then works from registers, so the
// tensor pipe runs beside the epilogue. (One thread doing all of it between
// block barriers left the warps waiting for the MMAs.) Per 64 similarities a
// thread takes 32 packed FMAs and 32 three-input maxima; only when one of its
// four 16-column maxima beats its running best are those 16 searched for the
// first such column, which happens about log(n / 16) times per row. 197 us per
// launch at 32,400 cells (316 us with one thread driving the MMAs, a compare
// and two selects per similarity and a partial per tile); tensor pipe 44 %.
// ---------------------------------------------------------------------------
constexpr int kBestStages = 3;
constexpr int kNlRing = 8;  // log-sum-exp blocks: one is read while kBestStages + 2 later ones may be copied
constexpr int kRoleThreads = kTileThreads + 64;  // epilogue warps, the MMA warp, the copy warp
static_assert(kNlRing > kBestStages + 2, "a log-sum-exp block is read until its tile's epilogue is done");
struct BestSmem {
  uint4 a[2][kTileBytes / 16];
  uint4 b[kBestStages][kTileBytes / 16];
  float nl[kNlRing][kTile];  // negated log-sum-exps of the columns (-inf past n)
  unsigned long long a_full[2], a_free[2], b_full[kBestStages], b_free[kBestStages], nl_full[kNlRing];
  unsigned long long acc_full[2], acc_free[2];
  uint32_t tmem;
  int stop;
};
constexpr size_t kBestSmemBytes = 88 * 1024;  // keeps at most 2 CTAs (of 256 tensor-memory columns) on an SM
static_assert(sizeof(BestSmem) <= kBestSmemBytes && 3 * kBestSmemBytes > 228 * 1024, "tile shared memory");

// the first CTA of pass 2 that holds a tile of row block rb, and the most CTAs that hold tiles of one
__host__ __device__ __forceinline__ int best_first(int rb, int nb, int per) { return rb * nb / per; }
__host__ __device__ __forceinline__ int best_parts(int nb, int per) { return (nb - 1) / per + 2; }

__global__ void __launch_bounds__(kRoleThreads, 2) k_pmm_argmax(const unsigned char* __restrict__ ca,
                                                                const unsigned char* __restrict__ cb, int n, int nb,
                                                                int per, float s_two,
                                                                const float* __restrict__ nlse_c,
                                                                float* __restrict__ prow_v, int* __restrict__ prow_i,
                                                                int* __restrict__ err, int wait_limit) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  BestSmem& S = *reinterpret_cast<BestSmem*>(smem_raw);
  const int t0 = (int)blockIdx.x * per, nt = min(per, nb * nb - t0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)),
                 "r"(2 * kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      bar_init(smem_u32(&S.a_full[i]), 1);
      bar_init(smem_u32(&S.a_free[i]), 1);
      bar_init(smem_u32(&S.acc_full[i]), 1);
      bar_init(smem_u32(&S.acc_free[i]), kTileThreads / 32);
    }
    for (int i = 0; i < kBestStages; ++i) {
      bar_init(smem_u32(&S.b_full[i]), 1);
      bar_init(smem_u32(&S.b_free[i]), 1);
    }
    for (int i = 0; i < kNlRing; ++i) bar_init(smem_u32(&S.nl_full[i]), 1);
    S.stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;
  const volatile int* stop = &S.stop;
  // Every wait is bounded; one that runs out sets the error flag and `stop`,
  // which ends all roles. Each role then waits for what it has in flight.
  auto give_up = [&]() {
    atomicExch(err, 1);
    *(volatile int*)&S.stop = 1;
  };
  int rb = t0 / nb, c = t0 - rb * nb;  // row and column block of the tile at hand, kept by each role
  if (warp == 9) {
    if (lane == 0) {
      int k = 0, r = -1, s = 0;  // tile, row block of this CTA, stage
      uint32_t lap = 1;           // parity of the stage's last release
      bool ok = true;
      for (; k < nt; ++k) {
        if (k == 0 || c == 0) {
          const int q = (r + 1) & 1;
          if (r + 1 >= 2 && !mbar_wait_or(smem_u32(&S.a_free[q]), (uint32_t)(((r + 1) >> 1) - 1) & 1u, kWaitLimit, stop)) {
            ok = false;
            break;
          }
          ++r;
          bar_expect(smem_u32(&S.a_full[q]), kTileBytes);
          bulk_copy(smem_u32(S.a[q]), ca + (size_t)rb * kTileBytes, kTileBytes, smem_u32(&S.a_full[q]));
        }
        if (k >= kBestStages && !mbar_wait_or(smem_u32(&S.b_free[s]), lap, kWaitLimit, stop)) {
          ok = false;
          break;
        }
        bar_expect(smem_u32(&S.b_full[s]), kTileBytes);
        bulk_copy(smem_u32(S.b[s]), cb + (size_t)c * kTileBytes, kTileBytes, smem_u32(&S.b_full[s]));
        const uint32_t nl_bar = smem_u32(&S.nl_full[k % kNlRing]);
        bar_expect(nl_bar, kTile * 4);
        bulk_copy(smem_u32(S.nl[k % kNlRing]), nlse_c + (size_t)c * kTile, kTile * 4, nl_bar);
        if (++s == kBestStages) {
          s = 0;
          lap ^= 1u;
        }
        if (++c == nb) {
          c = 0;
          ++rb;
        }
      }
      if (!ok && !*stop) give_up();
      // copies in flight end before the shared memory is released
      for (int j = max(0, k - kNlRing); j < k; ++j)
        mbar_wait(smem_u32(&S.nl_full[j % kNlRing]), (uint32_t)(j / kNlRing) & 1u, kWaitLimit);
      for (int j = max(0, k - kBestStages); j < k; ++j)
        mbar_wait(smem_u32(&S.b_full[j % kBestStages]), (uint32_t)(j / kBestStages) & 1u, kWaitLimit);
      for (int j = max(0, r - 1); j <= r; ++j) mbar_wait(smem_u32(&S.a_full[j & 1]), (uint32_t)(j >> 1) & 1u, kWaitLimit);
    }
  } else if (warp == 8) {
    if (lane == 0) {
      int k = 0, r = -1, s = 0;
      uint32_t lap = 0;  // parity of the stage's present fill
      bool ok = true;
      for (; k < nt; ++k) {
        const int q = k & 1;
        if (k == 0 || c == 0) {
          ++r;
          ok = mbar_wait_or(smem_u32(&S.a_full[r & 1]), (uint32_t)(r >> 1) & 1u, kWaitLimit, stop);
        }
        ok = ok && mbar_wait_or(smem_u32(&S.b_full[s]), lap, kWaitLimit, stop);
        if (ok && k >= 2)
          ok = mbar_wait_or(smem_u32(&S.acc_free[q]), (uint32_t)((k >> 1) - 1) & 1u, kWaitLimit, stop);
        if (!ok) break;
        tc_fence_after();
        mma_tile(tmem + (uint32_t)q * kTmemCols, smem_u32(S.a[r & 1]), smem_u32(S.b[s]));
        mma_commit(smem_u32(&S.b_free[s]));
        if (++c == nb) {
          c = 0;
          mma_commit(smem_u32(&S.a_free[r & 1]));
        }
        mma_commit(smem_u32(&S.acc_full[q]));
        if (++s == kBestStages) {
          s = 0;
          lap ^= 1u;
        }
      }
      if (!ok && !*stop) give_up();
      // MMAs in flight end before tensor memory is freed
      if (k > 0) mbar_wait(smem_u32(&S.acc_full[(k - 1) & 1]), (uint32_t)((k - 1) >> 1) & 1u, kWaitLimit);
      for (int j = max(0, k - kBestStages); j < k; ++j)
        mbar_wait(smem_u32(&S.b_free[j % kBestStages]), (uint32_t)(j / kBestStages) & 1u, kWaitLimit);
    }
  } else {
    const int quarter = warp & 3, half = warp >> 2;
    const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 64);
    const float2 two = make_float2(s_two, s_two);
    float best = -INFINITY;
    int bidx = 0x7fffffff;
    for (int k = 0; k < nt; ++k) {
      const int q = k & 1;
      bool ok = mbar_wait_or(smem_u32(&S.acc_full[q]), (uint32_t)(k >> 1) & 1u, wait_limit, stop);
      ok = ok && mbar_wait_or(smem_u32(&S.nl_full[k % kNlRing]), (uint32_t)(k / kNlRing) & 1u, kWaitLimit, stop);
      if (!__all_sync(0xffffffffu, ok)) {
        if (!*stop) give_up();
        break;
      }
      tc_fence_after();
      uint32_t r[64];
      tmem_ld32(tbase + (uint32_t)q * kTmemCols, r);
      tmem_ld32(tbase + (uint32_t)q * kTmemCols + 32u, r + 32);
      tmem_wait(r);
      tc_fence_before();
      if (lane == 0) bar_arrive(smem_u32(&S.acc_free[q]));  // every lane's values are in registers (aligned load)
      const float4* nl4 = reinterpret_cast<const float4*>(S.nl[k % kNlRing] + half * 64);
      float2 v[32];
      float m[4];  // of each 16 columns
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 x = nl4[ch * 4 + i];
          const int e = 8 * ch + 2 * i;
          v[e] = __ffma2_rn(make_float2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])), two,
                            make_float2(x.x, x.y));
          v[e + 1] = __ffma2_rn(make_float2(__uint_as_float(r[2 * e + 2]), __uint_as_float(r[2 * e + 3])), two,
                                make_float2(x.z, x.w));
        }
        const float2* u = v + 8 * ch;
        m[ch] = max3(max3(u[0].x, u[0].y, u[1].x), max3(u[1].y, u[2].x, u[2].y),
                     max3(max3(u[3].x, u[3].y, u[4].x), max3(u[4].y, u[5].x, u[5].y),
                          max3(fmaxf(u[6].x, u[6].y), u[7].x, u[7].y)));
      }
      if (fmaxf(max3(m[0], m[1], m[2]), m[3]) > best) {
#pragma unroll
        for (int ch = 0; ch < 4; ++ch)
          if (m[ch] > best) {  // the first column that reaches it
            int i = 15;
#pragma unroll
            for (int e = 7; e >= 0; --e) {
              if (v[8 * ch + e].y == m[ch]) i = 2 * e + 1;
              if (v[8 * ch + e].x == m[ch]) i = 2 * e;
            }
            best = m[ch];
            bidx = c * kTile + half * 64 + ch * 16 + i;
          }
      }
      if (k == nt - 1 || c == nb - 1) {  // the row block ends here: one partial per column half
        const int row = rb * kTile + quarter * 32 + lane;
        const int part = 2 * ((int)blockIdx.x - best_first(rb, nb, per)) + half;
        if (row < n) {
          prow_v[(size_t)part * n + row] = best;
          prow_i[(size_t)part * n + row] = bidx;
        }
        best = -INFINITY;
        bidx = 0x7fffffff;
      }
      if (++c == nb) {
        c = 0;
        ++rb;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kTmemCols) : "memory");
  }
}

// Fixed-order reductions of the per-tile partials: a CTA takes 32 rows (or
// columns), warp g of its 8 the partials g, g + 8, ... in ascending order
// (coalesced over the 32 rows), then the 8 warp results are combined in order.
constexpr int kRedRows = 32;
constexpr int kRedWarps = 8;

__global__ void __launch_bounds__(kRedRows * kRedWarps) k_pmm_lse(const float* __restrict__ part, int nb, int n,
                                                                  float inv_tau, float* __restrict__ lse,
                                                                  float* __restrict__ nlse) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  __shared__ float sp[kRedWarps][kRedRows];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int i = blockIdx.x * kRedRows + lane;
  float s = 0.0f;
  if (i < n) {
#pragma unroll 4
    for (int b = g; b < nb; b += kRedWarps) s += part[(size_t)b * n + i];
  }
  sp[g][lane] = s;
  __syncthreads();
  if (g == 0) {
    float t = sp[0][lane];
#pragma unroll
    for (int k = 1; k < kRedWarps; ++k) t += sp[k][lane];
    const float l = inv_tau + logf(t);  // log sum exp(M / tau) = 1 / tau + log sum exp((M - 1) / tau)
    if (i < n) lse[i] = l;
    nlse[i] = i < n ? -l : -INFINITY;  // whole blocks of kTile: no column past n is ever the best
  }
}

// the best of a row's partials: two from each CTA that holds tiles of its row block
__global__ void k_pmm_best(const float* __restrict__ pv, const int* __restrict__ pi, int nb, int per, int n,
                           int* __restrict__ best) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int rb = i / kTile, parts = 2 * ((rb * nb + nb - 1) / per - best_first(rb, nb, per) + 1);
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  for (int b = 0; b < parts; ++b) {
    const float v = pv[(size_t)b * n + i];
    const int x = pi[(size_t)b * n + i];
    if (better(v, x, bv, bi)) {
      bv = v;
      bi = x;
    }
  }
  best[i] = bi;
}

// the coarse similarity of two split codes, with the three products of the
// tiles; 16-byte loads (two-byte ones made this chain of 128 dependent loads
// the whole kernel: 20 us for 32,400 cells)
__device__ __forceinline__ float dot_codes(const __nv_bfloat16* a, const __nv_bfloat16* b) {
  uint4 ua[kCode / 8], ub[kCode / 8];
#pragma unroll
  for (int k = 0; k < kCode / 8; ++k) {
    ua[k] = reinterpret_cast<const uint4*>(a)[k];
    ub[k] = reinterpret_cast<const uint4*>(b)[k];
  }
  auto val = [](const uint4 (&u)[kCode / 8], int k) {  // bf16 k as binary32
    const uint4 v = u[k >> 3];
    const int q = (k >> 1) & 3;
    const uint32_t x = q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w;
    return __uint_as_float((k & 1) ? x & 0xffff0000u : x << 16);
  };
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < kC; ++k) {
    const float ah = val(ua, k), al = val(ua, kC + k), bh = val(ub, k), bl = val(ub, kC + k);
    s = fmaf(ah, bh, fmaf(al, bh, fmaf(ah, bl, s)));
  }
  return s;
}

// mutual nearest neighbours: flag[i] = 1 when query cell i and rendered cell
// row_best[i] are each other's argmax, with P_M of the pair (an argmax left at
// its sentinel by non-finite features matches nothing). After a timed-out
// tile pass (*err set) nothing matches, so the fine level has no work.
__global__ void k_pmm_mnn(int n, const int* __restrict__ row_best, const int* __restrict__ col_best,
                          const __nv_bfloat16* __restrict__ cq, const __nv_bfloat16* __restrict__ cr,
                          const float* __restrict__ lse_row, const float* __restrict__ lse_col, float s_two,
                          int* __restrict__ flag, float* __restrict__ prob, const int* __restrict__ err) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (*err) {
    flag[i] = 0;
    return;
  }
  const int j = row_best[i];
  const bool mutual = j >= 0 && j < n && col_best[j] == i;
  flag[i] = mutual ? 1 : 0;
  if (mutual) prob[i] = expf(dot_codes(cq + (size_t)i * kCode, cr + (size_t)j * kCode) * s_two - lse_row[i] - lse_col[j]);
}

// the matches at their scanned positions, in ascending query order
__global__ void k_pmm_mnn_scatter(int n, const int* __restrict__ row_best, const int* __restrict__ flag,
                                  const int* __restrict__ off, const float* __restrict__ prob_in,
                                  int* __restrict__ coarse, float* __restrict__ prob) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || !flag[i]) return;
  const int pos = off[i];
  coarse[2 * pos] = i;
  coarse[2 * pos + 1] = row_best[i];
  prob[pos] = prob_in[i];
}

// ---------------------------------------------------------------------------
// fine level: one CTA of 64 threads per coarse match. Both windows (8 x 8
// pixels x 32 channels) arrive by TMA, one box each, channel-major as the
// product reads them. The 64 x 64 similarities are a register-tiled product:
// thread (ti, tj) of the 8 x 8 thread grid holds rows 4 ti + {0..3},
// 32 + 4 ti + {0..3} times the same of tj's columns: four 16-byte shared reads
// per channel for 64 FMAs in packed pairs. Every similarity is one FMA chain in
// channel order. The window sums run along the rows and down the columns in
// order from shared memory, on exponentials taken once; both argmaxes stay in
// registers.
// What bounds it is the shared-memory pipe: a 16-byte read takes four
// wavefronts whatever its lanes share, so 64 accumulators from 16-byte
// broadcasts of one side (306 us for 23,448 windows) lost to the 8 x 8 tile
// (295 us), and loading the windows through registers cost more wavefronts than
// the product. Now 263 us;
// 418 us with the windows loaded through registers, a row pair per
// thread against broadcast columns and the exponentials taken twice.
// ---------------------------------------------------------------------------
constexpr int kEs = kWin + 4;  // row stride of the 64 x 64 buffer: 16-byte rows, float4 reads by row conflict-free

// (value, index) argmax across the lanes that differ in bit `o`
__device__ __forceinline__ void best_xor(float& v, int& i, int o) {
  const float ov = __shfl_xor_sync(0xffffffffu, v, o);
  const int oi = __shfl_xor_sync(0xffffffffu, i, o);
  if (better(ov, oi, v, i)) {
    v = ov;
    i = oi;
  }
}

// the box of one window: 8 x 8 pixels at (x, y), all channels
__device__ __forceinline__ void load_window(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(0), "r"(bar)
      : "memory");
}

__global__ void __launch_bounds__(kWin, 8) k_pmm_fine(const __grid_constant__ CUtensorMap map_q,
                                                      const __grid_constant__ CUtensorMap map_r, int W, int Wc,
                                                      const int* __restrict__ coarse, float inv_tau, float s_exp,
                                                      float s_two, int* __restrict__ slot_r, float* __restrict__ slot_p,
                                                      int* __restrict__ win_count, const int* __restrict__ n_coarse,
                                                      int* __restrict__ err) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  // the unit vectors, channel-major (query, then rendered); then the window's
  // exponentials; then its similarities
  __shared__ __align__(128) float buf[kWin * kEs];
  __shared__ unsigned long long load_bar;
  __shared__ __align__(16) float lr[kWin], lc[kWin];
  __shared__ float cv[2][kWin];  // column argmax of each warp's rows
  __shared__ int ci_s[2][kWin];
  __shared__ int rbest[kWin], cbest[kWin];
  static_assert(2 * kC * kWin <= kWin * kEs, "the unit vectors fit in the window buffer");
  const int k = blockIdx.x, a = threadIdx.x;
  if (k >= *n_coarse) return;  // launched for every cell; the coarse count is known on the device only
  const int ci = coarse[2 * k], cj = coarse[2 * k + 1];
  float* qT = buf;
  float* rT = buf + kC * kWin;
  const uint32_t bar = smem_u32(&load_bar);
  if (a == 0) {
    bar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    bar_expect(bar, 2 * kC * kWin * 4);
    load_window(smem_u32(qT), &map_q, (ci % Wc) * kRatio, (ci / Wc) * kRatio, bar);
    load_window(smem_u32(rT), &map_r, (cj % Wc) * kRatio, (cj / Wc) * kRatio, bar);
  }
  __syncthreads();
  if (__syncthreads_or(!mbar_wait(bar, 0u, kWaitLimit))) {  // the windows never arrived: reported, drained
    if (a == 0) atomicExch(err, 1);
    win_count[k] = 0;
    mbar_wait(bar, 0u, kWaitLimit);
    return;
  }
  {  // thread a normalises query vector a and rendered vector a in place (fp32, channel order)
    float vq[kC], vr[kC];
    float sq = 0.0f, sr = 0.0f;
#pragma unroll
    for (int c = 0; c < kC; ++c) {
      vq[c] = qT[c * kWin + a];
      vr[c] = rT[c * kWin + a];
    }
#pragma unroll
    for (int c = 0; c < kC; ++c) {
      sq = fmaf(vq[c], vq[c], sq);
      sr = fmaf(vr[c], vr[c], sr);
    }
    const float iq = sq > 0.0f ? 1.0f / sqrtf(sq) : 0.0f, ir = sr > 0.0f ? 1.0f / sqrtf(sr) : 0.0f;
#pragma unroll
    for (int c = 0; c < kC; ++c) {
      qT[c * kWin + a] = vq[c] * iq;
      rT[c * kWin + a] = vr[c] * ir;
    }
  }
  __syncthreads();
  const int ti = a >> 3, tj = a & 7;
  float2 M[8][4];  // row i of the thread's eight; column pairs (0,1), (2,3) of each four
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) M[i][j] = make_float2(0.0f, 0.0f);
#pragma unroll 4
  for (int c = 0; c < kC; ++c) {
    const float4* q4 = reinterpret_cast<const float4*>(qT + c * kWin);
    const float4* r4 = reinterpret_cast<const float4*>(rT + c * kWin);
    const float4 qa = q4[ti], qb = q4[8 + ti], ra = r4[tj], rb = r4[8 + tj];
    const float q[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
    const float2 r[4] = {make_float2(ra.x, ra.y), make_float2(ra.z, ra.w), make_float2(rb.x, rb.y),
                         make_float2(rb.z, rb.w)};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 qq = make_float2(q[i], q[i]);
#pragma unroll
      for (int j = 0; j < 4; ++j) M[i][j] = __ffma2_rn(qq, r[j], M[i][j]);
    }
  }
  __syncthreads();  // the unit vectors are read: the buffer takes the exponentials
  auto row_of = [&](int i) { return i < 4 ? 4 * ti + i : 28 + 4 * ti + i; };
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float4* e4 = reinterpret_cast<float4*>(buf + row_of(i) * kEs);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 x = M[i][2 * h], y = M[i][2 * h + 1];
      e4[8 * h + tj] = make_float4(ex2_ftz((x.x - 1.0f) * s_exp), ex2_ftz((x.y - 1.0f) * s_exp),
                                   ex2_ftz((y.x - 1.0f) * s_exp), ex2_ftz((y.y - 1.0f) * s_exp));
    }
  }
  __syncthreads();
  {  // thread a: row a (its two column halves in order) and column a, each in ascending order
    const float4* e4 = reinterpret_cast<const float4*>(buf + a * kEs);
    float rs[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float s = 0.0f;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 x = e4[8 * h + q];
        s += x.x;
        s += x.y;
        s += x.z;
        s += x.w;
      }
      rs[h] = s;
    }
    lr[a] = inv_tau + logf(rs[0] + rs[1]);
    float cs = 0.0f;
#pragma unroll 16
    for (int i = 0; i < kWin; ++i) cs += buf[i * kEs + a];
    lc[a] = inv_tau + logf(cs);
  }
  __syncthreads();
  {
    const float4* lc4 = reinterpret_cast<const float4*>(lc);
    const float4* lr4 = reinterpret_cast<const float4*>(lr);
    const float4 ca = lc4[tj], cb = lc4[8 + tj], ra = lr4[ti], rb = lr4[8 + ti];
    const float lcv[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
    const float lrv[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
    float bv[8];
    int bi[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      bv[j] = -INFINITY;
      bi[j] = 0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = row_of(i);
      float rv = -INFINITY;
      int ri = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {  // ascending columns (rows): the first maximum stays
        const float m = (j & 1) ? M[i][j >> 1].y : M[i][j >> 1].x;
        const float vr = fmaf(m, s_two, -lcv[j]), vc = fmaf(m, s_two, -lrv[i]);
        if (vr > rv) {
          rv = vr;
          ri = j < 4 ? 4 * tj + j : 28 + 4 * tj + j;
        }
        if (vc > bv[j]) {
          bv[j] = vc;
          bi[j] = row;
        }
      }
      best_xor(rv, ri, 1);
      best_xor(rv, ri, 2);
      best_xor(rv, ri, 4);
      if (tj == i) rbest[row] = ri;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      best_xor(bv[j], bi[j], 8);
      best_xor(bv[j], bi[j], 16);
      const int col = j < 4 ? 4 * tj + j : 28 + 4 * tj + j;
      if ((ti & 3) == (j & 3)) {
        cv[a >> 5][col] = bv[j];
        ci_s[a >> 5][col] = bi[j];
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float4* m4 = reinterpret_cast<float4*>(buf + row_of(i) * kEs);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        m4[8 * h + tj] = make_float4(M[i][2 * h].x, M[i][2 * h].y, M[i][2 * h + 1].x, M[i][2 * h + 1].y);
    }
  }
  __syncthreads();
  cbest[a] = better(cv[1][a], ci_s[1][a], cv[0][a], ci_s[0][a]) ? ci_s[1][a] : ci_s[0][a];
  __syncthreads();
  const int b = rbest[a];
  const bool mutual = cbest[b] == a;
  const int by = (cj / Wc) * kRatio + b / kRatio, bx = (cj % Wc) * kRatio + b % kRatio;
  slot_r[(size_t)k * kWin + a] = mutual ? by * W + bx : -1;
  slot_p[(size_t)k * kWin + a] = mutual ? expf(buf[a * kEs + b] * s_two - lr[a] - lc[b]) : 0.0f;
  const unsigned bal = __ballot_sync(0xffffffffu, mutual);
  if ((a & 31) == 0) rbest[a] = __popc(bal);  // this warp's rows are read (its own entries): reuse for the warp counts
  __syncthreads();
  if (a == 0) win_count[k] = rbest[0] + rbest[32];
}

// exclusive scan of n_win counts (one CTA): offsets and the total. A warp takes
// 1,024 consecutive counts, eight 16-byte loads per lane all in flight at once
// (one load per step of a serial loop: 11 us for 32,400 counts).
constexpr int kScanSteps = 8;
__global__ void __launch_bounds__(kScanThreads) k_pmm_scan(int n_win, const int* __restrict__ cnt,
                                                           int* __restrict__ off, int* __restrict__ total,
                                                           const int* __restrict__ n_dev) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  __shared__ uint32_t wsum[2][32];
  if (n_dev) n_win = *n_dev;  // a count produced on the device (the coarse matches)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t carry = 0;
  int buf = 0;
  for (int base = 0; base < n_win; base += kScanThreads * 4 * kScanSteps, buf ^= 1) {  // block-uniform
    const int k0 = base + w * (128 * kScanSteps) + 4 * lane;
    int4 c[kScanSteps];
#pragma unroll
    for (int i = 0; i < kScanSteps; ++i) {
      const int k = k0 + 128 * i;
      c[i] = make_int4(0, 0, 0, 0);
      if (k + 3 < n_win) {
        c[i] = *reinterpret_cast<const int4*>(cnt + k);
      } else {
        if (k < n_win) c[i].x = cnt[k];
        if (k + 1 < n_win) c[i].y = cnt[k + 1];
        if (k + 2 < n_win) c[i].z = cnt[k + 2];
      }
    }
    uint32_t excl[kScanSteps], run = 0;  // before this lane's four of step i, in the warp
#pragma unroll
    for (int i = 0; i < kScanSteps; ++i) {
      const uint32_t t4 = (uint32_t)(c[i].x + c[i].y + c[i].z + c[i].w);
      uint32_t incl = t4;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      excl[i] = run + incl - t4;
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) wsum[buf][w] = run;
    __syncthreads();
    const uint32_t x = wsum[buf][lane];
    uint32_t y = x;  // every warp scans the 32 warp sums
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += t;
    }
    const uint32_t before = carry + __shfl_sync(0xffffffffu, y - x, w);
    carry += __shfl_sync(0xffffffffu, y, 31);
#pragma unroll
    for (int i = 0; i < kScanSteps; ++i) {
      const int k = k0 + 128 * i;
      const int a = (int)(before + excl[i]), b = a + c[i].x, d = b + c[i].y, e = d + c[i].z;
      if (k + 3 < n_win) {
        *reinterpret_cast<int4*>(off + k) = make_int4(a, b, d, e);
      } else {
        if (k < n_win) off[k] = a;
        if (k + 1 < n_win) off[k + 1] = b;
        if (k + 2 < n_win) off[k + 2] = d;
      }
    }
  }
  if (threadIdx.x == 0) *total = (int)carry;
}

// fine matches of window k at its offset, in query-pixel order: two warps per
// window, kScatterWins windows per CTA
constexpr int kScatterWins = 4;
__global__ void __launch_bounds__(kScatterWins* kWin) k_pmm_fine_scatter(
    int W, int Wc, const int* __restrict__ coarse, const int* __restrict__ slot_r, const float* __restrict__ slot_p,
    const int* __restrict__ off, int* __restrict__ fine, float* __restrict__ prob, const int* __restrict__ n_coarse) {
  gsr::pdl_wait();
  gsr::pdl_trigger();
  __shared__ int first[kScatterWins];  // matches of each window's first warp
  const int wi = threadIdx.x / kWin, a = threadIdx.x % kWin, k = blockIdx.x * kScatterWins + wi;
  const bool in = k < *n_coarse;
  const int r = in ? slot_r[(size_t)k * kWin + a] : -1;
  const unsigned bal = __ballot_sync(0xffffffffu, r >= 0);
  if (a == 0) first[wi] = __popc(bal);
  __syncthreads();
  if (r < 0) return;
  const int pos = off[k] + (a >= 32 ? first[wi] : 0) + __popc(bal & ((1u << (a & 31)) - 1u));
  const int ci = coarse[2 * k];
  const int qy = (ci / Wc) * kRatio + a / kRatio, qx = (ci % Wc) * kRatio + a % kRatio;
  fine[3 * pos] = k;
  fine[3 * pos + 1] = qy * W + qx;
  fine[3 * pos + 2] = r;
  prob[pos] = slot_p[(size_t)k * kWin + a];
}

}  // namespace

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
struct gs_pmm {
  int device = 0, sm_count = 1;
  int C = 0, H = 0, W = 0, Hc = 0, Wc = 0, n = 0, nb = 0;
  int per = 1;  // tiles per CTA of pass 2
  void* arena = nullptr;
  __nv_bfloat16 *codes_q = nullptr, *codes_r = nullptr;
  // the codes in the tensor-core operand layout; paired_q: rows of pass 1
  unsigned char *tiled_q = nullptr, *tiled_r = nullptr, *paired_q = nullptr;
  float *prow_v = nullptr, *pcol_v = nullptr, *lse_row = nullptr, *lse_col = nullptr;
  float *nlse_row = nullptr, *nlse_col = nullptr;  // negated, whole blocks of kTile
  int *prow_i = nullptr, *row_best = nullptr, *col_best = nullptr;
  int *coarse = nullptr, *fine = nullptr, *slot_r = nullptr, *counters = nullptr, *win_cnt = nullptr,
      *win_off = nullptr;
  float *coarse_p = nullptr, *fine_p = nullptr, *slot_p = nullptr;
  int* host = nullptr;  // pinned: counts and error flag
  int wait_limit = kWaitLimit;  // polls of a tensor-core completion wait
};

namespace {

gs_status pmm_fail(gs_status st, const std::string& msg) {
  gsr::set_last_error(msg);
  return st;
}

#define PMM_CUDA(x)                                                                    \
  do {                                                                                 \
    const cudaError_t e_ = (x);                                                        \
    if (e_ != cudaSuccess) return pmm_fail(GS_ERR_CUDA, std::string(#x) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// the driver's tensor-map encoder, looked up once
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

// a (kC, H, W) binary32 map read in boxes of one window
bool window_map(const float* F, int H, int W, CUtensorMap* map) {
  const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
  if (!encode) return false;
  const cuuint64_t dim[3] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)kC};
  const cuuint64_t stride[2] = {(cuuint64_t)W * 4, (cuuint64_t)W * H * 4};  // bytes; W is a multiple of 8
  const cuuint32_t box[3] = {kRatio, kRatio, kC}, step[3] = {1, 1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(F), dim, stride, box, step,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

extern "C" {

gs_status gs_pmm_create(int channels, int height, int width, gs_pmm** out) {
  if (!out) return pmm_fail(GS_ERR_INVALID_ARG, "out is required");
  *out = nullptr;
  if (channels != kC) return pmm_fail(GS_ERR_INVALID_ARG, "PMM needs 32 feature channels");
  if (height < kRatio || width < kRatio || height % kRatio || width % kRatio || height > 8192 || width > 8192)
    return pmm_fail(GS_ERR_INVALID_ARG, "feature maps must be 8..8192 pixels, multiples of 8");
  const int Hc = height / kRatio, Wc = width / kRatio, n = Hc * Wc;
  if (n > kMaxCells) return pmm_fail(GS_ERR_INVALID_ARG, "more than 2^18 coarse cells");
  gs_pmm* m = new gs_pmm();
  m->C = channels;
  m->H = height;
  m->W = width;
  m->Hc = Hc;
  m->Wc = Wc;
  m->n = n;
  m->nb = (n + kTile - 1) / kTile;
  cudaError_t e = cudaGetDevice(&m->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, m->device);
  // the tile passes' shared memory, on this matcher's device
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_pmm_sums, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSumSmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_pmm_argmax, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBestSmemBytes);
  // pass 2: two CTAs per SM, equal runs of tiles
  const int tiles = m->nb * m->nb, ctas = std::min(tiles, 2 * m->sm_count);
  m->per = (tiles + ctas - 1) / ctas;
  const size_t nn = (size_t)n, part = (size_t)m->nb * nn;
  const size_t bpart = std::max<size_t>(m->nb, 2 * best_parts(m->nb, m->per)) * nn;  // pass 2's partials
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align_up(off + bytes);
    return o;
  };
  const size_t o_cq = take(nn * kCode * 2), o_cr = take(nn * kCode * 2);
  const size_t tiled_bytes = (size_t)m->nb * kTileBytes;  // whole blocks: rows past n stay zero
  const size_t o_tq = take(tiled_bytes), o_pq = take(tiled_bytes + kTileBytes), o_tr = take(tiled_bytes);
  const size_t o_prv = take(bpart * 4), o_pri = take(bpart * 4), o_pcv = take(part * 4);
  const size_t o_nlr = take((size_t)m->nb * kTile * 4), o_nlc = take((size_t)m->nb * kTile * 4);
  const size_t o_lr = take(nn * 4), o_lc = take(nn * 4), o_rb = take(nn * 4), o_cb = take(nn * 4);
  const size_t o_co = take(nn * 8), o_cp = take(nn * 4);
  const size_t o_sr = take(nn * kWin * 4), o_sp = take(nn * kWin * 4);
  const size_t o_fi = take(nn * kWin * 12), o_fp = take(nn * kWin * 4);
  const size_t o_wc = take(nn * 4), o_wo = take(nn * 4);
  const size_t o_ct = take(4 * 4);
  if (e == cudaSuccess) e = cudaMalloc(&m->arena, off);
  // rows of the tiled codes past n are never written: zero operands of the ragged last block
  if (e == cudaSuccess) e = cudaMemset(static_cast<char*>(m->arena) + o_tq, 0, o_tr + tiled_bytes - o_tq);
  if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&m->host), 4 * sizeof(int));
  if (e != cudaSuccess) {
    gs_pmm_destroy(m);
    return pmm_fail(e == cudaErrorMemoryAllocation ? GS_ERR_OOM : GS_ERR_CUDA,
                    std::string("gs_pmm_create: ") + cudaGetErrorString(e));
  }
  char* base = static_cast<char*>(m->arena);
  m->codes_q = reinterpret_cast<__nv_bfloat16*>(base + o_cq);
  m->codes_r = reinterpret_cast<__nv_bfloat16*>(base + o_cr);
  m->tiled_q = reinterpret_cast<unsigned char*>(base + o_tq);
  m->tiled_r = reinterpret_cast<unsigned char*>(base + o_tr);
  m->paired_q = reinterpret_cast<unsigned char*>(base + o_pq);
  m->prow_v = reinterpret_cast<float*>(base + o_prv);
  m->prow_i = reinterpret_cast<int*>(base + o_pri);
  m->pcol_v = reinterpret_cast<float*>(base + o_pcv);
  m->nlse_row = reinterpret_cast<float*>(base + o_nlr);
  m->nlse_col = reinterpret_cast<float*>(base + o_nlc);
  m->lse_row = reinterpret_cast<float*>(base + o_lr);
  m->lse_col = reinterpret_cast<float*>(base + o_lc);
  m->row_best = reinterpret_cast<int*>(base + o_rb);
  m->col_best = reinterpret_cast<int*>(base + o_cb);
  m->coarse = reinterpret_cast<int*>(base + o_co);
  m->coarse_p = reinterpret_cast<float*>(base + o_cp);
  m->slot_r = reinterpret_cast<int*>(base + o_sr);
  m->slot_p = reinterpret_cast<float*>(base + o_sp);
  m->fine = reinterpret_cast<int*>(base + o_fi);
  m->fine_p = reinterpret_cast<float*>(base + o_fp);
  m->win_cnt = reinterpret_cast<int*>(base + o_wc);
  m->win_off = reinterpret_cast<int*>(base + o_wo);
  m->counters = reinterpret_cast<int*>(base + o_ct);
  *out = m;
  return GS_OK;
}

gs_status gs_pmm_set_wait_limit(gs_pmm* m, int polls) {
  if (!m) return pmm_fail(GS_ERR_INVALID_ARG, "matcher is NULL");
  if (polls < 0) return pmm_fail(GS_ERR_INVALID_ARG, "polls must be >= 0");
  m->wait_limit = polls;
  return GS_OK;
}

gs_status gs_pmm_shape(const gs_pmm* m, int* channels, int* height, int* width) {
  if (!m) return pmm_fail(GS_ERR_INVALID_ARG, "matcher is NULL");
  if (channels) *channels = m->C;
  if (height) *height = m->H;
  if (width) *width = m->W;
  return GS_OK;
}

void gs_pmm_destroy(gs_pmm* m) {
  if (!m) return;
  cudaSetDevice(m->device);
  if (m->arena) {
    cudaDeviceSynchronize();
    cudaFree(m->arena);
  }
  if (m->host) cudaFreeHost(m->host);
  delete m;
}

gs_status gs_pmm_match(gs_pmm* m, const float* feat_query, const float* feat_render, float tau,
                       gs_pmm_result* out, void* stream) {
  gsr::set_last_error("");
  if (!m || !feat_query || !feat_render || !out) return pmm_fail(GS_ERR_INVALID_ARG, "matcher, maps and out are required");
  if (((uintptr_t)feat_query | (uintptr_t)feat_render) & 15u)
    return pmm_fail(GS_ERR_INVALID_ARG, "feature maps must be 16-byte aligned");
  if (!(tau >= 0.025f) || !std::isfinite(tau)) return pmm_fail(GS_ERR_INVALID_ARG, "tau must be finite and >= 0.025");
  PMM_CUDA(cudaSetDevice(m->device));
  const cudaStream_t st = (cudaStream_t)stream;
  const int n = m->n, nb = m->nb;
  CUtensorMap map_q, map_r;
  if (!window_map(feat_query, m->H, m->W, &map_q) || !window_map(feat_render, m->H, m->W, &map_r))
    return pmm_fail(GS_ERR_CUDA, "cuTensorMapEncodeTiled failed");
  const float inv_tau = 1.0f / tau;
  const float s_exp = 1.4426950408889634f * inv_tau;  // exp(x / tau) = exp2(x log2(e) / tau)
  const float s_two = 2.0f * inv_tau;
  PMM_CUDA(cudaMemsetAsync(m->counters, 0, 4 * sizeof(int), st));
  const dim3 cgrid((unsigned)((m->Wc + 31) / 32), (unsigned)m->Hc, 2);
  const CodeMap mq{feat_query, reinterpret_cast<unsigned short*>(m->codes_q), m->tiled_q, m->paired_q};
  const CodeMap mr{feat_render, reinterpret_cast<unsigned short*>(m->codes_r), m->tiled_r, nullptr};
  k_pmm_codes<<<cgrid, 1024, 0, st>>>(mq, mr, m->H, m->W, m->Wc);
  PMM_CUDA(cudaGetLastError());
  const int tiles = nb * nb;
  const unsigned char* cq = m->tiled_q;
  const unsigned char* cr = m->tiled_r;
  int* err = m->counters + 3;
  const int rg = (n + 255) / 256;
  // pass 1: row and column exp sums, then the log-sum-exps
  const int stiles = (nb + 1) / 2 * nb;
  const int sctas = std::min(stiles, 2 * m->sm_count), sper = (stiles + sctas - 1) / sctas;
  // every kernel from here on starts early: thirteen short and long ones in a
  // row, whose launches and block scheduling hide behind one another (1080p maps
  // 1331 -> 1301 us, three localisations of 960 x 540 views, with the solver's
  // early starts, 2335 -> 2174 us)
  auto go = [&](auto kernel, int grid, int block, size_t smem, auto... args) -> cudaError_t {
    return gsr::launch_dependent(true, kernel, dim3((unsigned)grid), block, smem, st, args...);
  };
  PMM_CUDA(go(k_pmm_sums, (stiles + sper - 1) / sper, kSumThreads, kSumSmemBytes, m->paired_q, cr, n, nb, sper, s_exp,
              m->prow_v, m->pcol_v, err, m->wait_limit));
  const int rd = nb * (kTile / kRedRows);
  PMM_CUDA(go(k_pmm_lse, rd, kRedRows * kRedWarps, 0, m->prow_v, nb, n, inv_tau, m->lse_row, m->nlse_row));
  PMM_CUDA(go(k_pmm_lse, rd, kRedRows * kRedWarps, 0, m->pcol_v, nb, n, inv_tau, m->lse_col, m->nlse_col));
  // pass 2: row argmax of log P_M, then (operands swapped) its column argmax
  const int per = m->per, bgrid = (tiles + per - 1) / per;
  PMM_CUDA(go(k_pmm_argmax, bgrid, kRoleThreads, kBestSmemBytes, cq, cr, n, nb, per, s_two, m->nlse_col, m->prow_v,
              m->prow_i, err, m->wait_limit));
  PMM_CUDA(go(k_pmm_best, rg, 256, 0, m->prow_v, m->prow_i, nb, per, n, m->row_best));
  PMM_CUDA(go(k_pmm_argmax, bgrid, kRoleThreads, kBestSmemBytes, cr, cq, n, nb, per, s_two, m->nlse_row, m->prow_v,
              m->prow_i, err, m->wait_limit));
  PMM_CUDA(go(k_pmm_best, rg, 256, 0, m->prow_v, m->prow_i, nb, per, n, m->col_best));
  // mutual nearest neighbours in ascending query order
  PMM_CUDA(go(k_pmm_mnn, rg, 256, 0, n, m->row_best, m->col_best, m->codes_q, m->codes_r, m->lse_row, m->lse_col,
              s_two, m->win_cnt, m->slot_p, err));
  PMM_CUDA(go(k_pmm_scan, 1, kScanThreads, 0, n, m->win_cnt, m->win_off, m->counters, nullptr));
  PMM_CUDA(go(k_pmm_mnn_scatter, rg, 256, 0, n, m->row_best, m->win_cnt, m->win_off, m->slot_p, m->coarse, m->coarse_p));
  // fine level without a round trip: one CTA per cell (the most coarse matches
  // there can be); those past the device-side coarse count return at once
  PMM_CUDA(go(k_pmm_fine, n, kWin, 0, map_q, map_r, m->W, m->Wc, m->coarse, inv_tau, s_exp, s_two, m->slot_r,
              m->slot_p, m->win_cnt, m->counters, err));
  PMM_CUDA(go(k_pmm_scan, 1, kScanThreads, 0, 0, m->win_cnt, m->win_off, m->counters + 1, m->counters));
  PMM_CUDA(go(k_pmm_fine_scatter, (n + kScatterWins - 1) / kScatterWins, kScatterWins * kWin, 0, m->W, m->Wc, m->coarse,
              m->slot_r, m->slot_p, m->win_off, m->fine, m->fine_p, m->counters));
  PMM_CUDA(cudaMemcpyAsync(m->host, m->counters, 4 * sizeof(int), cudaMemcpyDeviceToHost, st));
  PMM_CUDA(cudaStreamSynchronize(st));
  if (m->host[3])
    return pmm_fail(GS_ERR_TIMEOUT, "a tensor-core completion wait ran out of polls (limit " +
                                        std::to_string(m->wait_limit) + "); the matcher stays usable");
  const int n_coarse = m->host[0];
  out->n_cells = n;
  out->codes_q = reinterpret_cast<const uint16_t*>(m->codes_q);
  out->codes_r = reinterpret_cast<const uint16_t*>(m->codes_r);
  out->lse_row = m->lse_row;
  out->lse_col = m->lse_col;
  out->row_best = m->row_best;
  out->col_best = m->col_best;
  out->n_coarse = n_coarse;
  out->coarse = m->coarse;
  out->coarse_prob = m->coarse_p;
  out->n_fine = m->host[1];
  out->fine = m->fine;
  out->fine_prob = m->fine_p;
  return GS_OK;
}

}  // extern "C"
