// Chains of weight products for a decode step, without split-K partial sums in global memory.
//
// What bounds it: HBM.  A step's products are short (a 4096 x 4096 matrix is 5 us of HBM time), so
// what matters beside the stream itself is how long HBM idles where one product hands over to the
// next.  The kernels of kernels_gemv.cu cut every product over all threadblocks along K and meet
// in L2: partial sums out, a grid-wide counter, the combine, a second counter, the next
// product's activations - 6 to 10 us per product, more at large batches.  Here a product is cut
// along its ROWS, and along K only between the two threadblocks of a cluster, whose halves meet in
// distributed shared memory: no partial sum touches global memory, one grid-wide counter per
// product is left, and the last product of a launch needs no combine kernel behind it.
//
// Rows are cut in units of 4 + 4 (rows i .. i + 3 and i + 64 .. i + 67 of a 128-row tile: gate / up
// partners and the two halves of a rotary pair stay together), because 148 SMs do not divide the
// 32 - 48 row tiles of a short product: 512 units over 74 clusters are 6.92 each (98.8 %).  A
// weight block stores its rows one after the other (128 bytes each), so a run of units is two
// contiguous pieces of every block of the row tile.  In shared memory a run of up to 16 (or 8)
// units is an IMAGE of a row tile: unit u sits where it sits in its tile, modulo 16 (8), lower
// rows first, upper rows behind them, so a run that crosses a tile boundary wraps around and
// always costs two to four bulk copies.  An image is the A operand of tcgen05.mma (M = 128); rows
// of it that are not this threadblock's are whatever shared memory holds there - they only reach
// accumulator lanes that nobody reads.  Images of 8 units come in twos, k blocks kb and kb + 1
// behind each other, and are multiplied with M = 64.  (Both as one operand of M = 128 against both
// activation tiles side by side took fewer MMAs and the same time, but half of its results were
// nobody's: at batch 32 the GPU is at its power limit, and a step of 4690 us became one of 4640.)
//
// One threadblock per SM.  Up to 32 batch rows it takes 147 KiB of shared memory and 88 registers per
// thread at most: a threadblock of the attention kernel before and after it on the stream fits beside it, and
// the weights of the first product are in place when the kernel before it ends.  A ring of 64 KiB
// per SM already saturates HBM (measured with bulk copies of 2 - 16 KiB: 48 KiB 6.3, 64 KiB 6.8, 80
// - 112 KiB 6.9, 192 KiB 6.4 - 6.7 TB/s), so sharing the SM costs no bandwidth.  Larger batches take
// the whole SM: their activation tiles are up to 32 KiB each.
//
// Warps: 0 and 3 weight producers (a pipeline each, or every other stage: one warp's instruction latency
// would bound the stream of a product whose stages are four or eight copies), 1 activation producer, 2 MMA
// issue and tensor-memory allocation, 4 and up epilogue, behind them (up to 128 rows) the second
// pipeline's MMA issue and (128 rows) activation producer.  Producers and MMA warps run warp-uniform code
// and elect a lane for the copy or MMA itself: inside an if (lane == 0) every operand goes through a
// vector register (measured: a group of four MMAs and a commit 293 cycles against 212, a bulk copy 64
// against 25).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>

#include "device_common.cuh"
#include "host_common.h"

namespace {

using namespace boostk;

constexpr uint32_t kRowTile = 128;
constexpr uint32_t kBlockBytes = 16384;                        // 128 rows x 64 columns of bf16
constexpr uint32_t kBlocksPerPage = kPageBytes / kBlockBytes;  // 128
constexpr uint32_t kUnitsPerTile = 16;                         // units of 4 + 4 rows
constexpr uint32_t kEpiWarp0 = 4;                              // warps 0 - 3: producers, the first MMA warp; then epilogue, the second MMA warp
constexpr uint32_t kStageBytes = kBlockBytes;                  // one image of 16 units, or two k blocks of an image of 8
constexpr uint32_t kMaxStages = 12, kMaxXSlots = 12;
constexpr uint32_t kMaxPhases = 4;

struct PairPhase {
  const void* const* w_page_ptr;
  const uint32_t* w_order;
  uint32_t n_pages, n_host_pages;
  uint32_t N, K, k_blocks, n_units;
  const __nv_bfloat16* x;
  uint32_t split;            // 2: the cluster's threadblocks take half of K each; 1: every threadblock has rows of its own
  uint32_t image;            // units of an image: 16, or 8 where no worker has more (then a stage holds two k blocks)
  uint32_t max_images;       // images of the widest worker
  uint32_t mode;             // an accumulator holds a quarter of a k block (0), a k block (1), several (2)
  uint32_t slot_blocks;      // k blocks of a slot of accumulators
  void* y;
  int y_dtype;
  const __nv_bfloat16* residual;
  uint32_t epi;              // BOOST_EPI_*
  const float* ssq_in;       // [ssq_parts][ssq_stride] sums of squares of the rows of x, or null
  uint32_t ssq_parts, ssq_stride;
  float x_cols, rms_eps;
  float* ssq_out;            // [ssq_parts_of][kN]: the same for the rows of y (bf16 output), or null
  __nv_bfloat16* q_out;
  const void* const *k_page_ptr, *const *v_page_ptr, *const *k_page_ptr2, *const *v_page_ptr2;
  const int32_t *block_table, *ctx_lens;
  uint32_t n_pool_blocks, max_blocks, Hq, Hkv;
  const float* rope_table;
};

struct PairParams {
  uint32_t n_phases, M_b, nb, n_stages, x_slots;   // nb: activation rows of a tile (the batch rounded up)
  uint32_t early;  // weights and their page tables may be read while the kernel ahead on the stream still runs
  uint32_t* ws;    // workspace header
  uint32_t* bar;   // [0] threadblocks past their last wait, [1] phases finished, summed over the threadblocks; zero at rest
  PairPhase ph[kMaxPhases];
  alignas(64) CUtensorMap x_map[kMaxPhases];   // more than 32 batch rows
};

// kN: the batch class of an instantiation (8, 16, 32, 64, 128, 256 rows).
// Activations by tiled TMA copies, or by one warp's 16-byte copies (measured when both were built: TMA 1.7 % slower
// for a step at batch 1, 1.2 % at 8, 0.8 % at 32; more rows are too many copies for one warp).
__host__ __device__ constexpr bool x_by_tma(uint32_t n) { return n > 32; }
// k blocks of an activation slot.
__host__ __device__ constexpr uint32_t x_blocks(uint32_t n) { return n >= 128 ? 1 : 2; }
// The tensor cores' fp32 adder truncates: every MMA that adds to an accumulator takes about 2.7e-8 of
// what it holds, always towards zero, so a sum over n MMAs is off by n / 2 times that (2-norm against
// fp64, normal inputs, 32 / 128 / 256 MMAs: 4.5e-7, 2.1e-6, 4.4e-6).  An accumulator therefore holds a PART
// of the columns only (plan_parts), and the epilogue warps take the parts out of tensor
// memory as they come and add them up where additions round to nearest.
// Parts of part_cols columns (an M = 128 product has at least 16) change hands in slots of up to
// slot_parts; as many slots as tensor memory holds are in flight.
// Up to 128 rows there are two pipelines (a weight producer, a ring of stages and one of activation slots, an MMA
// warp and accumulators each), which take the chunks of a slot's k blocks in turn: a part that holds several
// blocks has every other chunk.  At 256 rows there is one: its MMAs take longer than what the issuing
// warp does between them, and tensor memory holds two accumulators only.
__host__ __device__ constexpr uint32_t pipes_of(uint32_t n) { return n <= 128 ? 2 : 1; }
__host__ __device__ constexpr uint32_t part_cols(uint32_t n) { return n < 16 ? 16 : n; }
__host__ __device__ constexpr uint32_t slot_parts(uint32_t n) { return n <= 8 ? 16 : n <= 64 ? 4 : n <= 128 ? 2 : 1; }
__host__ __device__ constexpr uint32_t slot_cols(uint32_t n) { return part_cols(n) * slot_parts(n); }
constexpr uint32_t kMaxAccSlots = 8;
__host__ __device__ constexpr uint32_t acc_slots(uint32_t n) { return 512 / slot_cols(n) < kMaxAccSlots ? 512 / slot_cols(n) : kMaxAccSlots; }
__host__ __device__ constexpr uint32_t tmem_cols(uint32_t n) { return acc_slots(n) * slot_cols(n); }
// k blocks of a chunk.  (A slot holds a multiple of that, but at the end of K.)
__host__ __device__ constexpr uint32_t chunk_blocks(uint32_t n, uint32_t image) {
  return pipes_of(n) == 1 ? 1 : image == 8 || x_blocks(n) == 2 ? 2 : 1;
}
// Slots of one chunk go to the pipelines in turn.  (128 rows, images of 8, a k block to an accumulator.  All to the first pipeline,
// half of the ring idle: fp32 results at batch 80, 1000 x 1024 10.65 us, 2048 x 1536 12.9; in turn 10.3, 12.5.)
__host__ __device__ constexpr bool slots_in_turn(uint32_t n, uint32_t image, uint32_t slot_blocks) {
  return n == 128 && slot_blocks == chunk_blocks(n, image);
}
// Activation producers.  (At 128 rows one is too slow for both pipelines: 375 cycles a slot, where the tensor cores take
// 256 and HBM 275; down product 34.2 -> 30.2 us with two.  Fewer rows: slots of two blocks; batch 64 was 0.6 % slower with two.)
__host__ __device__ constexpr uint32_t x_warps(uint32_t n) { return n == 128 ? 2 : 1; }
// Epilogue warps: a short product's last accumulator is finished by all of them at the end of a phase,
// which at large batches is bound by their instruction latency.
__host__ __device__ constexpr uint32_t epi_warps(uint32_t n) { return n <= 32 ? 8 : 16; }
__host__ __device__ constexpr uint32_t threads_of(uint32_t n) { return (kEpiWarp0 + epi_warps(n) + pipes_of(n) - 1 + x_warps(n) - 1) * 32; }
// Sums on their way from tensor memory to the threads that finish them, fp32 [columns][128 lanes].
// Rows of one threadblock: at most this many columns at a time (32 in two buffers in turn were 1.5 % slower than 64
// for a step at batch 250).  128 rows: 32, so that shared memory holds six stages and six activation slots
// (6-layer step at batch 128: 1477 us; six and four 1569, four and eight 1600).  256 rows: 64 or 32 (see wide_chunk).
[[maybe_unused]] __host__ __device__ constexpr uint32_t chunk_cols(uint32_t n) { return n < 64 ? n : n == 128 ? 32 : 64; }
// Rows that two threadblocks share: each finishes half of the columns, in this many rounds.  The
// columns of a round, this threadblock's sums and the peer's, are kept in the chunk buffers
// (up to 32 rows), or this threadblock's in the activation slots, which are idle then, and the peer's in the
// chunk buffer where they fit (64 and 128 rows).
__host__ __device__ constexpr uint32_t rounds_of(uint32_t n) { return n >= 256 ? 2 : 1; }
__host__ __device__ constexpr uint32_t sums_bytes(uint32_t chunk) { return chunk * kRowTile * 4; }

template <auto kValue>
struct Const { static constexpr auto value = kValue; };

// Rows [u0, u1) (in units) of worker w of W.
__host__ __device__ inline void worker_range(uint32_t n_units, uint32_t w, uint32_t W, uint32_t& u0, uint32_t& u1) {
  u0 = (uint32_t)((uint64_t)n_units * w / W);
  u1 = (uint32_t)((uint64_t)n_units * (w + 1) / W);
}

__device__ __forceinline__ uint32_t mapa(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
// Store to another threadblock's shared memory, counted in bytes on a barrier of that threadblock.
__device__ __forceinline__ void st_async_f32(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)),
               "r"(bar)
               : "memory");
}
// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// D[tmem] (+)= A[smem] B[smem]^T, K = 16.  The operands' descriptors (umma_desc_k_sw128) by their low
// words, which hold the address: the issuing warp computes with those alone.  (Without the lane mask
// of umma_bf16, whose four registers cost issue time.)
constexpr uint32_t kDescHigh = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_low(uint32_t smem_addr) { return ((smem_addr >> 4) & 0x3FFFu) | (1u << 16); }
__device__ __forceinline__ void umma_low(uint32_t d_tmem, uint32_t a_low, uint32_t b_low, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_low), "r"(b_low), "r"(idesc), "r"(accumulate), "n"(kDescHigh)
      : "memory");
}
// Columns of this warp's 32 tensor-memory lanes, with the wait for them in the same statement, so that
// nothing is done with the registers before it: 8 at one address, 4, 8 at each of two, 2 at each of eight.
__device__ __forceinline__ void tmem_ld_8(uint32_t addr, float (&v)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
      : "r"(addr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_4(uint32_t addr, float (&v)[4]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
      : "r"(addr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_2x8(uint32_t addr0, uint32_t addr1, float (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=&f"(v[0]), "=&f"(v[1]), "=&f"(v[2]), "=&f"(v[3]), "=&f"(v[4]), "=&f"(v[5]), "=&f"(v[6]), "=&f"(v[7]), "=&f"(v[8]), "=&f"(v[9]),
        "=&f"(v[10]), "=&f"(v[11]), "=&f"(v[12]), "=&f"(v[13]), "=&f"(v[14]), "=&f"(v[15])
      : "r"(addr0), "r"(addr1)
      : "memory");
}
template <uint32_t kStep>
__device__ __forceinline__ void tmem_ld_8x2(uint32_t addr, float (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%16];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%2,%3}, [%17];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%4,%5}, [%18];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%6,%7}, [%19];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%8,%9}, [%20];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%10,%11}, [%21];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%12,%13}, [%22];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%14,%15}, [%23];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=&f"(v[0]), "=&f"(v[1]), "=&f"(v[2]), "=&f"(v[3]), "=&f"(v[4]), "=&f"(v[5]), "=&f"(v[6]), "=&f"(v[7]), "=&f"(v[8]), "=&f"(v[9]),
        "=&f"(v[10]), "=&f"(v[11]), "=&f"(v[12]), "=&f"(v[13]), "=&f"(v[14]), "=&f"(v[15])
      : "r"(addr), "r"(addr + kStep), "r"(addr + 2 * kStep), "r"(addr + 3 * kStep), "r"(addr + 4 * kStep), "r"(addr + 5 * kStep),
        "r"(addr + 6 * kStep), "r"(addr + 7 * kStep)
      : "memory");
}
__device__ __forceinline__ void tmem_st_8(uint32_t addr, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};" ::"f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]),
               "f"(v[5]), "f"(v[6]), "f"(v[7]), "r"(addr)
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Two fp32 additions (round to nearest) in one instruction.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return add2(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float bf16_round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// Barrier operations and copies on shared-memory addresses (the loops below step through them).
__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void arrive_remote(uint32_t bar) {   // bar: an address from mapa
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const uint8_t* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes),
               "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tma_tile(uint32_t dst, const void* map, int32_t c0, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
               "l"(map), "r"(bar), "r"(c0), "r"(0)
               : "memory");
}
__device__ __forceinline__ void cp_async_16s(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// The slow part of a bounded wait: the barrier had not completed at the first try.
__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t* status) {
  const long long limit = wait_limit_of(status);
  const long long t0 = clock64();
  while (!try_wait(bar, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > limit) {
      atomicOr(status, kErrWaitTimeout);
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}

// Schedule log only: bytes of units [u0, u1), blocks [kb0, kb1) of every row, that lie in host pages.
__device__ __noinline__ uint32_t host_bytes_of_range(const PairPhase& q, uint32_t u0, uint32_t u1, uint32_t kb0, uint32_t kb1) {
  uint32_t bytes = 0;
  for (uint32_t t = u0 / kUnitsPerTile; t * kUnitsPerTile < u1; ++t) {
    const uint32_t units = min(u1, (t + 1) * kUnitsPerTile) - max(u0, t * kUnitsPerTile);
    for (uint32_t b = t * q.k_blocks + kb0; b < t * q.k_blocks + kb1;) {
      const uint32_t page = b / kBlocksPerPage, here = min(t * q.k_blocks + kb1 - b, kBlocksPerPage - b % kBlocksPerPage);
      bool host = false;
      for (uint32_t i = 0; i < q.n_host_pages && !host; ++i) host = q.w_order[i] == page;
      if (host) bytes += here * units * 1024u;
      b += here;
    }
  }
  return bytes;
}

// Registers: beside an attention threadblock (up to 32 rows) and within an SM (64, 128) as many as measured best (32 rows: 80 / 88,
// hidden 256, 18 - 30 sequences of 20 - 100 tokens 1.015 / 1.002 of the time before the second pipeline).
template <uint32_t kN, uint32_t kChunk>
__global__ void __maxnreg__(kN >= 256 ? 96 : kN == 32 ? 88 : 80) gemv_pair_kernel(const __grid_constant__ PairParams p) {
  constexpr uint32_t kXB = x_blocks(kN), kSlots = acc_slots(kN), kSlotCols = slot_cols(kN), kPipes = pipes_of(kN);
  constexpr bool kTmaX = x_by_tma(kN);
  constexpr uint32_t kEpiWarps = epi_warps(kN), kEpiThreads = kEpiWarps * 32;
  constexpr bool kBig = kN >= 64;
  constexpr uint32_t CW = kChunk, CH = kBig ? 8 : kN / 2, HG = kEpiWarps / 4;   // columns of a group; warps that share lanes
  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t n_stages = p.n_stages, x_slots = p.x_slots;
  const uint32_t nb = kN <= 32 ? kN : p.nb;               // activation rows of a k block
  const uint32_t x_block = nb * 128u, x_slot = kXB * x_block;
  uint8_t* x_ring = ring + n_stages * kStageBytes;
  // (an 8-row activation tile is read as 16 rows: 1 KiB behind the slots)
  float* sums = reinterpret_cast<float*>(x_ring + x_slot * x_slots + 1024u);
  __shared__ uint64_t w_full[kMaxStages], w_empty[kMaxStages], x_full[kMaxXSlots], x_empty[kMaxXSlots];
  __shared__ uint64_t acc_full[kMaxAccSlots], acc_empty[kMaxAccSlots], xch_full, xch_free, drained[2];
  // The phases after the first may start.  One barrier each: a second activation producer that fills no slot of a
  // phase holds nobody up in it, so its look at one barrier for all could come after the next phase's arrival, where the
  // parity reads as not arrived yet and the wait would not end.
  __shared__ uint64_t go[kMaxPhases - 1];
  __shared__ uint32_t s_tmem;
  __shared__ uint32_t s_rec[kMaxPhases];
  __shared__ float s_rs[kN], s_red[kEpiThreads];
  __shared__ unsigned long long s_dst[2][kN], s_dst2[2][kN];   // rope: rows of the new token, per row tile of the image and sequence
  __shared__ volatile uint32_t s_abort;   // a bounded wait ran out: waits that would block fail at once from then on

  const uint32_t tid = threadIdx.x, lane = tid & 31;
  const uint32_t warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  uint32_t* status = p.ws + kWsStatus;
  const uint32_t n_cta = gridDim.x;

  pdl_launch_dependents();
  auto init_stage = [&](uint32_t s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], 1); };
  auto init_x = [&](uint32_t s) { mbar_init(&x_full[s], kTmaX ? 1 : 32); mbar_init(&x_empty[s], 1); };
  auto init_acc = [&](uint32_t s) { mbar_init(&acc_full[s], kPipes); mbar_init(&acc_empty[s], kEpiWarps); };
  // A lane per barrier (one thread for all 40: short products up to 0.2 us slower).  32 rows: one thread (6-layer 8B steps of
  // 20 / 24 / 32 sequences 896 / 923 / 979 us, with a lane each 899 / 929 / 982).
  if constexpr (kN == 32) {
    if (tid == 0) {
      for (uint32_t s = 0; s < n_stages; ++s) init_stage(s);
      for (uint32_t s = 0; s < x_slots; ++s) init_x(s);
      for (uint32_t s = 0; s < kSlots; ++s) init_acc(s);
      mbar_init(&xch_full, 1);
      mbar_init(&xch_free, 1);
      for (uint32_t i = 0; i < kMaxPhases - 1; ++i) mbar_init(&go[i], 1);
      mbar_init(&drained[0], 1);
      mbar_init(&drained[1], 1);
      s_abort = 0;
      fence_barrier_init();
    }
  } else if (warp == 0) {
    if (lane < n_stages) init_stage(lane);
    if (lane < x_slots) init_x(lane);
    if (lane < kSlots) init_acc(lane);
    if (lane < kMaxPhases - 1) mbar_init(&go[lane], 1);
    if (lane < 2) mbar_init(&drained[lane], 1);
    if (lane == 0) {
      mbar_init(&xch_full, 1);
      mbar_init(&xch_free, 1);
      s_abort = 0;
    }
    fence_barrier_init();
  }
  if (warp == 2) tmem_alloc(&s_tmem, tmem_cols(kN));
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  // (the peer's barriers must exist before anything is stored to it)
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  const uint32_t tmem = s_tmem;

  auto wait = [&](uint32_t bar, uint32_t parity) -> bool { return try_wait(bar, parity) || wait_slow(bar, parity, &s_abort, status); };
  // This threadblock's part of a phase: units [u0, u1) of the rows in images of `run` units (as even as
  // they come: a stage then takes HBM longer than the instructions around it), blocks [kb0, kb1) of K.
  struct Part { uint32_t u0, u1, run, kb0, kb1; };
  auto part_of = [&](const PairPhase& q) -> Part {
    Part r;
    const bool two = q.split == 2;
    worker_range(q.n_units, two ? blockIdx.x >> 1 : blockIdx.x, two ? n_cta >> 1 : n_cta, r.u0, r.u1);
    const uint32_t units = r.u1 - r.u0, images = (units + q.image - 1) / q.image;
    r.run = images ? (units + images - 1) / images : 1u;
    r.kb0 = two ? q.k_blocks * rank / 2 : 0u;
    r.kb1 = two ? q.k_blocks * (rank + 1) / 2 : q.k_blocks;
    return r;
  };
  // A pipeline's stages (activation slots) are behind each other.
  const uint32_t pipe_stages = n_stages / kPipes, pipe_slots = x_slots / kPipes;
  constexpr uint32_t kMma1 = kEpiWarp0 + kEpiWarps, kX1 = kMma1 + 1;   // the second pipeline's MMA warp and activation producer
  // Where a producer warp stands: the stage (activation slot) it would fill next, the parity of its wait for
  // it (one activation producer for two pipelines: stage1, parity1 for the second), and whether it is this
  // warp's turn.  Known at the end of the kernel too, for the wind-down.
  uint32_t stage = 0, parity = 1;
  [[maybe_unused]] uint32_t stage1 = 0, parity1 = 1;
  bool my_turn = kPipes == 2 || warp != 3;

  if (warp == 0 || warp == 3) {
    // ------------------------------------------------------------------ weight producers
    const uint32_t pipe = kPipes == 2 && warp == 3 ? 1u : 0u, first = pipe * pipe_stages;
    const uint32_t ring_a = smem_u32(ring) + first * kStageBytes, full_a = smem_u32(w_full) + first * 8, empty_a = smem_u32(w_empty) + first * 8;
    if (!p.early) {
      pdl_wait();
      fence_proxy_async_all();   // pages written with ordinary stores are read through the TMA unit
    }
    unsigned long long* const log = sched_log_of(p.ws);
    // Two pipelines: each of the two warps has one.  One: they take its stages in turn.
    // Per stage: wait, announce the bytes, copy.  Everything else is kept out of the loop: the lanes
    // hold the pieces' addresses (part of the run x lower / upper rows; x k block of an image of 8), and
    // step through K on their own.
    auto produce = [&](const PairPhase& q, uint32_t ph) -> bool {
      const Part w = part_of(q);
      const uint32_t image = q.image, k_blocks = q.k_blocks, n_pages = q.n_pages;
      [[maybe_unused]] const uint32_t slot_n = q.slot_blocks, chunk = chunk_blocks(kN, image), in_turn = slots_in_turn(kN, image, slot_n);
      const void* const* const page_ptr = q.w_page_ptr;
      const bool twos = image == 8;
      if (warp == 0 && lane == 0) {
        s_rec[ph] = kNoRecord;
        if (log && w.u0 < w.u1)
          s_rec[ph] = sched_log_begin(log, BOOST_SCHED_KIND_GEMV | (ph << 8), blockIdx.x, (w.u1 - w.u0) * (w.kb1 - w.kb0) * 1024u,
                                      q.n_host_pages ? host_bytes_of_range(q, w.u0, w.u1, w.kb0, w.kb1) : 0u);
      }
      __syncwarp();
      const uint32_t step = twos ? 2u : 1u;
      const uint32_t sub = lane >> 2, part = (lane >> 1) & 1u, half = lane & 1u;
      for (uint32_t ua = w.u0; ua < w.u1; ua += w.run) {
        // this lane's piece: units [a, b) of the image's run (its part before or behind the wrap), lower or upper rows, k block kb + second
        const uint32_t second = twos ? sub & 1u : 0u;
        const uint32_t ub = min(w.u1, ua + w.run), mid = min(ub, (ua / image + 1) * image);
        const uint32_t a = part ? mid : ua, b = part ? ub : mid;
        bool mine = sub < step && a < b;
        uint32_t bytes = (b - a) * 512u;
        if (mine && b - a == kUnitsPerTile) {   // a whole row tile is one copy
          bytes = kBlockBytes;
          mine = half == 0;
        }
        const uint32_t to = ring_a + second * (kStageBytes / 2) + half * image * 512u + (a % image) * 512u;
        const uint32_t in_block = (half * 64u + (a % kUnitsPerTile) * 4u) * 128u;
        const uint32_t tile = a / kUnitsPerTile * k_blocks;   // the row tile's first block
        uint32_t page = 0xFFFFFFFFu;
        const uint8_t *base = nullptr, *next = nullptr;   // the page of this piece's block, and the one after it
        const uint32_t tx = (ub - ua) * 1024u * step;
        auto fill = [&](uint32_t kb) -> bool {   // the next stage: block kb (and the next of an image of 8; an odd last one is its own partner: it meets zeros, or nothing)
          if (!wait(empty_a + stage * 8, parity)) return false;
          const uint32_t full = full_a + stage * 8;
          if (lane == 0) expect_tx(full, tx);
          __syncwarp();
          if (mine) {
            const uint32_t blk = tile + min(kb + second, w.kb1 - 1), pg = blk / kBlocksPerPage;
            if (pg != page) {   // (at the start, and where K runs into another page)
              base = pg == page + 1 && next ? next : static_cast<const uint8_t*>(page_ptr[pg]);
              page = pg;
              next = pg + 1 < n_pages ? static_cast<const uint8_t*>(page_ptr[pg + 1]) : nullptr;
            }
            bulk_copy(to + stage * kStageBytes, base + (size_t)(blk % kBlocksPerPage) * kBlockBytes + in_block, bytes, full);
          }
          return true;
        };
        auto next_stage = [&]() { if (++stage == pipe_stages) { stage = 0; parity ^= 1u; } };
        if constexpr (kPipes == 2) {
          uint32_t turn = pipe;   // 0: the slot's first chunk
          for (uint32_t k0 = w.kb0; k0 < w.kb1; k0 += slot_n, turn ^= in_turn) {
            const uint32_t k1 = min(k0 + slot_n, w.kb1);
            for (uint32_t kb = k0 + turn * chunk; kb < k1; kb += 2 * chunk)
              for (uint32_t j = kb; j < min(kb + chunk, k1); j += step) {
                if (!fill(j)) return false;
                next_stage();
              }
          }
        } else {
          for (uint32_t kb = w.kb0; kb < w.kb1; kb += step) {
            if (my_turn && !fill(kb)) return false;
            my_turn = !my_turn;
            next_stage();
          }
        }
      }
      return true;
    };
    for (uint32_t ph = 0; ph < p.n_phases; ++ph)
      if (!produce(p.ph[ph], ph)) break;
  } else if (warp == 1 || (x_warps(kN) == 2 && warp == kX1)) {
    // ------------------------------------------------------------------ activation producers
    // Up to 32 rows: 16-byte copies through the load/store path (the TMA unit works in order, and an
    // activation tile would queue behind the weight copies of a full ring).  Rows beyond the batch are
    // left as they are: they only reach accumulator columns that nobody reads.
    const uint32_t pipe = x_warps(kN) == 1 || warp == 1 ? 0u : 1u;
    const uint32_t x_a = smem_u32(x_ring), full_a = smem_u32(x_full), empty_a = smem_u32(x_empty);
    if constexpr (kTmaX) {
      if (elect_one())
        for (uint32_t ph = 0; ph < p.n_phases; ++ph) tma_prefetch_map(&p.x_map[ph]);
      __syncwarp();
    }
    pdl_wait();
    // fill(kb, xs): the k blocks of slot xs, from kb on.  For every slot of a phase that this warp fills.
    auto each_slot = [&](const PairPhase& q, const Part& w, auto fill) -> bool {
      [[maybe_unused]] auto put = [&](uint32_t kb, uint32_t kb_end, uint32_t first) -> bool {   // into the next slots of this warp's pipeline
        for (; kb < kb_end; kb += kXB) {
          if (!wait(empty_a + (first + stage) * 8, parity)) return false;
          fill(kb, first + stage);
          if (++stage == pipe_slots) { stage = 0; parity ^= 1u; }
        }
        return true;
      };
      for (uint32_t pa = w.u0; pa < w.u1; pa += w.run) {
        if constexpr (kPipes == 1) {
          if (!put(w.kb0, w.kb1, 0)) return false;
        } else {
          const uint32_t chunk = chunk_blocks(kN, q.image), slot_n = q.slot_blocks, in_turn = slots_in_turn(kN, q.image, slot_n);
          uint32_t turn = pipe;
          for (uint32_t k0 = w.kb0; k0 < w.kb1; k0 += slot_n, turn ^= in_turn) {
            const uint32_t k1 = min(k0 + slot_n, w.kb1);
            if constexpr (kXB == 2) {   // a chunk is a slot, and this warp fills both pipelines'
              static_assert(chunk_blocks(kN, 8) == 2 && chunk_blocks(kN, 16) == 2 && x_warps(kN) == 1);
              if constexpr (kN == 32) {   // (6-layer 8B step of 32 sequences 979 us, with the loop below 987; small models of up to 16: that 0.3 - 1 % faster)
                for (uint32_t c = k0; c < k1; c += 4) {
                  if (!wait(empty_a + stage * 8, parity)) return false;
                  fill(c, stage);
                  if (++stage == pipe_slots) { stage = 0; parity ^= 1u; }
                  if (c + 2 < k1) {
                    if (!wait(empty_a + (pipe_slots + stage1) * 8, parity1)) return false;
                    fill(c + 2, pipe_slots + stage1);
                    if (++stage1 == pipe_slots) { stage1 = 0; parity1 ^= 1u; }
                  }
                }
              } else {
                for (uint32_t c = k0; c < k1; c += 2) {
                  const bool second = ((c - k0) & 2u) != 0;
                  const uint32_t at = second ? stage1 : stage, slot = at + (second ? pipe_slots : 0u);
                  if (!wait(empty_a + slot * 8, second ? parity1 : parity)) return false;
                  fill(c, slot);
                  const bool wrap = at + 1 == pipe_slots;
                  if (second) { stage1 = wrap ? 0u : at + 1; parity1 ^= wrap; } else { stage = wrap ? 0u : at + 1; parity ^= wrap; }
                }
              }
            } else {
              static_assert(x_warps(kN) == 2);
              for (uint32_t c = k0 + turn * chunk; c < k1; c += 2 * chunk)
                if (!put(c, min(c + chunk, k1), pipe * pipe_slots)) return false;
            }
          }
        }
      }
      return true;
    };
    auto produce = [&](const PairPhase& q, uint32_t ph) -> bool {
      const Part w = part_of(q);
      const uint32_t K = q.K;
      if constexpr (kTmaX) {
        fence_proxy_async_all();   // x was written with ordinary stores and is read through the TMA unit
        return each_slot(q, w, [&](uint32_t kb, uint32_t xs) {
          if (elect_one()) {
            const uint32_t full = full_a + xs * 8, dst = x_a + xs * x_slot;
            expect_tx(full, x_slot);
            tma_tile(dst, &p.x_map[ph], (int32_t)(kb * 64u), full);
            // (behind an odd last block: columns outside the tensor, which arrive as zeros)
            if constexpr (kXB == 2) tma_tile(dst + x_block, &p.x_map[ph], (int32_t)((kb + 1 < w.kb1 ? kb + 1 : q.k_blocks) * 64u), full);
          }
          __syncwarp();
        });
      } else {
        const uint32_t c = lane & 7, r0 = lane >> 3, M_b = p.M_b;
        const uint32_t to0 = x_a + r0 * 128u + ((c ^ r0) << 4), to1 = x_a + (r0 + 4) * 128u + ((c ^ (r0 + 4)) << 4);   // rows 8 i + r0, 8 i + 4 + r0
        const __nv_bfloat16* const x0 = q.x + (size_t)r0 * K + (c * 8u < K ? c * 8u : 0u);
        return each_slot(q, w, [&](uint32_t kb, uint32_t xs) {
          const uint32_t at = xs * x_slot;
          uint32_t n[kXB], off[kXB];   // bytes and columns; behind the last block, and behind the last column in it, zeros
#pragma unroll
          for (uint32_t b = 0; b < kXB; ++b) {
            const bool in = kb + b < w.kb1 && (kb + b) * 64u + c * 8u < K;
            n[b] = in ? 16u : 0u;
            off[b] = in ? b * 64u : 0u;
          }
          const __nv_bfloat16* src = x0 + (n[0] ? kb * 64u : 0u);
#pragma unroll
          for (uint32_t i = 0; i < kN / 8; ++i) {
            if (i * 8 + r0 < M_b) {
#pragma unroll
              for (uint32_t b = 0; b < kXB; ++b) cp_async_16s(to0 + at + i * 1024u + b * x_block, src + off[b], n[b]);
            }
            src += (size_t)4 * K;
            if (i * 8 + 4 + r0 < M_b) {
#pragma unroll
              for (uint32_t b = 0; b < kXB; ++b) cp_async_16s(to1 + at + i * 1024u + b * x_block, src + off[b], n[b]);
            }
            src += (size_t)4 * K;
          }
          asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(full_a + xs * 8) : "memory");
        });
      }
    };
    for (uint32_t ph = 0; ph < p.n_phases; ++ph) {
      if (ph > 0) {
        // one lane polls; the barrier orders the other lanes' reads behind what it has acquired
        if (x_warps(kN) == 2 && pipe) wait(smem_u32(&go[ph - 1]), 0);
        else if (lane == 0) {
          if (!s_abort && !grid_counter_wait(p.bar + 1, ph * n_cta, status)) s_abort = 1;
          mbar_arrive(&go[ph - 1]);   // the epilogue warps (and the second producer) may read what the phase before wrote
          // The last threadblock past the last of these waits - everybody has arrived, nobody reads the
          // counters any more - puts them back to zero for the next launch.  (Here and not at the end of
          // the kernel, where the round trip would hold up the kernel that waits for this one.)
          if (ph + 1 == p.n_phases && atomicAdd(p.bar, 1u) == n_cta - 1) {
            p.bar[0] = 0u;
            p.bar[1] = 0u;
          }
        }
        __syncwarp();
      }
      if (!produce(p.ph[ph], ph)) break;
    }
    if constexpr (!kTmaX) cp_async_wait_all();   // (nothing in flight when the shared memory goes away)
  } else if (warp == 2 || warp == kMma1) {
    // ------------------------------------------------------------------ MMA issue
    // A warp cannot run ahead of the tensor cores by more than an MMA or two, so everything it does between
    // two groups of MMAs - barriers polled, commits (the second of a pair alone 73 cycles), the loop - adds
    // to their time unless another warp's MMAs fill it: hence the second pipeline.  Cycles per k block
    // (4 MMAs) with the operands always in place, 64 x 8 / 128 x 16 / 128 x 128 / 128 x 256 results: one warp
    // 383 / 428 / 473 / 535, two 192 / 216 / 256 / 512; the MMAs themselves take 92 / 156 / 256 / 512, and HBM
    // delivers the weights of one in 275 / 490 / 490 / 490.
    // (A pipeline's barriers have one consumer.  Two warps that took the stages of one ring in turn would poll
    // barriers whose earlier phases they have not seen, which a parity cannot tell from the one meant.)
    // (idesc64: an image of 8 alone, 64 rows)
    const uint32_t pipe = warp == 2 ? 0u : 1u, first = pipe * pipe_stages, first_x = pipe * pipe_slots;
    const uint32_t idesc = umma_idesc_bf16_f32(kRowTile, nb < 16 ? 16 : nb);
    const uint32_t idesc64 = umma_idesc_bf16_f32(kRowTile / 2, nb);
    const uint32_t full_a = smem_u32(w_full) + first * 8, empty_a = smem_u32(w_empty) + first * 8;
    const uint32_t xfull_a = smem_u32(x_full) + first_x * 8, xempty_a = smem_u32(x_empty) + first_x * 8;
    const uint32_t x_step = x_slot / 16, x_half = x_block / 16;
    const uint32_t w_low = desc_low(smem_u32(ring) + first * kStageBytes), x_low = desc_low(smem_u32(x_ring) + first_x * x_slot);
    const uint32_t afull_a = smem_u32(acc_full), aempty_a = smem_u32(acc_empty);
    uint32_t stage = 0, parity = 0, xs = 0, xpar = 0, as = 0, apar = 1;
    auto next_stage = [&]() { if (++stage == pipe_stages) { stage = 0; parity ^= 1u; } };
    auto next_slot = [&]() { if (++xs == pipe_slots) { xs = 0; xpar ^= 1u; } };
    auto next_acc = [&]() { if (++as == kSlots) { as = 0; apar ^= 1u; } };
    // odd lanes poll one barrier, even lanes the other
    auto wait_two = [&](uint32_t bar0, uint32_t par0, uint32_t bar1, uint32_t par1) -> bool {
      const uint32_t bar = (lane & 1u) ? bar1 : bar0, par = (lane & 1u) ? par1 : par0;
      bool ok = try_wait(bar, par);
      if (__all_sync(0xFFFFFFFFu, ok)) return true;
      if (!ok) ok = wait_slow(bar, par, &s_abort, status);
      return __all_sync(0xFFFFFFFFu, ok) != 0;
    };
    auto wait_one = [&](uint32_t bar, uint32_t par) -> bool { return wait_two(bar, par, bar, par); };
    // image8: images of 8 units (two k blocks a stage).  mode: see PairPhase.  (Compile-time, for this
    // warp's instruction latency.)
    auto multiply = [&](const PairPhase& q, auto image8, auto mode) -> bool {
      constexpr bool kImage8 = decltype(image8)::value;
      constexpr uint32_t kMode = decltype(mode)::value;
      // k blocks of an iteration (one pipeline: of an image of 8 in slots of one block, half a stage)
      constexpr uint32_t kStep = kPipes == 1 ? (kImage8 && kMode == 2 ? 2 : 1) : chunk_blocks(kN, kImage8 ? 8 : 16);
      constexpr bool kHalves = kImage8 && kStep == 1;
      const Part w = part_of(q);
      const uint32_t slot_n = q.slot_blocks, id = kImage8 ? idesc64 : idesc, in_turn = kPipes == 2 && slots_in_turn(kN, kImage8 ? 8 : 16, slot_n);
      constexpr uint32_t kBlockCols = kMode == 2 ? 0 : kMode == 1 ? part_cols(kN) : 4 * part_cols(kN), kNext = kMode == 0 ? part_cols(kN) : 0;
      // One k block: 4 MMAs.  (16 columns on: 32 bytes, 2 in a descriptor's address field, which counts in 16 bytes)
      auto mma_block = [&](uint32_t d, uint32_t wl, uint32_t xl, uint32_t accumulate) {
#pragma unroll
        for (uint32_t ks = 0; ks < 4; ++ks)
          umma_low(d + ks * kNext, wl + 2 * ks, xl + 2 * ks, id, kMode == 0 ? 0u : ks == 0 ? accumulate : 1u);
      };
      for (uint32_t ua = w.u0; ua < w.u1; ua += w.run) {
        uint32_t turn = pipe;
        for (uint32_t k0 = w.kb0; k0 < w.kb1; k0 += slot_n, turn ^= in_turn) {   // a slot of accumulators: the epilogue warps have read what was there
          const uint32_t k1 = min(k0 + slot_n, w.kb1), done = afull_a + as * 8;
          uint32_t d = tmem + as * kSlotCols + turn * (kMode == 2 ? part_cols(kN) : kStep * kBlockCols), accumulate = 0;
          if (!wait_one(aempty_a + as * 8, apar)) return false;
          for (uint32_t kb = k0 + turn * kStep; kb < k1; kb += kPipes * kStep, d += kPipes * kStep * kBlockCols) {
            const bool both = kStep == 2 && kb + 1 < k1, second = kHalves && ((kb - w.kb0) & 1u), last = !kHalves || second || kb + 1 == w.kb1;
            const uint32_t wl = w_low + stage * (kStageBytes / 16) + (second ? kStageBytes / 32 : 0u), xl = x_low + xs * x_step;
            const uint32_t free_w = empty_a + stage * 8, free_x = xempty_a + xs * 8;
            if (!wait_two(full_a + stage * 8, parity, xfull_a + xs * 8, xpar)) return false;
            if constexpr (!kTmaX) fence_proxy_async_smem();   // (activations that came through the load/store path)
            tc_fence_after_sync();
            if (last) next_stage();
            next_slot();
            if constexpr (kStep == 1 || (kImage8 && kXB == 2)) {   // one stage, one activation slot
              if (elect_one()) {
                mma_block(d, wl, xl, accumulate);
                if (both) mma_block(d + kBlockCols, wl + kStageBytes / 32, xl + x_half, kMode == 2);
                if (last) commit(free_w);
                commit(free_x);
              }
              __syncwarp();
            } else {   // two stages of one k block, or (from 128 rows on) two activation slots of one
              if (elect_one()) {
                mma_block(d, wl, xl, accumulate);
                if (!kImage8 || !both) commit(free_w);
                if (kXB == 1 || !both) commit(free_x);
              }
              __syncwarp();
              if (both) {
                const uint32_t wl1 = kImage8 ? wl + kStageBytes / 32 : w_low + stage * (kStageBytes / 16), free_w1 = kImage8 ? free_w : empty_a + stage * 8;
                const uint32_t xl1 = kXB == 2 ? xl + x_half : x_low + xs * x_step, free_x1 = kXB == 2 ? free_x : xempty_a + xs * 8;
                if (!(kImage8 ? wait_one(xfull_a + xs * 8, xpar) : wait_one(full_a + stage * 8, parity))) return false;
                tc_fence_after_sync();
                if constexpr (kImage8) next_slot(); else next_stage();
                if (elect_one()) {
                  mma_block(d + kBlockCols, wl1, xl1, kMode == 2);
                  commit(free_w1);
                  commit(free_x1);
                }
                __syncwarp();
              }
            }
            accumulate = kMode == 2;
          }
          if (elect_one()) commit(done);   // (a warp that had no chunk arrives all the same)
          __syncwarp();
          next_acc();
        }
      }
      return true;
    };
    auto multiply_phase = [&](const PairPhase& q) -> bool {
      auto with_mode = [&](auto mode) { return q.image == 8 ? multiply(q, Const<true>(), mode) : multiply(q, Const<false>(), mode); };
      if constexpr (kN == 8)
        if (q.mode == 0) return with_mode(Const<0u>());
      return q.mode == 1 ? with_mode(Const<1u>()) : with_mode(Const<2u>());
    };
    for (uint32_t ph = 0; ph < p.n_phases; ++ph)
      if (!multiply_phase(p.ph[ph])) break;
  } else if (warp >= kEpiWarp0) {
    // ------------------------------------------------------------------ epilogue
    // An image's accumulators are added up as they come, and the sums go to shared memory (half of the
    // columns to the peer's where two threadblocks share the rows), and from there to all epilogue
    // threads, which finish a pair of rows 64 apart (gate / up, the two halves of a rotary pair) for a
    // few sequences each.
    const uint32_t et = tid - kEpiWarp0 * 32, quarter = warp & 3u, hh = (warp - kEpiWarp0) >> 2;
    const uint32_t l128 = quarter * 32u + lane;   // tensor-memory lane
    uint32_t as = 0, apar = 0, n_xch = 0, n_free = 0;
    pdl_wait();
    const uint32_t skip = et == 0 ? skip_arrivals_of(p.ws) : 0u;
    for (uint32_t ph = 0; ph < p.n_phases; ++ph) {
      const PairPhase& q = p.ph[ph];
      const Part w = part_of(q);
      const bool two = q.split == 2;
      const uint32_t image = q.image, worker = two ? blockIdx.x >> 1 : blockIdx.x;
      const uint32_t epi = q.epi, N = q.N, M_b = p.M_b;
      if (ph > 0) {   // (one thread polls, the others wait in the hardware barrier)
        if (et == 0) wait(smem_u32(&go[ph - 1]), 0);
        // After a wait that gave up, everybody leaves before the next phase: a barrier whose peer never
        // came is not armed a second time.
        if (named_barrier_or(1, kEpiThreads, s_abort != 0)) break;
      }
      if (q.ssq_in && w.u0 < w.u1) {
        // row scales of this phase's activations: the parts in kGroups interleaved groups, then the groups in order
        constexpr uint32_t kGroups = kEpiThreads / kN;
        const uint32_t m = et % kN, g = et / kN;
        float s = 0.f;
        if (m < M_b)
#pragma unroll 8
          for (uint32_t i = g; i < q.ssq_parts; i += kGroups) s += __ldcg(q.ssq_in + (size_t)i * q.ssq_stride + m);
        s_red[et] = s;
        named_barrier_sync(1, kEpiThreads);
        if (et < kN) {
          float t = 0.f;
          for (uint32_t i = 0; i < kGroups; ++i) t += s_red[i * kN + et];
          s_rs[et] = rsqrtf(t / q.x_cols + q.rms_eps);
        }
        named_barrier_sync(1, kEpiThreads);
      }
      // This thread's place: row `pos` of the image's lower (and upper) half, columns col, col + m_step, ... of a chunk or round
      const uint32_t n_pos = 4 * image, pos = et % n_pos, m_step = kEpiThreads / n_pos, col = et / n_pos;
      constexpr uint32_t G = kBig ? 4 : kN / 8;                                      // columns a thread finishes at a time
      uint32_t ua, ub, u, d, n;   // the image: its run of units; the unit that sits at this position, and its rows of the weight
      bool valid;
      auto place = [&](uint32_t first) {
        ua = first;
        ub = min(w.u1, ua + w.run);
        u = ua + ((pos / 4 - ua) & (image - 1));
        d = (u % kUnitsPerTile) * 4u + (pos & 3u);   // row inside the half tile
        n = (u / kUnitsPerTile) * kRowTile + d;
        valid = u < ub;
      };
      // rope: where the new row of every sequence goes, for the (one or two) heads of the image
      auto row_table = [&]() {
        for (uint32_t e = et; e < 2 * kN; e += kEpiThreads) {
          const uint32_t m = e % kN, head = ua / kUnitsPerTile + e / kN;
          unsigned long long dst = 0, dst2 = 0;   // (the slot of the token rides in the low bits: rows are 256-byte aligned)
          const int32_t ctx = (m < M_b && head * kUnitsPerTile < ub) ? q.ctx_lens[m] : 0;
          if (ctx > 0) {
            if (head < q.Hq) {
              dst = reinterpret_cast<unsigned long long>(q.q_out + ((size_t)m * q.Hq + head) * kRowTile);
            } else {
              const uint32_t at = (uint32_t)ctx - 1u, bi = at / BOOST_KV_BLOCK_TOKENS, slot = at % BOOST_KV_BLOCK_TOKENS;
              const int32_t b = bi < q.max_blocks ? q.block_table[(size_t)m * q.max_blocks + bi] : -1;
              if (b < 0 || (uint32_t)b >= q.n_pool_blocks) {
                atomicOr(status, kErrBadIndex);
              } else {
                const bool is_k = head < q.Hq + q.Hkv;
                const size_t off = ((size_t)(head - q.Hq - (is_k ? 0u : q.Hkv)) * q.n_pool_blocks + (uint32_t)b) * 4096u + slot * 256u;
                const void* const* pages = is_k ? q.k_page_ptr : q.v_page_ptr;
                const void* const* pages2 = is_k ? q.k_page_ptr2 : q.v_page_ptr2;
                dst = reinterpret_cast<unsigned long long>(pages[off / kPageBytes]) + off % kPageBytes + slot;
                if (pages2) dst2 = reinterpret_cast<unsigned long long>(pages2[off / kPageBytes]) + off % kPageBytes + slot;
              }
            }
          }
          s_dst[e / kN][m] = dst;
          s_dst2[e / kN][m] = dst2;
        }
      };
      // What does not depend on the sums, for the G columns from i0 on of a range [mb, mb + cols) of sequences.
      float aux_a[G], aux_b[G];
      auto load_aux = [&](uint32_t mb, uint32_t cols, uint32_t i0) {
#pragma unroll
        for (uint32_t g = 0; g < G; ++g) {
          const uint32_t c = col + (i0 + g) * m_step, m = mb + c;
          const bool live = c < cols && m < M_b;
          if (epi == BOOST_EPI_PLAIN) {
            if (q.residual) {
              const unsigned short* r = reinterpret_cast<const unsigned short*>(q.residual) + (size_t)m * N + n;
              aux_a[g] = (valid && live && n < N) ? bf16_lo((uint32_t)__ldcg(r)) : 0.f;
              aux_b[g] = (valid && live && n + 64 < N) ? bf16_lo((uint32_t)__ldcg(r + 64)) : 0.f;
            }
          } else if (epi == BOOST_EPI_ROPE_APPEND) {
            const float2 cs = live ? __ldcg(reinterpret_cast<const float2*>(q.rope_table) + (size_t)m * 64 + d) : make_float2(1.f, 0.f);
            aux_a[g] = cs.x;
            aux_b[g] = cs.y;
          }
        }
      };
      // Finish columns [0, cols) = sequences [mb, mb + cols) of an image: own sums, the peer's sums (or null; a column in_lanes apart).  aux of the first G columns is loaded.
      auto finish = [&](const float* own, const float* in, uint32_t in_lanes, uint32_t mb, uint32_t cols, uint32_t image_no) {
        for (uint32_t i0 = 0; i0 * m_step < cols; i0 += G) {   // G at a time, so that their loads and arithmetic overlap
          if (i0) load_aux(mb, cols, i0);
          float lo[G], hi[G];
          bool live[G];
#pragma unroll
          for (uint32_t g = 0; g < G; ++g) {
            const uint32_t c = col + (i0 + g) * m_step, at = (c < cols ? c : 0u) * kRowTile + pos;
            live[g] = valid && c < cols && mb + c < M_b;
            lo[g] = own[at];
            hi[g] = own[at + n_pos];
            if (in) {
              if constexpr (kBig) {
                const float* const peer = in + (c < cols ? c : 0u) * in_lanes + pos;
                lo[g] += peer[0];
                hi[g] += peer[n_pos];
              } else {
                lo[g] += in[at];
                hi[g] += in[at + n_pos];
              }
            }
          }
          const uint32_t m0 = mb + col + i0 * m_step;
          if (q.ssq_in) {
#pragma unroll
            for (uint32_t g = 0; g < G; ++g) {
              const float rs = s_rs[min(m0 + g * m_step, kN - 1)];
              lo[g] *= rs;
              hi[g] *= rs;
            }
          }
          if (epi == BOOST_EPI_PLAIN) {
            if (q.residual) {
#pragma unroll
              for (uint32_t g = 0; g < G; ++g) { lo[g] += aux_a[g]; hi[g] += aux_b[g]; }
            }
            const bool in_lo = n < N, in_hi = n + 64 < N;
            const size_t idx = (size_t)m0 * N + n, step = (size_t)m_step * N;
            if (q.y_dtype == 0) {
              float* y = static_cast<float*>(q.y) + idx;
#pragma unroll
              for (uint32_t g = 0; g < G; ++g, y += step) {
                if (live[g] && in_lo) y[0] = lo[g];
                if (live[g] && in_hi) y[64] = hi[g];
              }
            } else {
              __nv_bfloat16* y = static_cast<__nv_bfloat16*>(q.y) + idx;
#pragma unroll
              for (uint32_t g = 0; g < G; ++g, y += step) {
                const __nv_bfloat16 ol = __float2bfloat16_rn(lo[g]), oh = __float2bfloat16_rn(hi[g]);
                const float fl = __bfloat162float(ol), fh = __bfloat162float(oh);
                lo[g] = 0.f;
                if (live[g] && in_lo) { y[0] = ol; lo[g] = fl * fl; }
                if (live[g] && in_hi) { y[64] = oh; lo[g] = fmaf(fh, fh, lo[g]); }
              }
              if (q.ssq_out) {   // sums of squares over the 32 rows (and their partners) of this warp
#pragma unroll
                for (uint32_t o = 16; o >= 1; o /= 2)
#pragma unroll
                  for (uint32_t g = 0; g < G; ++g) lo[g] += __shfl_xor_sync(0xFFFFFFFFu, lo[g], o);
                float* out = q.ssq_out + (size_t)((worker * q.max_images + image_no) * (image / 8) + pos / 32) * kN + m0;
#pragma unroll
                for (uint32_t g = 0; g < G; ++g)
                  if (lane == 0 && col + (i0 + g) * m_step < cols) out[g * m_step] = lo[g];
              }
            }
          } else if (epi == BOOST_EPI_SWIGLU) {
            __nv_bfloat16* y = static_cast<__nv_bfloat16*>(q.y) + (size_t)m0 * (N / 2) + (size_t)(u / kUnitsPerTile) * 64 + d;
            const size_t step = (size_t)m_step * (N / 2);
#pragma unroll
            for (uint32_t g = 0; g < G; ++g) {
              const float gate = bf16_round(lo[g]), up = bf16_round(hi[g]);
              lo[g] = gate / (1.f + expf(-gate)) * up;
            }
#pragma unroll
            for (uint32_t g = 0; g < G; ++g, y += step)
              if (live[g]) *y = __float2bfloat16_rn(lo[g]);
          } else {
            const uint32_t head = u / kUnitsPerTile, which = (head - ua / kUnitsPerTile) & 1u;
            const bool rotate = head < q.Hq + q.Hkv;
#pragma unroll
            for (uint32_t g = 0; g < G; ++g) {
              const uint32_t m = m0 + g * m_step;
              const float x1 = bf16_round(lo[g]), x2 = bf16_round(hi[g]), a = aux_a[g], b = aux_b[g];
              const __nv_bfloat16 y1 = __float2bfloat16_rn(rotate ? x1 * a - x2 * b : x1), y2 = __float2bfloat16_rn(rotate ? x2 * a + x1 * b : x2);
              if (live[g]) {
                const unsigned long long rows[2] = {s_dst[which][m], s_dst2[which][m]};
#pragma unroll
                for (uint32_t r = 0; r < 2; ++r) {
                  if (!rows[r]) continue;
                  // elements d, d + 64 of a 256-byte row whose 16-byte pieces are swizzled by the slot (query rows: slot 0)
                  uint8_t* at = reinterpret_cast<uint8_t*>(rows[r] & ~15ull) + (d & 7u) * 2u;
                  const uint32_t sw = (uint32_t)rows[r] & 7u;
                  *reinterpret_cast<__nv_bfloat16*>(at + (((d >> 3) ^ sw) << 4)) = y1;
                  *reinterpret_cast<__nv_bfloat16*>(at + (((d >> 3) ^ sw ^ 8u) << 4)) = y2;
                }
              }
            }
          }
        }
      };
      // The accumulator row of this lane.  Of an M = 64 product, 16 rows lie in the first 16 lanes of every 32.
      const bool m64 = image == 8, holds = !m64 || lane < 16;
      const uint32_t row = m64 ? quarter * 16u + lane : l128;
      // The sums of an image: group i is the CH columns from column(i) on.
      constexpr uint32_t kGroups = kN / (HG * CH);
      auto column = [&](uint32_t i) { return hh * CH + i * (HG * CH); };
      const uint32_t lane_base = tmem + ((quarter * 32u) << 16);
      const uint32_t mode = q.mode, slot_n = q.slot_blocks;
      // Parts of a slot with this many k blocks.
      auto parts_of = [&](uint32_t blocks) -> uint32_t {
        if (mode != 2) return mode ? blocks : 4 * blocks;
        return kPipes == 2 && blocks > chunk_blocks(kN, image) ? 2u : 1u;
      };
      auto wait_slot = [&]() {
        wait(smem_u32(&acc_full[as]), apar);
        __syncwarp();
        tc_fence_after_sync();
      };
      auto next_slot = [&]() { if (++as == kSlots) { as = 0; apar ^= 1u; } };
      // From 128 rows on the sums would be up to half of a thread's registers: they stay in tensor memory, in
      // the slot of the last part added, which is given back when the epilogue has read them.  (Registers:
      // 244 - 508 bytes of spills at 256 rows, 6-layer step at batch 250 2147 - 2350 us instead of 2045.)
      constexpr bool kParkSums = kN >= 128;
      float sum[kParkSums ? 1 : kGroups][CH];
      uint32_t parked = 0;   // the slot kept
      [[maybe_unused]] bool parked_two = false;   // it holds two parts, whose sum is still to be taken
      auto release_slot = [&](uint32_t slot) {
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[slot]);
      };
      auto add = [&](float* to, const float* v, uint32_t n) {
#pragma unroll
        for (uint32_t j = 0; j < n; j += 2) {
          const float2 t = add2(make_float2(to[j], to[j + 1]), make_float2(v[j], v[j + 1]));
          to[j] = t.x;
          to[j + 1] = t.y;
        }
      };
      auto group_sums = [&](uint32_t i, float (&v)[CH]) {   // i: a constant, except where the sums are parked
        if constexpr (kParkSums) {
          const uint32_t at = lane_base + parked * kSlotCols + column(i);
          if (kPipes == 2 && parked_two) {
            float both[16];
            tmem_ld_2x8(at, at + part_cols(kN), both);
            add(both, both + 8, 8);
#pragma unroll
            for (uint32_t e = 0; e < 8; ++e) v[e] = both[e];
          } else {
            tmem_ld_8(at, v);
          }
        } else {
#pragma unroll
          for (uint32_t e = 0; e < CH; ++e) v[e] = sum[i][e];
        }
      };
      // Every part of the image's columns, as its slot comes.  take(from, n): the n parts at tensor-memory address `from`.
      auto each_slot = [&](auto take) {
        for (uint32_t kb = w.kb0; kb < w.kb1; kb += slot_n) {
          wait_slot();
          if (column(0) < M_b) take(lane_base + as * kSlotCols + column(0), parts_of(min(slot_n, w.kb1 - kb)));
          release_slot(as);
          next_slot();
        }
      };
      auto accumulate = [&]() {
        if constexpr (kParkSums) {
          for (uint32_t kb = w.kb0; kb < w.kb1; kb += slot_n) {   // (one or two parts a slot)
            wait_slot();
            const bool two_parts = parts_of(min(slot_n, w.kb1 - kb)) == 2;
            if (kb != w.kb0) {   // the sum so far, from the slot before, goes on top of this slot's first part
              const uint32_t before = lane_base + parked * kSlotCols, here = lane_base + as * kSlotCols;
#pragma unroll
              for (uint32_t i = 0; i < kGroups; ++i) {
                if (column(i) >= M_b) continue;   // (columns beyond the batch: nobody's)
                float v[16];
                tmem_ld_2x8(before + column(i), here + column(i), v);
                add(v, v + 8, 8);
                if constexpr (kPipes == 2) {
                  if (parked_two) {
                    tmem_ld_8(before + part_cols(kN) + column(i), reinterpret_cast<float(&)[8]>(v[8]));
                    add(v, v + 8, 8);
                  }
                  if (two_parts) {
                    tmem_ld_8(here + part_cols(kN) + column(i), reinterpret_cast<float(&)[8]>(v[8]));
                    add(v, v + 8, 8);
                  }
                }
                tmem_st_8(here + column(i), v);
              }
              tmem_st_wait();
              release_slot(parked);
            }
            parked = as;
            parked_two = two_parts && kb == w.kb0;
            next_slot();
          }
        } else {
#pragma unroll
          for (uint32_t i = 0; i < kGroups; ++i)
#pragma unroll
            for (uint32_t j = 0; j < CH; ++j) sum[i][j] = 0.f;
          if constexpr (kN == 8) {
            if (mode == 0) {
              // batches of 1 and 2, whose sums compare with those of CUDA cores: four parts added up pairwise,
              // then a compensated sum (Knuth's two-sum: t + error = s + p exactly)
              float2 s = make_float2(0.f, 0.f), lost = s;
              each_slot([&](uint32_t from, uint32_t n_parts) {
#pragma unroll 1
                for (uint32_t a0 = 0; a0 < n_parts; a0 += 8) {
                  float v[16];
                  tmem_ld_8x2<part_cols(kN)>(from + a0 * part_cols(kN), v);
                  if (n_parts - a0 < 8) {   // (parts that are not there)
#pragma unroll
                    for (uint32_t a = 1; a < 8; ++a)
                      if (a0 + a >= n_parts) v[2 * a] = v[2 * a + 1] = 0.f;
                  }
                  float2 p[8];
#pragma unroll
                  for (uint32_t a = 0; a < 8; ++a) p[a] = make_float2(v[2 * a], v[2 * a + 1]);
#pragma unroll
                  for (uint32_t a = 0; a < 8; a += 4) {
                    const float2 four = add2(add2(p[a], p[a + 1]), add2(p[a + 2], p[a + 3]));
                    const float2 t = add2(s, four), d = sub2(t, s);
                    lost = add2(lost, add2(sub2(s, sub2(t, d)), sub2(four, d)));
                    s = t;
                  }
                }
              });
              // (an infinite sum has no remainder)
              sum[0][0] = fabsf(s.x) <= 3.402823466e38f ? s.x + lost.x : s.x;
              sum[0][1] = fabsf(s.y) <= 3.402823466e38f ? s.y + lost.y : s.y;
              return;
            }
          }
          each_slot([&](uint32_t from, uint32_t n_parts) {
#pragma unroll 1
            for (uint32_t a = 0; a < n_parts; ++a, from += part_cols(kN)) {
              if constexpr (CH == 4) {
                float v[4];
                tmem_ld_4(from, v);
                add(sum[0], v, 4);
              } else if constexpr (CH == 8 && kGroups == 1) {
                float v[8];
                tmem_ld_8(from, v);
                add(sum[0], v, 8);
              } else if constexpr (CH == 16) {
                float v[16];
                tmem_ld_2x8(from, from + 8, v);
                add(sum[0], v, 16);
              } else {
                static_assert(kN != 64 || (kGroups == 2 && CH == 8), "two groups of 8");
                float v[16];
                tmem_ld_2x8(from, from + HG * CH, v);
                add(sum[0], v, 8);
                add(sum[kGroups - 1], v + 8, 8);
              }
            }
          });
        }
      };
      uint32_t image_no = 0;
      if (two) {
        if (w.u0 < w.u1) {
          constexpr uint32_t kRounds = rounds_of(kN);
          const uint32_t half = nb / 2 / kRounds;                             // columns of a round that one threadblock finishes
          const uint32_t lanes = m64 ? 64u : kRowTile;                        // that hold sums
          float* own = kBig ? reinterpret_cast<float*>(x_ring) : sums;
          // At 64 and 128 rows the peer's sums arrive in the chunk buffer, idle here, where they fit; else in the activation slots,
          // once this threadblock's products have read them, which the peer is told (a microsecond: down product at
          // batch 64 / 128 25.2 -> 24.2, 30.3 -> 29.3 us without).
          const bool roomy = !kBig || (kRounds == 1 && half * lanes * 4u <= sums_bytes(CW));
          const uint32_t in_lanes = kBig && kRounds == 1 ? lanes : kRowTile;
          float* in = kBig && roomy ? sums : own + half * kRowTile;
          place(w.u0);
          if (epi == BOOST_EPI_ROPE_APPEND) row_table();
          // (All rounds' operands are asked for ahead of the sums: about 1 % of a step.  A second round's wait in the chunk
          // buffer, idle here: in registers, which are short above 128 rows, they cost products of few k blocks 1 - 2 %.)
          float* const kept = sums + et;
          static_assert(kRounds == 1 || 2 * G * kEpiThreads <= CW * kRowTile, "operands fit the chunk buffer");
          if constexpr (kRounds == 2) {
            load_aux((2 + rank) * half, half, 0);
#pragma unroll
            for (uint32_t g = 0; g < G; ++g) { kept[2 * g * kEpiThreads] = aux_a[g]; kept[(2 * g + 1) * kEpiThreads] = aux_b[g]; }
          }
          load_aux(rank * half, half, 0);
          if (et == 0) mbar_arrive_expect_tx(&xch_full, lanes * half * kRounds * 4u);
          accumulate();
          if (!roomy) {
            if (et == 0) {
              arrive_remote(mapa(smem_u32(&xch_free), rank ^ 1u));
              wait(smem_u32(&xch_free), n_free & 1u);
            }
            ++n_free;
            named_barrier_sync(1, kEpiThreads);
          }
          if (!__any_sync(0xFFFFFFFFu, s_abort != 0)) {   // the peer's columns, of all rounds
            const uint32_t to = mapa(smem_u32(in), rank ^ 1u), bar = mapa(smem_u32(&xch_full), rank ^ 1u);
#pragma unroll
            for (uint32_t i = 0; i < kGroups; ++i) {
              const uint32_t share = column(i) / half, c = column(i) - share * half + (share >> 1) * half;
              if ((share & 1u) == rank || share >= 2 * kRounds) continue;
              float v[CH];
              group_sums(i, v);
              if (holds) {
#pragma unroll
                for (uint32_t e = 0; e < CH; ++e) st_async_f32(to + ((c + e) * in_lanes + row) * 4u, v[e], bar);
              }
            }
          }
          for (uint32_t r = 0; r < kRounds; ++r) {
            const uint32_t mb = (2 * r + rank) * half;
            if (kRounds == 2 && r == 1) {
#pragma unroll
              for (uint32_t g = 0; g < G; ++g) { aux_a[g] = kept[2 * g * kEpiThreads]; aux_b[g] = kept[(2 * g + 1) * kEpiThreads]; }
            }
#pragma unroll
            for (uint32_t i = 0; i < kGroups; ++i) {   // this threadblock's columns of the round
              const uint32_t share = column(i) / half, c = column(i) - share * half;
              if (share != 2 * r + rank) continue;
              float v[CH];
              group_sums(i, v);
              if (holds) {
#pragma unroll
                for (uint32_t e = 0; e < CH; ++e) own[(c + e) * kRowTile + row] = v[e];
              }
            }
            if (kParkSums && r + 1 == kRounds) release_slot(parked);
            if (et == 0 && r == 0) wait(smem_u32(&xch_full), n_xch & 1u);
            named_barrier_sync(1, kEpiThreads);
            finish(own, in + r * half * in_lanes, in_lanes, mb, half, 0);
            if constexpr (kBig) {
              fence_proxy_async_smem();   // (the activation slots are written by TMA copies again)
              named_barrier_sync(1, kEpiThreads);
            }
          }
          ++n_xch;
          image_no = 1;
        }
      } else {
        constexpr uint32_t J = CW / (HG * CH);   // groups of a chunk
        const uint32_t n_chunks = (M_b + CW - 1) / CW;
        for (uint32_t ua0 = w.u0; ua0 < w.u1; ua0 += w.run, ++image_no) {
          place(ua0);
          if (epi == BOOST_EPI_ROPE_APPEND) row_table();
          load_aux(0, CW, 0);
          accumulate();
          for (uint32_t ch = 0; ch < n_chunks; ++ch) {
            if (ch) load_aux(ch * CW, CW, 0);
#pragma unroll
            for (uint32_t j = 0; j < J; ++j) {
              float v[CH];
              group_sums(kParkSums ? ch * J + j : j, v);   // (not parked: there is one chunk)
              if (holds) {
#pragma unroll
                for (uint32_t e = 0; e < CH; ++e) sums[(column(j) + e) * kRowTile + row] = v[e];
              }
            }
            if (kParkSums && ch + 1 == n_chunks) release_slot(parked);
            named_barrier_sync(1, kEpiThreads);
            finish(sums, nullptr, 0, ch * CW, CW, image_no);
            named_barrier_sync(1, kEpiThreads);   // (the buffer and the row table are written again)
          }
        }
      }
      if (q.ssq_out) {   // images this worker does not have: their share of the statistics is zero
        for (uint32_t j = image_no * (image / 8); j < q.max_images * (image / 8); ++j)
          for (uint32_t m = et; m < M_b; m += kEpiThreads)
            if (!two || (((m / (nb / 2 / rounds_of(kN))) & 1u) == rank)) q.ssq_out[(size_t)(worker * q.max_images * (image / 8) + j) * kN + m] = 0.f;
      }
      named_barrier_sync(1, kEpiThreads);   // everybody's outputs before the release
      if (et == 0) {
        if (ph + 1 < p.n_phases && blockIdx.x >= skip) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p.bar + 1), "r"(1u) : "memory");
        if (w.u0 < w.u1 && s_rec[ph] != kNoRecord) sched_log_end(sched_log_of(p.ws), s_rec[ph]);
      }
    }
  }
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  if (s_abort) {
    // A wait gave up somewhere (every role is past its last wait now, so nobody starts anything new): nothing
    // may be in the tensor cores' pipeline or on its way to shared memory when that goes away.  Each
    // issuer waits, as long as any other wait, for what it has started.  (A fixed time would not do: over
    // the host link the copies in flight of all threadblocks are a third of a millisecond.)
    if (warp == 2 || warp == kMma1) {
      uint64_t* const bar = &drained[warp == 2 ? 0 : 1];
      if (elect_one()) commit(smem_u32(bar));
      __syncwarp();
      mbar_wait(bar, 0, status);
    } else if (warp == 0 || warp == 3 || (kTmaX && (warp == 1 || warp == kX1))) {
      // the last use of every stage, backwards from the next one (uses before the first count as landed)
      const bool weights = warp == 0 || warp == 3, second = kPipes == 2 && (warp == 3 || warp == kX1);
      const uint32_t n = weights ? pipe_stages : pipe_slots;
      uint64_t* const full = (weights ? w_full : x_full) + (second ? n : 0);
      for (uint32_t i = 0; i < n; ++i) {
        if (stage == 0) { stage = n; parity ^= 1u; }
        --stage;
        if (kPipes == 1 && weights) my_turn = !my_turn;
        if (my_turn) mbar_wait(full + stage, parity ^ 1u, status);
        if (kPipes == 2 && x_warps(kN) == 1 && !weights) {
          if (stage1 == 0) { stage1 = n; parity1 ^= 1u; }
          --stage1;
          mbar_wait(full + n + stage1, parity1 ^ 1u, status);
        }
      }
    }
    __syncthreads();
    // Nor may the peer store here any more.  (Without a failed wait, what it stores and signals here has been waited for.)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  if (warp == 2) tmem_dealloc(tmem, tmem_cols(kN));
}

uint32_t units_bound(uint32_t n_units, uint32_t W) { return (n_units + W - 1) / W; }
uint32_t images_bound(uint32_t n_units, uint32_t W) { return (units_bound(n_units, W) + 15) / 16; }

// The k blocks of an accumulator, and with them the slots.  Every hand-over costs the MMA warps 350
// cycles and more, so accumulators hold as many as the results allow:
//   fp32 results   0.9 of the threadblocks' segments in the kernels of kernels_gemv.cu (two per SM up
//                  to 128 rows, one above; none longer than a row tile's columns): the sums are then no
//                  further from the exact ones than theirs.  Batches of 1 and 2, whose segments are
//                  summed on CUDA cores there: a quarter of a block.
//   bf16 results   at least 4096 columns (as many as those segments have at most): 4.4e-6 of the sum,
//                  where the rounding behind it is 1.7e-3.
// An even number (up to 16 rows a multiple of four), or 1.  A slot has an accumulator per pipeline.
void plan_parts(PairPhase& q, uint32_t clusters, uint32_t n_class, uint32_t M_b) {
  const bool fp32 = q.epi == BOOST_EPI_PLAIN && q.y_dtype == 0;
  q.mode = fp32 && M_b <= 2 ? 0 : 1;
  q.slot_blocks = q.mode == 0 ? slot_parts(n_class) / 4 : slot_parts(n_class);
  const uint64_t blocks = (uint64_t)(q.n_units / kUnitsPerTile) * q.k_blocks, segments = (uint64_t)clusters * (M_b <= 128 ? 4 : 2);
  uint32_t n = (uint32_t)(9 * (blocks < segments * q.k_blocks ? blocks : segments * q.k_blocks) / (10 * segments));
  if (!fp32 && n < 64) n = 64;
  const uint32_t unit = M_b <= 16 ? 4 : 2;
  n = n / unit * unit * pipes_of(n_class);
  if (q.mode == 0 || n == 0) return;
  q.mode = 2;
  const uint32_t own = (q.k_blocks + q.split - 1) / q.split, slots = (own + n - 1) / n;   // slots as even as they come
  const uint32_t round = pipes_of(n_class) == 2 ? 2 * chunk_blocks(n_class, q.image) : 2;
  q.slot_blocks = ((own + slots - 1) / slots + round - 1) / round * round;
}

// How a phase is cut.  Two threadblocks share the rows of a cluster, half of K each, where those rows
// fit one image: little crosses between them, and the rows divide evenly (4096 rows over 74
// clusters: 98.8 % of the SMs' time, over 148 threadblocks 86 %).  Longer products (gate / up, LM head)
// have rows enough for every threadblock on its own (97 % and more) and nothing to exchange.
void plan_phase(PairPhase& q, uint32_t clusters, uint32_t n_class, uint32_t M_b) {
  q.split = (q.k_blocks >= 2 && units_bound(q.n_units, clusters) <= 16) ? 2u : 1u;
  const uint32_t W = q.split == 2 ? clusters : 2 * clusters;
  q.image = units_bound(q.n_units, W) <= 8 ? 8u : 16u;
  q.max_images = images_bound(q.n_units, W);
  plan_parts(q, clusters, n_class, M_b);
}
uint32_t ssq_parts_of(const PairPhase& q, uint32_t clusters) { return (q.split == 2 ? clusters : 2 * clusters) * q.max_images * (q.image / 8); }

// Shared memory of an instantiation.  More than half an SM, so that no two threadblocks of this kernel
// share one (the grid counts on one threadblock per SM).  Up to 32 rows a threadblock of the
// attention kernel fits beside it (measured when it was chosen: a step at batch 1 is 2.8 % slower with
// 180 KiB, at batch 32 0.3 %); above, the activation tiles need the room.
constexpr uint32_t smem_total(uint32_t n) { return (n <= 32 ? 147u : 214u) * 1024u; }

// Clusters of two that the current device holds at once, one threadblock per SM (0: none, or an error, which
// is left in `rc`).  Set up once per device; every rule about how a product is cut starts from here.
template <uint32_t kN, uint32_t kChunk = chunk_cols(kN)>
uint32_t clusters_of(int& rc) {
  static std::atomic<uint32_t> known[boosth::kMaxDevices];   // count + 1; threads that meet here find the same
  const int dev = boosth::device_slot(), sms = boosth::sm_count();
  rc = dev < 0 || sms <= 0 ? BOOST_ERR_CUDA : BOOST_OK;
  if (rc != BOOST_OK) return 0;
  const uint32_t seen = known[dev].load(std::memory_order_acquire);
  if (seen) return seen - 1;
  rc = boosth::check(cudaFuncSetAttribute(gemv_pair_kernel<kN, kChunk>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_total(kN)));
  if (rc != BOOST_OK) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(threads_of(kN));
  cfg.dynamicSmemBytes = smem_total(kN);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  rc = boosth::check(cudaOccupancyMaxActiveClusters(&n, gemv_pair_kernel<kN, kChunk>, &cfg));
  if (rc != BOOST_OK) return 0;
  const uint32_t clusters = (uint32_t)n < (uint32_t)sms / 2 ? (uint32_t)n : (uint32_t)sms / 2;
  known[dev].store(clusters + 1, std::memory_order_release);
  return clusters;
}

uint32_t batch_class(uint32_t M_b) { return M_b <= 8 ? 8 : M_b <= 16 ? 16 : M_b <= 32 ? 32 : M_b <= 64 ? 64 : M_b <= 128 ? 128 : 256; }

// The same by batch, for sizes and rules (without a device: a B200's 74).
uint32_t clusters_for(uint32_t M_b) {
  int rc = BOOST_OK;
  uint32_t n = 0;
  switch (boosth::device_slot() < 0 ? 0 : batch_class(M_b)) {
    case 0: break;
    case 8: n = clusters_of<8>(rc); break;
    case 16: n = clusters_of<16>(rc); break;
    case 32: n = clusters_of<32>(rc); break;
    case 64: n = clusters_of<64>(rc); break;
    case 128: n = clusters_of<128>(rc); break;
    default: n = clusters_of<256>(rc);
  }
  return n ? n : 74;
}

// 129 - 256 rows: 64 columns to an epilogue's chunk, or 32?  Where four activation slots fit beside 64 that is better (tiles of
// up to 192 rows: 6-layer step at batch 180 1511 us, with 32 and a stage more 1523).  Tiles of 224 rows: 32, and
// a fourth slot in the room that leaves (batch 200: 1763 -> 1610).  Of 256 rows: the fourth slot pays where a product waits
// for activations (batch 250: 1903 -> 1820), and 64 columns, with three slots, where rows that are one threadblock's
// have few k blocks, so that the epilogue is most of its time.  Measured at batch 232 - 256, weights from HBM, by the
// average number of blocks of 8 rows x 64 columns in an image.  Products on their own (9600 - 60000 rows x 1024 - 4096
// columns): the times meet at 330 - 430 blocks for fp32 results, 390 - 460 for bf16, the lower ones where there is another
// image, whose MMAs hide the epilogue (28672 x 1024, 194 blocks: 32 columns 30.6 us, 64 27.7; 14336 x 4096, 775: 41.5, 45.1).
// Steps: six models of 300 - 540 blocks 0 - 2 % faster with 64, one of 775 (the 8B model) 4 % with 32.
// Where all rows of a step's launch are shared and its K is short, 64 (hidden 256 / 512, batch 200 - 240: 1.8 / 0.5 % faster); a
// step's first launch, a product on its own, is counted as one too: two forms of the kernel in turn cost 2 us a step.
bool wide_chunk(const PairParams& p) {
  if (p.nb <= 192) return true;
  const uint32_t clusters = clusters_for(p.M_b);
  const bool step = p.early || p.n_phases > 1;
  bool own_rows = false, shared_short = step;
  for (uint32_t i = 0; i < p.n_phases; ++i) {
    PairPhase q = p.ph[i];
    plan_phase(q, clusters, 256, p.M_b);
    if (q.split == 2) {
      shared_short = shared_short && q.k_blocks <= 32;
      continue;
    }
    if (p.nb < 256) return false;
    const bool fp32 = q.epi == BOOST_EPI_PLAIN && q.y_dtype == 0;
    const uint32_t most = step ? 600u : q.max_images > 1 ? (fp32 ? 330u : 390u) : fp32 ? 372u : 440u;
    if ((uint64_t)q.n_units * q.k_blocks > (uint64_t)most * 2 * clusters * q.max_images) return false;
    own_rows = true;
  }
  return own_rows || shared_short;
}

// Row statistics between the phases of one launch live in two buffers of the workspace; a phase's
// ssq_in is matched to the earlier phase that produces it by the caller's ssq_out pointer.
template <uint32_t kN, uint32_t kChunk = chunk_cols(kN)>
int launch_pair(PairParams& p, float* stats, size_t stats_bytes, cudaStream_t stream) {
  int rc;
  const uint32_t clusters = clusters_of<kN, kChunk>(rc);
  if (rc != BOOST_OK) return rc;
  if (clusters == 0) return BOOST_ERR_UNSUPPORTED;
  // activation slots: more than a microsecond of a short product's stream (a k block per 155 ns); from
  // 128 rows on half of the shared memory and more, since the tiles are as large as the weight stages.  Above 128 rows
  // four tiles, five where that leaves five stages (batch 150: 1424 -> 1384 us for 6 layers; 180: four 1511, five 1652), and
  // of 256 rows three where the chunks have 64 columns.
  const uint32_t slot_bytes = x_blocks(kN) * p.nb * 128u;
  const uint32_t x_budget = kN <= 16 ? 6 * slot_bytes : kN == 32 ? 4 * slot_bytes : kN == 64 ? 64u * 1024u : kN == 128 ? 96u * 1024u : (p.nb <= 160 ? 5 : p.nb == 256 && kChunk == 64 ? 3 : 4) * slot_bytes;
  p.x_slots = x_budget / slot_bytes < kMaxXSlots ? x_budget / slot_bytes : kMaxXSlots;
  p.x_slots = p.x_slots / pipes_of(kN) * pipes_of(kN);
  const uint32_t fixed = 2048u + p.x_slots * slot_bytes + sums_bytes(kChunk);
  p.n_stages = (smem_total(kN) - fixed) / kStageBytes;
  if (p.n_stages > kMaxStages) p.n_stages = kMaxStages;
  p.n_stages = p.n_stages / pipes_of(kN) * pipes_of(kN);
  const size_t smem = smem_total(kN);
  // (the caller's ssq pointers stand in for the buffers until here)
  const float* key[kMaxPhases];
  uint32_t n_stats = 0;
  for (uint32_t i = 0; i < p.n_phases; ++i) {
    PairPhase& q = p.ph[i];
    plan_phase(q, clusters, kN, p.M_b);
    for (int j = (int)i - 1; j >= 0; --j)
      if (q.ssq_in && key[j] == q.ssq_in) {
        q.ssq_in = p.ph[j].ssq_out;
        q.ssq_parts = ssq_parts_of(p.ph[j], clusters);
        q.ssq_stride = kN;
        break;
      }
    key[i] = q.ssq_out;
    if (q.ssq_out) {
      const size_t bytes = (size_t)ssq_parts_of(q, clusters) * kN * 4;
      if (2 * bytes > stats_bytes) return BOOST_ERR_CAPACITY;
      q.ssq_out = stats + (n_stats++ & 1u) * (stats_bytes / 8);
    }
  }
  return boosth::launch_chained_cluster(gemv_pair_kernel<kN, kChunk>, dim3(2 * clusters), dim3(threads_of(kN)), smem, 2, stream, p);
}

}  // namespace

size_t boosth::pair_stats_bytes(uint32_t N, uint32_t M_b) {
  // two buffers, for whichever way plan_phase cuts the rows; a workspace may serve smaller batches too
  const uint32_t units = (N + kRowTile - 1) / kRowTile * kUnitsPerTile;
  size_t most = 0;
  for (uint32_t n = 8; n <= batch_class(M_b); n *= 2) {
    const uint32_t workers = 2 * clusters_for(n);
    const size_t bytes = (size_t)2 * workers * images_bound(units, workers) * 2 * n * 4;
    most = bytes > most ? bytes : most;
  }
  return most;
}

boosth::PairCut boosth::pair_cut(uint32_t N, uint32_t K, uint32_t M_b) {
  PairPhase q = {};
  q.k_blocks = (K + 63) / 64;
  q.n_units = (N + kRowTile - 1) / kRowTile * kUnitsPerTile;
  const uint32_t clusters = clusters_for(M_b);
  plan_phase(q, clusters, batch_class(M_b), M_b);
  return {2 * clusters, q.split, units_bound(q.n_units, q.split == 2 ? clusters : 2 * clusters)};
}

int boosth::gemv_pair_launch(const boost_gemv_call_t* calls, uint32_t n_calls, uint32_t M_b, void* workspace, size_t workspace_bytes,
                             uint32_t header_row_tiles, uint32_t* sync_words, bool early, void* stream) {
  if (!calls || n_calls == 0 || n_calls > kMaxPhases || M_b == 0 || M_b > 256) return BOOST_ERR_INVALID;
  const size_t header = boosth::gemv_header_bytes(header_row_tiles);
  if (!workspace || workspace_bytes < header) return workspace ? BOOST_ERR_CAPACITY : BOOST_ERR_INVALID;
  float* stats = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + header);
  const size_t stats_bytes = (workspace_bytes - header) / 16 * 16;
  const uint32_t n_class = batch_class(M_b);
  PairParams p;
  p.n_phases = n_calls;
  p.M_b = M_b;
  p.nb = n_class <= 32 ? n_class : M_b <= 128 ? (M_b + 15) / 16 * 16 : (M_b + 31) / 32 * 32;
  p.ws = static_cast<uint32_t*>(workspace);
  p.bar = sync_words;
  p.early = early ? 1u : 0u;
  for (uint32_t i = 0; i < n_calls; ++i) {
    const boost_gemv_call_t& c = calls[i];
    const boost_gemv_epilogue_t& e = c.epilogue;
    int rc = boosth::gemv_check_call(c, M_b, workspace, workspace_bytes, header_row_tiles);
    if (rc == BOOST_OK && x_by_tma(n_class)) rc = boosth::encode_activation_map(&p.x_map[i], c.x, M_b, c.w.K, p.nb);
    if (rc != BOOST_OK) return rc;
    PairPhase& q = p.ph[i];
    q = PairPhase{};
    q.w_page_ptr = c.w.page_ptr;
    q.w_order = c.w.order;
    q.n_pages = (uint32_t)c.w.n_pages;
    q.n_host_pages = (uint32_t)c.w.n_host_pages;
    q.N = c.w.N;
    q.K = c.w.K;
    q.x = static_cast<const __nv_bfloat16*>(c.x);
    q.k_blocks = (c.w.K + 63) / 64;
    q.n_units = (c.w.N + kRowTile - 1) / kRowTile * kUnitsPerTile;
    q.y = c.y;
    q.y_dtype = c.y_dtype;
    q.residual = static_cast<const __nv_bfloat16*>(c.residual);
    q.epi = BOOST_EPI_PLAIN;
    q.x_cols = (float)c.w.K;
    if (c.has_epilogue) {
      q.epi = (uint32_t)e.mode;
      q.ssq_in = e.ssq_in;
      q.ssq_parts = e.ssq_in_tiles;
      q.ssq_stride = e.ssq_stride;
      q.rms_eps = e.rms_eps;
      q.ssq_out = e.ssq_out;
      q.q_out = static_cast<__nv_bfloat16*>(e.q_out);
      q.k_page_ptr = e.k_page_ptr;
      q.v_page_ptr = e.v_page_ptr;
      q.k_page_ptr2 = e.k_page_ptr2;
      q.v_page_ptr2 = e.v_page_ptr2;
      q.block_table = e.block_table;
      q.ctx_lens = e.ctx_lens;
      q.n_pool_blocks = e.n_pool_blocks;
      q.max_blocks = e.max_blocks;
      q.Hq = e.n_q_heads;
      q.Hkv = e.n_kv_heads;
      q.rope_table = e.rope_table;
    }
  }
  cudaStream_t st = (cudaStream_t)stream;
  switch (n_class) {
    case 8: return launch_pair<8>(p, stats, stats_bytes, st);
    case 16: return launch_pair<16>(p, stats, stats_bytes, st);
    case 32: return launch_pair<32>(p, stats, stats_bytes, st);
    case 64: return launch_pair<64>(p, stats, stats_bytes, st);
    case 128: return launch_pair<128>(p, stats, stats_bytes, st);
    default: return wide_chunk(p) ? launch_pair<256>(p, stats, stats_bytes, st) : launch_pair<256, 32>(p, stats, stats_bytes, st);
  }
}
