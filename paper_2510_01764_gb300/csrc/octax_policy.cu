// The actor-critic network of §4.1 on the tensor cores (tcgen05, TMEM), and
// the rollout that runs it between environment steps on the device.
//
// Network (§4.1): the 4-frame stack in the (frame, x, y) = (4, 64, 32)
// orientation; conv1 32 filters (8,4)/(4,2) -> 15 x 15; conv2 64 filters 4/2
// -> 6 x 6; conv3 64 filters 3/1 -> 4 x 4; ReLU after each; flatten; actor
// and critic heads of 256 ReLU units; n_logits actor outputs and one value.
// VALID convolutions; weights and stored activations in bfloat16, products
// accumulated in fp32 (TMEM), heads' output layers in fp32 on the CUDA cores.
//
// Conv kernel (persistent, one CTA per SM). A batch of kP = 8
// instances is processed at a time; the rows of every GEMM are
// (grid position, instance) with the instance fastest, so one 8-row core
// matrix of the tcgen05 no-swizzle K-major layout is one grid position of
// all 8 instances, and a position shift is a shift of the descriptor's start
// address by whole core matrices. Every convolution is then a sum over its
// kernel taps of GEMMs whose A operand is the layer input at a shifted start:
// no im2col copies.
//  - conv1 works on 4 x 2-pixel blocks: with stride (4, 2) its (8, 4) kernel
//    covers 2 x 2 blocks, so it is 4 taps of K = 32 (4 frames x 8 pixels)
//    over a 16 x 16 grid of blocks, expanded from the packed frame bits to
//    bf16 0/1; two output rows (16 positions x 8 instances = 128 rows each)
//    share one accumulator fed by the three block rows they read.
//  - conv2 (stride 2) reads conv1's output split by the parity of x and y:
//    tap (kx, ky) reads sub-grid (kx & 1, ky & 1) at offset (kx >> 1,
//    ky >> 1) of a 7-wide grid. The taps kx and kx + 2 read the same
//    sub-grid one position apart, so they are stacked along N (N = 128) and
//    the drain adds columns 64..127 of row g + 1 to columns 0..63 of row g.
//    The sub-grids are a band of six grid rows, written round and round; each M
//    tile covers two output rows and reads three grid rows.
//  - conv3 (stride 1) follows when the CTA's batches are through conv2; its A
//    operand is conv2's output in three copies, shifted by kx, so that the M
//    tile is the 16 output positions and nothing else.
//  Rows whose grid position lies outside conv1's or conv2's output are computed
//  and discarded (they read padding or neighbouring positions, always inside
//  the buffers).
// What bounds it: the chains of MMAs that add into one accumulator (12 of conv1
// per pair of rows, 16 of conv2 per tile; links of one chain alone were seen 85
// cycles apart, 12 of conv3's N = 64 in 1,010, and two chains side by side gave
// an MMA every 42) and their hand-overs; 9.6 K cycles a batch for conv1 and conv2,
// of which the tensor pipe needs 5.8 K, and 2.4 K for conv3 (1.7 K of operand
// reads). Against the form before it (a CTA took each batch through all
// phases, conv3's output positions 22 of 32 rows; 150 us for 16,384
// instances): 75 us for conv1 and conv2 and about 18 us for conv3. Its steps:
// roles that run ahead of each other, also over a batch's end (forward 173.5
// -> 126.5 us); a wait that seldom reads the timer, blocks expanded before the
// wait, a band whose rows are rewritten five rows later (112.5); MMAs issued
// by whole warps, whose operands need no moves to uniform registers (issuing 12
// took 1.25 K, now 0.75 K cycles of the warp; 101.8); conv3 in the same kernel
// (99.2). The microseconds of a forward here are of three policies in turn; one
// after another it takes 108 us (174 and 195 before all of them). No
// gain: a ring of 7 block rows with four accumulators; conv1's A operand in
// TMEM; conv1's two rows as separate chains.
// Heads kernel: a head of one or two 128-instance tiles per CTA; K = 1024
// streamed in 64-wide slices; the actor CTA also draws the action. Bound by the
// MMAs (16.4 K cycles for two tiles) and the first slice's arrival (2.4 K).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "octax_internal.h"

struct octax_policy {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int n_logits = 0;
  int64_t max_envs = 0;
  int sms = 0;
  void *w1 = nullptr, *w2 = nullptr, *w3 = nullptr, *wh = nullptr;  // packed bf16
  float *fp = nullptr;        // biases and output layers (fp32), see FpLayout
  uint8_t *act2 = nullptr;    // conv2 output of one conv launch, batches of 8 instances
  uint8_t *act3 = nullptr;    // flattened features, heads' A-operand tiles
  uint64_t *ring = nullptr;   // rollout: two packed observation slots [2][max_envs][4][32]
  unsigned int *err = nullptr;
  int stall = 0;              // octax_policy_debug_stall
};

namespace octax {

cudaStream_t env_stream(const octax_env *e);
int env_device(const octax_env *e);

namespace {

constexpr int kP = 8;            // instances per conv batch
// conv kernel, conv1 and conv2: warps by role; a draining warp reads the TMEM lane quarter warp & 3
constexpr int kDrain1Warps = 8, kDrain2Warps = 4, kBuildWarps = 4, kIssueWarps = 3;
constexpr int kIssueWarp = kDrain1Warps + kDrain2Warps + kBuildWarps;  // the first of them
constexpr int kConvThreads = 32 * (kIssueWarp + kIssueWarps);
// conv3, by the same warps: draining, then a warp each for the copies and the MMAs of even and of odd batches
constexpr int kDrain3Warps = 8;
constexpr int kMaxLogits = 17;   // 16 keys + the no-op
constexpr uint64_t kMaxWaitNs = 1000000000ull;
constexpr uint32_t kMaxPolls = 1u << 24;

// ---- conv1 / conv2 shared memory (bytes) ------------------------------
constexpr uint32_t kW1Off = 0;                             // conv1 B: [j 3][dx 2][chunk 4][n 64][8]
constexpr uint32_t kW1Bytes = 6 * 4 * 64 * 16;
constexpr uint32_t kW2Off = kW1Off + kW1Bytes;             // conv2 B: [ky 4][kx & 1][chunk 4][n 128][8]
constexpr uint32_t kW2Bytes = 4 * 2 * 4 * 128 * 16;
constexpr uint32_t kAct1Off = kW2Off + kW2Bytes;           // band: 4 parity sub-grids of six grid rows of 7
constexpr uint32_t kBandSlots = 6, kSlotBytes = 7 * 512;   // position: 4 chunks x 8 instances x 16 B
constexpr uint32_t kSubBytes = kBandSlots * kSlotBytes;
constexpr uint32_t kAct1Bytes = 4 * kSubBytes;
constexpr uint32_t kBlkRows = 5;                           // ring of block rows; a batch's 15 go round it three times
constexpr uint32_t kBlkOff = kAct1Off + kAct1Bytes;        // 16 positions each, and one that only discarded rows read
constexpr uint32_t kBlkBytes = (kBlkRows * 16 + 1) * 512;
constexpr uint32_t kFrOff = kBlkOff + kBlkBytes;           // frames [32 rows][4][8] u64
constexpr uint32_t kXbOff = kFrOff + 8192;
// conv2 drain exchange: row g + 1 of the warps that hold the last positions
// of a TMEM lane quarter comes from the next quarter's warp: [supplier 3]
// [lane 8][36 floats] (rows padded to 144 B: 16-byte aligned, and 8 lanes'
// rows start in distinct bank groups).
constexpr int kXbPitch = 36;
constexpr uint32_t kConvSmem = kXbOff + 3 * 8 * kXbPitch * 4;
static_assert(kConvSmem + 1024 <= 227 * 1024, "conv kernel shared memory (with 1 KB of static shared data)");
constexpr uint32_t kAct2Bytes = 36 * 1024;                 // conv2 output of a batch: position: 8 chunks x 8 x 16 B
// Most batches per CTA of one conv launch; more instances take several launches
// over the same act2, which so stays within 350 MB (without a limit it took 4.6
// KB of each instance, more than all else that a policy keeps of one). A launch
// costs its weights' copy and the pipeline's start: 131,072 instances 798 us in
// one launch, 809 in two of 54 batches, 841 with at most 24 and 846 with at most
// 16, whose act2 (88 MB) stays in L2: that gains nothing. A multiple of 16, so
// that a launch of the most begins at a tile of the features.
constexpr int kMaxRounds = 64;
static_assert(kMaxRounds * kP % 128 == 0, "launches begin at a tile of 128 instances");
// TMEM columns (fp32): conv1: 2 buffers x 2 output rows x 32; conv2: 2 buffers x 128
constexpr uint32_t kD1Col = 0, kD2Col = 128, kConvTmemCols = 512;

// ---- conv3 --------------------------------------------------------------------
constexpr uint32_t kW3Bytes = 3 * 8 * 192 * 16;            // conv3 B: [ky 3][chunk 8][n = 64 kx + o][8]
constexpr int kStages3 = 6;                                // ring of one kx each: 6 rows x 4 positions x 1 KB
constexpr uint32_t kStage3Bytes = 24 * 1024;
static_assert(kW3Bytes + kStages3 * kStage3Bytes <= kConvSmem, "conv3's weights and stages over the others' operands");

// ---- heads kernel -----------------------------------------------------------
constexpr uint32_t kHA = 128 * 64 * 2;                // A slice: 128 rows x 64 K (bf16) = 8 chunk planes
constexpr uint32_t kHB = 256 * 64 * 2;                // B slice: 256 rows x 64 K
constexpr uint32_t kHeadRing = 192 * 1024;            // stages | output layer [output][256] | biases, hidden and output
constexpr uint32_t kHeadSmem = kHeadRing + kMaxLogits * 256 * 4 + (256 + 32) * 4;
static_assert(kHeadSmem + 1024 <= 227 * 1024, "heads kernel shared memory (with 1 KB of static shared data)");
static_assert(2 * 8 * kMaxLogits * 128 * 4 <= kHeadRing, "the sums fit the ring");
constexpr uint32_t kAct3TileBytes = 128 * 1024 * 2;   // [slice 16][chunk 8][row 128][16 B]

// fp32 parameter block: b1 32 | b2 64 | b3 64 | bh [2][256] | wa2 [17][256] | ba2 [17] | wc2 [256] | bc2
struct FpLayout {
  static constexpr int b1 = 0, b2 = 32, b3 = 96, bh = 160, wa2 = 672, ba2 = wa2 + kMaxLogits * 256,
                       wc2 = ba2 + kMaxLogits, bc2 = wc2 + 256, total = bc2 + 1;
};

// ---- PTX helpers -------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  // the timer is read rarely: a read takes longer than the waits of a pipeline that runs
  if (mbar_try(bar, parity)) return true;
  uint64_t t0 = 0;
  for (uint32_t i = 0; i < kMaxPolls; ++i) {
#pragma unroll 1
    for (int k = 0; k < 32; ++k)
      if (mbar_try(bar, parity)) return true;
    const uint64_t now = global_ns();
    if (i == 0) t0 = now;
    if (now - t0 > kMaxWaitNs) break;
  }
  return false;
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bulk copy global -> shared (16-byte aligned, size a multiple of 16), completing on `bar`.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor, no swizzle: start, leading-dimension (K
// direction) and stride-dimension (M/N direction, between 8-row core
// matrices) byte offsets; bits 46-48 hold the fixed value 0b001.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         (1ull << 46);
}
// The descriptor of the same layout `bytes` further on: shared addresses stay
// below 2^18, so the 14-bit start field takes the offset without a carry, and
// the MMA-issuing loops add compile-time offsets to a base built once.
__device__ __forceinline__ uint64_t sdesc_at(uint64_t base, uint32_t bytes) { return base + (bytes >> 4); }
// Instruction descriptor, kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(uint32_t M, uint32_t N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
// The same from a whole warp in step: one lane issues. All operands are the
// same in every lane and known to be, so they need no moves to uniform
// registers behind every instruction.
__device__ __forceinline__ void mma_bf16_warp(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\telect.sync _|e, 0xFFFFFFFF;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_commit_warp(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\telect.sync _|e, 0xFFFFFFFF;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 32 consecutive fp32 columns of this thread's TMEM lane (warp w reads lanes 32w..32w+31).
__device__ __forceinline__ void tmem_ld32(uint32_t addr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
  // the wait names the loaded registers, so no use of them is scheduled before it
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
        "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
        "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :
      : "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}
// Two 16-column loads (one per address) behind a single wait, in one asm
// statement so that no use of the registers can be scheduled before the wait.
__device__ __forceinline__ void tmem_ld16x2(uint32_t a0, uint32_t a1, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(a0), "r"(a1)
      : "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}
// 32 columns at each of a0 and a1 of this thread's TMEM lane, behind one wait.
__device__ __forceinline__ void tmem_ld32x2(uint32_t a0, uint32_t a1, float (&v)[32], float (&w)[32]) {
  uint32_t r[32], q[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(a0));
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]), "=r"(q[8]),
        "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]), "=r"(q[15]), "=r"(q[16]),
        "=r"(q[17]), "=r"(q[18]), "=r"(q[19]), "=r"(q[20]), "=r"(q[21]), "=r"(q[22]), "=r"(q[23]), "=r"(q[24]),
        "=r"(q[25]), "=r"(q[26]), "=r"(q[27]), "=r"(q[28]), "=r"(q[29]), "=r"(q[30]), "=r"(q[31])
      : "r"(a1));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
        "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
        "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :
      : "memory");
  asm volatile(""
      : "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]), "+r"(q[6]), "+r"(q[7]),
        "+r"(q[8]), "+r"(q[9]), "+r"(q[10]), "+r"(q[11]), "+r"(q[12]), "+r"(q[13]), "+r"(q[14]), "+r"(q[15]),
        "+r"(q[16]), "+r"(q[17]), "+r"(q[18]), "+r"(q[19]), "+r"(q[20]), "+r"(q[21]), "+r"(q[22]), "+r"(q[23]),
        "+r"(q[24]), "+r"(q[25]), "+r"(q[26]), "+r"(q[27]), "+r"(q[28]), "+r"(q[29]), "+r"(q[30]), "+r"(q[31])
      :
      : "memory");  // after the wait (volatile statements keep their order)
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    v[j] = __uint_as_float(r[j]);
    w[j] = __uint_as_float(q[j]);
  }
}
// 32 floats to / from one 16-byte aligned exchange row, as 8 vector accesses.
__device__ __forceinline__ void xrow_put(float *row, const float (&v)[32]) {
#pragma unroll
  for (int c = 0; c < 8; ++c)
    reinterpret_cast<float4 *>(row)[c] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
}
__device__ __forceinline__ void xrow_get(const float *row, float (&v)[32]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float4 f = reinterpret_cast<const float4 *>(row)[c];
    v[4 * c] = f.x;
    v[4 * c + 1] = f.y;
    v[4 * c + 2] = f.z;
    v[4 * c + 3] = f.w;
  }
}
__device__ __forceinline__ uint64_t f32x2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
// bias (pairs) + ReLU on 8 values, packed to one 16-byte chunk of 8 bf16.
// Rounding keeps order and sign, so the maximum with 0 may follow it, two
// values at a time.
__device__ __forceinline__ uint4 relu_chunk(const float *v, const uint64_t *bias) {
  uint32_t o[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint64_t s;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(s) : "l"(f32x2(v[2 * j], v[2 * j + 1])), "l"(bias[j]));
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(s));
    const __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(lo, hi), __floats2bfloat162_rn(0.0f, 0.0f));
    o[j] = *reinterpret_cast<const uint32_t *>(&h);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}
// Barrier `id` of kN threads that also says whether all of them are ok.
template <int kN>
__device__ __forceinline__ bool all_ok(int id, bool ok) {
  uint32_t any_fail;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.eq.u32 p, %1, 0;\n\tbarrier.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(any_fail)
      : "r"((uint32_t)ok), "r"(id), "r"(kN)
      : "memory");
  return !any_fail;
}
// The band slot of the row after row pr (of a batch's seven): past the last
// slot comes the first, or, if that holds row pr again, the second.
__device__ __forceinline__ uint32_t next_slot(uint32_t slot, int pr) {
  return slot < kBandSlots - 1 ? slot + 1 : pr < 6 ? 1 : 0;
}
__device__ __forceinline__ uint32_t philox_w0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                              uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
  return c0;
}

struct ConvArgs {
  const uint64_t *obs_words;  // [n][4][32] packed frames (or null)
  const uint8_t *obs_u8;      // [n][4][32][64] uint8 frames (or null)
  int64_t n;
  const uint8_t *w1, *w2, *w3;  // packed bf16 B operands
  const float *fp;            // FpLayout
  uint8_t *act2;              // [batches][6 py][6 px][8 chunks][8 instances][16 B]
  uint8_t *act3;              // [tiles][16][8][128][16 B]
  unsigned int *err;
  int stall;                  // diagnostic: the first conv1 commit is skipped (its wait runs out)
};

struct Conv3Smem {
  uint64_t full[kStages3], empty[kStages3], done[2], freed[2], bar_w, fin[2];
  int issued[2], landed[2];  // stages whose copies were issued / waited for, even and odd batches
};

// conv3 of the CTA's batches, from conv2's output as this CTA wrote it: the M
// tile is the 4 x 4 output positions of 8 instances exactly. Tap (kx, ky) reads
// input positions (qx + kx, qy + ky): the stages hold, for one kx, columns kx ..
// kx + 3 of the six rows (24 positions; each row is one bulk copy of 4 KB), and
// ky shifts the start by one row of them. Even and odd batches have three
// stages, an accumulator buffer, a copying and an issuing thread each: the
// MMAs of one accumulator run at one per ~85 cycles, of two side by side at
// one per 42. Returns this thread's outcome.
__device__ __forceinline__ bool conv3_batches(const ConvArgs &a, uint8_t *sm, Conv3Smem &S, const float *bias3,
                                              uint32_t tmem, int my_batches) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = smem_u32(sm);
  bool ok = true;
  if (warp < kDrain3Warps) {
    // drain: warps w and w + 4 read lane quarter w & 3 (four positions), 32 of the 64 channels each
    const int half = warp >> 2, m = 4 * (warp & 3) + (lane >> 3), ri = lane & 7;  // m = qx + 4 qy
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    for (int bi = 0; bi < my_batches; ++bi) {
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(&S.done[bi & 1]), (bi >> 1) & 1));
      if (!ok) break;
      tc_fence_after();
      float v[32], w[32];
      const uint32_t d = tmem + lane_base + 256 * (bi & 1) + 32 * half;
      tmem_ld32x2(d + 64, d + 128, v, w);
#pragma unroll
      for (int c = 0; c < 32; ++c) w[c] += v[c];
      tmem_ld32(d, v);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&S.freed[bi & 1]));
#pragma unroll
      for (int c = 0; c < 32; ++c) v[c] += w[c];
      const int64_t inst = (blockIdx.x + (int64_t)bi * gridDim.x) * kP + ri;
      if (inst < a.n) {
        // feature slice m: k = 64 m + channel
        uint8_t *dst = a.act3 + (inst >> 7) * (int64_t)kAct3TileBytes + m * 16384 + (inst & 127) * 16;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const ulonglong2 *const b3 = reinterpret_cast<const ulonglong2 *>(bias3 + 32 * half + 8 * c);
          const uint64_t bias[4] = {b3[0].x, b3[0].y, b3[1].x, b3[1].y};
          *reinterpret_cast<uint4 *>(dst + (4 * half + c) * 2048) = relu_chunk(v + 8 * c, bias);
        }
      }
    }
  } else if (lane == 0 && warp < kDrain3Warps + 2) {  // copies of this thread's batches: even or odd
    const int who = warp - kDrain3Warps;
    if (who == 0) {
      mbar_expect_tx(smem_u32(&S.bar_w), kW3Bytes);
      for (uint32_t o = 0; o < kW3Bytes; o += 24576) bulk_g2s(sbase + o, a.w3 + o, 24576, smem_u32(&S.bar_w));
    }
    int issued = 0;
    for (int bi = who; bi < my_batches && ok; bi += 2) {
      const uint8_t *const src = a.act2 + (blockIdx.x + (int64_t)bi * gridDim.x) * kAct2Bytes;
      for (int kx = 0; kx < 3; ++kx) {
        const int st = 3 * who + kx;
        if (bi >= 2) ok = mbar_wait(smem_u32(&S.empty[st]), ((bi >> 1) - 1) & 1);  // the stage's previous MMAs are done
        if (!ok) break;
        const uint32_t f = smem_u32(&S.full[st]), dst = sbase + kW3Bytes + st * kStage3Bytes;
        mbar_expect_tx(f, kStage3Bytes);
#pragma unroll
        for (int py = 0; py < 6; ++py) bulk_g2s(dst + py * 4096, src + (kx + 6 * py) * 1024, 4096, f);
        ++issued;
      }
    }
    grid_dependents_launch();  // (earlier, the next kernel's waiting CTAs would keep the SMs from other streams)
    S.issued[who] = issued;
  } else if (lane == 0 && warp < kDrain3Warps + 4) {  // MMAs of this thread's batches
    const int who = warp - kDrain3Warps - 2;
    const uint64_t a3d = sdesc(sbase + kW3Bytes + 3 * who * kStage3Bytes, 128, 1024), b3d = sdesc(sbase, 3072, 128);
    ok = mbar_wait(smem_u32(&S.bar_w), 0);
    int landed = 0;
    for (int bi = who; bi < my_batches && ok; bi += 2) {
      if (bi >= 2) ok = mbar_wait(smem_u32(&S.freed[who]), ((bi >> 1) - 1) & 1);
      for (int kx = 0; kx < 3 && ok; ++kx) {
        ok = mbar_wait(smem_u32(&S.full[3 * who + kx]), (bi >> 1) & 1);
        if (!ok) break;
        ++landed;
        tc_fence_after();
        const uint64_t at = sdesc_at(a3d, kx * kStage3Bytes), bt = sdesc_at(b3d, kx * 1024);
        const uint32_t d = tmem + 256 * who + 64 * kx;  // an accumulator per kx, summed by the drain
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_bf16(d, sdesc_at(at, ky * 4096 + kk * 256), sdesc_at(bt, ky * 24576 + kk * 6144), idesc_bf16(128, 64),
                     (ky | kk) != 0);
        mma_commit(smem_u32(&S.empty[3 * who + kx]));
      }
      if (ok) mma_commit(smem_u32(&S.done[who]));
    }
    S.landed[who] = landed;
  }
  return ok;
}

// The convolutions of batches blockIdx.x, blockIdx.x + gridDim.x, ...: conv1 and
// conv2 of all of them, then conv3 (conv3_batches). In the first part every
// role runs its own loop over the batches' steps and meets the others through
// mbarriers only, so that the roles work on different steps (and, around a
// batch's end, on different batches) at the same time:
//   builders     wait c1[P & 1] (pair P - 2's MMAs: its block rows are free)  arrive blk[P & 1]
//   conv1 issue  wait blk[P & 1], d1f[P & 1] (accumulator drained)           commit c1[P & 1]
//   conv1 drain  wait c1[P & 1], c2[.] where band rows are rewritten         arrive d1f[P & 1], band[T & 1]
//   conv2 issue  wait band[T & 1], d2f[T & 1]                                commit c2[T & 1]
//   conv2 drain  wait c2[T & 1]                                              arrive d2f[T & 1]
// P counts conv1 pairs (7 per batch), T conv2 tiles (3 per batch). A barrier
// never gets two phases ahead of any of its waiters: pair P + 2 needs pair P
// drained and its blocks rebuilt, tile T + 2 needs tile T drained, and the
// conv1 drain waits for every tile before it completes the rows of the tile
// after next.
// The band: each conv1 grid row goes to the next of six slots, round and
// round. A tile reads its three rows as two pairs of neighbours, so a row that
// falls on the last slot is also written to the first, where its pair with the
// row after it is. A slot is rewritten five rows later at the earliest: when
// rows 0, 2 and 5 of a batch are written the tiles before last have to be done
// (the previous batch's 1 and 2, this one's 0), which leaves a tile two pairs'
// time. Every wait is bounded; a role whose wait runs out leaves
// its loop, and the others run into their own limits.
template <bool kU8>
__global__ void __launch_bounds__(kConvThreads, 1) policy_conv_kernel(const ConvArgs a) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ __align__(8) uint64_t bars[16];
  __shared__ uint32_t tmem_s;
  __shared__ __align__(16) float sb[160];    // b1 | b2 | b3
  __shared__ __align__(8) Conv3Smem s3;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const uint32_t sbase = smem_u32(sm);
  auto bar = [&](int j) { return smem_u32(&bars[j]); };
  // pairs of barriers, by the parity of the pair / tile
  constexpr int kBarC1 = 0, kBarBlk = 2, kBarD1f = 4, kBarC2 = 6, kBarD2f = 8, kBarBand = 10, kBarW = 12, kBarFin = 13;

  for (int j = t; j < 160; j += kConvThreads) sb[j] = a.fp[j];
  if (t == 0) {
    for (int j = 0; j < 2; ++j) {
      mbar_init(bar(kBarC1 + j), 1);
      mbar_init(bar(kBarBlk + j), kBuildWarps);
      mbar_init(bar(kBarD1f + j), kDrain1Warps);
      mbar_init(bar(kBarC2 + j), 1);
      mbar_init(bar(kBarD2f + j), kDrain2Warps);
      mbar_init(bar(kBarBand + j), kDrain1Warps);
    }
    for (int s = 0; s < kStages3; ++s) {
      mbar_init(smem_u32(&s3.full[s]), 1);
      mbar_init(smem_u32(&s3.empty[s]), 1);
    }
    for (int j = 0; j < 2; ++j) {
      mbar_init(smem_u32(&s3.done[j]), 1);
      mbar_init(smem_u32(&s3.freed[j]), kDrain3Warps);
      mbar_init(smem_u32(&s3.fin[j]), 1);
      s3.issued[j] = s3.landed[j] = 0;
    }
    mbar_init(smem_u32(&s3.bar_w), 1);
    for (int j = kBarW; j < 16; ++j) mbar_init(bar(j), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)),
                 "r"(kConvTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_s;
  const int64_t n_batches = (a.n + kP - 1) / kP;
  const int my_batches = (int)((n_batches - blockIdx.x + gridDim.x - 1) / gridDim.x);
  const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;  // a warp reads TMEM lane quarter warp & 3
  const int g = 4 * (warp & 3) + (lane >> 3), ri = lane & 7;     // grid position in the M tile, instance in the batch
  bool ok = true;

  if (warp < kDrain1Warps) {
    // ---- conv1 drain: warps w and w + 4 read the same lane quarter, each 16
    // channels of both output rows of a pair; bias, ReLU, bf16, band
    const int half = warp >> 2, ox = g;
    uint64_t bias[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) bias[j] = f32x2(sb[16 * half + 2 * j], sb[16 * half + 2 * j + 1]);
    uint8_t *const dst0 = sm + kAct1Off + (ox & 1) * kSubBytes + (ox >> 1) * 512 + ri * 16 + 2 * half * 128;
    uint32_t P = 0, slot = 0;
    for (int bi = 0; bi < my_batches && ok; ++bi) {
      for (int pr = 0; pr < 7; ++pr, ++P) {
        ok = mbar_wait(bar(kBarC1 + (P & 1)), (P >> 1) & 1);
        if (bi > 0 ? pr == 0 || pr == 2 || pr == 5 : pr == 5) {  // the last tile that read the slot
          const uint32_t T = 3 * bi + (pr == 0 ? -2 : pr == 2 ? -1 : 0);
          ok = ok && mbar_wait(bar(kBarC2 + (T & 1)), (T >> 1) & 1);
        }
        if (!__all_sync(0xFFFFFFFFu, ok)) {
          ok = false;
          break;
        }
        tc_fence_after();
        float v[32];  // columns 16 half .. of row 2 pr (v[0..15]) and of row 2 pr + 1 (v[16..31])
        const uint32_t d = tmem + lane_base + kD1Col + 64 * (P & 1) + 16 * half;
        tmem_ld16x2(d, d + 32, v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kBarD1f + (P & 1)));
        if (ox <= 13) {  // conv2 reads x <= 13
          uint8_t *const dst = dst0 + slot * kSlotBytes;
          const bool twice = slot == kBandSlots - 1 && pr < 6;
#pragma unroll
          for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              const uint4 o = relu_chunk(v + 16 * s2 + 8 * c, bias + 4 * c);
              uint8_t *const q = dst + 2 * s2 * kSubBytes + c * 128;
              *reinterpret_cast<uint4 *>(q) = o;
              if (twice) *reinterpret_cast<uint4 *>(q - (kBandSlots - 1) * kSlotBytes) = o;
            }
        }
        slot = next_slot(slot, pr);
        if (pr == 2 || pr == 4 || pr == 6) {  // three rows of a tile are there
          fence_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(kBarBand + ((3 * bi + (pr >> 1) - 1) & 1)));
        }
      }
    }
  } else if (warp < kDrain1Warps + kDrain2Warps) {
    // ---- conv2 drain: positions g = px + 7 (row of the tile), outputs at px <
    // 6, which add position g + 1's second half: by a shuffle, or from the next
    // lane quarter through the exchange buffer
    const int px = g % 7, qt = warp & 3;
    const bool valid = px < 6 && g < 14;
    float *const xb = reinterpret_cast<float *>(sm + kXbOff) + (lane & 7) * kXbPitch;
    uint32_t T = 0;
    for (int bi = 0; bi < my_batches && ok; ++bi) {
      const int64_t batch = blockIdx.x + (int64_t)bi * gridDim.x;
      for (int tt = 0; tt < 3 && ok; ++tt, ++T) {
        ok = all_ok<kDrain2Warps * 32>(1, mbar_wait(bar(kBarC2 + (T & 1)), (T >> 1) & 1));
        if (!ok) break;
        tc_fence_after();
        uint8_t *const dst = a.act2 + batch * (int64_t)kAct2Bytes + (px + 6 * (2 * tt + g / 7)) * 1024 + ri * 16;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[32], w[32];
          const uint32_t d = tmem + lane_base + kD2Col + 128 * (T & 1) + 32 * h;
          tmem_ld32x2(d, d + 64, v, w);
          if (h == 1) {  // accumulator read: tile T + 2 may have it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarD2f + (T & 1)));
            asm volatile("bar.sync 1, %0;" ::"r"(kDrain2Warps * 32) : "memory");  // the other half's rows were read
          }
          if (qt > 0 && lane < 8) xrow_put(xb + (qt - 1) * 8 * kXbPitch, w);
#pragma unroll
          for (int c = 0; c < 32; ++c) w[c] = __shfl_down_sync(0xFFFFFFFFu, w[c], 8);
          asm volatile("bar.sync 1, %0;" ::"r"(kDrain2Warps * 32) : "memory");
          if (qt < 3 && lane >= 24) xrow_get(xb + qt * 8 * kXbPitch, w);
#pragma unroll
          for (int c = 0; c < 32; ++c) v[c] += w[c];
          if (valid) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const ulonglong2 *const b2 = reinterpret_cast<const ulonglong2 *>(sb + 32 + 32 * h + 8 * c);
              const uint64_t bias[4] = {b2[0].x, b2[0].y, b2[1].x, b2[1].y};
              *reinterpret_cast<uint4 *>(dst + (4 * h + c) * 128) = relu_chunk(v + 8 * c, bias);
            }
          }
        }
      }
    }
  } else if (warp < kIssueWarp) {
    // ---- builders. A batch's frames lie in shared memory as packed rows (bit
    // x of row word y = pixel (x, y)), [row y][frame c][instance i], so that
    // the 32 lanes of a warp building one block position read 32 consecutive
    // words. Thread tb holds rows 2 y2, 2 y2 + 1 of all four frames of one
    // instance of the next batch in registers.
    const int bw = warp - kDrain1Warps - kDrain2Warps, tb = 32 * bw + lane, fi = tb & 7, y2 = tb >> 3;
    uint64_t *const fr = reinterpret_cast<uint64_t *>(sm + kFrOff);
    uint8_t *const blk = sm + kBlkOff + 4 * bw * 512 + lane * 16;
    // The observations may have been written by the kernel ahead in the stream
    // while this one was set up, so they are read with ordinary loads, which stay
    // behind the dependency wait; the read-only path is for memory that nothing
    // writes during the whole kernel. (Not past L1: a thread's eight 16-byte
    // loads of uint8 rows share a line.)
    uint64_t pf[8];  // [frame c][row 2 y2, 2 y2 + 1]
    auto load_words = [&](int64_t first) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        ulonglong2 v = make_ulonglong2(0, 0);
        if (first + fi < a.n)
          v = *reinterpret_cast<const ulonglong2 *>(a.obs_words + (first + fi) * 128 + c * 32 + 2 * y2);
        pf[2 * c] = v.x;
        pf[2 * c + 1] = v.y;
      }
    };
    // uint8 frames: frame c's two rows are 128 bytes, on their way while the
    // pairs between are built, then packed (nonzero -> 1)
    uint4 raw[8];
    auto load_bytes = [&](int64_t first, int c) {
#pragma unroll
      for (int q = 0; q < 8; ++q)
        raw[q] = first + fi < a.n
                     ? reinterpret_cast<const uint4 *>(a.obs_u8 + ((first + fi) * 128 + c * 32 + 2 * y2) * 64)[q]
                     : make_uint4(0, 0, 0, 0);
    };
    auto pack_bytes = [&](int c) {
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        uint32_t bits[2] = {0, 0};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 r = raw[4 * y + q];
          const uint32_t w4[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            // bit 0 of each byte that is not zero; the product gathers the four in its top byte
            const uint32_t m = ((((w4[e] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w4[e]) >> 7) & 0x01010101u;
            bits[q >> 1] |= ((m * 0x01020408u) >> 24) << (16 * (q & 1) + 4 * e);
          }
        }
        pf[2 * c + y] = (uint64_t)bits[0] | (uint64_t)bits[1] << 32;
      }
    };
    // block row: pixel rows 2 row, 2 row + 1; this warp's 4 of 16 positions
    auto expand_row = [&](int row, uint4(&o)[4]) {
      // 16 pixels of either pixel row: the even ones stay, the odd ones move up
      // to bit 16 and on, so a mask and a product give two bf16 (1.0 is 0x3F80)
      const uint16_t *const px = reinterpret_cast<const uint16_t *>(fr + 2 * row * 32 + lane) + bw;
      const uint32_t u0 = px[0], u1 = px[4 * 32];
      const uint32_t s0 = (u0 & 0x5555u) | (u0 & 0xAAAAu) << 15, s1 = (u1 & 0x5555u) | (u1 & 0xAAAAu) << 15;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t e0 = s0 >> (8 * (j >> 1)), e1 = s1 >> (8 * (j >> 1));
        const uint32_t m = 0x00010001u << (4 * (j & 1)), one = 0x3F80u >> (4 * (j & 1));
        o[j] = make_uint4((e0 & m) * one, (e0 & (m << 2)) * (one >> 2), (e1 & m) * one, (e1 & (m << 2)) * (one >> 2));
      }
    };
    auto put_row = [&](int row, const uint4(&o)[4]) {
#pragma unroll
      for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4 *>(blk + (16 * (row % (int)kBlkRows) + j) * 512) = o[j];
    };
    grid_dependency_wait();  // the observations
    if (kU8) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        load_bytes((int64_t)blockIdx.x * kP, c);
        pack_bytes(c);
      }
    } else {
      load_words((int64_t)blockIdx.x * kP);
    }
    uint32_t P = 0;
    for (int bi = 0; bi < my_batches; ++bi) {
      const int64_t next = (blockIdx.x + (int64_t)(bi + 1) * gridDim.x) * kP;  // past the end: rows of zeros
      ok = all_ok<kBuildWarps * 32>(2, ok);  // every builder has read the previous frames
      if (!ok) break;
#pragma unroll
      for (int k = 0; k < 8; ++k) fr[((2 * y2 + (k & 1)) * 4 + (k >> 1)) * 8 + fi] = pf[k];
      asm volatile("bar.sync 2, %0;" ::"r"(kBuildWarps * 32) : "memory");
#pragma unroll
      for (int pr = 0; pr < 7; ++pr, ++P) {
        // rows 2 pr + 1 and 2 pr + 2 take the places of rows that pair P - 2 read
        // last, a batch's rows 0 .. 2 those of the previous batch's last two pairs
        // (the pixels are expanded before the wait: what follows it delays the
        // pair's MMAs, and with them the pair after next)
        uint4 o0[4], o1[4], o2[4];
        if (pr == 0) expand_row(0, o0);
        expand_row(2 * pr + 1, o1);
        expand_row(2 * pr + 2, o2);
        if (ok && P >= 2) ok = mbar_wait(bar(kBarC1 + (P & 1)), ((P - 2) >> 1) & 1);
        if (pr == 0) {
          put_row(0, o0);
          put_row(1, o1);
          if (ok && P >= 1) ok = mbar_wait(bar(kBarC1 + ((P - 1) & 1)), ((P - 1) >> 1) & 1);
        } else {
          put_row(2 * pr + 1, o1);
        }
        put_row(2 * pr + 2, o2);
        fence_async_smem();
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (ok && lane == 0) mbar_arrive(bar(kBarBlk + (P & 1)));
        // (not before the first pair's fence, which would wait for them)
        if (!kU8 && pr == 1) load_words(next);
        if (kU8) {
          if (pr == 2) pack_bytes(0);
          if (pr == 4) pack_bytes(1);
          if (pr == 5) pack_bytes(2);
          if (pr == 0) load_bytes(next, 0);
          if (pr == 2) load_bytes(next, 1);
          if (pr == 4) load_bytes(next, 2);
          if (pr == 5) load_bytes(next, 3);
        }
      }
      if (kU8) pack_bytes(3);
    }
  } else {
    // ---- issuing warps: whole warps in step, one lane of which issues
    const int who = __shfl_sync(0xFFFFFFFFu, warp - kIssueWarp, 0);  // 0, 1: conv1 pairs of that parity; 2: conv2
    if (who == 0 && lane == 0) {
      mbar_expect_tx(bar(kBarW), kW1Bytes + kW2Bytes);
      bulk_g2s(sbase + kW1Off, a.w1, kW1Bytes, bar(kBarW));
      for (uint32_t o = 0; o < kW2Bytes; o += 16384) bulk_g2s(sbase + kW2Off + o, a.w2 + o, 16384, bar(kBarW));
    }
    __syncwarp();
    const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem, 0);
    ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar(kBarW), 0));
    if (who < 2) {
      // Both output rows of a pair in one N = 64 accumulator: block row j (shift
      // dx) feeds row 2p through tap (dx, dy = j) and row 2p + 1 through tap (dx,
      // dy = j - 1); W1 holds, per (j, dx), those two taps stacked over n (zeros
      // where a tap does not apply), so the MMAs of j = 1 read their A tile once
      // for 64 outputs. Those of j = 0 and 2 take the half that is not zero,
      // but for the first, which also clears row 2p + 1.
      const uint64_t a1d = sdesc(sbase + kBlkOff, 128, 512), b1d = sdesc(sbase + kW1Off, 1024, 128);
      const uint32_t d = tm + kD1Col + 64 * who;
      uint32_t pr = who;
      const uint32_t pairs = 7 * (uint32_t)my_batches;
      for (uint32_t P = who; P < pairs && ok; P += 2) {
        uint64_t ad[3];
        uint32_t slot = 2 * pr % kBlkRows;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          ad[j] = sdesc_at(a1d, slot * 16 * 512);
          slot = slot + 1 == kBlkRows ? 0 : slot + 1;
        }
        ok = __all_sync(0xFFFFFFFFu, (P < 2 || mbar_wait(bar(kBarD1f + who), ((P >> 1) - 1) & 1)) &&
                                         mbar_wait(bar(kBarBlk + who), (P >> 1) & 1));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
          for (int dx = 0; dx < 2; ++dx)
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
              mma_bf16_warp(d + (j == 2 ? 32 : 0), sdesc_at(ad[j], dx * 512 + kk * 256),
                       sdesc_at(b1d, (2 * j + dx) * 4096 + kk * 2048 + (j == 2 ? 32 * 16 : 0)),
                       idesc_bf16(128, j == 1 || (j | dx | kk) == 0 ? 64 : 32), (j | dx | kk) != 0);
        if (!(a.stall && P == 0)) mma_commit_warp(bar(kBarC1 + who));
        pr = pr >= 5 ? pr - 5 : pr + 2;
      }
    } else {
      const uint64_t a2d = sdesc(sbase + kAct1Off, 128, 512), b2d = sdesc(sbase + kW2Off, 2048, 128);
      const uint32_t tiles = 3 * (uint32_t)my_batches;
      int tt = 0;
      uint32_t slot = 0, s0 = 0, s1 = 0, s2 = 0;  // the next row's, and those of the tile's rows 0 .. 2
      for (uint32_t T = 0; T < tiles && ok; ++T) {
        s0 = s2;
        if (tt == 0) {
          s0 = slot;
          slot = next_slot(slot, 0);
        }
        s1 = slot;
        slot = next_slot(slot, 2 * tt + 1);
        s2 = slot;
        slot = next_slot(slot, 2 * tt + 2);
        const uint64_t at[2] = {sdesc_at(a2d, s0 % (kBandSlots - 1) * kSlotBytes), sdesc_at(a2d, s1 % (kBandSlots - 1) * kSlotBytes)};
        ok = __all_sync(0xFFFFFFFFu, (T < 2 || mbar_wait(bar(kBarD2f + (T & 1)), ((T >> 1) - 1) & 1)) &&
                                         mbar_wait(bar(kBarBand + (T & 1)), (T >> 1) & 1));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tm + kD2Col + 128 * (T & 1);
#pragma unroll
        for (int ky = 0; ky < 4; ++ky)
#pragma unroll
          for (int px = 0; px < 2; ++px)  // taps (px, ky) and (px + 2, ky)
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
              mma_bf16_warp(d, sdesc_at(at[ky >> 1], (px + 2 * (ky & 1)) * kSubBytes + kk * 256),
                       sdesc_at(b2d, (ky * 2 + px) * 8192 + kk * 4096), idesc_bf16(128, 128), (ky | px | kk) != 0);
        mma_commit_warp(bar(kBarC2 + (T & 1)));
        tt = tt == 2 ? 0 : tt + 1;
      }
    }
  }
  // conv2's output, written above, is read by bulk copies below, into shared
  // memory that was written and read above
  asm volatile("fence.proxy.async;" ::: "memory");
  tc_fence_before();
  ok = !__syncthreads_or(!ok);
  tc_fence_after();
  const bool third = ok;
  if (third) ok = conv3_batches(a, sm, s3, sb + 96, tmem, my_batches);
  ok = !__syncthreads_or(!ok);
  if (!ok) {  // the MMAs and copies of every issuing thread land before TMEM and shared memory go
    if (t == 0) atomicOr(a.err, 1u);
    if (warp >= kIssueWarp) {
      mma_commit_warp(bar(kBarFin + warp - kIssueWarp));
      mbar_wait(bar(kBarFin + warp - kIssueWarp), 0);
      if (warp == kIssueWarp) mbar_wait(bar(kBarW), 0);
    }
    if (third && warp >= kDrain3Warps && warp < kDrain3Warps + 2 && lane == 0) {
      const int who = warp - kDrain3Warps;
      mbar_wait(smem_u32(&s3.bar_w), 0);
      for (int q = s3.landed[who]; q < s3.issued[who]; ++q) mbar_wait(smem_u32(&s3.full[3 * who + q % 3]), (q / 3) & 1);
    }
    if (third && warp >= kDrain3Warps + 2 && warp < kDrain3Warps + 4 && lane == 0) {
      mma_commit(smem_u32(&s3.fin[warp - kDrain3Warps - 2]));
      mbar_wait(smem_u32(&s3.fin[warp - kDrain3Warps - 2]), 0);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kConvTmemCols));
}

struct HeadsArgs {
  const uint8_t *act3;
  int64_t n;
  const uint8_t *wh;     // [2][16 slices][8 chunks][256][16 B]
  const float *fp;       // FpLayout
  int L;
  float *logits;         // [n][L] or null
  float *value;          // [n] or null
  uint8_t *actions;      // [n] or null
  uint32_t key0, key1, step;
  unsigned int *err;
};

// MT tiles of 128 instances by a head's 256 hidden units per CTA; blockIdx.y: 0
// actor, 1 critic. K = 1024 comes in slices of 64 through a ring of stages (one
// thread issues the copies, another the MMAs).
template <int MT>
__global__ void __launch_bounds__(256 * MT, 1) policy_heads_kernel(const HeadsArgs a) {
  constexpr uint32_t kStage = MT * kHA + kHB, kCols = MT * 256;
  constexpr int kStages = kHeadRing / kStage, kSlices = 16, kThreads = 256 * MT;
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages], fin;
  __shared__ uint32_t tmem_s;
  __shared__ int s_landed;  // slices whose copies the MMA thread has waited for
  const int t = threadIdx.x, warp = t >> 5;
  const int head = blockIdx.y;
  const int64_t tile = (int64_t)blockIdx.x * MT;
  const uint32_t sbase = smem_u32(sm);
  float *wout = reinterpret_cast<float *>(sm + kHeadRing);        // actor [L][256] or critic [256]
  float *bias = wout + kMaxLogits * 256;                           // [256] hidden biases, then outputs'
  if (t == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    mbar_init(smem_u32(&fin), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_s;
  const uint8_t *A = a.act3 + tile * (int64_t)kAct3TileBytes;
  const uint8_t *B = a.wh + (int64_t)head * kSlices * kHB;
  bool ok = true;
  // Thread 0 issues the copies, thread 32 the MMAs: each runs its own chain of
  // waits and issues (a bulk copy or an MMA costs far more latency on the
  // issuing thread than its bytes or its share of the tensor pipe).
  int loaded = 0;           // thread 0: slices whose copies were issued
  if (t == 0) {
    // the first slices' weights need not wait for conv3
    for (int s = 0; s < kStages && s < kSlices; ++s) {
      const uint32_t f = smem_u32(&full[s]);
      mbar_expect_tx(f, kStage);
      bulk_g2s(sbase + s * kStage + MT * kHA, B + (int64_t)s * kHB, kHB, f);
    }
    grid_dependency_wait();  // conv3's features
    for (int s = 0; s < kSlices && ok; ++s) {
      const int st = s % kStages;
      const uint32_t f = smem_u32(&full[st]);
      if (s >= kStages) {  // stage st last held slice s - kStages: its MMAs must be done
        ok = mbar_wait(smem_u32(&empty[st]), ((s / kStages) - 1) & 1);
        if (!ok) break;
        mbar_expect_tx(f, kStage);
        bulk_g2s(sbase + st * kStage + MT * kHA, B + (int64_t)s * kHB, kHB, f);
      }
#pragma unroll
      for (int m = 0; m < MT; ++m)
        bulk_g2s(sbase + st * kStage + m * kHA, A + m * (int64_t)kAct3TileBytes + (int64_t)s * kHA, kHA, f);
      loaded = s + 1;
    }
  } else if (t == 32) {
    int landed = 0;
    for (int s = 0; s < kSlices && ok; ++s) {
      const int st = s % kStages;
      ok = mbar_wait(smem_u32(&full[st]), (s / kStages) & 1);
      if (!ok) break;
      landed = s + 1;
      tc_fence_after();
      const uint64_t a0 = sdesc(sbase + st * kStage, 2048, 128);
      const uint64_t b0 = sdesc(sbase + st * kStage + MT * kHA, 256 * 16, 128);
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_bf16(tmem + m * 256, sdesc_at(a0, m * kHA + kk * 2 * 2048), sdesc_at(b0, kk * 2 * 256 * 16),
                   idesc_bf16(128, 256), (s | kk) != 0);
      mma_commit(smem_u32(&empty[st]));
    }
    // the last slice's MMAs complete -> every earlier one has too
    if (ok) ok = mbar_wait(smem_u32(&empty[(kSlices - 1) % kStages]), ((kSlices - 1) / kStages) & 1);
    if (!ok) {  // let this thread's MMAs land before TMEM goes
      mma_commit(smem_u32(&fin));
      mbar_wait(smem_u32(&fin), 0);
    }
    s_landed = landed;
  } else if (warp >= 2) {  // meanwhile the output layers
    const int outs = head == 0 ? a.L : 1;
    const float *const w = a.fp + (head == 0 ? FpLayout::wa2 : FpLayout::wc2);
    const float *const b = a.fp + (head == 0 ? FpLayout::ba2 : FpLayout::bc2);
    for (int j = t - 64; j < outs * 256; j += kThreads - 64) wout[j] = w[j];
    for (int j = t - 64; j < 256; j += kThreads - 64) bias[j] = a.fp[FpLayout::bh + 256 * head + j];
    for (int j = t - 64; j < outs; j += kThreads - 64) bias[256 + j] = b[j];
  }
  ok = !__syncthreads_or(!ok);
  if (!ok && t == 0)  // copies issued but never waited for land before shared memory goes
    for (int q = s_landed; q < loaded; ++q) mbar_wait(smem_u32(&full[q % kStages]), (q / kStages) & 1);
  tc_fence_after();
  // A TMEM lane quarter (warp & 3) and half of the hidden units per warp;
  // the products of 32 hidden units with an output's weights meet in the stages'
  // shared memory, [tile][32 units][output][row]. Loops stay rolled: every
  // instruction here runs a few times only, so fetching it is what it costs
  // (unrolled over the outputs this took 10 K cycles of a tile pair's 33 K).
  const int row = t & 127, hh = (warp >> 2) & 1, m = warp >> 3;
  const int64_t inst = (tile + m) * 128 + row;
  const int outs = head == 0 ? a.L : 1;
  float *const sums = reinterpret_cast<float *>(sm) + m * (8 * kMaxLogits * 128) + row;
  if (ok) {
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
      const int unit = 128 * hh + 32 * c;
      float h[32];
      tmem_ld32(tmem + lane_base + m * 256 + unit, h);
      const float4 *const b4 = reinterpret_cast<const float4 *>(bias + unit);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 b = b4[j];
        h[4 * j] = fmaxf(h[4 * j] + b.x, 0.0f);
        h[4 * j + 1] = fmaxf(h[4 * j + 1] + b.y, 0.0f);
        h[4 * j + 2] = fmaxf(h[4 * j + 2] + b.z, 0.0f);
        h[4 * j + 3] = fmaxf(h[4 * j + 3] + b.w, 0.0f);
      }
#pragma unroll 1
      for (int o = 0; o < outs; ++o) {  // the weights as 8 vector loads, four independent partial sums
        const float4 *const w4 = reinterpret_cast<const float4 *>(wout + o * 256 + unit);
        float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 ww = w4[q];
          s0 = fmaf(h[4 * q], ww.x, s0);
          s1 = fmaf(h[4 * q + 1], ww.y, s1);
          s2 = fmaf(h[4 * q + 2], ww.z, s2);
          s3 = fmaf(h[4 * q + 3], ww.w, s3);
        }
        sums[((unit >> 5) * kMaxLogits + o) * 128] = (s0 + s1) + (s2 + s3);
      }
    }
  }
  __syncthreads();
  if (ok && !hh && inst < a.n) {
    float top = -INFINITY;
#pragma unroll 1
    for (int o = 0; o < outs; ++o) {
      float lo = 0.0f, hi = 0.0f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        lo += sums[(c * kMaxLogits + o) * 128];
        hi += sums[((4 + c) * kMaxLogits + o) * 128];
      }
      lo += hi;
      lo += bias[256 + o];
      top = fmaxf(top, lo);
      sums[o * 128] = lo;  // (this thread's own)
      if (head == 0) {
        if (a.logits) a.logits[inst * a.L + o] = lo;
      } else if (a.value) {
        a.value[inst] = lo;
      }
    }
    if (head == 0 && a.actions) {
      // inverse CDF: the first index whose cumulative weight exceeds u * total
      const uint32_t w = philox_w0((uint32_t)inst, a.step, 0u, 0u, a.key0, a.key1);
      const float u = (float)(w >> 8) * 5.9604644775390625e-08f;  // 2^-24
      float tot = 0.0f, run = 0.0f;
#pragma unroll 1
      for (int o = 0; o < outs; ++o) {
        const float e = expf(sums[o * 128] - top);
        sums[o * 128] = e;
        tot += e;
      }
      const float target = u * tot;
      int pick = 0;
#pragma unroll 1
      for (; pick < outs - 1; ++pick) {
        run += sums[pick * 128];
        if (target < run) break;
      }
      a.actions[inst] = (uint8_t)pick;
    }
  }
  if (!ok && t == 0) atomicOr(a.err, 1u);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
}

// ---- host: weight packing ----------------------------------------------------
uint16_t bf16_bits(float f) {
  __nv_bfloat16 h = __float2bfloat16_rn(f);
  uint16_t b;
  std::memcpy(&b, &h, 2);
  return b;
}

template <class Args>
cudaError_t launch(void (*kernel)(const Args), dim3 grid, int block, size_t smem, cudaStream_t s, Args &args) {
  void *list[] = {&args};
  return launch_kernel((const void *)kernel, grid, dim3((unsigned)block), list, smem, s, true);
}

int launch_forward(octax_policy *p, int64_t n, const uint64_t *obs_words, const uint8_t *obs_u8, uint64_t seed,
                   uint32_t step, float *logits, float *value, uint8_t *actions, cudaStream_t s) {
  if (n < 1 || n > p->max_envs) {
    set_error("octax_policy: need 1 <= n_envs <= max_envs of the policy");
    return OCTAX_EINVAL;
  }
  HeadsArgs h{p->act3, n, (const uint8_t *)p->wh, p->fp, p->n_logits, logits, value, actions,
              (uint32_t)seed, (uint32_t)(seed >> 32), step, p->err};
  // launches of about the same number of whole rounds, which begin at a tile of 128 instances
  const int64_t round = (int64_t)p->sms * kP, launches = (n + kMaxRounds * round - 1) / (kMaxRounds * round);
  const int64_t rounds = (n + launches * round - 1) / (launches * round);
  const int64_t per = std::min(((rounds + 1) / 2 * 2 * round + 127) / 128 * 128, kMaxRounds * round);  // instances of one
  cudaError_t r = cudaSuccess;
  for (int64_t i = 0; i < n; i += per) {
    const int64_t m = std::min(per, n - i);
    ConvArgs c{obs_words ? obs_words + i * 128 : nullptr, obs_u8 ? obs_u8 + i * 8192 : nullptr, m,
               (const uint8_t *)p->w1, (const uint8_t *)p->w2, (const uint8_t *)p->w3, p->fp, p->act2,
               p->act3 + i / 128 * (int64_t)kAct3TileBytes, p->err, p->stall};
    const unsigned grid = (unsigned)std::min<int64_t>((m + kP - 1) / kP, p->sms);
    r = obs_u8 ? launch(policy_conv_kernel<true>, dim3(grid), kConvThreads, kConvSmem, s, c)
               : launch(policy_conv_kernel<false>, dim3(grid), kConvThreads, kConvSmem, s, c);
    if (r != cudaSuccess) return cuda_fail(r, "policy conv launch");
  }
  // A CTA holds an SM's shared memory, so they run in waves of one per SM: one
  // tile each as long as that makes one wave, else two (the weights then come
  // in once for both).
  const unsigned tiles = (unsigned)((n + 127) / 128);
  r = 2 * (int64_t)tiles <= p->sms ? launch(policy_heads_kernel<1>, dim3(tiles, 2), 256, kHeadSmem, s, h)
                                   : launch(policy_heads_kernel<2>, dim3((tiles + 1) / 2, 2), 512, kHeadSmem, s, h);
  if (r != cudaSuccess) return cuda_fail(r, "policy heads launch");
  return OCTAX_OK;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace
}  // namespace octax

using namespace octax;

extern "C" {

int octax_policy_create(const octax_policy_params *prm, int64_t max_envs, int device, void *cuda_stream,
                        octax_policy **out) {
  if (!out || !prm || max_envs < 1 || max_envs > ((int64_t)1 << 31) || prm->n_logits < 1 ||
      prm->n_logits > kMaxLogits) {
    set_error("octax_policy_create: need params, out, 1 <= max_envs <= 2^31, 1 <= n_logits <= 17");
    return OCTAX_EINVAL;
  }
  *out = nullptr;
  const float *need[] = {prm->w1, prm->b1, prm->w2, prm->b2, prm->w3, prm->b3, prm->wa1,
                         prm->ba1, prm->wa2, prm->ba2, prm->wc1, prm->bc1, prm->wc2, prm->bc2};
  for (const float *q : need)
    if (!q) {
      set_error("octax_policy_create: every parameter array is required");
      return OCTAX_EINVAL;
    }
  cudaError_t r = cudaSetDevice(device);
  if (r != cudaSuccess) return cuda_fail(r, "octax_policy_create: cudaSetDevice");
  const int L = prm->n_logits;
  // conv1 B, per block row j (0..2) and shift dx: [j][dx][chunk = frame c][n 64][k' = kx + 4 ky];
  // n < 32: w1[n][c][4 dx + kx][2 j + ky] (tap dy = j, for j <= 1), n >= 32: w1[n - 32][c][4 dx + kx][2 (j - 1) + ky]
  // (tap dy = j - 1, for j >= 1), zero otherwise
  std::vector<uint16_t> w1p(6 * 4 * 64 * 8, 0);
  for (int j = 0; j < 3; ++j)
    for (int dx = 0; dx < 2; ++dx)
      for (int c = 0; c < 4; ++c)
        for (int n = 0; n < 64; ++n) {
          const int dy = n < 32 ? j : j - 1, o = n & 31;
          if (dy < 0 || dy > 1) continue;
          for (int k = 0; k < 8; ++k) {
            const int kx = 4 * dx + (k & 3), ky = 2 * dy + (k >> 2);
            w1p[(((j * 2 + dx) * 4 + c) * 64 + n) * 8 + k] = bf16_bits(prm->w1[((o * 4 + c) * 8 + kx) * 4 + ky]);
          }
        }
  // conv2 B: [ky][px = kx & 1][chunk j][n = 64 (kx >> 1) + o][e] = w2[o][8 j + e][kx][ky]
  // (taps kx and kx + 2 stacked along N)
  std::vector<uint16_t> w2p(4 * 2 * 4 * 128 * 8);
  for (int ky = 0; ky < 4; ++ky)
    for (int px = 0; px < 2; ++px)
      for (int j = 0; j < 4; ++j)
        for (int n = 0; n < 128; ++n)
          for (int e = 0; e < 8; ++e) {
            const int kx = px + 2 * (n >> 6), o = n & 63;
            w2p[((((ky * 2 + px) * 4 + j) * 128 + n) * 8) + e] =
                bf16_bits(prm->w2[((o * 32 + 8 * j + e) * 4 + kx) * 4 + ky]);
          }
  // conv3 B: [ky][chunk j][n = 64 kx + o][e] = w3[o][8 j + e][kx][ky] (the three taps of a
  // kernel row stacked along N)
  std::vector<uint16_t> w3p(3 * 8 * 192 * 8);
  for (int ky = 0; ky < 3; ++ky)
    for (int j = 0; j < 8; ++j)
      for (int n = 0; n < 192; ++n)
        for (int e = 0; e < 8; ++e) {
          const int kx = n >> 6, o = n & 63;
          w3p[((ky * 8 + j) * 192 + n) * 8 + e] = bf16_bits(prm->w3[((o * 64 + 8 * j + e) * 3 + kx) * 3 + ky]);
        }
  // heads B: [head][slice q (16)][chunk j][n 256][e]; feature k = 64 q + channel (q = qx + 4 qy),
  // the caller's flatten index is channel * 16 + qx * 4 + qy
  std::vector<uint16_t> whp(2 * 16 * 8 * 256 * 8);
  for (int head = 0; head < 2; ++head) {
    const float *W = head ? prm->wc1 : prm->wa1;
    for (int q = 0; q < 16; ++q)
      for (int j = 0; j < 8; ++j)
        for (int n = 0; n < 256; ++n)
          for (int e = 0; e < 8; ++e) {
            const int ch = 8 * j + e, qx = q & 3, qy = q >> 2;
            whp[((((size_t)head * 16 + q) * 8 + j) * 256 + n) * 8 + e] =
                bf16_bits(W[(size_t)n * 1024 + ch * 16 + qx * 4 + qy]);
          }
  }
  std::vector<float> fp(FpLayout::total, 0.0f);
  std::memcpy(&fp[FpLayout::b1], prm->b1, 32 * 4);
  std::memcpy(&fp[FpLayout::b2], prm->b2, 64 * 4);
  std::memcpy(&fp[FpLayout::b3], prm->b3, 64 * 4);
  std::memcpy(&fp[FpLayout::bh], prm->ba1, 256 * 4);
  std::memcpy(&fp[FpLayout::bh + 256], prm->bc1, 256 * 4);
  std::memcpy(&fp[FpLayout::wa2], prm->wa2, (size_t)L * 256 * 4);
  std::memcpy(&fp[FpLayout::ba2], prm->ba2, (size_t)L * 4);
  std::memcpy(&fp[FpLayout::wc2], prm->wc2, 256 * 4);
  fp[FpLayout::bc2] = prm->bc2[0];

  octax_policy *p = new octax_policy();
  p->device = device;
  p->n_logits = L;
  p->max_envs = max_envs;
  cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, device);
  if (p->sms < 1) p->sms = 1;
  const int64_t tiles = (max_envs + 255) / 256 * 2;  // (the heads kernel reads them in pairs)
  auto fail = [&](cudaError_t e, const char *what) {
    octax_policy_destroy(p);
    return cuda_fail(e, what);
  };
  if ((r = cudaMalloc(&p->w1, w1p.size() * 2)) != cudaSuccess) return fail(r, "octax_policy_create: alloc");
  if ((r = cudaMalloc(&p->w2, w2p.size() * 2)) != cudaSuccess) return fail(r, "octax_policy_create: alloc");
  if ((r = cudaMalloc(&p->w3, w3p.size() * 2)) != cudaSuccess) return fail(r, "octax_policy_create: alloc");
  if ((r = cudaMalloc(&p->wh, whp.size() * 2)) != cudaSuccess) return fail(r, "octax_policy_create: alloc");
  if ((r = cudaMalloc((void **)&p->fp, fp.size() * 4)) != cudaSuccess) return fail(r, "octax_policy_create: alloc");
  const int64_t batches = std::min<int64_t>((max_envs + kP - 1) / kP, (int64_t)kMaxRounds * p->sms);
  if ((r = cudaMalloc((void **)&p->act2, (size_t)batches * kAct2Bytes)) != cudaSuccess)
    return fail(r, "octax_policy_create: alloc");
  if ((r = cudaMalloc((void **)&p->act3, (size_t)tiles * kAct3TileBytes)) != cudaSuccess)
    return fail(r, "octax_policy_create: alloc");
  if ((r = cudaMalloc((void **)&p->ring, (size_t)2 * max_envs * 1024)) != cudaSuccess)
    return fail(r, "octax_policy_create: alloc");
  if ((r = cudaMalloc((void **)&p->err, 4)) != cudaSuccess) return fail(r, "octax_policy_create: alloc");
  if (cuda_stream) {
    p->stream = static_cast<cudaStream_t>(cuda_stream);
  } else {
    if ((r = cudaStreamCreateWithFlags(&p->stream, cudaStreamNonBlocking)) != cudaSuccess)
      return fail(r, "octax_policy_create: stream");
    p->own_stream = true;
  }
  r = cudaMemcpy(p->w1, w1p.data(), w1p.size() * 2, cudaMemcpyHostToDevice);
  if (r == cudaSuccess) r = cudaMemcpy(p->w2, w2p.data(), w2p.size() * 2, cudaMemcpyHostToDevice);
  if (r == cudaSuccess) r = cudaMemcpy(p->w3, w3p.data(), w3p.size() * 2, cudaMemcpyHostToDevice);
  if (r == cudaSuccess) r = cudaMemcpy(p->wh, whp.data(), whp.size() * 2, cudaMemcpyHostToDevice);
  if (r == cudaSuccess) r = cudaMemcpy(p->fp, fp.data(), fp.size() * 4, cudaMemcpyHostToDevice);
  if (r == cudaSuccess) r = cudaMemset(p->act3, 0, (size_t)tiles * kAct3TileBytes);
  if (r == cudaSuccess) r = cudaMemset(p->ring, 0, (size_t)2 * max_envs * 1024);
  if (r == cudaSuccess) r = cudaMemset(p->err, 0, 4);
  if (r == cudaSuccess)
    r = cudaFuncSetAttribute(policy_conv_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvSmem);
  if (r == cudaSuccess)
    r = cudaFuncSetAttribute(policy_conv_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvSmem);
  if (r == cudaSuccess)
    r = cudaFuncSetAttribute(policy_heads_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kHeadSmem);
  if (r == cudaSuccess)
    r = cudaFuncSetAttribute(policy_heads_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kHeadSmem);
  if (r != cudaSuccess) return fail(r, "octax_policy_create: upload");
  *out = p;
  return OCTAX_OK;
}

int octax_policy_forward(octax_policy *p, int64_t n_envs, const uint64_t *obs_words_dev, uint64_t seed, uint32_t step,
                         float *logits_dev, float *value_dev, uint8_t *actions_dev) {
  if (!p || !obs_words_dev || !aligned16(obs_words_dev)) {
    set_error("octax_policy_forward: need a policy and 16-byte aligned packed observations");
    return OCTAX_EINVAL;
  }
  cudaError_t r = cudaSetDevice(p->device);
  if (r != cudaSuccess) return cuda_fail(r, "octax_policy_forward: cudaSetDevice");
  return launch_forward(p, n_envs, obs_words_dev, nullptr, seed, step, logits_dev, value_dev, actions_dev,
                        p->stream);
}

int octax_policy_forward_u8(octax_policy *p, int64_t n_envs, const uint8_t *obs_dev, uint64_t seed, uint32_t step,
                            float *logits_dev, float *value_dev, uint8_t *actions_dev) {
  if (!p || !obs_dev || !aligned16(obs_dev)) {
    set_error("octax_policy_forward_u8: need a policy and 16-byte aligned observations");
    return OCTAX_EINVAL;
  }
  cudaError_t r = cudaSetDevice(p->device);
  if (r != cudaSuccess) return cuda_fail(r, "octax_policy_forward_u8: cudaSetDevice");
  return launch_forward(p, n_envs, nullptr, obs_dev, seed, step, logits_dev, value_dev, actions_dev, p->stream);
}

int octax_rollout_policy(octax_env *e, octax_policy *p, int n_steps, uint64_t seed, uint32_t step0,
                         uint64_t *obs_words_dev, uint8_t *actions_dev, float *logits_dev, float *value_dev,
                         float *reward_dev, uint8_t *done_dev) {
  if (!e || !p || n_steps < 1 || !obs_words_dev || !aligned16(obs_words_dev) || !actions_dev || !value_dev ||
      !reward_dev || !done_dev) {
    set_error("octax_rollout_policy: need env, policy, n_steps >= 1, aligned obs_words, actions, value, "
              "reward and done");
    return OCTAX_EINVAL;
  }
  const int64_t n = octax_num_envs(e);
  if (octax_stack_frames(e) != 4 || octax_variant(e) != OCTAX_VARIANT_CHIP8 || n > p->max_envs ||
      env_device(e) != p->device) {
    set_error("octax_rollout_policy: the network takes CHIP-8 environments with 4 stacked frames, at most "
              "max_envs instances, on the policy's device");
    return OCTAX_EINVAL;
  }
  cudaError_t r = cudaSetDevice(p->device);
  if (r != cudaSuccess) return cuda_fail(r, "octax_rollout_policy: cudaSetDevice");
  cudaStream_t s = env_stream(e);
  const size_t obs_bytes = (size_t)n * 1024;
  uint64_t *slot[2] = {p->ring, p->ring + (size_t)p->max_envs * 128};
  r = cudaMemcpyAsync(slot[0], obs_words_dev, obs_bytes, cudaMemcpyDeviceToDevice, s);
  if (r != cudaSuccess) return cuda_fail(r, "octax_rollout_policy: observation copy");
  int cur = 0;
  for (int k = 0; k < n_steps; ++k) {
    uint8_t *act = actions_dev + (size_t)k * n;
    int rc = launch_forward(p, n, slot[cur], nullptr, seed, step0 + (uint32_t)k,
                            logits_dev ? logits_dev + (size_t)k * n * p->n_logits : nullptr,
                            value_dev + (size_t)k * n, act, s);
    if (rc) return rc;
    rc = octax_step_n_packed(e, 1, act, slot[cur ^ 1], reward_dev + (size_t)k * n, done_dev + (size_t)k * n);
    if (rc) return rc;
    cur ^= 1;
  }
  r = cudaMemcpyAsync(obs_words_dev, slot[cur], obs_bytes, cudaMemcpyDeviceToDevice, s);
  if (r != cudaSuccess) return cuda_fail(r, "octax_rollout_policy: observation copy");
  return OCTAX_OK;
}

int octax_policy_sync(octax_policy *p) {
  if (!p) {
    set_error("octax_policy_sync: need a policy");
    return OCTAX_EINVAL;
  }
  cudaError_t r = cudaSetDevice(p->device);
  if (r == cudaSuccess) r = cudaStreamSynchronize(p->stream);
  if (r == cudaSuccess) r = cudaDeviceSynchronize();
  if (r != cudaSuccess) return cuda_fail(r, "octax_policy_sync");
  unsigned int h = 0;
  r = cudaMemcpy(&h, p->err, 4, cudaMemcpyDeviceToHost);
  if (r != cudaSuccess) return cuda_fail(r, "octax_policy_sync");
  if (h) {
    cudaMemset(p->err, 0, 4);
    set_error("octax_policy_sync: a policy kernel gave up a bounded wait; its outputs are incomplete");
    return OCTAX_ECUDA;
  }
  return OCTAX_OK;
}

int octax_policy_debug_stall(octax_policy *p, int on) {
  if (!p) {
    set_error("octax_policy_debug_stall: need a policy");
    return OCTAX_EINVAL;
  }
  p->stall = on != 0;
  return OCTAX_OK;
}

void octax_policy_destroy(octax_policy *p) {
  if (!p) return;
  cudaSetDevice(p->device);
  if (p->stream) cudaStreamSynchronize(p->stream);
  for (void *q : {p->w1, p->w2, p->w3, p->wh, (void *)p->fp, (void *)p->act2, (void *)p->act3, (void *)p->ring, (void *)p->err})
    if (q) cudaFree(q);
  if (p->own_stream && p->stream) cudaStreamDestroy(p->stream);
  delete p;
}

}  // extern "C"
