// Internal declarations shared by the liboctax translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "octax.h"

namespace octax {

constexpr int kRamBytes = 4096;
constexpr int kPageShift = 6;               // 64-byte RAM pages: 64 pages -> one u64 mask
// Written-address range of an instance, lo | hi << 16 (lo > hi: nothing written).
constexpr uint32_t kNoWrites = 0x0FFFu;
constexpr int kFrameBytes = 32 * 64;        // one uint8 CHIP-8 observation frame
constexpr int kSchipFrameBytes = 64 * 128;  // one uint8 SCHIP observation frame (the 128x64 buffer)
constexpr uint32_t kBigFontAddr = 0x0A0;    // SCHIP 8x10 glyphs, 10 bytes each
// Packed display words (u64) per instance: 32 rows x 1 (CHIP-8), 64 rows x 2 (SCHIP).
constexpr int kDispWords = 32;
constexpr int kSchipDispWords = 128;
__host__ __device__ inline int frame_bytes(int schip) { return schip ? kSchipFrameBytes : kFrameBytes; }
__host__ __device__ inline int disp_words(int schip) { return schip ? kSchipDispWords : kDispWords; }
// A packed observation frame: the display words themselves (u64, bit x of a
// word = pixel x of its 64-pixel run).
__host__ __device__ inline int packed_frame_bytes(int schip) { return 8 * disp_words(schip); }
constexpr int kMaxBlock = 256;

// Game descriptor as the kernels read it (one per game, device memory).
struct TermDev {
  uint8_t src, xform;
  uint16_t idx;
  int32_t arg;
};
struct ClauseDev {
  TermDev lhs;
  int32_t cmp;
  int32_t rhs;
};
struct alignas(16) GameDev {
  uint32_t K, frameskip, n_actions, n_score, n_term, max_steps, startup, sticky;
  uint32_t max_noops, variant, pad[2];
  uint8_t action_set[16];
  TermDev score[4];
  ClauseDev term[4];
};
static_assert(sizeof(GameDev) <= 192, "GameDev must fit its shared-memory slot");
constexpr int kGameSmem = 192;
constexpr int kLutSmem = 256 * 8;            // byte of pixels -> 8 output bytes
// What a CTA stages of its game, one contiguous blob per game in device
// memory, in this order: RAM image | descriptor | pixel table | coefficients |
// micro-ops (one per even address from table_base on, to the end of the longest
// ROM, and a sentinel; 8 bytes of each, then 4 bytes of each).
constexpr int kBlobLut = kRamBytes + kGameSmem;
constexpr int kBlobCoef = kBlobLut + kLutSmem;
constexpr int kBlobUops = kBlobCoef + 64;
__host__ __device__ constexpr uint32_t blob_bytes(uint32_t n_uops) {
  return ((uint32_t)kBlobUops + 12 * (n_uops + 1) + 15) & ~15u;
}
// First address of a table of n_uops micro-ops: that of the ROM, or 0 where the
// longest ROM has more than 3,072 bytes. Programs that fall through into the
// memory below the ROM (random ones end up there: 7 of 10 of their instructions
// after 200 steps) then leave the datapath no more; the 3 KB this takes are a
// seventh of what such an environment's CTAs stage. 262,144 random programs of
// 3,584 bytes, 2,000 steps: 414 us a step with the ROM's addresses alone, 397
// with all; 16,384 and 65,536 of them 1-5 % faster, template programs padded to
// that length 0.7 % faster to 1 % slower. At 3,072 bytes neither side leads
// (0.94-1.04); at 1,024, where a CTA of 32 instances loses one of eight resident
// ones, template programs lose 5 %.
constexpr int kLongTable = 3072 / 2;
__host__ __device__ constexpr uint32_t table_base(uint32_t n_uops) { return n_uops > (uint32_t)kLongTable ? 0u : 0x200u; }
inline size_t blob_stride(int n_uops) { return ((size_t)blob_bytes((uint32_t)n_uops) + 255) & ~(size_t)255; }

// Emulator state: one record of 32-bit words per slot (slot = index), the same
// words in device memory and, while a CTA steps the instance, in shared memory:
// a warp moves the records of its instances as one run of 16-byte pieces.
// Words, after the packed display (64, SCHIP 256):
//   +0 V0-VF  +4 DT | last action | ST | 15 (bytes)  +5 PC | I << 16
//   +6 SP | hires << 7 | status << 8 | game << 16  +7 written range  +8 dirty pages (u64)
//   +10 episode steps  +11 env steps  +12 stack (16 x u16)  +20 uid  +21 Philox key (2)
//   +23 output row  [SCHIP: +24 flag registers (16 bytes)]
// The lengths, 92 and 284 words, are 28 mod 32: instances next to each other
// start four banks apart.
constexpr int kRecTail = 28;
template <bool kS>
struct Rec {
  static constexpr int kV = kS ? 256 : 64;
  static constexpr int kPseudo = kV + 4, kPcI = kV + 5, kMisc = kV + 6, kWrange = kV + 7, kDirty = kV + 8, kEp = kV + 10,
                       kEnv = kV + 11, kStack = kV + 12, kUid = kV + 20, kKey = kV + 21, kRow = kV + 23, kRpl = kV + 24,
                       kWords = kV + kRecTail;
};
static_assert(Rec<false>::kWords % 4 == 0 && Rec<true>::kWords % 4 == 0, "records move as 16-byte pieces");
__host__ __device__ inline int rec_words(int schip) { return schip ? Rec<true>::kWords : Rec<false>::kWords; }

struct DevState {
  int64_t n;              // slots
  uint32_t *rec;          // [n][rec_words]
  uint8_t *ram;           // [n][4096] per-instance RAM (valid on dirty pages only)
  int schip;              // 1: SCHIP layout
};

// Every per-slot array is set (checked on the host before each launch).
inline bool state_complete(const DevState &s) { return s.n > 0 && s.rec && s.ram; }

// A group: up to block/32*ipw consecutive slots that share one game (one CTA's work).
struct Group {
  uint32_t slot0;
  uint16_t count;
  uint16_t game;
  uint32_t io;            // index into the IO table (0 when launched with io0)
  uint32_t row0;          // output row of slot0 within its request (serving resets)
};

// Where one request's per-step inputs and outputs live.
struct IO {
  const uint8_t *actions;  // [steps][rows]
  uint8_t *obs;            // [steps][rows][S][H][W]
  float *reward;           // [steps][rows]
  uint8_t *done;           // [steps][rows]
  int64_t rows;            // rows per step
  int32_t packed;          // 1: obs frames are the packed display words (packed_frame_bytes)
  int32_t pad;
};

struct StepLaunch {
  DevState st;
  const uint8_t *blobs;    // [n_games][blob_stride(n_uops)]
  int n_uops;              // micro-ops per game
  uint32_t stride;         // blob_stride of the table as built
  const Group *groups;
  int n_groups;
  IO io0;                  // used when io_table == nullptr
  const IO *io_table;
  int step0;               // output step index of this launch's first step
  int steps;               // env steps in this launch
  int S;                   // stack frames
  uint32_t quirks;
  int ipw;                 // instances emulated per warp (1..32)
  int writers;             // >0: warp-specialised kernel with this many writer warps
  unsigned int *work_counter;  // non-null: persistent CTAs pull groups from it
  unsigned int *err;       // set when a bounded barrier wait gives up (specialised kernel)
  int wrappers;            // 1: some game uses sticky actions or no-op reset (kernel variant)
  int stall_writers;       // diagnostic: writer warps skip the hand-over (specialised kernel)
};

struct ResetLaunch {
  DevState st;
  const uint8_t *blobs;
  int n_uops;
  uint32_t stride;
  const Group *groups;
  int n_groups;
  const uint8_t *mask;     // [n_out_rows] by out_row, nullable = all
  uint8_t *obs;            // [rows][S][32][64] by out_row, nullable
  int S;
  uint32_t quirks;
  int ipw;
  int init;                // 1: also set key/uid/env_steps/status (creation)
  uint64_t seed;
  const uint32_t *row_of_slot;  // used when init (nullable = group.row0 + lane)
  const uint32_t *uid_of_slot;  // used when init (nullable = the row)
  const uint64_t *seed_of_group;  // init: per-group seed (nullable = seed)
};

// Dynamic shared memory of a step CTA with a table of n_uops micro-ops.
size_t step_smem_bytes(int block, int ipw, int schip, int n_uops);
// Warp-specialised kernel: `block` emulator threads plus 32 * writers writer threads.
size_t step_ws_smem_bytes(int block, int ipw, int n_uops);
size_t max_dynamic_smem();
// The launch shapes that are accepted: what a CTA's instances may take of shared memory.
bool shape_fits(int block, int ipw, int schip, int writers);
// Instances per warp, at most ipw, that an accepted shape launches beside a table of n_uops micro-ops.
int fit_ipw(int block, int ipw, int schip, int writers, int n_uops);
// Fills the pixel table and the micro-ops of every blob from its RAM image.
cudaError_t launch_tables(uint8_t *blobs, size_t stride, int n_games, int n_uops, int schip, uint32_t quirks,
                          cudaStream_t s);
cudaError_t launch_step(const StepLaunch &p, int grid, int block, cudaStream_t s);
cudaError_t launch_reset(const ResetLaunch &p, int block, cudaStream_t s);
cudaError_t launch_hash(const DevState &st, const uint8_t *blobs, size_t stride, const uint32_t *slot_of_row,
                        int64_t rows, uint64_t *out, cudaStream_t s);
cudaError_t launch_records(const DevState &st, const uint8_t *blobs, size_t stride, const uint32_t *slot_of_row,
                           int64_t first, int64_t count, octax_state_record *out, cudaStream_t s);
cudaError_t launch_set_records(const DevState &st, const uint8_t *blobs, size_t stride, const uint32_t *slot_of_row,
                               int64_t first, int64_t count, const octax_state_record *in, cudaStream_t s);
int max_resident_ctas(int block, int ipw, int writers, int wrappers, int schip, int n_uops);
// True when a game enables the sticky-action or no-op-reset wrapper.
inline int uses_wrappers(const GameDev *games, size_t n) {
  for (size_t i = 0; i < n; ++i)
    if (games[i].sticky != 0u || games[i].max_noops != 0u) return 1;
  return 0;
}
// Bytes of device memory that a server's budget is charged per slot; the
// record and the RAM take 4,464 (SCHIP 5,232) of them.
constexpr size_t kSlotStateBytes = 4468, kSchipSlotStateBytes = 5236;
inline size_t slot_state_bytes(int schip) { return schip ? kSchipSlotStateBytes : kSlotStateBytes; }
static_assert(4 * Rec<false>::kWords + kRamBytes <= kSlotStateBytes, "slot fits its charge");
static_assert(4 * Rec<true>::kWords + kRamBytes <= kSchipSlotStateBytes, "slot fits its charge");
cudaError_t alloc_state(DevState &st, int64_t n, int schip, void **block_out, size_t *bytes_out);
// Append one step launch to a graph (after `dep`, if non-null).
cudaError_t add_step_node(cudaGraph_t g, cudaGraphNode_t *node, cudaGraphNode_t dep, const StepLaunch &p,
                          int grid, int block);

// Validate game descriptors; build device descriptors and 4 KB RAM images.
int build_games(const octax_game *games, int n_games, std::vector<GameDev> &dev,
                std::vector<uint8_t> &images);
// Micro-op table length for these games (entries to the end of the longest ROM).
int table_uops(const octax_game *games, int n_games);
// Upload the blobs of `games` (device memory of n * blob_stride bytes) and build their tables.
cudaError_t upload_blobs(const std::vector<GameDev> &games, const std::vector<uint8_t> &images, int n_uops, int schip,
                         uint32_t quirks, uint8_t *blobs, cudaStream_t s);

// Instances per warp for n instances on `sms` SMs.
int spread_ipw(int64_t n, int sms, int schip);
// The most it gives.
inline int most_spread_ipw(int schip) { return schip ? 8 : 16; }

// Programmatic dependent launch: a kernel launched with `dependent` may be set
// up before the one ahead of it in the stream has ended. It touches nothing
// that another kernel may write before its grid_dependency_wait(), which
// returns when the kernels ahead have ended, and lets its own successor be set
// up (grid_dependents_launch()) only after that, or where all it writes follows
// from data read after that: so no two kernels of a stream run side by side
// but for their set-up.
#ifdef __CUDACC__
__device__ __forceinline__ void grid_dependents_launch() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif
inline cudaError_t launch_kernel(const void *fn, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t s,
                                 bool dependent) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// Error reporting (thread-local message).
void set_error(const std::string &msg);
int cuda_fail(cudaError_t e, const char *what);

}  // namespace octax
