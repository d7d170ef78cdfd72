// liboctax device code: the vectorised CHIP-8 environment step for sm_103a.
//
// Mapping (one CTA = one group of block/32 * ipw instances of one game):
//  - each warp emulates `ipw` instances with L = 32 / ipw lanes each (rounded
//    to a power of two). The L lanes of an instance execute the same
//    instructions on the same values; they split what has parts: the rows of a
//    sprite, a clear, a copy. Display row y belongs to lane y mod L;
//  - an instance's state is one record of 32-bit words, in device memory and in
//    shared memory alike, so that a warp fetches and returns the records of its
//    instances as one run of 16-byte pieces. PC/I/SP/status, the 64-bit
//    dirty-page mask and the written-address range live in registers; V0-VF and
//    the timers as bytes in shared memory, a copy per lane (20 bytes apart:
//    five banks, so lanes on the same register never collide), which keeps
//    lanes from ever waiting for one another over a register;
//  - the game's initial 4 KB RAM image (font + ROM) is staged once per CTA in
//    shared memory and is read-only; an instance's writes go to 64-byte pages
//    of its own RAM in global memory, tracked by the dirty mask. Sprites and
//    fetches use the image whenever their bytes lie outside the range of
//    addresses written since the reset (data packed next to a score buffer);
//    other reads unless their page is dirty. A reset only clears the mask and
//    the range;
//  - dispatch limits divergence: the common opcodes (jumps, skips, loads,
//    adds, 8XYN ALU, key tests, timers, FX29) run through one branch-free
//    datapath that every lane executes together: one signed byte dot product
//    (VX, VY, VX & VY, VX >> 1) . coefficients + immediate, whose low byte is
//    the result, whose bit 8 is the flag and which decides a skip by being
//    zero; the next PC is one of two that the micro-op carries. Micro-ops are
//    decoded once per environment (tables_kernel) for every even address of
//    the ROM (of a long ROM, from address 0 on: table_base) and staged with the
//    image. DXYN has a branch of its own; the
//    rest (CXNN, calls and returns, 00E0, BCD and bulk memory ops, odd or
//    written addresses, undefined encodings, the Super-CHIP forms) takes a
//    divergent switch;
//  - observation frames are expanded from the packed rows by the whole warp
//    together (a byte of pixels becomes 8 bytes through a 256-entry table in
//    shared memory): every store is a 16-byte streaming store and each store
//    instruction writes complete 64-byte image rows (CHIP-8) or 128-byte rows
//    (Super-CHIP). They can also be written one bit per pixel (the display
//    words themselves), 8x fewer bytes.
// Each instance runs exactly K instructions per frame, so all lanes of a warp
// meet at every frame boundary.
//
// What bounds it: below a few thousand instances the dependent chain of one
// instruction (micro-op load, register loads, compare, next offset); in the
// middle the warp instructions per emulated instruction; above, the frame
// stores. Measured against the form before it (a lane per instance with the
// others idle, 8- or 16-byte micro-ops decoded by every CTA, registers as
// 32-bit words interleaved over the CTA, coefficient rows and separate
// selects per instruction class): one step of 64 template instances 11.0 ->
// 6.2 us, of 16,384 34.2 -> 20.9 us (7.0 TB/s), 16 packed steps of 12,289
// shooter instances 352 -> 163 us, 8 Super-CHIP steps of 8,192 492 -> 303 us,
// 8 steps of 65,536 over 16 ROMs 978 -> 836 us, 4 steps of 262,144 random
// programs 1,472 -> 1,391 us. The micro-ops take 12 bytes and not 16 so that
// a CTA of 64 instances with a 3.5 KB ROM keeps four CTAs per SM (random
// programs 1,683 us with 16); the pixel table stays because expanding by
// multiplication costs the issue-bound cases 1 % (it gains 7 % on one step of
// 16,384); three CTAs of 256 threads per SM (80 registers) lose 8 % there.
#include <algorithm>
#include <map>
#include <mutex>
#include <cstring>

#include "octax_internal.h"

namespace octax {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// The CTA's dynamic shared memory: the game's blob (its RAM image first),
// the records, the lanes' registers. Reading the image
// through this array (not through a pointer) keeps those loads in the shared
// state space.
extern __shared__ __align__(16) uint8_t g_smem[];

__device__ __forceinline__ uint32_t img_byte(uint32_t a) { return g_smem[a]; }

struct Regs {
  uint32_t pc, I, sp, status;
  uint64_t dirty;
  uint32_t draws, phase, env_steps;
  uint32_t hires;     // SCHIP: 1 in 128x64 mode
  uint32_t wrange;    // lowest | highest << 16 RAM address written since the reset
  uint32_t wbase, wspan;  // the same as micro-op offsets (set_range): a fetch at offset o may read a
                          // written byte if o - wbase <= wspan
};

struct Ctx {
  uint8_t *V;          // shared: this lane's V0-VF, DT, last action, ST, 15
  uint32_t *rec;       // shared: this instance's record
  uint8_t *ram;        // global: this instance's 4 KB RAM (dirty pages)
  uint32_t n_uops;     // entries of the micro-op table (the sentinel follows)
  uint32_t base;       // address of the first one
  uint32_t sub, L;     // this lane among the L of its instance
  uint32_t gmask;      // those lanes
};

constexpr uint32_t kDT = 16, kLastAct = 17, kST = 18, kFifteen = 19;  // bytes behind V0-VF
constexpr int kLaneBytes = 20;

// Packed display words per instance and bytes per observation frame.
template <bool kS>
struct Disp {
  static constexpr int kWords = kS ? kSchipDispWords : kDispWords;
  static constexpr int kFrame = kS ? kSchipFrameBytes : kFrameBytes;
};

__device__ __forceinline__ uint64_t *disp_of(const Ctx &C) { return reinterpret_cast<uint64_t *>(C.rec); }
__device__ __forceinline__ uint32_t getV(const Ctx &C, uint32_t x) { return C.V[x]; }
__device__ __forceinline__ void setV(const Ctx &C, uint32_t x, uint32_t val) { C.V[x] = (uint8_t)val; }
__device__ __forceinline__ void setVF(const Ctx &C, uint32_t f) { C.V[15] = (uint8_t)f; }

__device__ __forceinline__ uint32_t dirty_bit(uint64_t dirty, uint32_t a) {
  return (uint32_t)(dirty >> ((a & 0xFFFu) >> kPageShift)) & 1u;
}

// Micro-op offset (8 bytes per even address) of a PC; the sentinel's for an
// odd PC or one outside the table.
__device__ __forceinline__ uint32_t to_off(uint32_t pc, const Ctx &C) {
  const uint32_t d = pc - C.base;
  return min(__funnelshift_r(d, d, 1), C.n_uops) << 3;
}
__device__ __forceinline__ uint32_t off_pc(uint32_t off, const Ctx &C) { return C.base + (off >> 2); }

// A fetch at offset o reads the two bytes from off_pc(o) on; the range starts
// one byte early for that. Nothing written: an offset no fetch has.
__device__ __forceinline__ void set_range(Regs &R, const Ctx &C, uint32_t wrange) {
  const uint32_t lo = wrange & 0xFFFFu, hi = wrange >> 16;
  R.wrange = wrange;
  R.wbase = lo > hi ? 0x40000000u : (lo - 1u - C.base) << 2;
  R.wspan = lo > hi ? 0u : ((hi - lo + 1u) << 2) + 3u;
}

// Page copy-on-write keeps one 64-bit mask in registers, and beside it the
// range of RAM addresses written since the reset, so a sprite or an
// instruction on a dirty page but outside that range (beside a score buffer,
// say) is still read from the shared image. Other reads of a dirty page use
// its complete copy.
// True when every byte of [a, a + len) (len <= 32, a + len <= 4096) is as in the image.
__device__ __forceinline__ bool unwritten(const Regs &R, uint32_t a, uint32_t len) {
  if (a + len - 1u < (R.wrange & 0xFFFFu) || a > (R.wrange >> 16)) return true;
  return !(dirty_bit(R.dirty, a) | dirty_bit(R.dirty, a + len - 1u));
}

// A byte of RAM: a dirty page's copy is complete.
__device__ __forceinline__ uint32_t rd8(const Regs &R, const Ctx &C, uint32_t a) {
  a &= 0xFFFu;
  return dirty_bit(R.dirty, a) ? (uint32_t)C.ram[a] : img_byte(a);
}

// All lanes of the instance store the same byte. The page copy must be
// finished by all of them before any stores into it.
__device__ __forceinline__ void wr8(Regs &R, const Ctx &C, uint32_t a, uint32_t val) {
  a &= 0xFFFu;
  const uint32_t page = a >> kPageShift;
  if (!((R.dirty >> page) & 1u)) {  // first write to this page: copy it from the image
    const uint4 *src = reinterpret_cast<const uint4 *>(g_smem + (page << kPageShift));
    uint4 *dst = reinterpret_cast<uint4 *>(C.ram + (page << kPageShift));
    dst[0] = src[0];
    dst[1] = src[1];
    dst[2] = src[2];
    dst[3] = src[3];
    R.dirty |= 1ull << page;
    __syncwarp(C.gmask);
  }
  set_range(R, C, min(R.wrange & 0xFFFFu, a) | max(R.wrange >> 16, a) << 16);
  C.ram[a] = (uint8_t)val;
}

// Philox4x32-10 (Salmon et al., SC'11); word 0 of the output block.
__device__ __forceinline__ uint32_t philox_w0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                              uint32_t k0, uint32_t k1) {
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

__device__ __forceinline__ void tick(const Ctx &C) {
  uint32_t *w = reinterpret_cast<uint32_t *>(C.V + kDT);
  uint32_t t = *w;  // DT | last action << 8 | ST << 16 | 15 << 24
  t -= (t & 0xFFu) != 0u;
  t -= (t & 0xFF0000u) != 0u ? 0x10000u : 0u;
  *w = t;
}

// DXYN: XOR an 8-wide, n-row sprite at (vx mod 64, vy mod 32); VF = collision.
// Each lane draws the screen rows it owns.
__device__ __forceinline__ void draw(Regs &R, const Ctx &C, uint32_t vx, uint32_t vy, uint32_t n,
                                     uint32_t quirks) {
  const uint32_t x0 = vx & 63u, y0 = vy & 31u, I = R.I;
  const bool wrap = quirks & OCTAX_QUIRK_WRAP_SPRITES;
  const uint32_t rows = wrap ? n : min(n, 32u - y0);  // rows below the screen clip
  const uint32_t r0 = (C.sub - y0) & (C.L - 1u);      // the first row of this lane
  uint64_t *const disp = disp_of(C);
  uint64_t hit = 0;
  // the sprite is read from the image unless a byte of it may have been written
  if (!wrap && I + n <= (uint32_t)kRamBytes && (n == 0 || unwritten(R, I, n))) {
    for (uint32_t r = r0; r < rows; r += C.L) {
      const uint64_t s = (uint64_t)(__brev(img_byte(I + r)) >> 24) << x0;  // pixel j -> bit x0 + j, right edge clips
      const uint64_t old = disp[y0 + r];
      hit |= old & s;
      disp[y0 + r] = old ^ s;
    }
  } else {
    for (uint32_t r = r0; r < rows; r += C.L) {
      const uint64_t rev = __brev(rd8(R, C, I + r)) >> 24;  // pixel j of the sprite -> bit j
      uint64_t s = rev << x0;
      if (wrap && x0 > 56u) s |= rev >> (64u - x0);
      uint64_t *row = disp + ((y0 + r) & 31u);
      const uint64_t old = *row;
      hit |= old & s;
      *row = old ^ s;
    }
  }
  setVF(C, (__ballot_sync(C.gmask, hit != 0ull) & C.gmask) != 0u);
}

// Each of the low 16 bits of v doubled (bit j -> bits 2j and 2j + 1).
__device__ __forceinline__ uint32_t double_bits(uint32_t v) {
  v = (v | (v << 8)) & 0x00FF00FFu;
  v = (v | (v << 4)) & 0x0F0F0F0Fu;
  v = (v | (v << 2)) & 0x33333333u;
  v = (v | (v << 1)) & 0x55555555u;
  return v | (v << 1);
}

// SCHIP DXYN / DXY0 on the 128x64 buffer (word 2y + h of an instance holds
// pixels 64h..64h+63 of row y, bit x = pixel 64h + x). In hires mode sprite
// pixels are buffer pixels; in lores mode the grid is 64x32 and each sprite
// pixel covers a 2x2 block. N = 0: 16x16 sprite, two bytes per row. VF = any
// lit buffer pixel turned off. Clipping (or the wrap quirk) on the grid.
__device__ __forceinline__ void draw_schip(Regs &R, const Ctx &C, uint32_t vx, uint32_t vy, uint32_t n,
                                           uint32_t quirks) {
  const bool wrap = quirks & OCTAX_QUIRK_WRAP_SPRITES;
  const uint32_t unit = R.hires ? 1u : 2u;               // buffer pixels per grid pixel
  const uint32_t gw = 128u / unit, gh = 64u / unit;      // grid
  const uint32_t x0 = vx & (gw - 1u), y0 = vy & (gh - 1u);
  const uint32_t rows = n ? n : 16u, width = n ? 8u : 16u;
  const uint32_t bx = x0 * unit, bits_w = width * unit;  // buffer column, pattern width (<= 32)
  // sprite bytes from the shared image unless one of them may have been written
  const uint32_t I = R.I, nbytes = n ? n : 32u;
  const bool from_img = I + nbytes <= (uint32_t)kRamBytes && unwritten(R, I, nbytes);
  uint64_t hit = 0;
  // buffer rows b below the sprite's top; each lane draws the rows it owns
  const uint32_t top = y0 * unit;
  for (uint32_t b = (C.sub - top) & (C.L - 1u); b < rows * unit; b += C.L) {
    uint32_t by = top + b;
    if (by >= 64u) {
      if (!wrap) break;
      by -= 64u;
    }
    const uint32_t r = b >> (unit - 1u);
    uint32_t bits;
    if (from_img) bits = n ? img_byte(I + r) : (img_byte(I + 2u * r) << 8) | img_byte(I + 2u * r + 1u);
    else bits = n ? rd8(R, C, I + r) : ((rd8(R, C, I + 2u * r) << 8) | rd8(R, C, I + 2u * r + 1u));
    const uint32_t rev = __brev(bits) >> (32u - width);   // sprite pixel j -> bit j
    const uint64_t pat = unit == 1u ? (uint64_t)rev : (uint64_t)double_bits(rev);
    // pat << bx as a 128-bit value (lo, hi); bits past column 127 drop
    uint64_t lo = bx < 64u ? pat << bx : 0ull;
    uint64_t hi = bx == 0u ? 0ull : bx < 64u ? pat >> (64u - bx) : pat << (bx - 64u);
    if (wrap && bx + bits_w > 128u) lo |= pat >> (128u - bx);  // wrapped part re-enters at column 0
    uint64_t *row = disp_of(C) + 2u * by;
    const uint64_t o0 = row[0], o1 = row[1];
    hit |= (o0 & lo) | (o1 & hi);
    row[0] = o0 ^ lo;
    row[1] = o1 ^ hi;
  }
  setVF(C, (__ballot_sync(C.gmask, hit != 0ull) & C.gmask) != 0u);
}

// SCHIP scrolls of the 128x64 buffer by buffer pixels; vacated pixels clear.
__device__ __forceinline__ void scroll_down(const Ctx &C, uint32_t k) {
  // rows change owners: one lane moves them all, between two meetings of the instance's lanes
  uint64_t *d = disp_of(C);
  __syncwarp(C.gmask);
  if (C.sub == 0)
    for (int w = 127; w >= 0; --w) d[w] = (uint32_t)w >= 2u * k ? d[w - 2 * (int)k] : 0ull;
  __syncwarp(C.gmask);
}
__device__ __forceinline__ void scroll_right(const Ctx &C, uint32_t c) {  // 0 < c < 64
  uint64_t *d = disp_of(C);
  for (uint32_t y = C.sub; y < 64u; y += C.L) {
    const uint64_t lo = d[2 * y], hi = d[2 * y + 1];
    d[2 * y] = lo << c;
    d[2 * y + 1] = (hi << c) | (lo >> (64u - c));
  }
}
__device__ __forceinline__ void scroll_left(const Ctx &C, uint32_t c) {  // 0 < c < 64
  uint64_t *d = disp_of(C);
  for (uint32_t y = C.sub; y < 64u; y += C.L) {
    const uint64_t lo = d[2 * y], hi = d[2 * y + 1];
    d[2 * y] = (lo >> c) | (hi << (64u - c));
    d[2 * y + 1] = hi >> c;
  }
}
// Clear the rows this lane owns.
template <bool kS>
__device__ __forceinline__ void clear_display(const Ctx &C) {
  uint64_t *d = disp_of(C);
  constexpr uint32_t kPerRow = kS ? 2 : 1;
  for (uint32_t y = C.sub; y < Disp<kS>::kWords / kPerRow; y += C.L)
#pragma unroll
    for (uint32_t h = 0; h < kPerRow; ++h) d[kPerRow * y + h] = 0ull;
}

// ---- micro-ops ---------------------------------------------------------------
// Decoded form of the instruction at an even address, 12 bytes in two tables:
//   x: coefficients (offset in the table of them) | xs << 8 | ys << 16 (bytes behind Ctx::V), flags
//      in the top byte
//   y: offset of the next micro-op when the skip test holds | << 16 when it does not (equal: no skip);
//      a slow opcode: the opcode | kind << 16
//   z: immediate << 19 (13 bits, signed) | dst (a byte behind Ctx::V)
// res = coefficients . (VX, VY, VX & VY, VX >> 1) + immediate, then by flag:
constexpr uint32_t kUWrite = 1u << 24;  // V[dst] = low byte of res (dst may be DT or ST)
constexpr uint32_t kUFlag = 1u << 25;   // VF = bit 8 of res (8XY5 / 8XY7 add 256: NOT borrow)
constexpr uint32_t kUBit0 = 1u << 26;   // ... exclusive-or bit 0 of VX (8XY6)
constexpr uint32_t kUIndex = 1u << 27;  // I = res
constexpr uint32_t kUKey = 1u << 28;    // the immediate is the key term: skip when VX & 15 is the held key
constexpr uint32_t kUSlow = 1u << 29;   // not for the datapath: kind in y
constexpr uint32_t kKindDraw = 1u << 16, kKindRaw = 2u << 16;  // else the opcode as it is
// The key term of a step: -key, or 256 with no key held. VX + it, taken modulo
// 16 with the ninth bit, is zero just when VX & 15 is the key.
constexpr uint32_t kKeyMask = 0x10Fu, kSkipMask = 0x1FFu;

__device__ __forceinline__ constexpr uint32_t coef(int c0, int c1, int c2, int c3) {
  return (c0 & 0xFF) | (c1 & 0xFF) << 8 | (c2 & 0xFF) << 16 | (uint32_t)(c3 & 0xFF) << 24;
}
enum { kCZero, kCX, kCY, kCOr, kCAnd, kCXor, kCAdd, kCSub, kCShr, kCRsub, kCTwice, kCGlyph, kCBigGlyph };
__constant__ const uint32_t kCoefs[16] = {
    coef(0, 0, 0, 0), coef(1, 0, 0, 0),  coef(0, 1, 0, 0), coef(1, 1, -1, 0),  // x + y - (x & y) = x | y
    coef(0, 0, 1, 0), coef(1, 1, -2, 0),                                        // x + y - 2 (x & y) = x ^ y
    coef(1, 1, 0, 0), coef(1, -1, 0, 0), coef(0, 0, 0, 1), coef(-1, 1, 0, 0), coef(2, 0, 0, 0),
    coef(0, 0, 5, 0), coef(0, 0, 10, 0)};                                       // glyphs of 5 or 10 bytes

// Micro-op of `op` at table entry e. Successors and jump targets outside the
// table leave the instruction to the switch, which sets PC itself.
__device__ __forceinline__ uint3 make_uop(uint32_t op, uint32_t e, uint32_t base, uint32_t n_uops, uint32_t quirks,
                                          bool schip) {
  const uint32_t cls = op >> 12, x = (op >> 8) & 15u, y = (op >> 4) & 15u, n = op & 15u, nn = op & 0xFFu;
  const uint32_t nnn = op & 0xFFFu;
  const uint32_t next = (e + 1) << 3, skip = (e + 2) << 3;
  uint32_t flags = 0, dst = x, xs = x, ys = y, c = kCZero, t = next, f = next;
  int32_t imm = 0;
  bool fast = e + 1 < n_uops;
  auto skips = [&](bool negated) {
    t = negated ? next : skip;
    f = negated ? skip : next;
    fast &= e + 2 < n_uops;
  };
  switch (cls) {
    case 0x0:  // 0NNN is ignored; the rest goes to the switch
      fast &= !(op == 0x00E0u || op == 0x00EEu ||
                (schip && ((op & 0xFFF0u) == 0x00C0u || (op >= 0x00FBu && op <= 0x00FFu))));
      break;
    case 0x1:
      fast = nnn >= base && !(nnn & 1u) && ((nnn - base) >> 1) < n_uops;
      t = f = (nnn - base) << 2;
      break;
    case 0x3:
    case 0x4:
      c = kCX;
      imm = -(int32_t)nn;
      skips(cls == 0x4);
      break;
    case 0x5:
    case 0x9:
      c = kCSub;
      skips(cls == 0x9);
      fast &= n == 0;
      break;
    case 0x6:
      imm = (int32_t)nn;
      flags = kUWrite;
      break;
    case 0x7:
      c = kCX;
      imm = (int32_t)nn;
      flags = kUWrite;
      break;
    case 0x8:
      flags = kUWrite;
      if (n >= 1 && n <= 3 && (quirks & OCTAX_QUIRK_LOGIC_RESETS_VF)) flags |= kUFlag;  // bit 8 of those is 0
      if ((n == 6 || n == 14) && (quirks & OCTAX_QUIRK_SHIFT_USES_VY)) xs = y;
      switch (n) {
        case 0x0: c = kCY; break;
        case 0x1: c = kCOr; break;
        case 0x2: c = kCAnd; break;
        case 0x3: c = kCXor; break;
        case 0x4: c = kCAdd; flags |= kUFlag; break;
        case 0x5: c = kCSub; imm = 256; flags |= kUFlag; break;
        case 0x6: c = kCShr; flags |= kUFlag | kUBit0; break;
        case 0x7: c = kCRsub; imm = 256; flags |= kUFlag; break;
        case 0xE: c = kCTwice; flags |= kUFlag; break;
        default: fast = false; break;
      }
      break;
    case 0xA:
      imm = (int32_t)nnn;
      flags = kUIndex;
      break;
    case 0xE:
      c = kCX;
      flags = kUKey;
      skips(nn == 0xA1u);
      fast &= nn == 0x9Eu || nn == 0xA1u;
      break;
    case 0xF:
      if (nn == 0x07u) {
        c = kCX;
        xs = kDT;
        flags = kUWrite;
      } else if (nn == 0x15u || nn == 0x18u) {
        c = kCX;
        dst = nn == 0x15u ? kDT : kST;
        flags = kUWrite;
      } else if (nn == 0x29u || (schip && nn == 0x30u)) {
        c = nn == 0x29u ? kCGlyph : kCBigGlyph;
        ys = kFifteen;
        imm = nn == 0x29u ? 0x50 : (int32_t)kBigFontAddr;
        flags = kUIndex;
      } else {
        fast = false;
      }
      break;
    default:
      fast = false;
      break;
  }
  if (fast) return make_uint3(c << 2 | xs << 8 | ys << 16 | flags, t | f << 16, (uint32_t)imm << 19 | dst);
  return make_uint3(x << 8 | y << 16 | kUSlow, op | (cls == 0xDu ? kKindDraw : 0u), 0u);
}

// 4 pixels (bits 0..3) -> 4 bytes of value 0/1 (byte j = bit j).
__device__ __forceinline__ uint32_t spread4(uint32_t nib) { return (nib * 0x00204081u) & 0x01010101u; }

// One CTA per game: its blob's pixel table and micro-ops from its RAM image.
__global__ void tables_kernel(uint8_t *blobs, uint64_t stride, uint32_t n_uops, int schip, uint32_t quirks) {
  uint8_t *b = blobs + blockIdx.x * stride;
  uint2 *lut = reinterpret_cast<uint2 *>(b + kBlobLut);
  for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) lut[i] = make_uint2(spread4(i & 15u), spread4(i >> 4));
  if (threadIdx.x < 16) reinterpret_cast<uint32_t *>(b + kBlobCoef)[threadIdx.x] = kCoefs[threadIdx.x];
  uint2 *xy = reinterpret_cast<uint2 *>(b + kBlobUops);
  uint32_t *z = reinterpret_cast<uint32_t *>(xy + n_uops + 1);
  const uint32_t base = table_base(n_uops);
  for (uint32_t e = threadIdx.x; e <= n_uops; e += blockDim.x) {
    uint3 u = make_uint3(kUSlow, kKindRaw, 0u);  // the sentinel
    if (e < n_uops)
      u = make_uop((uint32_t)b[base + 2 * e] << 8 | b[base + 2 * e + 1], e, base, n_uops, quirks, schip != 0);
    xy[e] = make_uint2(u.x, u.y);
    z[e] = u.z;
  }
}

// Any instruction: the rare / heavy ones, undefined encodings, and every one
// from an odd, written or far address. PC has already been advanced.
// The lanes of the instance meet here first: those ahead wait before they
// change the stack, RAM or the flag registers, which the lanes share.
// kS: the SCHIP variant (128x64 buffer, extra 00xx and FXxx forms).
template <bool kS>
__device__ __forceinline__ void exec_slow(Regs &R, const Ctx &C, uint32_t op, uint32_t pc, int key,
                                       uint32_t quirks) {
  const uint32_t x = (op >> 8) & 15u, y = (op >> 4) & 15u, n = op & 15u, nn = op & 0xFFu;
  const uint32_t nnn = op & 0xFFFu;
  uint16_t *const stack = reinterpret_cast<uint16_t *>(C.rec + Rec<kS>::kStack);
  uint8_t *const rpl = kS ? reinterpret_cast<uint8_t *>(C.rec + Rec<kS>::kRpl) : nullptr;
  __syncwarp(C.gmask);
  const uint32_t vx = getV(C, x), vy = getV(C, y);
  switch (op >> 12) {
    case 0x0:
      if (op == 0x00E0u) {
        clear_display<kS>(C);
      } else if (kS && (op & 0xFFF0u) == 0x00C0u) {  // scroll down N
        scroll_down(C, n * (R.hires ? 1u : 2u));
      } else if (kS && op == 0x00FBu) {  // scroll right 4
        scroll_right(C, R.hires ? 4u : 8u);
      } else if (kS && op == 0x00FCu) {  // scroll left 4
        scroll_left(C, R.hires ? 4u : 8u);
      } else if (kS && op == 0x00FDu) {  // exit: stay here
        R.status |= OCTAX_STATUS_EXIT;
        R.pc = pc;
      } else if (kS && (op == 0x00FEu || op == 0x00FFu)) {  // lores / hires, buffer kept
        R.hires = op & 1u;
      } else if (op == 0x00EEu) {
        if (R.sp == 0) {
          R.status |= OCTAX_STATUS_STACK_FAULT;
          R.sp = 16;
        }
        R.sp -= 1;
        R.pc = stack[R.sp];
      }
      break;
    case 0x1:
      R.pc = nnn;
      break;
    case 0x2:
      if (R.sp == 16) {
        R.status |= OCTAX_STATUS_STACK_FAULT;
        R.sp = 0;
      }
      stack[R.sp] = (uint16_t)R.pc;
      R.sp += 1;
      R.pc = nnn;
      break;
    case 0x3:
      if (vx == nn) R.pc = (R.pc + 2u) & 0xFFFu;
      break;
    case 0x4:
      if (vx != nn) R.pc = (R.pc + 2u) & 0xFFFu;
      break;
    case 0x5:
      if (n) R.status |= OCTAX_STATUS_BAD_OP;
      else if (vx == vy) R.pc = (R.pc + 2u) & 0xFFFu;
      break;
    case 0x6:
      setV(C, x, nn);
      break;
    case 0x7:
      setV(C, x, vx + nn);
      break;
    case 0x8:
      switch (n) {
        case 0x0: setV(C, x, vy); break;
        case 0x1:
          setV(C, x, vx | vy);
          if (quirks & OCTAX_QUIRK_LOGIC_RESETS_VF) setVF(C, 0);
          break;
        case 0x2:
          setV(C, x, vx & vy);
          if (quirks & OCTAX_QUIRK_LOGIC_RESETS_VF) setVF(C, 0);
          break;
        case 0x3:
          setV(C, x, vx ^ vy);
          if (quirks & OCTAX_QUIRK_LOGIC_RESETS_VF) setVF(C, 0);
          break;
        case 0x4: {
          const uint32_t s = vx + vy;
          setV(C, x, s);
          setVF(C, s >> 8);
          break;
        }
        case 0x5:
          setV(C, x, vx - vy);
          setVF(C, vx >= vy);
          break;
        case 0x6: {
          const uint32_t src = (quirks & OCTAX_QUIRK_SHIFT_USES_VY) ? vy : vx;
          setV(C, x, src >> 1);
          setVF(C, src & 1u);
          break;
        }
        case 0x7:
          setV(C, x, vy - vx);
          setVF(C, vy >= vx);
          break;
        case 0xE: {
          const uint32_t src = (quirks & OCTAX_QUIRK_SHIFT_USES_VY) ? vy : vx;
          setV(C, x, src << 1);
          setVF(C, src >> 7);
          break;
        }
        default:
          R.status |= OCTAX_STATUS_BAD_OP;
          break;
      }
      break;
    case 0x9:
      if (n) R.status |= OCTAX_STATUS_BAD_OP;
      else if (vx != vy) R.pc = (R.pc + 2u) & 0xFFFu;
      break;
    case 0xA:
      R.I = nnn;
      break;
    case 0xB:
      R.pc = (nnn + ((quirks & OCTAX_QUIRK_JUMP_VX) ? vx : getV(C, 0))) & 0xFFFu;
      break;
    case 0xC: {
      const uint32_t rnd = philox_w0(C.rec[Rec<kS>::kUid], R.env_steps, pc | ((R.draws & 0xFFFFu) << 16), R.phase,
                                     C.rec[Rec<kS>::kKey], C.rec[Rec<kS>::kKey + 1]);
      R.draws += 1;
      setV(C, x, rnd & nn);
      break;
    }
    case 0xD:
      if (kS) draw_schip(R, C, vx, vy, n, quirks);
      else draw(R, C, vx, vy, n, quirks);
      break;
    case 0xE: {
      const bool pressed = key >= 0 && (uint32_t)key == (vx & 15u);
      if (nn == 0x9Eu) {
        if (pressed) R.pc = (R.pc + 2u) & 0xFFFu;
      } else if (nn == 0xA1u) {
        if (!pressed) R.pc = (R.pc + 2u) & 0xFFFu;
      } else {
        R.status |= OCTAX_STATUS_BAD_OP;
      }
      break;
    }
    default:  // 0xF
      switch (nn) {
        case 0x07: setV(C, x, getV(C, kDT)); break;
        case 0x0A:
          if (key >= 0) setV(C, x, (uint32_t)key);
          else R.pc = pc;
          break;
        case 0x15: setV(C, kDT, vx); break;
        case 0x18: setV(C, kST, vx); break;
        case 0x1E: {
          const uint32_t s = R.I + vx;
          R.I = s & 0xFFFFu;
          if (quirks & OCTAX_QUIRK_FX1E_VF) setVF(C, s > 0xFFFu);
          break;
        }
        case 0x29: R.I = 0x50u + 5u * (vx & 15u); break;
        case 0x30:
          if (kS) R.I = kBigFontAddr + 10u * (vx & 15u);
          else R.status |= OCTAX_STATUS_BAD_OP;
          break;
        case 0x75:
          if (kS) {
            for (uint32_t i = 0; i <= x; ++i) rpl[i] = (uint8_t)getV(C, i);
          } else {
            R.status |= OCTAX_STATUS_BAD_OP;
          }
          break;
        case 0x85:
          if (kS) {
            for (uint32_t i = 0; i <= x; ++i) setV(C, i, rpl[i]);
          } else {
            R.status |= OCTAX_STATUS_BAD_OP;
          }
          break;
        case 0x33:
          wr8(R, C, R.I, vx / 100u);
          wr8(R, C, R.I + 1u, (vx / 10u) % 10u);
          wr8(R, C, R.I + 2u, vx % 10u);
          break;
        case 0x55:
          for (uint32_t i = 0; i <= x; ++i) wr8(R, C, R.I + i, getV(C, i));
          if (quirks & OCTAX_QUIRK_LOADSTORE_INC_I) R.I = (R.I + x + 1u) & 0xFFFFu;
          break;
        case 0x65:
          for (uint32_t i = 0; i <= x; ++i) setV(C, i, rd8(R, C, R.I + i));
          if (quirks & OCTAX_QUIRK_LOADSTORE_INC_I) R.I = (R.I + x + 1u) & 0xFFFFu;
          break;
        default:
          R.status |= OCTAX_STATUS_BAD_OP;
          break;
      }
      break;
  }
}

// a (unsigned bytes) . b (signed bytes) + c
__device__ __forceinline__ int32_t dot4(uint32_t a, uint32_t b, int32_t c) {
  int32_t d;
  asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// Run `count` instructions from R.pc on. key: held CHIP-8 key or -1.
// The loop carries the micro-op offset; R.pc holds the PC whenever the offset
// is the sentinel's.
template <bool kS>
__device__ __forceinline__ void run_instrs(Regs &R, const Ctx &C, int key, uint32_t quirks, uint32_t count) {
  const uint8_t *const uops = g_smem + kBlobUops;
  const uint32_t sentinel = C.n_uops << 3;
  const uint8_t *const imms = uops + sentinel + 8;
  const int32_t keyterm = key >= 0 ? -key : 256;
  uint32_t off = to_off(R.pc, C);
  // Not unrolled: on divergent programs a second copy of the datapath costs
  // more in instruction fetch than the loop overhead it saves.
#pragma unroll 1
  for (uint32_t k = 0; k < count; ++k) {
    uint2 u = *reinterpret_cast<const uint2 *>(uops + off);
    const uint32_t z = *reinterpret_cast<const uint32_t *>(imms + (off >> 1));
    if (off - R.wbase <= R.wspan && dirty_bit(R.dirty, off_pc(off, C))) u = make_uint2(kUSlow, kKindRaw);  // written
    const uint32_t vx = C.V[(u.x >> 8) & 0xFFu], vy = C.V[(u.x >> 16) & 0xFFu];
    if (!(u.x & kUSlow)) {
      const uint32_t c = *reinterpret_cast<const uint32_t *>(g_smem + kBlobCoef + (u.x & 0xFFu));
      const bool by_key = u.x & kUKey;
      const int32_t res = dot4(vx + (vy << 8) + ((vx & vy) << 16) + ((vx >> 1) << 24), c,
                               by_key ? keyterm : (int32_t)z >> 19);
      off = ((uint32_t)res & (by_key ? kKeyMask : kSkipMask)) == 0u ? u.y & 0xFFFFu : u.y >> 16;
      if (u.x & kUWrite) C.V[z & 31u] = (uint8_t)res;
      // after VX: with X = F the flag wins
      if (u.x & kUFlag) C.V[15] = (uint8_t)((((uint32_t)res >> 8) ^ ((u.x & kUBit0) ? vx : 0u)) & 1u);
      if (u.x & kUIndex) R.I = (uint32_t)res;
    } else {
      const uint32_t pc = off == sentinel ? R.pc : off_pc(off, C);
      R.pc = (pc + 2u) & 0xFFFu;
      if (u.y & kKindDraw) {
        if (kS) draw_schip(R, C, vx, vy, u.y & 15u, quirks);
        else draw(R, C, vx, vy, u.y & 15u, quirks);
      } else {
        const uint32_t op = (u.y & kKindRaw) ? rd8(R, C, pc) << 8 | rd8(R, C, pc + 1u) : u.y;
        exec_slow<kS>(R, C, op, pc, key, quirks);
      }
      off = to_off(R.pc, C);
    }
  }
  if (off != sentinel) R.pc = off_pc(off, C);
}

__device__ __forceinline__ int32_t term_value(const Regs &R, const Ctx &C, const TermDev &t) {
  const int32_t v = t.src == OCTAX_SRC_REG ? (int32_t)getV(C, t.idx & 15u) : (int32_t)rd8(R, C, t.idx);
  switch (t.xform) {
    case OCTAX_X_RAW: return v;
    case OCTAX_X_NEG: return -v;
    case OCTAX_X_DEC_TENS: return v / 10;
    case OCTAX_X_DEC_ONES: return v % 10;
    case OCTAX_X_DEC_TENS_MINUS_ONES: return v / 10 - v % 10;
    case OCTAX_X_NIB_HI_MINUS_LO: return (v >> 4) - (v & 15);
    case OCTAX_X_ZERO_IF_GT: return v > t.arg ? 0 : v;
    default: return 0;
  }
}

__device__ __forceinline__ int32_t score(const Regs &R, const Ctx &C, const GameDev &G) {
  int32_t s = 0;
  for (uint32_t i = 0; i < G.n_score; ++i) s += term_value(R, C, G.score[i]);
  return s;
}

__device__ __forceinline__ bool terminated(const Regs &R, const Ctx &C, const GameDev &G) {
  bool hit = false;
  for (uint32_t i = 0; i < G.n_term; ++i) {
    const ClauseDev &c = G.term[i];
    const int32_t v = term_value(R, C, c.lhs);
    switch (c.cmp) {
      case OCTAX_CMP_EQ: hit |= v == c.rhs; break;
      case OCTAX_CMP_NE: hit |= v != c.rhs; break;
      case OCTAX_CMP_GE: hit |= v >= c.rhs; break;
      case OCTAX_CMP_GT: hit |= v > c.rhs; break;
      case OCTAX_CMP_LE: hit |= v <= c.rhs; break;
      case OCTAX_CMP_LT: hit |= v < c.rhs; break;
      default: break;
    }
  }
  return hit;
}

// Power-on state + the game's startup instructions (no key, timers tick every
// K), then the no-op reset wrapper (§3.2): a drawn number of no-key env steps
// of frameskip frames each, unobserved. The previous action becomes the no-op.
// kWrap = false compiles the wrapper out (no game of the launch uses it).
// The lanes of the instance meet here first: the stack and the flag registers
// are one copy for all of them, and a lane behind may still be at the last
// instructions of its step (a return reads the stack).
template <bool kWrap, bool kS>
__device__ __forceinline__ void reset_instance(Regs &R, const Ctx &C, const GameDev &G, uint32_t quirks) {
  __syncwarp(C.gmask);
  uint32_t *const V = reinterpret_cast<uint32_t *>(C.V);
#pragma unroll
  for (int i = 0; i < 4; ++i) V[i] = 0;
  V[4] = 15u << 24;  // DT, ST = 0
  R.pc = 0x200;
  R.I = 0;
  R.sp = 0;
  R.dirty = 0;
  set_range(R, C, kNoWrites);
#pragma unroll
  for (int i = 0; i < 8; ++i) C.rec[Rec<kS>::kStack + i] = 0;
  clear_display<kS>(C);
  R.hires = 0;  // SCHIP: every episode starts in lores with clear flag registers
  if (kS)
    for (int i = 0; i < 4; ++i) C.rec[Rec<kS>::kRpl + i] = 0;
  // Startup: full chunks of K (each followed by a tick), then the remainder
  // (no tick); after it, the no-op frames (K instructions and a tick each).
  // One loop, so that the interpreter is inlined here only once.
  const uint32_t noop_frames =
      !kWrap || G.max_noops == 0u ? 0u
                        : philox_w0(C.rec[Rec<kS>::kUid], R.env_steps, 0u, 3u, C.rec[Rec<kS>::kKey],
                                    C.rec[Rec<kS>::kKey + 1]) % (G.max_noops + 1u) * G.frameskip;
  const uint32_t full = G.startup / G.K, rem = G.startup - full * G.K;
  const uint32_t chunks = full + (rem != 0u) + noop_frames;
  R.phase = 1;
  R.draws = 0;
  for (uint32_t i = 0; i < chunks; ++i) {
    const bool partial = i == full && rem != 0u;
    run_instrs<kS>(R, C, -1, quirks, partial ? rem : G.K);
    if (!partial) tick(C);
  }
  C.V[kLastAct] = (uint8_t)G.n_actions;
  R.phase = 0;
  R.draws = 0;
}

// Pixels 16q..16q+15 of a packed row -> 16 bytes of 0/1, through a
// per-CTA table that maps a byte of pixels to its 8 output bytes.
__device__ __forceinline__ uint4 expand16(uint64_t row, uint32_t q) {
  const uint2 *const lut = reinterpret_cast<const uint2 *>(g_smem + kBlobLut);
  const uint32_t bits = (uint32_t)(row >> (16u * q)) & 0xFFFFu;
  const uint2 lo = lut[bits & 0xFFu], hi = lut[bits >> 8];
  return make_uint4(lo.x, lo.y, hi.x, hi.y);
}

// Whole-warp frame write of the warp's `ipw` instances (records at `recs`).
// frame (per lane, 0 = skip) points at the frame of that lane's own instance,
// whose lanes start at instance << lane_sh.
// 16-byte pieces of a row: 4 (CHIP-8) or 8 (SCHIP) lanes write one row, so the
// warp writes 8 (4) rows at a time: one row of each of 8 (4) instances, or, with
// fewer instances, several rows of each.
template <bool kS>
__device__ __forceinline__ void capture_frame(const uint32_t *recs, uint8_t *frame, int lane, int ipw, int lane_sh) {
  constexpr int kPer = kS ? 8 : 4, kLogAll = kS ? 2 : 3;  // lanes per row, log2(rows at a time)
  constexpr int kRows = kS ? 64 : 32, kRowBytes = kS ? 128 : 64;
  const uint64_t mine = reinterpret_cast<uint64_t>(frame);
  const uint32_t q = lane & (kPer - 1);
  const int lg = min(5 - lane_sh, kLogAll);   // log2(instances at a time)
  const int step = 1 << (kLogAll - lg);       // rows of one instance at a time
  const int place = lane / kPer;              // row of the 8 (4)
  const int r0 = place & (step - 1);
  for (int m = 0; m < ipw; m += 1 << lg) {
    const int src = m + (place >> (kLogAll - lg));
    const uint64_t base = __shfl_sync(kFull, mine, (src << lane_sh) & 31);
    if (src < ipw && base) {
      const uint64_t *row = reinterpret_cast<const uint64_t *>(recs + src * Rec<kS>::kWords);
      if (kS) row += q >> 2;
      uint8_t *dst = reinterpret_cast<uint8_t *>(base) + q * 16u;
      for (int r = r0; r < kRows; r += 4 * step)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int y = r + u * step;
          __stcs(reinterpret_cast<uint4 *>(dst + y * kRowBytes), expand16(row[kS ? 2 * y : y], q & 3u));
        }
    }
  }
}

// Packed frame of every instance of the warp with a non-null `frame`: its
// display words copied as they are, two per 16-byte streaming store.
template <bool kS>
__device__ __forceinline__ void capture_packed(const uint32_t *recs, uint8_t *frame, int lane, int ipw, int lane_sh) {
  constexpr int kPieces = Disp<kS>::kWords / 2;  // 16-byte stores per instance-frame: 16 or 64
  constexpr int kAtOnce = kS ? 1 : 2;            // instances
  const uint64_t mine = reinterpret_cast<uint64_t>(frame);
  for (int m = 0; m < ipw; m += kAtOnce) {
    const int src = m + (kS ? 0 : lane >> 4);
    const uint64_t base = __shfl_sync(kFull, mine, (src << lane_sh) & 31);
    if (src < ipw && base)
      for (int c = lane & (kS ? 31 : 15); c < kPieces; c += 32)
        __stcs(reinterpret_cast<uint4 *>(base) + c, reinterpret_cast<const uint4 *>(recs + src * Rec<kS>::kWords)[c]);
  }
}

// Packed reset observation of the instances in `which` (every stack slot).
template <bool kS>
__device__ __forceinline__ void write_reset_packed(const uint32_t *recs, uint8_t *obs, int S, unsigned which, int lane,
                                                   int lane_sh) {
  constexpr int kPieces = Disp<kS>::kWords / 2;
  const uint64_t mine = reinterpret_cast<uint64_t>(obs);
  while (which) {  // bit of an instance's first lane
    const int src = __ffs(which) - 1;
    which &= which - 1;
    uint4 *const base = reinterpret_cast<uint4 *>(__shfl_sync(kFull, mine, src));
    const uint4 *const d = reinterpret_cast<const uint4 *>(recs + (src >> lane_sh) * Rec<kS>::kWords);
    for (int c = lane; c < kPieces; c += 32)
      for (int s = 0; s < S; ++s) __stcs(base + s * kPieces + c, d[c]);
  }
}

// Reset observation of the instances in `which`: the display in every stack slot.
template <bool kS>
__device__ __forceinline__ void write_reset_obs(const uint32_t *recs, uint8_t *obs, int S, unsigned which, int lane,
                                                int lane_sh) {
  const uint64_t mine = reinterpret_cast<uint64_t>(obs);
  constexpr int kChunks = Disp<kS>::kFrame / 16;  // 16-byte chunks per frame
  while (which) {  // bit of an instance's first lane
    const int src = __ffs(which) - 1;
    which &= which - 1;
    const uint64_t base = __shfl_sync(kFull, mine, src);
    const uint64_t *const d = reinterpret_cast<const uint64_t *>(recs + (src >> lane_sh) * Rec<kS>::kWords);
#pragma unroll
    for (int it = 0; it < kChunks / 32; ++it) {
      const int c = it * 32 + lane;  // 16-byte chunk of the frame: word c / 4 of the display
      const uint4 o = expand16(d[c >> 2], c & 3);
      for (int s = 0; s < S; ++s)
        __stcs(reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(base) + s * Disp<kS>::kFrame + c * 16), o);
    }
  }
}

__device__ __forceinline__ void copy16_async(void *smem, const void *gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Shared memory of a CTA: the game's blob | records [instances] | registers [emulator lanes][20].
__device__ __forceinline__ uint32_t *smem_recs(uint32_t n_uops) {
  return reinterpret_cast<uint32_t *>(g_smem + blob_bytes(n_uops));
}
__device__ __forceinline__ const GameDev &smem_game() { return *reinterpret_cast<const GameDev *>(g_smem + kRamBytes); }

// Starts the copy of a game's blob (all threads; copy_wait and a barrier follow).
__device__ __forceinline__ void stage_game(const uint8_t *blobs, uint32_t stride, int game, uint32_t n_uops) {
  const uint8_t *src = blobs + (size_t)game * stride;
  for (uint32_t i = 16 * threadIdx.x; i < blob_bytes(n_uops); i += 16 * blockDim.x) copy16_async(g_smem + i, src + i);
}

// The lanes of a warp and what it emulates: ipw instances, each by 1 << sh lanes.
struct Warp {
  int lane, w, ipw, sh;  // w: among the CTA's emulator warps
  int J;                 // instances of the CTA
  int i, j;              // this lane's instance within the warp / the CTA
  uint32_t *recs;        // the warp's records
  bool active;           // this lane emulates an instance
  int count;             // instances of this warp
};

__device__ __forceinline__ Warp make_warp(int ipw, int emu_warps, const Group &g, uint32_t n_uops, int words) {
  Warp W;
  W.lane = threadIdx.x & 31;
  W.w = threadIdx.x >> 5;
  W.ipw = ipw;
  W.sh = ipw <= 1 ? 5 : __clz(ipw - 1) - 27;  // 5 - ceil(log2(ipw))
  W.J = emu_warps * ipw;
  W.i = W.lane >> W.sh;
  W.j = W.w * ipw + W.i;
  W.count = min(max((int)g.count - W.w * ipw, 0), ipw);
  W.active = W.i < W.count;
  W.recs = smem_recs(n_uops) + W.w * ipw * words;
  return W;
}

template <bool kS>
__device__ __forceinline__ Ctx make_ctx(const Warp &W, const DevState &st, int64_t slot, uint32_t n_uops, uint32_t base) {
  Ctx C;
  C.rec = W.recs + (W.active ? W.i : 0) * Rec<kS>::kWords;
  C.V = reinterpret_cast<uint8_t *>(smem_recs(n_uops) + W.J * Rec<kS>::kWords) + threadIdx.x * kLaneBytes;
  C.ram = st.ram + slot * (int64_t)kRamBytes;
  C.n_uops = n_uops;
  C.base = base;
  C.L = 1u << W.sh;
  C.sub = W.lane & (C.L - 1u);
  C.gmask = (W.sh == 5 ? kFull : (1u << C.L) - 1u) << (W.lane - C.sub);
  return C;
}

// Starts the copy of the warp's records (copy_wait and a warp barrier follow).
template <bool kS>
__device__ __forceinline__ void fetch_records(const Warp &W, const DevState &st, const Group &g) {
  const uint32_t *src = st.rec + ((int64_t)g.slot0 + W.w * W.ipw) * Rec<kS>::kWords;
  for (int c = 4 * W.lane; c < W.count * Rec<kS>::kWords; c += 128) copy16_async(W.recs + c, src + c);
}

template <bool kS>
__device__ __forceinline__ void load_regs(Regs &R, const Ctx &C) {
  const uint32_t pcI = C.rec[Rec<kS>::kPcI], misc = C.rec[Rec<kS>::kMisc];
  R.pc = pcI & 0xFFFFu;
  R.I = pcI >> 16;
  R.sp = misc & 0x7Fu;
  R.hires = kS ? (misc >> 7) & 1u : 0u;
  R.status = (misc >> 8) & 0xFFu;
  R.dirty = *reinterpret_cast<const uint64_t *>(C.rec + Rec<kS>::kDirty);
  set_range(R, C, C.rec[Rec<kS>::kWrange]);
  R.env_steps = C.rec[Rec<kS>::kEnv];
  R.draws = 0;
  R.phase = 0;
#pragma unroll
  for (int k = 0; k < 5; ++k) reinterpret_cast<uint32_t *>(C.V)[k] = C.rec[Rec<kS>::kV + k];
}

// Back into the record (every lane of the instance stores the same words).
template <bool kS>
__device__ __forceinline__ void store_regs(const Regs &R, const Ctx &C, uint32_t ep) {
  C.rec[Rec<kS>::kPcI] = R.pc | (R.I << 16);
  C.rec[Rec<kS>::kMisc] = (C.rec[Rec<kS>::kMisc] & 0xFFFF0000u) | R.status << 8 | R.hires << 7 | R.sp;
  C.rec[Rec<kS>::kWrange] = R.wrange;
  *reinterpret_cast<uint64_t *>(C.rec + Rec<kS>::kDirty) = R.dirty;
  C.rec[Rec<kS>::kEp] = ep;
  C.rec[Rec<kS>::kEnv] = R.env_steps;
#pragma unroll
  for (int k = 0; k < 5; ++k) C.rec[Rec<kS>::kV + k] = reinterpret_cast<const uint32_t *>(C.V)[k];
}

// The warp's records back to device memory; `which` (bits of first lanes): of those instances only.
template <bool kS>
__device__ __forceinline__ void return_records(const Warp &W, const DevState &st, const Group &g, unsigned which) {
  __syncwarp();
  uint32_t *dst = st.rec + ((int64_t)g.slot0 + W.w * W.ipw) * Rec<kS>::kWords;
  for (int c = 4 * W.lane; c < W.count * Rec<kS>::kWords; c += 128)
    if ((which >> ((c / Rec<kS>::kWords) << W.sh)) & 1u)
      *reinterpret_cast<uint4 *>(dst + c) = *reinterpret_cast<const uint4 *>(W.recs + c);
}

// The key an action index holds down (-1: none).
__device__ __forceinline__ int key_of(Regs &R, const GameDev &G, uint32_t a) {
  if (a < G.n_actions) return G.action_set[a] & 15;
  if (a > G.n_actions) R.status |= OCTAX_STATUS_BAD_ACTION;
  return -1;
}

// Sticky actions (§3.2): repeat the previous step's action with probability sticky / 2^32.
template <bool kWrap, bool kS>
__device__ __forceinline__ uint32_t applied_action(const Regs &R, const Ctx &C, const GameDev &G, uint32_t a) {
  if (kWrap && G.sticky != 0u &&
      philox_w0(C.rec[Rec<kS>::kUid], R.env_steps, 0u, 2u, C.rec[Rec<kS>::kKey], C.rec[Rec<kS>::kKey + 1]) < G.sticky)
    a = C.V[kLastAct];
  C.V[kLastAct] = (uint8_t)a;
  return a;
}

template <bool kWrap, bool kS, uint32_t kBase>
__device__ void run_group(const StepLaunch &p, const Group &g, const Warp &W) {
  const DevState &st = p.st;
  const GameDev &G = smem_game();
  const int64_t slot = (int64_t)g.slot0 + (W.active ? W.j : 0);
  const IO io = p.io_table ? p.io_table[g.io] : p.io0;
  const uint32_t quirks = p.quirks;
  const Ctx C = make_ctx<kS>(W, st, slot, (uint32_t)p.n_uops, kBase);
  const int frame = io.packed ? 8 * Disp<kS>::kWords : Disp<kS>::kFrame;
  Regs R;
  load_regs<kS>(R, C);
  const int64_t row = (int64_t)C.rec[Rec<kS>::kRow];
  uint32_t ep = C.rec[Rec<kS>::kEp];
  int32_t prev = W.active ? score(R, C, G) : 0;
  const uint32_t K = G.K, FS = G.frameskip, first_kept = FS - (uint32_t)p.S;
  uint32_t a_next = W.active ? io.actions[(int64_t)p.step0 * io.rows + row] : 0u;
  __syncwarp();

  for (int s = 0; s < p.steps; ++s) {
    const int64_t io_row = (int64_t)(p.step0 + s) * io.rows + row;
    int key = -1;
    uint8_t *my_obs = nullptr;
    if (W.active) {
      key = key_of(R, G, applied_action<kWrap, kS>(R, C, G, a_next));
      my_obs = io.obs + io_row * (int64_t)p.S * frame;
      if (s + 1 < p.steps) a_next = io.actions[io_row + io.rows];  // in flight during this step
    }
    R.draws = 0;
    R.phase = 0;
    for (uint32_t f = 0; f < FS; ++f) {
      if (W.active) {
        run_instrs<kS>(R, C, key, quirks, K);
        tick(C);
      }
      if (f >= first_kept) {
        __syncwarp();
        uint8_t *const dst = my_obs ? my_obs + (f - first_kept) * frame : nullptr;
        if (io.packed) capture_packed<kS>(W.recs, dst, W.lane, W.ipw, W.sh);
        else capture_frame<kS>(W.recs, dst, W.lane, W.ipw, W.sh);
        __syncwarp();
      }
    }
    // little is left of the launch: its successor may be set up (earlier, its
    // waiting CTAs would keep the SMs from other streams' kernels)
    if (s + 1 == p.steps) grid_dependents_launch();
    bool done = false;
    if (W.active) {
      const int32_t sc = score(R, C, G);
      ep += 1;
      R.env_steps += 1;
      done = terminated(R, C, G) || (G.max_steps != 0 && ep >= G.max_steps);
      if (C.sub == 0) {
        io.reward[io_row] = (float)(sc - prev);
        io.done[io_row] = done ? 1 : 0;
      }
      if (done) {
        reset_instance<kWrap, kS>(R, C, G, quirks);
        ep = 0;
        prev = score(R, C, G);
      } else {
        prev = sc;
      }
    }
    const unsigned which = __ballot_sync(kFull, done && C.sub == 0);
    if (which) {
      __syncwarp();
      if (io.packed) write_reset_packed<kS>(W.recs, my_obs, p.S, which, W.lane, W.sh);
      else write_reset_obs<kS>(W.recs, my_obs, p.S, which, W.lane, W.sh);
      __syncwarp();
    }
  }

  if (W.active) store_regs<kS>(R, C, ep);
  return_records<kS>(W, st, g, kFull);
}

// One CTA's loop over groups (a persistent CTA pulls them off the queue).
// Every step kernel is held to 128 registers (two 256-thread CTAs per SM).
// kWrap: the sticky-action / no-op-reset variant (games without the wrappers
// run the kernel without them); kS: the Super-CHIP display layout; kBase: the
// table's first address (computed in the kernel it costs the issue-bound cases
// 0.3-0.7 % and random programs 0.9 %).
template <bool kWrap, bool kS, uint32_t kBase>
__global__ void __launch_bounds__(kMaxBlock, 2) step_kernel(const StepLaunch p) {
  __shared__ int s_group;
  int cur_game = -1;
  int gi = blockIdx.x;
  for (;;) {
    if (p.work_counter) {
      if (threadIdx.x == 0) s_group = (int)atomicAdd(p.work_counter, 1u);
      __syncthreads();
      gi = s_group;
    }
    if (gi >= p.n_groups) break;
    const Group g = p.groups[gi];
    const Warp W = make_warp(p.ipw, blockDim.x >> 5, g, (uint32_t)p.n_uops, Rec<kS>::kWords);
    if ((int)g.game != cur_game) {
      stage_game(p.blobs, p.stride, g.game, (uint32_t)p.n_uops);
      cur_game = g.game;
    }
    grid_dependency_wait();  // states, actions and output buffers from here on
    fetch_records<kS>(W, p.st, g);
    copy_wait();
    __syncthreads();
    run_group<kWrap, kS, kBase>(p, g, W);
    if (!p.work_counter) break;
    __syncthreads();  // shared memory is reused by the next group
  }
}


// ---------------------------------------------------------------------------
// Warp-specialised step: the first block/32 warps emulate (as in run_group),
// the last `writers` warps only write observations. At every kept frame the
// emulators copy their packed display rows into one slot of a two-slot ring
// in shared memory and go on emulating; the writers expand that slot to
// uint8 frames and stream them out, so interpreter and stores overlap. After
// each step a last message carries the done flags and reset displays; the
// writer thread that wrote an address earlier in the step is the one that
// overwrites it with the reset observation, so program order keeps them
// ordered. Slots hand over through mbarriers (full: all emulator threads
// arrive; empty: all writer threads arrive); every wait polls a bounded
// number of times for at most kMaxWaitNs of the global timer and, if it
// gives up, records the failure in p.err. The lanes of a warp decide together
// whether a wait ran out (those of an instance meet in the interpreter, which
// has no limit), and what one warp gave up ends the CTA's work on later groups.

constexpr uint32_t kMaxPolls = 1u << 22;
constexpr uint64_t kMaxWaitNs = 1000000000ull;  // one second

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(b))
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, unsigned int *err) {
  const uint64_t t0 = global_ns();
  for (uint32_t i = 0; i < kMaxPolls; ++i) {
    if (mbar_try(b, parity)) return true;
    if (global_ns() - t0 > kMaxWaitNs) break;
  }
  atomicOr(err, 1u);
  return false;
}

struct WsSmem {
  uint64_t *ring;    // [2][J][33] snapshots of packed display rows (33: rows of neighbours in other banks)
  uint8_t *done;     // [2][J] done flags of the end-of-step message
  uint64_t *full;    // [2]
  uint64_t *empty;   // [2]
};
constexpr int kRingPitch = 33;

// behind the records and registers: ring | done flags | barriers
__device__ __forceinline__ WsSmem carve_ws(uint32_t n_uops, int J, int emu_warps) {
  WsSmem w;
  uint8_t *p = reinterpret_cast<uint8_t *>(smem_recs(n_uops) + J * Rec<false>::kWords) + emu_warps * 32 * kLaneBytes;
  w.ring = reinterpret_cast<uint64_t *>(p);
  w.done = reinterpret_cast<uint8_t *>(w.ring + 2 * kRingPitch * J);
  w.full = reinterpret_cast<uint64_t *>(w.done + ((2 * J + 15) & ~15));
  w.empty = w.full + 2;
  return w;
}

// The rows this lane owns into slot b of the ring.
__device__ __forceinline__ void ring_put(const WsSmem &W, const Ctx &C, int J, int j, uint32_t b) {
  uint64_t *dst = W.ring + (b * J + j) * kRingPitch;
  for (uint32_t r = C.sub; r < 32u; r += C.L) dst[r] = disp_of(C)[r];
}

// Emulator side of one group. `msg` counts messages of this CTA.
__device__ void run_group_emu(const StepLaunch &p, const Group &g, const Warp &W, const WsSmem &X, uint32_t &msg,
                              bool &failed) {
  const DevState &st = p.st;
  const GameDev &G = smem_game();
  const int64_t slot = (int64_t)g.slot0 + (W.active ? W.j : 0);
  const IO io = p.io_table ? p.io_table[g.io] : p.io0;
  const uint32_t quirks = p.quirks;
  const Ctx C = make_ctx<false>(W, st, slot, (uint32_t)p.n_uops, table_base((uint32_t)p.n_uops));
  Regs R;
  load_regs<false>(R, C);
  const int64_t row = (int64_t)C.rec[Rec<false>::kRow];
  uint32_t ep = C.rec[Rec<false>::kEp];
  int32_t prev = W.active ? score(R, C, G) : 0;
  const uint32_t K = G.K, FS = G.frameskip, first_kept = FS - (uint32_t)p.S;

  for (int s = 0; s < p.steps && !failed; ++s) {
    const int64_t io_row = (int64_t)(p.step0 + s) * io.rows + row;
    int key = -1;
    if (W.active) key = key_of(R, G, applied_action<true, false>(R, C, G, io.actions[io_row]));
    R.draws = 0;
    R.phase = 0;
    for (uint32_t f = 0; f < FS && !failed; ++f) {
      if (W.active) {
        run_instrs<false>(R, C, key, quirks, K);
        tick(C);
      }
      if (f >= first_kept) {  // hand the frame to the writers
        const uint32_t b = msg & 1u, use = msg >> 1;
        failed = !__all_sync(kFull, mbar_wait(X.empty + b, (use & 1u) ^ 1u, p.err));
        if (failed) break;
        if (W.active) ring_put(X, C, W.J, W.j, b);
        mbar_arrive(X.full + b);
        ++msg;
      }
    }
    if (failed) break;
    bool done = false;
    if (W.active) {
      const int32_t sc = score(R, C, G);
      ep += 1;
      R.env_steps += 1;
      done = terminated(R, C, G) || (G.max_steps != 0 && ep >= G.max_steps);
      if (C.sub == 0) {
        io.reward[io_row] = (float)(sc - prev);
        io.done[io_row] = done ? 1 : 0;
      }
      if (done) {
        reset_instance<true, false>(R, C, G, quirks);
        ep = 0;
        prev = score(R, C, G);
      } else {
        prev = sc;
      }
    }
    // end-of-step message: done flags and the reset displays
    const uint32_t b = msg & 1u, use = msg >> 1;
    failed = !__all_sync(kFull, mbar_wait(X.empty + b, (use & 1u) ^ 1u, p.err));
    if (failed) break;
    if (W.active) {
      X.done[b * W.J + W.j] = done ? 1 : 0;
      if (done) ring_put(X, C, W.J, W.j, b);
    }
    mbar_arrive(X.full + b);
    ++msg;
  }

  // a failed wait fails the whole warp's group: its records stay as they were
  if (failed) return;
  if (W.active) store_regs<false>(R, C, ep);
  return_records<false>(W, st, g, kFull);
}

// Writer side of one group: writer warp ww owns instances
// [ww * J/W, (ww + 1) * J/W); lane -> instance 8m + lane/4, quarter lane%4.
__device__ void run_group_writer(const StepLaunch &p, const Group &g, const WsSmem &W, uint32_t &msg,
                                 bool &failed) {
  if (p.stall_writers) return;  // diagnostic: never hand slots back (see octax_debug_stall_writers)
  const int t = threadIdx.x, lane = t & 31;
  const int E = (int)(blockDim.x >> 5) - p.writers;
  const int J = E * p.ipw;
  const int per = J / p.writers, passes = per >> 3;  // per in {8, 16, 32}
  const int ww = (t >> 5) - E;
  const uint32_t q = lane & 3u;
  const IO io = p.io_table ? p.io_table[g.io] : p.io0;
  const int S_ = p.S;
  int jj[4];
  int64_t orow[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    jj[m] = ww * per + 8 * m + (lane >> 2);
    const bool act = m < passes && jj[m] < (int)g.count;
    orow[m] = act ? (int64_t)p.st.rec[((int64_t)g.slot0 + jj[m]) * Rec<false>::kWords + Rec<false>::kRow] : -1;
  }
  const GameDev &G = smem_game();
  const uint32_t FS = G.frameskip, first_kept = FS - (uint32_t)S_;
  for (int s = 0; s < p.steps && !failed; ++s) {
    const int64_t step_row = (int64_t)(p.step0 + s) * io.rows;
    for (uint32_t f = first_kept; f <= FS; ++f) {  // FS - S frames, then the end-of-step message
      const uint32_t b = msg & 1u, use = msg >> 1;
      failed = !__all_sync(kFull, mbar_wait(W.full + b, use & 1u, p.err));
      if (failed) break;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (m >= passes || orow[m] < 0) continue;
        uint8_t *obs = io.obs + (step_row + orow[m]) * (int64_t)S_ * kFrameBytes + q * 16u;
        const uint64_t *rows = W.ring + (b * J + jj[m]) * kRingPitch;
        if (f < FS) {
          uint8_t *dst = obs + (f - first_kept) * kFrameBytes;
#pragma unroll 8
          for (int r = 0; r < 32; ++r) __stcs(reinterpret_cast<uint4 *>(dst + r * 64), expand16(rows[r], q));
        } else if (W.done[b * J + jj[m]]) {
          for (int r = 0; r < 32; ++r) {
            const uint4 o = expand16(rows[r], q);
            for (int k = 0; k < S_; ++k)
              __stcs(reinterpret_cast<uint4 *>(obs + k * kFrameBytes + r * 64), o);
          }
        }
      }
      mbar_arrive(W.empty + b);
      ++msg;
    }
  }
}

__global__ void step_kernel_ws(const StepLaunch p) {
  const int E = (int)(blockDim.x >> 5) - p.writers;
  const WsSmem X = carve_ws((uint32_t)p.n_uops, E * p.ipw, E);
  __shared__ int s_group;
  if (threadIdx.x == 0) {
    mbar_init(X.full + 0, (uint32_t)E * 32u);
    mbar_init(X.full + 1, (uint32_t)E * 32u);
    mbar_init(X.empty + 0, (uint32_t)p.writers * 32u);
    mbar_init(X.empty + 1, (uint32_t)p.writers * 32u);
  }
  __syncthreads();
  const bool writer = (int)(threadIdx.x >> 5) >= E;
  uint32_t msg = 0;
  bool failed = false;
  int cur_game = -1;
  int gi = blockIdx.x;
  for (;;) {
    if (p.work_counter) {
      if (threadIdx.x == 0) s_group = (int)atomicAdd(p.work_counter, 1u);
      __syncthreads();
      gi = s_group;
    }
    if (gi >= p.n_groups) break;
    const Group g = p.groups[gi];
    const Warp W = make_warp(p.ipw, E, g, (uint32_t)p.n_uops, Rec<false>::kWords);
    if ((int)g.game != cur_game) {
      stage_game(p.blobs, p.stride, g.game, (uint32_t)p.n_uops);
      cur_game = g.game;
    }
    grid_dependency_wait();  // states, actions and output buffers from here on
    if (!writer) fetch_records<false>(W, p.st, g);
    copy_wait();
    __syncthreads();
    if (!failed) {
      if (writer) run_group_writer(p, g, X, msg, failed);
      else run_group_emu(p, g, W, X, msg, failed);
    }
    failed = __syncthreads_or(failed);  // (and shared memory is reused by the next group)
    if (!p.work_counter) break;
  }
}

template <bool kS>
__global__ void __launch_bounds__(kMaxBlock, 2) reset_kernel(const ResetLaunch p) {
  using T = Rec<kS>;
  const Group g = p.groups[blockIdx.x];
  const Warp W = make_warp(p.ipw, blockDim.x >> 5, g, (uint32_t)p.n_uops, T::kWords);
  if (!p.init) fetch_records<kS>(W, p.st, g);
  stage_game(p.blobs, p.stride, g.game, (uint32_t)p.n_uops);
  copy_wait();
  __syncthreads();
  const DevState &st = p.st;
  const GameDev &G = smem_game();
  const int64_t slot = (int64_t)g.slot0 + (W.active ? W.j : 0);
  const Ctx C = make_ctx<kS>(W, st, slot, (uint32_t)p.n_uops, table_base((uint32_t)p.n_uops));
  Regs R;
  if (p.init) {
    const uint64_t seed = p.seed_of_group ? p.seed_of_group[blockIdx.x] : p.seed;
    R.status = 0;
    R.env_steps = 0;
    if (W.active) {
      const uint32_t row = p.row_of_slot ? p.row_of_slot[slot] : g.row0 + (uint32_t)W.j;
      for (int k = T::kRow + 1; k < T::kWords; ++k) C.rec[k] = 0;
      C.rec[T::kMisc] = (uint32_t)g.game << 16;
      C.rec[T::kKey] = (uint32_t)(seed & 0xFFFFFFFFu);
      C.rec[T::kKey + 1] = (uint32_t)(seed >> 32);
      C.rec[T::kUid] = p.uid_of_slot ? p.uid_of_slot[slot] : row;
      C.rec[T::kRow] = row;
    }
    __syncwarp();
  } else {
    load_regs<kS>(R, C);
  }
  const uint32_t row = C.rec[T::kRow];
  const bool doit = W.active && (p.mask == nullptr || p.mask[row] != 0);
  if (doit) reset_instance<true, kS>(R, C, G, p.quirks);
  const unsigned which = __ballot_sync(kFull, doit && C.sub == 0);
  if (p.obs && which) {
    __syncwarp();
    write_reset_obs<kS>(W.recs, doit ? p.obs + (int64_t)row * p.S * Disp<kS>::kFrame : nullptr, p.S, which, W.lane, W.sh);
  }
  __syncwarp();
  if (doit) store_regs<kS>(R, C, 0u);
  return_records<kS>(W, st, g, which);
}

// RAM byte of a slot as the program sees it.
__device__ __forceinline__ uint8_t ram_byte(const DevState &st, const uint8_t *img, int64_t slot,
                                            uint64_t dirty, uint32_t a) {
  return ((dirty >> (a >> kPageShift)) & 1u) ? st.ram[slot * (int64_t)kRamBytes + a] : img[a];
}

__device__ __forceinline__ uint64_t fnv_byte(uint64_t h, uint32_t b) {
  return (h ^ (uint64_t)(b & 0xFFu)) * 1099511628211ull;
}
__device__ __forceinline__ uint64_t fnv_word(uint64_t h, uint32_t w) {
  for (int b = 0; b < 4; ++b) h = fnv_byte(h, w >> (8 * b));
  return h;
}

__global__ void hash_kernel(const DevState st, const uint8_t *blobs, size_t stride, const uint32_t *slot_of_row,
                            int64_t rows, uint64_t *out) {
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= rows) return;
  const int64_t slot = slot_of_row[row];
  const uint32_t *rec = st.rec + slot * rec_words(st.schip);
  const uint32_t *t = rec + 2 * disp_words(st.schip);  // the words behind the display
  const uint32_t misc = t[6];
  const uint8_t *img = blobs + (misc >> 16) * stride;
  uint64_t h = 14695981039346656037ull;
  for (int j = 0; j < 4; ++j) h = fnv_word(h, t[j]);
  const uint32_t I = t[5] >> 16, PC = t[5] & 0xFFFFu;
  h = fnv_word(h, I | PC << 16);
  h = fnv_word(h, (misc & 0x7Fu) | (t[4] & 0xFFu) << 8 | (t[4] & 0xFF0000u) | (misc & 0xFF00u) << 16);  // SP DT ST status
  for (int i = 0; i < 8; ++i) h = fnv_word(h, t[12 + i]);
  for (int r = 0; r < 2 * disp_words(st.schip); ++r) h = fnv_word(h, rec[r]);  // SCHIP words run [y][h], as in the record
  const uint64_t dirty = t[8] | (uint64_t)t[9] << 32;
  for (uint32_t a = 0; a < (uint32_t)kRamBytes; ++a) h = fnv_byte(h, ram_byte(st, img, slot, dirty, a));
  h = fnv_word(h, t[10]);
  h = fnv_word(h, t[11]);
  h = fnv_byte(h, t[4] >> 8);
  if (st.schip) {
    h = fnv_byte(h, (misc >> 7) & 1u);
    for (int i = 0; i < 4; ++i) h = fnv_word(h, t[24 + i]);
  }
  out[row] = h;
}

__global__ void records_kernel(const DevState st, const uint8_t *blobs, size_t stride, const uint32_t *slot_of_row,
                               int64_t first, int64_t count, octax_state_record *out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int64_t slot = slot_of_row[first + i];
  const uint32_t *w = st.rec + slot * rec_words(st.schip);
  const uint32_t *t = w + 2 * disp_words(st.schip);
  octax_state_record &rec = out[i];
  for (int j = 0; j < 16; ++j) rec.V[j] = (uint8_t)(t[j >> 2] >> (8 * (j & 3)));
  const uint32_t pcI = t[5], misc = t[6], timers = t[4];
  rec.PC = (uint16_t)(pcI & 0xFFFFu);
  rec.I = (uint16_t)(pcI >> 16);
  rec.SP = (uint8_t)(misc & 0x7Fu);
  rec.DT = (uint8_t)timers;
  rec.ST = (uint8_t)(timers >> 16);
  rec.status = (uint8_t)(misc >> 8);
  for (int k = 0; k < 16; ++k) rec.stack[k] = (uint16_t)(t[12 + (k >> 1)] >> (16 * (k & 1)));
  const uint64_t *disp = reinterpret_cast<const uint64_t *>(w);
  for (int y = 0; y < 64; ++y)
    for (int hw = 0; hw < 2; ++hw)
      rec.display[y][hw] = st.schip ? disp[2 * y + hw] : (y < 32 && hw == 0 ? disp[y] : 0ull);
  const uint8_t *img = blobs + (misc >> 16) * stride;
  const uint64_t dirty = t[8] | (uint64_t)t[9] << 32;
  for (uint32_t a = 0; a < (uint32_t)kRamBytes; ++a) rec.ram[a] = ram_byte(st, img, slot, dirty, a);
  rec.episode_steps = t[10];
  rec.env_steps = t[11];
  rec.last_action = (uint8_t)(timers >> 8);
  rec.hires = st.schip ? (misc >> 7) & 1u : 0;
  for (int k = 0; k < 6; ++k) rec.pad[k] = 0;
  for (int k = 0; k < 16; ++k) rec.rpl[k] = st.schip ? (uint8_t)(t[24 + (k >> 2)] >> (8 * (k & 3))) : 0;
}

__global__ void set_records_kernel(const DevState st, const uint8_t *blobs, size_t stride,
                                   const uint32_t *slot_of_row, int64_t first, int64_t count,
                                   const octax_state_record *in) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int64_t slot = slot_of_row[first + i];
  const octax_state_record &rec = in[i];
  uint32_t *w = st.rec + slot * rec_words(st.schip);
  uint32_t *t = w + 2 * disp_words(st.schip);
  for (int j = 0; j < 4; ++j) {
    uint32_t v = 0;
    for (int b = 0; b < 4; ++b) v |= (uint32_t)rec.V[4 * j + b] << (8 * b);
    t[j] = v;
  }
  t[4] = (uint32_t)rec.DT | (uint32_t)rec.last_action << 8 | (uint32_t)rec.ST << 16 | 15u << 24;
  t[5] = (uint32_t)(rec.PC & 0xFFFu) | ((uint32_t)rec.I << 16);
  t[6] = (t[6] & 0xFFFF0000u) | (uint32_t)rec.status << 8 | (st.schip && rec.hires ? 0x80u : 0u) | (uint32_t)rec.SP;
  for (int k = 0; k < 8; ++k) t[12 + k] = (uint32_t)rec.stack[2 * k] | (uint32_t)rec.stack[2 * k + 1] << 16;
  uint64_t *disp = reinterpret_cast<uint64_t *>(w);
  for (int r = 0; r < disp_words(st.schip); ++r) disp[r] = st.schip ? rec.display[r >> 1][r & 1] : rec.display[r][0];
  if (st.schip)
    for (int k = 0; k < 4; ++k) {
      uint32_t v = 0;
      for (int b = 0; b < 4; ++b) v |= (uint32_t)rec.rpl[4 * k + b] << (8 * b);
      t[24 + k] = v;
    }
  const uint8_t *img = blobs + (t[6] >> 16) * stride;
  uint64_t dirty = 0;
  uint32_t lo = 0xFFFu, hi = 0u;
  uint8_t *ram = st.ram + slot * (int64_t)kRamBytes;
  for (int page = 0; page < kRamBytes >> kPageShift; ++page) {
    bool differs = false;
    for (int b = 0; b < (1 << kPageShift); ++b) {
      const int a = (page << kPageShift) + b;
      if (rec.ram[a] != img[a]) {
        differs = true;
        lo = a < (int)lo ? (uint32_t)a : lo;
        hi = (uint32_t)a;
      }
    }
    if (differs) {
      dirty |= 1ull << page;
      for (int b = 0; b < (1 << kPageShift); ++b) ram[(page << kPageShift) + b] = rec.ram[(page << kPageShift) + b];
    }
  }
  t[7] = lo | hi << 16;  // the bytes that differ from the image lie in [lo, hi]
  t[8] = (uint32_t)dirty;
  t[9] = (uint32_t)(dirty >> 32);
  t[10] = rec.episode_steps;
  t[11] = rec.env_steps;
}

}  // namespace

size_t step_smem_bytes(int block, int ipw, int schip, int n_uops) {
  const size_t J = (size_t)(block / 32) * ipw;
  return blob_bytes(n_uops) + J * 4 * rec_words(schip) + (size_t)block * kLaneBytes;
}

// Opt-in dynamic shared memory limit of the current device (less 1 KB for
// static shared memory), queried once per device ordinal.
size_t max_dynamic_smem() {
  static std::mutex mu;
  static std::map<int, size_t> per_dev;
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  auto it = per_dev.find(dev);
  if (it != per_dev.end()) return it->second;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || optin <= 0)
    optin = 99 * 1024;
  const size_t v = (size_t)optin - 1024;
  per_dev[dev] = v;
  return v;
}

size_t step_ws_smem_bytes(int block, int ipw, int n_uops) {
  const size_t J = (size_t)(block / 32) * ipw;
  return step_smem_bytes(block, ipw, 0, n_uops) + 2 * kRingPitch * 8 * J + ((2 * J + 15) & ~(size_t)15) + 4 * 8;
}

// The accepted shapes: 23,232 bytes for the game and 384 (SCHIP 1,152) per
// instance, with the writers' ring 512 more and the hand-over's flags.
bool shape_fits(int block, int ipw, int schip, int writers) {
  const size_t J = (size_t)(block / 32) * ipw;
  size_t need = 23232 + J * (schip ? 1152 : 384);
  if (writers > 0) need += 512 * J + ((2 * J + 15) & ~(size_t)15) + 32;
  return need <= max_dynamic_smem();
}

static size_t launch_smem(int block, int ipw, int schip, int writers, int n_uops) {
  return writers > 0 ? step_ws_smem_bytes(block, ipw, n_uops) : step_smem_bytes(block, ipw, schip, n_uops);
}

// Most instances per warp, up to ipw, whose records fit a CTA's shared memory
// beside the game's table. Of the accepted shapes one can lose some: 256 x 22
// of Super-CHIP games with a ROM over 3,072 bytes run as 256 x 21.
int fit_ipw(int block, int ipw, int schip, int writers, int n_uops) {
  while (ipw > 1 && launch_smem(block, ipw, schip, writers, n_uops) > max_dynamic_smem()) --ipw;
  return ipw;
}

// The step kernel instantiation for a launch (null: writer warps on SCHIP).
template <uint32_t kBase>
static const void *plain_fn(int wrappers, int schip) {
  if (schip) return wrappers ? (const void *)step_kernel<true, true, kBase> : (const void *)step_kernel<false, true, kBase>;
  return wrappers ? (const void *)step_kernel<true, false, kBase> : (const void *)step_kernel<false, false, kBase>;
}
static const void *step_fn(int writers, int wrappers, int schip, int n_uops) {
  if (writers > 0) return schip ? nullptr : (const void *)step_kernel_ws;
  return table_base((uint32_t)n_uops) == 0u ? plain_fn<0u>(wrappers, schip) : plain_fn<0x200u>(wrappers, schip);
}

// The dynamic shared memory attribute of a kernel applies to the current
// device only, so it is set once per device ordinal (under a lock: the
// serving thread and user threads launch concurrently).
static cudaError_t ensure_smem_attr() {
  static std::mutex mu;
  static std::map<int, bool> done;
  int dev = 0;
  cudaError_t de = cudaGetDevice(&dev);
  if (de != cudaSuccess) return de;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return cudaSuccess;
  const int cap = (int)max_dynamic_smem();
  const int kShort = 0, kLong = kLongTable + 1;  // micro-ops of tables at either base
  const void *fns[] = {step_fn(0, 0, 0, kShort),          step_fn(0, 1, 0, kShort), step_fn(0, 0, 1, kShort),
                       step_fn(0, 1, 1, kShort),          step_fn(0, 0, 0, kLong),  step_fn(0, 1, 0, kLong),
                       step_fn(0, 0, 1, kLong),           step_fn(0, 1, 1, kLong),  (const void *)reset_kernel<false>,
                       (const void *)reset_kernel<true>, (const void *)step_kernel_ws};
  for (const void *f : fns) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, cap);
    if (e != cudaSuccess) return e;
  }
  done[dev] = true;
  return cudaSuccess;
}

cudaError_t launch_step(const StepLaunch &p, int grid, int block, cudaStream_t s) {
  if (!state_complete(p.st)) return cudaErrorInvalidValue;
  cudaError_t e = ensure_smem_attr();
  if (e != cudaSuccess) return e;
  if (grid <= 0) return cudaSuccess;
  const void *fn = step_fn(p.writers, p.wrappers, p.st.schip, p.n_uops);
  if (!fn) return cudaErrorInvalidValue;
  StepLaunch copy = p;
  void *args[] = {&copy};
  const int threads = p.writers > 0 ? block + 32 * p.writers : block;
  return launch_kernel(fn, dim3((unsigned)grid), dim3((unsigned)threads), args,
                       launch_smem(block, p.ipw, p.st.schip, p.writers, p.n_uops), s, !p.work_counter);
}

cudaError_t launch_reset(const ResetLaunch &p, int block, cudaStream_t s) {
  if (!state_complete(p.st)) return cudaErrorInvalidValue;
  cudaError_t e = ensure_smem_attr();
  if (e != cudaSuccess) return e;
  if (p.n_groups <= 0) return cudaSuccess;
  const size_t smem = step_smem_bytes(block, p.ipw, p.st.schip, p.n_uops);
  if (p.st.schip) reset_kernel<true><<<p.n_groups, block, smem, s>>>(p);
  else reset_kernel<false><<<p.n_groups, block, smem, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_tables(uint8_t *blobs, size_t stride, int n_games, int n_uops, int schip, uint32_t quirks,
                          cudaStream_t s) {
  tables_kernel<<<n_games, 256, 0, s>>>(blobs, stride, (uint32_t)n_uops, schip, quirks);
  return cudaGetLastError();
}

cudaError_t launch_hash(const DevState &st, const uint8_t *blobs, size_t stride, const uint32_t *slot_of_row,
                        int64_t rows, uint64_t *out, cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  if (!state_complete(st)) return cudaErrorInvalidValue;
  const int tb = 128;
  hash_kernel<<<(unsigned)((rows + tb - 1) / tb), tb, 0, s>>>(st, blobs, stride, slot_of_row, rows, out);
  return cudaGetLastError();
}

cudaError_t launch_records(const DevState &st, const uint8_t *blobs, size_t stride, const uint32_t *slot_of_row,
                           int64_t first, int64_t count, octax_state_record *out, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  if (!state_complete(st)) return cudaErrorInvalidValue;
  const int tb = 128;
  records_kernel<<<(unsigned)((count + tb - 1) / tb), tb, 0, s>>>(st, blobs, stride, slot_of_row, first, count, out);
  return cudaGetLastError();
}

cudaError_t launch_set_records(const DevState &st, const uint8_t *blobs, size_t stride, const uint32_t *slot_of_row,
                               int64_t first, int64_t count, const octax_state_record *in, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  if (!state_complete(st)) return cudaErrorInvalidValue;
  const int tb = 128;
  set_records_kernel<<<(unsigned)((count + tb - 1) / tb), tb, 0, s>>>(st, blobs, stride, slot_of_row, first, count, in);
  return cudaGetLastError();
}

cudaError_t add_step_node(cudaGraph_t g, cudaGraphNode_t *node, cudaGraphNode_t dep, const StepLaunch &p,
                          int grid, int block) {
  if (!state_complete(p.st)) return cudaErrorInvalidValue;
  cudaError_t e = ensure_smem_attr();
  if (e != cudaSuccess) return e;
  const void *fn = step_fn(p.writers, p.wrappers, p.st.schip, p.n_uops);
  if (!fn) return cudaErrorInvalidValue;
  StepLaunch copy = p;
  void *args[] = {&copy};
  cudaKernelNodeParams kp;
  memset(&kp, 0, sizeof kp);
  kp.func = const_cast<void *>(fn);
  kp.gridDim = dim3((unsigned)grid);
  kp.blockDim = dim3((unsigned)(p.writers > 0 ? block + 32 * p.writers : block));
  kp.sharedMemBytes = (unsigned)launch_smem(block, p.ipw, p.st.schip, p.writers, p.n_uops);
  kp.kernelParams = args;
  return cudaGraphAddKernelNode(node, g, dep ? &dep : nullptr, dep ? 1 : 0, &kp);
}

cudaError_t alloc_state(DevState &st, int64_t n, int schip, void **block_out, size_t *bytes_out) {
  const size_t rec = ((size_t)n * 4 * rec_words(schip) + 255) & ~(size_t)255;
  const size_t total = rec + (size_t)n * kRamBytes;
  uint8_t *base = nullptr;
  cudaError_t e = cudaMalloc(&base, total);
  if (e != cudaSuccess) return e;
  st.rec = reinterpret_cast<uint32_t *>(base);
  st.ram = base + rec;
  st.n = n;
  st.schip = schip;
  *block_out = base;
  *bytes_out = total;
  return cudaSuccess;
}

int max_resident_ctas(int block, int ipw, int writers, int wrappers, int schip, int n_uops) {
  if (ensure_smem_attr() != cudaSuccess) return 0;
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const void *fn = step_fn(writers, wrappers, schip, n_uops);
  if (!fn) return 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block + 32 * writers,
                                                launch_smem(block, ipw, schip, writers, n_uops));
  return sms * per_sm;
}

}  // namespace octax
