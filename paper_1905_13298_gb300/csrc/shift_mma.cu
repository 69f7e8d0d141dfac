// Shift operators on the tensor cores, exact (sm_103a).
//
//   y[row][col] = sat32( bias[col] + sum_k s[col][k] * (A[row][k] >> -p[col][k]) )      (Eq. 1-3)
//
// A floor shift is not linear in x, but it is linear in the bits of x: with
// sh = -p in [0, 15],
//   x >> sh = sum_{i = sh}^{15} bit_i(x) 2^(i - sh)  +  (x >> 16) 2^(16 - sh),
// since bits 16 and up are never shifted out.  So the sum over k is an
// ordinary contraction of 16 bit features and one signed digit x >> 16 per
// input value with weights that are 0 or +-2^e: every operand is exact in 8-bit
// floating point and every product is a power of two times a small integer.
// It runs as tcgen05.mma kind::f8f6f4 at 8192 multiply-adds per clock and SM;
// 17 of them per term replace the two instructions (shift, multiply-add) that
// the CUDA cores issue at 128 per clock.
//
// Operands, per input value and weight (16 bytes each):
//   x   e4m3, word j = z & (0x01010101 << j) where byte q of z holds nibble q
//       of x in its low half: byte q of word j is bit 4q + j at bit position
//       j, which encodes 2^(j - 9) (subnormal up to j = 2)
//   w   e5m2, word j: byte q is s * 2^(4q - sh) if 4q + j >= sh, else 0
// and the digit, one byte per value: x >> 16 in [-16, 16] as e4m3 sign and
// magnitude (the codes 0..16 encode n * 2^-9) against s * 2^(16 - sh).
//
// Exactness.  Products are integers times one power of two per accumulator, and
// fp32 accumulation of integers is exact while every partial sum stays below
// 2^24, whatever the order.  Two accumulators share a tile: L takes the bit
// features, H the digits.  With a = sum_k |w| of a column,
//   L <= 2^16 a,   H <= max|digit| 2^16 a in units of 2.
// A tile whose columns keep both below 2^24 ("bounded": every layer whose shifts
// are centred for its fan-in) sums its whole reduction so.  Any other tile keeps
// the terms themselves small, whatever the codes: the digits of weights with
// sh >= 8 go to L instead (2^8 16 each), nibble 3 of the inputs of weights with
// sh < 4 goes to H as one more digit (2^(12 - sh)), so a term is at most 4351 in L
// and 2168 in H (units of 2^9), and runs of 3840 terms stay below 2^24; the integer
// sums are added between runs.  That is 19 tensor operations per 32 indices
// instead of 17.  Inputs beyond 2^20 take one pass per 4-bit digit of x >> 16, the
// lower digits unsigned.  The accumulator-width proof is the one of the other
// integer kernels: where it fails, sums are 64-bit (in tiles of 128 columns, half of
// them at a time, in two walks: all of them have no room) and saturated.
//
// CTA: 128 rows (tensor-memory lanes) x N columns; a pair of CTAs shares a tile
// of 256 rows, each decoding half of its weights (cta_group::2), since a tile's
// weight bytes are written to and read from shared memory once per 128 or 256
// rows.  23 warps (swapped roles, below: 27, two of them idle), with x as operand A:
//   warps 0-11   operand A, three groups of four: a thread gathers 16 values of
//                its row, expands them and writes them to tensor memory
//   warps 12-15  epilogue: accumulators to integer sums in shared memory, then
//                bias, saturation, residual, ReLU, max|y| and the output
//   warps 16-21  operand B, three groups of two: decode the packed codes of a
//                column through a table of weight bytes into shared memory
//   warp 22      issues the tensor operations (swapped roles: warp 16, B after it)
// FC layers of up to 128 rows, and others of few tiles, swap the operands' roles: the
// lanes are 128 weight columns, decoded into tensor memory, and N = 64 rows of x are
// expanded into shared memory, so that no lane is idle and a code is decoded once per
// 64 rows (VGG16 FC1 at batch 64: 0.361 ms with rows as lanes, 0.189 ms so).
// A ring of three slots of 16 reduction indices connects them; CTAs are
// persistent over tiles and the ring runs on across them.  A grid that leaves
// SMs idle splits the reduction over the CTAs of a cluster, which sum their
// partial tiles through distributed shared memory.  Every barrier wait of a role
// is bounded; on expiry the CTA stops and sets a flag, and no output is made from
// its sums.  The cluster barriers need no bound of their own: every CTA reaches
// them, since its roles' waits are bounded.
//
// Measured (GB300, back to back over changing inputs, with the max|x| pre-pass,
// CUDA-core kernels -> here): FC 8192 x 4096 x 4096 9.93 -> 1.53 ms (one input again and
// again: 1.47; about 760 clocks a slot of 16 indices, of which the operations alone
// take 608), ConvShift 64x56x56 3x3 at batch 32 with a residual 0.296 -> 0.110 ms,
// 256x14x14 -> 512 3x3/2 0.216 -> 0.051 ms, 1024x14x14 -> 256 1x1 at batch 64 0.301 -> 0.086
// ms, VGG16 FC1 at batch 64 0.565 -> 0.189 ms.  What bounds it: at
// N = 128 the ALU pipe (expanding x: 5-6 of its instructions a value, which run
// at 64 lanes a clock and SM) and the operations' issue; at N = 64 the issuing
// warp (about 590 clocks a slot with nothing else done, against 272 of
// operations) and operand A.  wait -> issue -> commit is a chain of single instructions.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>

#include "ds_common.cuh"
#include "tensor_core.cuh"

namespace ds {

__device__ int g_mma_fault;  // set when a bounded wait gives up

namespace {

namespace cg = cooperative_groups;

constexpr int kRows = 128;      // rows per tile: the lanes of tensor memory
constexpr int kSlotK = 16;      // reduction indices per ring slot
constexpr int kSlots = 3;
constexpr int kRunChunks = 120; // chunks of 32 per run of a tile with unbounded columns
constexpr int kAGroups = 3;     // four warps each; group g fills ring slot g
constexpr int kAWarps = 4 * kAGroups, kEpiWarps = 4;
static_assert(kAGroups == kSlots, "a group of operand-A warps per ring slot");
// warps 0-11 operand A, 12-15 epilogue, then operand B, then the tensor operations
constexpr int kFirstEpi = kAWarps, kFirstB = kFirstEpi + kEpiWarps;
// Operand B: three groups of two warps, or with swapped roles two of four.  23
// warps leave a thread 80 registers, from 25 on it is 72: with 72 the convolution's operand
// A spills in its loop (a version with 270 spilled bytes ran 15-30% slower).
__host__ __device__ constexpr int b_warps(bool swap) { return swap ? 8 : 6; }
__device__ __forceinline__ int swapped_b_warp(int warp) {
  return warp > kFirstB && (warp & 3) != 0 ? 3 * ((warp - kFirstB) >> 2) + (warp & 3) - 1 : 1 << 16;
}
// Swapped roles: the issuing warp is warp 16 and B's are 17-19, 21-23, 25 and 26 (20
// and 24 idle), so that no B warp is on its scheduler: VGG16 FC1 at batch 64 0.205
// -> 0.193 ms on one GPU in turn.  (Unswapped, two more warps would cost the 80 registers.)
__host__ __device__ constexpr int cta_threads(bool swap) { return 32 * (swap ? 27 : kFirstB + b_warps(false) + 1); }
constexpr int kCodeAhead = 4;   // slots of a B group whose codes are in flight
constexpr int kCodeBytes = kCodeAhead * b_warps(false) * 32 * 16;
constexpr int kMaxColTiles = 512;
constexpr int kMaxTaps = 121;
constexpr int kMaxCluster = 16;
constexpr long long kWaitCycles = 4000000000LL;  // about 2 s

// the wait limit of the next launches (a diagnostic can shorten it to make the waits run out)
std::atomic<long long> g_wait_cycles{kWaitCycles};

constexpr int kAccStride = kRows + 1;  // words between a column's sums and the next one's: no bank conflicts either way
constexpr int kXStride = 20;    // words per staged row of 16 values: 16-byte reads of 8 rows hit all banks

// Tensor-memory columns: accumulators L and H (two pairs when N = 64), then
// three operand slots of 64 columns and two buffers of 3 x 8 digit columns.
constexpr uint32_t kTmemSlots = 256, kTmemDigits = kTmemSlots + 64 * kSlots, kTmemCols = 512;

// Column-tile flags.
constexpr uint32_t kInt32 = 1;   // 32-bit sums are exact
constexpr uint32_t kBounded = 2;  // the columns' weights bound L and H over the whole reduction

struct PhaseInfo {
  FastDiv ohw, ow, ct;   // OH * OW, OW, column tiles
  int tile_end;          // tiles of the phases up to and including this one
  int col_tiles, flag_off, flag_tiles;
};

struct MmaSet {
  GemmParams p[kMaxGemmPhases];
  PhaseInfo info[kMaxGemmPhases];
  int n, splits, table_entries;  // table_entries: per phase
  long long wait_cycles;         // limit of a barrier wait before the CTA gives up
};

struct __align__(8) Bars {
  uint64_t full[kSlots], empty[kSlots], acc_full[2], acc_empty[2], done;
  long long wait_cycles;
  uint32_t tmem, amax;
  int abort;  // a wait of this CTA has given up
};

constexpr int kLutBytes = 64 * 128;
constexpr int kFlagOff = 512, kWalkOff = 1024, kBiasOff = 3072, kLutOff = 5120, kTableOff = kLutOff + 2 * kLutBytes;

template <int N, bool PAIR>
struct Layout {
  static constexpr int NL = PAIR ? N / 2 : N;           // columns whose weights one CTA holds
  static constexpr int slot_bytes = kSlotK * NL * 16;
  static constexpr int digit_bytes = 2 * NL * 16;       // 32 indices, one operand
  // 32-bit sums, or 64-bit sums of all columns where they have room (N = 64), else of half
  // of them, in a second walk over the tile.  One walk instead of two, inputs up to 2^31
  // (four digits), against the CUDA cores: 64x56x56 3x3 at batch 32 733 -> 395 us (567),
  // 256x56x56 -> 64 1x1 400 -> 243 (318), the 7x7 stem 903 -> 566 (615), VGG16 FC1 at batch 64
  // 1471 -> 754 (1169).  Tiles of 128 columns stay under them in two (1024x14x14 -> 256
  // 1x1 484 against 592).
  static constexpr bool halves = N > 64;
  static constexpr int acc_bytes = N * kAccStride * (halves ? 4 : 8);
  static constexpr int xrow_bytes = kAWarps * 2 * 32 * kXStride * 4;
  __host__ __device__ static int base(int table_entries, int phases) {
    return (kTableOff + 2 * (4 * table_entries + 32) * 4 * phases + 1023) / 1024 * 1024;
  }
  static size_t total(int table_entries, int phases, bool conv) {
    return (size_t)base(table_entries, phases) + kSlots * slot_bytes + 6 * digit_bytes + acc_bytes + kCodeBytes +
           (conv ? 0 : xrow_bytes);
  }
};

// A whole warp waits, and goes on or gives up as one: its lanes' looks at the
// barrier may differ, and what follows is warp-wide tensor-memory work.
__device__ __noinline__ bool slow_wait(uint64_t* bar, uint32_t parity, volatile Bars* bars) {
  const long long t0 = clock64();
  while (!tc::mbar_try_wait(bar, parity)) {
    if (bars->abort) return false;
    if (clock64() - t0 > bars->wait_cycles) {
      bars->abort = 1;
      atomicExch(&g_mma_fault, 1);
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ bool wait(uint64_t* bar, uint32_t parity, volatile Bars* bars) {
  return __all_sync(0xffffffffu, tc::mbar_try_wait(bar, parity) || slow_wait(bar, parity, bars));
}

// The walk over a CTA's tiles, and in each tile over its segments (column half,
// run, digit) and the 32-index chunks of a segment.  Every role walks alike.
template <int GROUP, bool SWAP, bool HALVES>
struct Walk {
  const MmaSet& S;
  const uint8_t* flags;
  int t, t_step, n_tiles;
  int digits;
  int split_half;  // -1: both halves of a 64-bit tile in turn (no split); else the half of this pass
  int rank;
  int ph, rt, ct;
  uint32_t fl;
  int half, run, runs, d;
  int cb, ce;        // the chunks of this CTA's share of the reduction
  int chunk, c_end;  // the chunks of the segment

  __device__ __forceinline__ Walk(const MmaSet& s, const uint8_t* f, int digits_, int split_half_)
      : S(s), flags(f), digits(digits_), split_half(split_half_) {
    n_tiles = s.info[s.n - 1].tile_end;
    rank = (int)blockIdx.x / GROUP % s.splits;
    t = (int)blockIdx.x / GROUP / s.splits;
    t_step = (int)gridDim.x / GROUP / s.splits;
  }
  __device__ __forceinline__ bool valid() const { return t < n_tiles; }
  __device__ __forceinline__ const GemmParams& P() const { return S.p[ph]; }
  __device__ __forceinline__ void start_tile() {
    ph = 0;
    while (t >= S.info[ph].tile_end) ++ph;
    const int local = t - (ph > 0 ? S.info[ph - 1].tile_end : 0);
    rt = fdiv(local, S.info[ph].ct);
    ct = local - rt * S.info[ph].col_tiles;
    fl = flags[S.info[ph].flag_off + (SWAP ? rt : ct)];
    const int n = (int)S.p[ph].n_chunks;
    cb = (int)((int64_t)n * rank / S.splits);
    ce = (int)((int64_t)n * (rank + 1) / S.splits);
    runs = (fl & kBounded) ? 1 : (ce - cb + kRunChunks - 1) / kRunChunks;
    half = split_half > 0 ? split_half : 0;
    run = 0;
    d = 0;
    start_segment();
  }
  __device__ __forceinline__ void start_segment() {
    chunk = (fl & kBounded) ? cb : cb + run * kRunChunks;
    c_end = (fl & kBounded) ? ce : min(ce, chunk + kRunChunks);
  }
  __device__ __forceinline__ bool first_segment() const { return run == 0 && d == 0; }
  __device__ __forceinline__ bool last_segment() const { return run == runs - 1 && d == digits - 1; }
  // Whether the last segment of the CTA's last tile (of its second half, if 64-bit) is being walked.
  __device__ __forceinline__ bool at_end() const {
    return last_segment() && t + t_step >= n_tiles && (one_walk() || half == 1);
  }
  // Whether all columns are summed in one walk (HALVES: only 64-bit sums of half of the columns have room).
  __device__ __forceinline__ bool one_walk() const { return !HALVES || (fl & kInt32); }
  // The place in the walk, kept in shared memory between a producer warp's
  // segments (its registers are needed in between); every lane has the same.
  static constexpr int kWords = 14;
  __device__ __forceinline__ void save(int* m) const {
    __syncwarp();
    m[0] = t; m[1] = ph; m[2] = rt; m[3] = ct; m[4] = (int)fl; m[5] = half; m[6] = run; m[7] = runs; m[8] = d;
    m[9] = cb; m[10] = ce; m[11] = chunk; m[12] = c_end;
    __syncwarp();
  }
  __device__ __forceinline__ void restore(const int* m) {
    t = m[0]; ph = m[1]; rt = m[2]; ct = m[3]; fl = (uint32_t)m[4]; half = m[5]; run = m[6]; runs = m[7]; d = m[8];
    cb = m[9]; ce = m[10]; chunk = m[11]; c_end = m[12];
  }
  // The next segment, or the first of the next tile; false at the end of the tile (t advanced).
  __device__ __forceinline__ bool next_segment() {
    if (++d == digits) {
      d = 0;
      if (++run == runs) {
        run = 0;
        if (one_walk() || split_half >= 0 || half == 1) {
          t += t_step;
          return false;
        }
        half = 1;
      }
    }
    start_segment();
    return true;
  }
};

template <int GROUP, bool SWAP, bool HALVES>
__device__ __forceinline__ bool next_segment_or_tile(Walk<GROUP, SWAP, HALVES>& w) {
  if (w.next_segment()) return true;
  if (!w.valid()) return false;
  w.start_tile();
  return true;
}

// 16 bit features of x as four words.
__device__ __forceinline__ void expand_x(uint32_t x, uint32_t* w) {
  const uint32_t z = __byte_perm(x, x << 4, 0x6150);
  w[0] = z & 0x01010101u;
  w[1] = z & 0x02020202u;
  w[2] = z & 0x04040404u;
  w[3] = z & 0x08080808u;
}
// Bytes 2 of four values (their digits, two's complement) as e4m3 sign and magnitude.
__device__ __forceinline__ uint32_t digit4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  const uint32_t v = __byte_perm(__byte_perm(a, b, 0x0062), __byte_perm(c, d, 0x0062), 0x5410);
  uint32_t m;  // 0xff in the negative bytes
  asm("prmt.b32 %0, %1, 0, 0xba98;" : "=r"(m) : "r"(v));
  return ((v ^ m) + (m & 0x01010101u)) | (m & 0x80808080u);
}
// Nibbles 3 (bits 12-15) of four values as e4m3 integers.
__device__ __forceinline__ uint32_t nibble4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  return (__byte_perm(__byte_perm(a, b, 0x0051), __byte_perm(c, d, 0x0051), 0x5410) >> 4) & 0x0F0F0F0Fu;
}
// Digit d of x >> 16 (4 bits each, the top one signed) at bit 16; the low 16 bits stay with digit 0.
__device__ __forceinline__ uint32_t pick_digit(uint32_t x, int d, int digits) {
  if (d == 0) return x & 0xFFFFFu;
  const int32_t t = (int32_t)x >> (16 + 4 * d);
  return (uint32_t)(d == digits - 1 ? t : (t & 15)) << 16;
}

// Bits 0, 2, 4, 6 of b as the top bits of bytes 0..3.  The partial products of
// the multiplication meet only at odd positions, so a carry lands on an even
// one and stops there.
__device__ __forceinline__ uint32_t spread(uint32_t b) { return ((b & 0x55u) * 0x02082080u) & 0x80808080u; }

// The tap at element offset off of the window at src; 0 where a bit of m (its kernel row and column) is set in nm.
__device__ __forceinline__ uint32_t load_tap(const int32_t* src, int off, uint32_t m, uint32_t nm) {
  uint32_t v;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
      "and.b32 t, %2, %3;\n\t"
      "setp.eq.u32 p, t, 0;\n\t"
      "mov.b32 %0, 0;\n\t"
      "@p ld.global.nc.b32 %0, [%1];\n\t}"
      : "=&r"(v)
      : "l"(src + off), "r"(m), "r"(nm));
  return v;
}

// The weight bytes of four codes, from the table at lut: n4 holds 15 - sh per
// byte, sg the sign and zr the zero-code flag in the top bits.  The code of
// byte i goes to dst + i * step.
template <int STEP>
__device__ __forceinline__ void decode4(uint32_t n4, uint32_t sg, uint32_t zr, uint32_t lut, uint32_t dst) {
  const uint32_t ix = n4 | (sg >> 3) | (zr >> 2);
  uint32_t w[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[i][0]), "=r"(w[i][1]), "=r"(w[i][2]), "=r"(w[i][3])
                 : "r"(lut + __byte_perm(ix, 0, 0x4440 + i) * 128));
#pragma unroll
  for (int i = 0; i < 4; ++i)
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + i * STEP), "r"(w[i][0]), "r"(w[i][1]),
                 "r"(w[i][2]), "r"(w[i][3])
                 : "memory");
}

// The digit weights of four codes.  Bounded tiles: hi takes all digits, in units
// of 2.  Others: hi those with sh < 8, lo those with sh >= 8, n3 the nibble-3
// weights 2^(12 - sh) of the codes with sh < 4.
__device__ __forceinline__ void digit_weights(uint32_t n4, uint32_t sg, uint32_t zr, bool bounded, uint32_t& hi,
                                              uint32_t& lo, uint32_t& n3) {
  const uint32_t nz = ~((zr >> 7) * 0xFFu), pk = n4 << 2;
  hi = ((pk + 0x20202020u) | sg) & nz;
  if (!bounded) {
    const uint32_t lt8 = ((n4 & 0x08080808u) >> 3) * 0xFFu;               // 0xff where sh < 8
    const uint32_t lt4 = ((n4 & (n4 << 1) & 0x08080808u) >> 3) * 0xFFu;   // 0xff where sh < 4
    lo = ((pk + 0x40404040u) | sg) & nz & ~lt8;
    n3 = ((pk + 0x10101010u) | sg) & nz & lt4;
    hi &= lt8;
  }
}

__device__ __forceinline__ int32_t sat32(long long v) {
  return (int32_t)(v > (long long)INT32_MAX ? (long long)INT32_MAX : (v < (long long)INT32_MIN ? (long long)INT32_MIN : v));
}

// A row's place in the input and output tensors.
struct RowPlace {
  int64_t x0;   // conv: element offset of the window's first tap; FC: of the row
  int64_t y0;   // element offset of column 0's output
  uint32_t nm;  // conv: complement of the valid kernel rows (bits 0-15) and columns (16-31)
  bool ok;
};

template <bool CONV>
__device__ __forceinline__ RowPlace row_place(const GemmParams& P, const PhaseInfo& I, int64_t row) {
  RowPlace r;
  r.ok = row < P.rows;
  r.nm = 0xffffffffu;
  r.x0 = 0;
  r.y0 = 0;
  if (!r.ok) return r;
  if (!CONV) {
    r.x0 = row * P.kred;
    r.y0 = row * P.cols;
    return r;
  }
  const int n = fdiv((int)row, I.ohw);
  const int pix = (int)row - n * P.OH * P.OW;
  const int oh = fdiv(pix, I.ow), ow = pix - oh * P.OW;
  const int ih = oh * P.sh - P.ph, iw = ow * P.sw - P.pw;
  r.x0 = (int64_t)n * P.C * P.H * P.W + (int64_t)ih * P.W + iw;
  // kernel rows [max(0, -ih), min(R, H - ih)) read inside the image, columns likewise
  uint32_t vr = 0, vc = 0;
  const int r0 = max(0, -ih), r1 = min(P.R, P.H - ih), c0 = max(0, -iw), c1 = min(P.S, P.W - iw);
  if (r1 > r0) vr = ((1u << r1) - 1) & ~((1u << r0) - 1);
  if (c1 > c0) vc = ((1u << c1) - 1) & ~((1u << c0) - 1);
  r.nm = ~(vr | (vc << 16));
  int64_t plane = (int64_t)P.OH * P.OW, off = pix;
  if (P.ys_h) {
    plane = (int64_t)P.yH * P.yW;
    off = (int64_t)(P.ys_h * oh + P.yph) * P.yW + P.ys_w * ow + P.ypw;
  }
  r.y0 = (int64_t)n * P.cols * plane + off;
  return r;
}

template <bool CONV>
__device__ __forceinline__ int64_t col_stride(const GemmParams& P) {
  return !CONV ? 1 : (P.ys_h ? (int64_t)P.yH * P.yW : (int64_t)P.OH * P.OW);
}

// The tensor operations of ring slot SLOT into accumulator pair BUF, and with
// the second half of a chunk those of its digits (buffer dbuf).  Every operand
// address is a constant or a base from the kernel's parameters, so the
// operations issue from uniform registers.  first: 0 for the segment's first chunk,
// whose operations overwrite the accumulators.
template <int N, bool PAIR, bool SWAP, int SLOT, int BUF, bool DIGITS>
__device__ __forceinline__ void issue_slot(uint64_t b0, uint64_t d0, bool dbuf, uint32_t first, bool bounded,
                                           uint64_t* empty, uint32_t pair_mask) {
  using L = Layout<N, PAIR>;
  // x is e4m3 (0), the weights e5m2 (1)
  constexpr uint32_t idesc = (1u << 4) | ((SWAP ? 1u : 0u) << 7) | ((SWAP ? 0u : 1u) << 10) |
                             ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kRows * (PAIR ? 2 : 1) >> 4) << 24);
  constexpr uint32_t acc = BUF * 2 * N, a = kTmemSlots + 64 * SLOT;
#pragma unroll
  for (int j = 0; j < kSlotK / 2; ++j)
    tc::mma_f8_ts<PAIR>(acc, a + 8 * j, b0 + (uint64_t)((SLOT * L::slot_bytes >> 4) + 2 * j * L::NL), idesc,
                        j == 0 && !DIGITS ? first : 1u);
  if constexpr (DIGITS) {
    auto digit = [&](uint32_t ad, uint64_t dd) {
      tc::mma_f8_ts<PAIR>(acc + N, ad, dd, idesc, first);
      if (!bounded) {
        // x digits with the lo weights into L, x nibbles with the n3 weights into H
        constexpr uint64_t step = L::digit_bytes >> 4;
        tc::mma_f8_ts<PAIR>(acc, ad + (SWAP ? 8 : 0), dd + (SWAP ? 0 : step), idesc, 1u);
        tc::mma_f8_ts<PAIR>(acc + N, ad + (SWAP ? 16 : 8), dd + (SWAP ? step : 2 * step), idesc, 1u);
      }
    };
    if (dbuf)
      digit(kTmemDigits + 24, d0 + (uint64_t)(3 * L::digit_bytes >> 4));
    else
      digit(kTmemDigits, d0);
  }
  tc::commit<PAIR>(empty + SLOT, pair_mask);
}

// A segment's n chunks, from ring slot 2 pos mod 3 on (pos = chunks so far mod 3;
// the chunk loop is unrolled over the three positions, so that every slot is a
// constant).  ring: bit s is the parity of slot s's next use.
template <int N, bool PAIR, bool SWAP, int BUF>
__device__ __forceinline__ bool issue_segment(Bars* bars, uint64_t b0, uint64_t d0, int n, int& pos, uint32_t& ring,
                                              bool& dbuf, bool bounded, uint32_t pair_mask) {
  uint32_t first = 0;
  auto chunk = [&](auto p) {
    constexpr int S0 = 2 * decltype(p)::value % 3, S1 = (S0 + 1) % 3;
    if (!wait(&bars->full[S0], (ring >> S0) & 1u, bars)) return false;
    tc::fence_after();
    if (tc::elect_one()) issue_slot<N, PAIR, SWAP, S0, BUF, false>(b0, d0, dbuf, first, bounded, bars->empty, pair_mask);
    __syncwarp();
    if (!wait(&bars->full[S1], (ring >> S1) & 1u, bars)) return false;
    tc::fence_after();
    if (tc::elect_one()) issue_slot<N, PAIR, SWAP, S1, BUF, true>(b0, d0, dbuf, first, bounded, bars->empty, pair_mask);
    __syncwarp();
    ring ^= (1u << S0) | (1u << S1);
    dbuf = !dbuf;
    first = 1u;
    return true;
  };
  while (true) {
    if (pos == 0) {
      if (!chunk(std::integral_constant<int, 0>{})) return false;
      pos = 1;
      if (--n == 0) return true;
    }
    if (pos == 1) {
      if (!chunk(std::integral_constant<int, 1>{})) return false;
      pos = 2;
      if (--n == 0) return true;
    }
    if (!chunk(std::integral_constant<int, 2>{})) return false;
    pos = 0;
    if (--n == 0) return true;
  }
}

template <int N, bool PAIR, bool CONV, bool VEC, bool SWAP>
__global__ void __launch_bounds__(cta_threads(SWAP), 1) shift_mma_kernel(const __grid_constant__ MmaSet S) {
  using L = Layout<N, PAIR>;
  using Tiles = Walk<PAIR ? 2 : 1, SWAP, L::halves>;
  constexpr int NL = L::NL;            // columns whose weights this CTA decodes
  constexpr int kAccBufs = 128 / N;
  constexpr int kGroupSize = PAIR ? 2 : 1;
  constexpr int kBWarps = b_warps(SWAP), kBSlotWarps = SWAP ? 4 : 2;  // B warps in all and per slot
  constexpr int kThreads = cta_threads(SWAP), kMmaWarp = SWAP ? kFirstB : kFirstB + kBWarps;
  extern __shared__ __align__(1024) unsigned char smem[];
  Bars* bars = reinterpret_cast<Bars*>(smem);
  uint8_t* flags = smem + kFlagOff;
  unsigned char* lut = smem + kLutOff;
  int32_t* tables = reinterpret_cast<int32_t*>(smem + kTableOff);
  unsigned char* bslots = smem + L::base(S.table_entries, S.n);
  unsigned char* bdigits = bslots + kSlots * L::slot_bytes;
  unsigned char* accs = bdigits + 6 * L::digit_bytes;
  unsigned char* codes = accs + L::acc_bytes;
  unsigned char* xrows = codes + kCodeBytes;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int cta = PAIR ? (int)(blockIdx.x & 1) : 0;  // place in the pair: its rows of the tile
  const uint32_t crank = blockIdx.x % (uint32_t)(S.splits * kGroupSize);  // rank in the cluster
  const uint32_t leader = crank - (uint32_t)cta;
  const uint32_t pair_mask = 3u << leader;

  // ---- setup: barriers, tensor memory, tables, column-tile flags ----
  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s) {
      tc::mbar_init(&bars->full[s], kGroupSize * (4 + kBSlotWarps));
      tc::mbar_init(&bars->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&bars->acc_full[b], 1);
      tc::mbar_init(&bars->acc_empty[b], kGroupSize * kEpiWarps);
    }
    tc::mbar_init(&bars->done, 1);
    bars->abort = 0;
    bars->wait_cycles = S.wait_cycles;
    bars->amax = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) tc::tmem_alloc<PAIR>(&bars->tmem, kTmemCols);
  const bool have_amax = S.p[0].amax_in != nullptr;
  const uint32_t amax = have_amax ? *S.p[0].amax_in : 0x80000000u;
  const int digits = amax <= (1u << 20) ? 1 : (amax <= (1u << 24) ? 2 : (amax <= (1u << 28) ? 3 : 4));
  // A convolution's column flags and tables are made by different warps side by
  // side (its launches are many and short: 1-2 us of each); FC's by all warps.
  constexpr int kFlagWarps = CONV ? 12 : kThreads / 32, kTableWarp = CONV ? kFlagWarps : 0;
  if (warp < kFlagWarps) {
    for (int ph = 0; ph < S.n; ++ph) {
      const GemmParams& P = S.p[ph];
      for (int ct = warp; ct < S.info[ph].flag_tiles; ct += kFlagWarps) {
        bool wide = !have_amax || (P.flags & DS_FORCE_INT64), free = false;
        constexpr int kTileCols = SWAP ? kRows : N;
        for (int c = lane; c < kTileCols; c += 32) {
          const int64_t col = (int64_t)ct * kTileCols + c;
          if (col >= P.cols) continue;
          const unsigned long long A = reinterpret_cast<const unsigned long long*>(P.blob + P.off_cola)[col];
          const unsigned long long nnz = reinterpret_cast<const uint32_t*>(P.blob + P.off_nnz)[col];
          const unsigned long long b = P.bias ? (unsigned long long)uabs(P.bias[col]) : 0ull;
          // 2^31 * A and every product below stay inside 64 bits for A < 2^32; a larger A fails both bounds
          const bool huge = (A >> 32) != 0;
          wide |= huge || ((((unsigned long long)amax * A + 32767ull) >> 15) + nnz + b > (unsigned long long)INT32_MAX);
          const unsigned long long u = digits > 1 ? 16u : (amax + 65535u) >> 16;  // max |digit|
          free |= huge || 2 * A > (1ull << 24) || u * A > (1ull << 24);
        }
        const uint32_t f =
            (__any_sync(0xffffffffu, wide) ? 0u : kInt32) | (__any_sync(0xffffffffu, free) ? 0u : kBounded);
        if (lane == 0) flags[S.info[ph].flag_off + ct] = (uint8_t)f;
      }
    }
  }
  if (warp >= kTableWarp) {
    // weight bytes by code: row sh ^ 15 | negative << 4 | zero << 5, eight copies
    // of 16 bytes per row, so that 8 lanes reading any rows hit all banks once
    // (the second table leaves nibble 3 out for sh < 4, see above)
    for (int i = tid - 32 * kTableWarp; i < 2 * 64 * 8; i += kThreads - 32 * kTableWarp) {
      const int row = (i >> 3) & 63, sh = 15 - (row & 15);
      // byte q: the weight 2^(4q - sh) as e5m2
      uint32_t e = 0x04040404u * (uint32_t)(15 - sh) + 0x30201000u;
      if (row & 16) e |= 0x80808080u;
      if (i >= 512 && sh < 4) e &= 0x00FFFFFFu;
      if (row >= 32) e = 0u;
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int cut = 8 * ((sh - j + 3) >> 2);  // bits of the bytes q with 4q + j < sh
        w[j] = cut < 32 ? e & (~0u << cut) : 0u;
      }
      *reinterpret_cast<uint4*>(lut + i * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    if (CONV) {
      // taps of 16 consecutive reduction indices: element offsets, then kernel
      // row / column bits.  Copy c = 0..3 starts at tap c, so that 16-byte reads can
      // start anywhere; the last 32 entries are the taps of the reduction's partial
      // last slot, its missing ones (and 16 more) marked as never valid.
      for (int ph = 0; ph < S.n; ++ph) {
        const GemmParams& P = S.p[ph];
        const int rs = P.R * P.S, te = S.table_entries, tail = (int)(P.kred % kSlotK);
        const int t0 = (int)((P.kred - tail) % rs);
        for (int e = tid - 32 * kTableWarp; e < 4 * te + 32; e += kThreads - 32 * kTableWarp) {
          const bool in_tail = e >= 4 * te;
          const int i = in_tail ? t0 + e - 4 * te : e / te + e % te;
          const int c = i / rs, tap = i - c * rs, r = tap / P.S, q = tap - r * P.S;
          const bool never = in_tail && e - 4 * te >= tail;
          int32_t* t = tables + ph * 2 * (4 * te + 32) + e;
          t[0] = never ? 0 : c * P.H * P.W + r * P.W + q;
          t[4 * te + 32] = never ? INT32_MIN : (int32_t)((1u << r) | (0x10000u << q));
        }
      }
    }
  }
  tc::fence_before();
  if constexpr (PAIR)
    cg::this_cluster().sync();  // the peer's barriers exist before anything arrives there
  else
    __syncthreads();
  tc::fence_after();
  constexpr uint32_t tmem = 0;  // all 512 columns are this CTA's, so they start at column 0
  // Arrivals at the barriers of the CTA that issues the tensor operations.  From the
  // other CTA of a pair they publish writes to that CTA's own shared and tensor memory,
  // which no thread of the issuing CTA reads: each SM's tensor unit reads its own
  // CTA's operands, and before its arrival a warp has waited for its tensor-memory
  // stores and fenced its shared-memory writes for the asynchronous proxy.  So the
  // instruction's default ordering (release at CTA scope) is left as it is; release
  // at cluster scope measured 830-1190 clocks an arrival instead of 5-15, FC of 4096 rows
  // 1766 us instead of 1150.
  auto arrive = [&](uint64_t* bar) {
    if constexpr (PAIR)
      tc::mbar_arrive_cluster(tc::map_rank(tc::smem_u32(bar), leader));
    else
      tc::mbar_arrive(bar);
  };

  int* ws = reinterpret_cast<int*>(smem + kWalkOff) + warp * Tiles::kWords;
  static_assert(kWalkOff + kThreads / 32 * Tiles::kWords * 4 <= kBiasOff, "one place per warp");
  const bool split = S.splits > 1;
  // a split tile of 64-bit sums goes in two passes where a walk sums half of the columns
  int n_pass = 1;
  if (L::halves && split) {
    Tiles w(S, flags, digits, 0);
    w.start_tile();
    n_pass = (w.fl & kInt32) ? 1 : 2;
  }
  // ring position (A, B, tensor operations) and accumulator position (tensor operations, epilogue)
  int slot = 0, seg_no = 0;
  uint32_t ring = 0, it = 0;  // parity of the slot's use, slots so far

  for (int pass = 0; pass < n_pass; ++pass) {
    if (SWAP && warp < kFirstEpi) {
      // ---- operand A, swapped roles: a lane is a weight column, its codes decoded into tensor memory ----
      const int q = warp & 3;
      slot = warp >> 2;
      if (pass == 0) it = (uint32_t)slot;
      const uint32_t a0 = tmem + ((uint32_t)(32 * q) << 16) + kTmemSlots + 64 * slot;
      const uint32_t d0 = tmem + ((uint32_t)(32 * q) << 16) + kTmemDigits;
      const uint32_t lut_a = tc::smem_u32(lut) + (lane & 7) * 16;
      uint4* cells = reinterpret_cast<uint4*>(xrows) + tid;  // kCodeAhead slots: 16 codes, sign and non-zero plane
      uint32_t issued = 0, used = 0, modes = 0;              // modes: bounded flags of the slots in flight
      int rem = 0, half = 0;
      uint32_t bounded = 0, in = 0;
      int64_t cols = 0;
      const unsigned char *nsrc = nullptr, *bsrc = nullptr;
      auto seek = [&](bool first, int n) {
        Tiles v(S, flags, digits, L::halves && split ? pass : -1);
        bool more = true;
        if (first) {
          v.start_tile();
          n -= pass * 2 * (v.ce - v.cb) * digits;  // the slots of the earlier passes
        } else {
          v.restore(ws);
          more = next_segment_or_tile(v);
        }
        while (more && n >= 2 * (v.c_end - v.chunk)) {
          n -= 2 * (v.c_end - v.chunk);
          more = next_segment_or_tile(v);
        }
        v.save(ws);
        if (!more) return false;
        const GemmParams& P = v.P();
        const int64_t c = (int64_t)v.rt * kRows + 32 * q + lane;
        cols = P.cols;
        in = c < cols;
        bounded = (v.fl & kBounded) ? 1u : 0u;
        rem = 2 * (v.c_end - v.chunk) - n;
        half = n & 1;
        const int64_t rec = (int64_t)(v.chunk + (n >> 1)) * cols + (in ? c : 0);
        nsrc = P.blob + P.off_nib + rec * 16;
        bsrc = P.blob + P.off_bits + rec * 8;
        return true;
      };
      bool more = seek(true, (int)it);
      auto issue = [&]() {
        if (more) {
          uint4* cell = cells + (issued % kCodeAhead) * 32 * kAWarps;
          cp_async8(cell, in ? nsrc + 8 * half : S.p[0].blob, in);
          cp_async8(reinterpret_cast<unsigned char*>(cell) + 8, in ? bsrc : S.p[0].blob, in);
          const uint32_t m = 1u << (issued % kCodeAhead), hm = m << 8;
          modes = (modes & ~(m | hm)) | (bounded ? m : 0u) | (half ? hm : 0u);
          ++issued;
          rem -= kAGroups;
          if (rem > 0) {
            half += kAGroups;
            nsrc += (half >> 1) * cols * 16;
            bsrc += (half >> 1) * cols * 8;
            half &= 1;
          } else {
            more = seek(false, -rem);
          }
        }
        cp_async_commit();
      };
#pragma unroll 1
      for (int i = 0; i < kCodeAhead - 1; ++i) issue();
      for (;;) {
        issue();
        if (used == issued) break;
        cp_async_wait<kCodeAhead - 1>();
        const uint4 cell = cells[(used % kCodeAhead) * 32 * kAWarps];
        const bool bnd = (modes >> (used % kCodeAhead)) & 1u;
        const int h = (modes >> (8 + used % kCodeAhead)) & 1u;
        ++used;
        const uint32_t la = lut_a + (bnd ? 0 : kLutBytes);
        const uint32_t sp = cell.z >> (16 * h), zp = ~cell.w >> (16 * h);
        const uint32_t ad = d0 + 12 * (it & 2) + 4 * h;
        if (!wait(&bars->empty[slot], ring ^ 1u, bars)) break;
        tc::fence_after();
#pragma unroll
        for (int w8 = 0; w8 < 2; ++w8) {
          const uint32_t nib = w8 ? cell.y : cell.x, sb = sp >> (8 * w8), zb = zp >> (8 * w8);
          const uint32_t ne = ~nib & 0x0F0F0F0Fu, no = ~(nib >> 4) & 0x0F0F0F0Fu;
          const uint32_t se = spread(sb), so = spread(sb >> 1), ze = spread(zb), zo = spread(zb >> 1);
          const uint32_t ie = ne | (se >> 3) | (ze >> 2), io = no | (so >> 3) | (zo >> 2);
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            uint32_t e[16];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint32_t row = __byte_perm((i & 1) ? io : ie, 0, 0x4440 + 2 * p + (i >> 1));
              asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                           : "=r"(e[4 * i]), "=r"(e[4 * i + 1]), "=r"(e[4 * i + 2]), "=r"(e[4 * i + 3])
                           : "r"(la + row * 128));
            }
            tc::st16(a0 + 32 * w8 + 16 * p, e);
          }
          uint32_t hi[2], lo[2], n3[2];
          digit_weights(ne, se, ze, bnd, hi[0], lo[0], n3[0]);
          digit_weights(no, so, zo, bnd, hi[1], lo[1], n3[1]);
          tc::st2(ad + 2 * w8, hi[0], hi[1]);
          if (!bnd) {
            tc::st2(ad + 8 + 2 * w8, lo[0], lo[1]);
            tc::st2(ad + 16 + 2 * w8, n3[0], n3[1]);
          }
        }
        tc::wait_st();
        tc::fence_before();
        __syncwarp();
        if (lane == 0) arrive(&bars->full[slot]);
        it += kAGroups;
        ring ^= 1u;
      }
    } else if (warp < kFirstEpi) {
      // ---- operand A: group g fills ring slot g: slots it = g, g + 3, ... of the CTA's sequence, two per chunk ----
      const int q = warp & 3;
      slot = warp >> 2;
      if (pass == 0) it = (uint32_t)slot;
      const uint32_t a0 = tmem + ((uint32_t)(32 * q) << 16) + kTmemSlots + 64 * slot;
      const uint32_t d0 = tmem + ((uint32_t)(32 * q) << 16) + kTmemDigits;
      int32_t* xbuf = reinterpret_cast<int32_t*>(xrows) + warp * 2 * 32 * kXStride;
      uint32_t x[CONV ? kSlotK : kSlotK / 2];
      // the position of the next load, kept up to date slot by slot
      int rem = 0;          // slots from there to the end of its segment
      uint32_t mode = 0;    // bit 0: bounded tile; bits 1..: digit
      const int32_t* src = nullptr;
      uint32_t nm = 0xffffffffu;          // FC: rows present
      int left = 0;                       // reduction indices from there on
      int t0 = 0, rs = 1, step_taps = 0;  // conv: tap, taps, taps and elements to the next slot
      int step = 0, chan_step = 0;
      const int32_t* tab = nullptr;
      // Moves n slots on, into later segments; false past the end of the sequence.
      auto seek = [&](bool first, int n) {
        Tiles v(S, flags, digits, L::halves && split ? pass : -1);
        bool more = true;
        if (first) {
          v.start_tile();
          n -= pass * 2 * (v.ce - v.cb) * digits;  // the slots of the earlier passes
        } else {
          v.restore(ws);
          more = next_segment_or_tile(v);
        }
        while (more && n >= 2 * (v.c_end - v.chunk)) {
          n -= 2 * (v.c_end - v.chunk);
          more = next_segment_or_tile(v);
        }
        v.save(ws);
        if (!more) return false;
        const GemmParams& P = v.P();
        const int64_t row0 = (int64_t)v.rt * (kRows * kGroupSize) + 128 * cta + 32 * q;
        const int64_t k0 = (int64_t)v.chunk * kChunk + n * kSlotK;
        rem = 2 * (v.c_end - v.chunk) - n;
        mode = ((v.fl & kBounded) ? 1u : 0u) | ((uint32_t)v.d << 1);
        left = (int)(P.kred - k0);
        if constexpr (CONV) {
          const RowPlace rp = row_place<true>(P, S.info[v.ph], row0 + lane);
          nm = rp.nm | 0x80000000u;  // kernel column 15 does not exist: the bit of the taps that are never valid
          rs = P.R * P.S;
          chan_step = P.H * P.W;
          step_taps = kAGroups * kSlotK % rs;
          step = kAGroups * kSlotK / rs * chan_step;
          const int c0 = (int)(k0 / rs);
          t0 = (int)k0 - c0 * rs;
          src = P.x + rp.x0 + (int64_t)c0 * chan_step;
          tab = tables + v.ph * 2 * (4 * S.table_entries + 32);
        } else {
          const int r = VEC ? lane >> 2 : 4 * (lane >> 4), kk = VEC ? 4 * (lane & 3) : (lane & 15);
          src = P.x + (row0 + r) * P.kred + k0 + kk;
          left -= kk;
          nm = 0;
#pragma unroll
          for (int i = 0; i < (VEC ? 4 : 16); ++i)
            if (row0 + r + (VEC ? 8 * i : (i & 3) + 8 * (i >> 2)) < P.rows) nm |= 1u << i;
        }
        return true;
      };
      // conv: loads the 16 values of the slot at the current position
      auto load = [&]() {
        const int te = S.table_entries;
        const int4* tb = reinterpret_cast<const int4*>(tab + (left >= kSlotK ? (t0 & 3) * te + (t0 & ~3)
                                                                             : 4 * te + (left > 0 ? 0 : kSlotK)));
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int4 o = tb[h], m = tb[te + 8 + h];
          x[4 * h] = load_tap(src, o.x, m.x, nm);
          x[4 * h + 1] = load_tap(src, o.y, m.y, nm);
          x[4 * h + 2] = load_tap(src, o.z, m.z, nm);
          x[4 * h + 3] = load_tap(src, o.w, m.w, nm);
        }
      };
      // FC: starts the copy of the warp's 32 rows x 16 values, row by row, to the warp's own buffer
      auto stage = [&](int buf) {
        int32_t* dst = xbuf + buf * 32 * kXStride;
        const int64_t row_step = S.p[0].kred;
        if constexpr (VEC) {
          dst += (lane >> 2) * kXStride + 4 * (lane & 3);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const bool ok = left > 0 && ((nm >> i) & 1u);
            cp_async16(dst + 8 * i * kXStride, ok ? src + 8 * i * row_step : S.p[0].x, ok);
          }
        } else {
          dst += 4 * (lane >> 4) * kXStride + (lane & 15);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int r = (i & 3) + 8 * (i >> 2);
            const bool ok = left > 0 && ((nm >> i) & 1u);
            cp_async4(dst + r * kXStride, ok ? src + r * row_step : S.p[0].x, ok);
          }
        }
        cp_async_commit();
      };
      bool more = seek(true, (int)it);
      if (more) {
        if constexpr (CONV) {
          load();
        } else {
          stage(0);
        }
      }
      int buf = 0;
      while (more) {
        const uint32_t now = mode;
        rem -= kAGroups;
        if (rem > 0) {
          left -= kAGroups * kSlotK;
          if constexpr (CONV) {
            t0 += step_taps;
            src += step;
            if (t0 >= rs) {
              t0 -= rs;
              src += chan_step;
            }
          } else {
            src += kAGroups * kSlotK;
          }
        } else {
          more = seek(false, -rem);
        }
        if constexpr (!CONV) {
          if (more) {
            stage(buf ^ 1);
            cp_async_wait<1>();
          } else {
            cp_async_wait<0>();
          }
          __syncwarp();
        }
        if (!wait(&bars->empty[slot], ring ^ 1u, bars)) break;
        tc::fence_after();
        const uint32_t ad = d0 + 12 * (it & 2) + 4 * (it & 1);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t* v = CONV ? x + 8 * hf : x;
          if constexpr (!CONV) {
            const int4* sx = reinterpret_cast<const int4*>(xbuf + buf * 32 * kXStride + lane * kXStride) + 2 * hf;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int4 t = sx[i];
              v[4 * i] = t.x;
              v[4 * i + 1] = t.y;
              v[4 * i + 2] = t.z;
              v[4 * i + 3] = t.w;
            }
          }
          if (__builtin_expect(digits > 1, 0)) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = pick_digit(v[i], (int)(now >> 1), digits);
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t e[16];
#pragma unroll
            for (int i = 0; i < 4; ++i) expand_x(v[4 * h + i], e + 4 * i);
            tc::st16(a0 + 32 * hf + 16 * h, e);
          }
          // even and odd values in separate words, as the weights' digits
          tc::st2(ad + 2 * hf, digit4(v[0], v[2], v[4], v[6]), digit4(v[1], v[3], v[5], v[7]));
          if (!(now & 1u)) tc::st2(ad + 8 + 2 * hf, nibble4(v[0], v[2], v[4], v[6]), nibble4(v[1], v[3], v[5], v[7]));
        }
        tc::wait_st();
        tc::fence_before();
        __syncwarp();  // (FC: the staging buffer has been read, too)
        if (lane == 0) arrive(&bars->full[slot]);
        if constexpr (CONV) {
          if (more) load();  // of the next slot, in flight until the ring gives one back
        }
        it += kAGroups;
        ring ^= 1u;
        buf ^= 1;
      }
    } else if (warp < kFirstB) {
      // ---- epilogue: accumulators to integer sums in shared memory (which frees them for the next
      // segment), then from there, after the tile's last segment, to the output ----
      Tiles w(S, flags, digits, L::halves && split ? pass : -1);
      w.start_tile();
      const int q = warp & 3, rowl = 32 * q + lane;
      int32_t* bias = reinterpret_cast<int32_t*>(smem + kBiasOff) + q * N;  // this warp's copy of the tile's biases
      uint32_t* acc32 = reinterpret_cast<uint32_t*>(accs) + rowl;
      long long* acc64 = reinterpret_cast<long long*>(accs) + rowl;
      bool more = true;
      while (more) {
        const GemmParams& P = w.P();
        const bool i32 = (w.fl & kInt32) != 0, first = w.first_segment();
        // split tiles' sums, and a convolution's last ones, are left to all of the CTA's warps
        const bool out = w.last_segment() && !split && !(CONV && w.at_end());
        const int c_lo = !L::halves || i32 ? 0 : w.half * (N / 2), c_hi = !L::halves || i32 ? N : c_lo + N / 2;
        const int b = seg_no % kAccBufs, sh = 4 * w.d;
        const uint32_t acc = tmem + ((uint32_t)(32 * q) << 16) + b * 2 * N;
        // H holds 2^-17 of the digit sums, multiples of 2 (bounded tiles) or of 2^9
        const int hshift = (w.fl & kBounded) ? 1 : 9;
        const float hscale = (w.fl & kBounded) ? 65536.f : 256.f;
        const int64_t col0 = (int64_t)w.ct * N;
        if (!SWAP && out) {
          for (int c = lane; c < N; c += 32)
            bias[c] = P.bias != nullptr && col0 + c < P.cols ? __ldg(P.bias + col0 + c) : 0;
          __syncwarp();
        }
        if (!wait(&bars->acc_full[b], (uint32_t)(seg_no / kAccBufs) & 1u, bars)) break;
        tc::fence_after();
        for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
          uint32_t rl[16], rh[16];
          tc::ld16(acc + c0, rl);
          tc::ld16(acc + N + c0, rh);
          tc::wait_ld(rl, rh);
          if (i32) {
            uint32_t* a = acc32 + c0 * kAccStride;
#pragma unroll
            for (int j = 0; j < 16; ++j)
              rl[j] = (uint32_t)__float2int_rn(__uint_as_float(rl[j]) * 512.f) +
                      ((uint32_t)__float2int_rn(__uint_as_float(rh[j]) * hscale) << hshift);
            if (__builtin_expect(!first || sh != 0, 0)) {
#pragma unroll
              for (int j = 0; j < 16; ++j) rl[j] = (rl[j] << sh) + (first ? 0u : a[j * kAccStride]);
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) a[j * kAccStride] = rl[j];
          } else {
            long long* a = acc64 + (c0 - c_lo) * kAccStride;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int lo = __float2int_rn(__uint_as_float(rl[j]) * 512.f);
              const int hi = __float2int_rn(__uint_as_float(rh[j]) * hscale);
              const long long v = ((long long)lo + (long long)hi * (1ll << hshift)) * (1ll << sh);
              a[j * kAccStride] = first ? v : a[j * kAccStride] + v;
            }
          }
        }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) arrive(&bars->acc_empty[b]);
        if (out) {
          uint32_t amax_local = 0;
          const bool relu = (P.flags & DS_RELU) != 0;
          const int64_t row0 = (int64_t)w.rt * (kRows * kGroupSize) + 128 * cta + 32 * q;
          const int nc = (int)min((int64_t)(c_hi - c_lo), P.cols - col0 - c_lo);  // columns of this half that exist
          if constexpr (SWAP) {
            // lanes along the columns already; the tile's N sums of a lane are rows
            const int64_t col = (int64_t)w.rt * kRows + rowl, r0 = (int64_t)w.ct * N + c_lo;
            const int nr = (int)min((int64_t)(c_hi - c_lo), P.rows - r0);
            if (col < P.cols) {
              const int32_t bc = P.bias != nullptr ? __ldg(P.bias + col) : 0;
              int32_t* y = P.y + r0 * P.cols + col;
              for (int r = 0; r < nr; ++r) {
                int32_t o = i32 ? (int32_t)(acc32[(c_lo + r) * kAccStride] + (uint32_t)bc)
                                : sat32(acc64[r * kAccStride] + bc);
                if (relu) o = max(o, 0);
                amax_local = max(amax_local, uabs(o));
                y[r * P.cols] = o;
              }
            }
          } else if constexpr (CONV) {
            // lanes along the rows (pixels)
            const RowPlace rp = row_place<true>(P, S.info[w.ph], row0 + lane);
            if (rp.ok) {
              const int64_t cs = col_stride<true>(P);
              const int64_t idx = rp.y0 + (col0 + c_lo) * cs;
              int32_t* y = P.y + idx;
              const bool resid = (P.flags & DS_RESIDUAL) != 0, want_max = P.amax_out != nullptr;
              const int32_t floor_v = relu ? 0 : INT32_MIN;
              int c0 = 0;
              if (i32) {
                const int32_t* rs = P.residual + idx;
                const uint32_t* a = acc32 + c_lo * kAccStride;
                for (; c0 + 8 <= nc; c0 += 8) {
                  int32_t o[8], res[8];
                  if (resid) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) res[j] = __ldg(rs + j * cs);
                    rs += 8 * cs;
                  }
                  const int4 b0 = *reinterpret_cast<const int4*>(bias + c_lo + c0);
                  const int4 b1 = *reinterpret_cast<const int4*>(bias + c_lo + c0 + 4);
                  const int32_t bj[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                  for (int j = 0; j < 8; ++j) o[j] = (int32_t)(a[j * kAccStride] + (uint32_t)bj[j]);
                  a += 8 * kAccStride;
                  if (resid) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) o[j] = add_sat(o[j], res[j]);
                  }
#pragma unroll
                  for (int j = 0; j < 8; ++j) {
                    o[j] = max(o[j], floor_v);
                    y[j * cs] = o[j];
                  }
                  y += 8 * cs;
                  if (want_max) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) amax_local = max(amax_local, uabs(o[j]));
                  }
                }
              }
              for (; c0 < nc; ++c0) {  // the columns' remainder, and 64-bit sums
                int32_t o = i32 ? (int32_t)(acc32[(c_lo + c0) * kAccStride] + (uint32_t)bias[c_lo + c0])
                                : sat32(acc64[c0 * kAccStride] + bias[c_lo + c0]);
                if (resid) o = add_sat(o, __ldg(P.residual + idx + c0 * cs));
                o = max(o, floor_v);
                amax_local = max(amax_local, uabs(o));
                *y = o;
                y += cs;
              }
            }
          } else {
            // lanes along the columns
            __syncwarp();  // the other lanes' sums
            const int nr = (int)min((int64_t)32, P.rows - row0);
            for (int c0 = 0; c0 < nc; c0 += 32) {
              const int c = c0 + lane;
              if (c >= nc) continue;
              const int32_t bc = bias[c_lo + c];
              int32_t* y = P.y + row0 * P.cols + col0 + c_lo + c;
#pragma unroll 4
              for (int r = 0; r < nr; ++r) {
                int32_t o = i32 ? (int32_t)((acc32 - lane)[(c_lo + c) * kAccStride + r] + (uint32_t)bc)
                                : sat32((acc64 - lane)[c * kAccStride + r] + bc);
                if (relu) o = max(o, 0);
                amax_local = max(amax_local, uabs(o));
                y[r * P.cols] = o;
              }
            }
          }
          __syncwarp();
          if (P.amax_out != nullptr) {
            amax_local = __reduce_max_sync(0xffffffffu, amax_local);
            if (lane == 0 && amax_local) atomicMax(P.amax_out, amax_local);
          }
        }
        ++seg_no;
        more = next_segment_or_tile(w);
      }
    } else if (SWAP && swapped_b_warp(warp) < kBWarps) {
      // ---- operand B, swapped roles: two groups of four warps; a thread expands 8 values of one row of x ----
      const int bwarp = swapped_b_warp(warp), tb = bwarp % kBSlotWarps * 32 + lane, g = bwarp / kBSlotWarps;
      const int n = tb % N, kw = tb / N;  // row of the tile, which 8 of the slot's 16 indices
      static_assert(!SWAP || N == 64, "128 threads: 64 rows x 16 indices");
      const uint32_t dst0 = tc::smem_u32(bslots) + n * 16 + kw * 8 * N * 16;
      const uint32_t dig0 = tc::smem_u32(bdigits) + n * 16 + kw * 8 + g * N * 16;
      if (pass == 0) {
        it = (uint32_t)g;
        slot = g;
      }
      // kCodeAhead slots of 8 values, in flight to this thread's own words
      int4* cells = reinterpret_cast<int4*>(xrows + kCodeAhead * kAWarps * 32 * 16) + (bwarp * 32 + lane);
      uint32_t issued = 0, used = 0, modes = 0;  // modes: a byte per slot in flight: bounded flag, digit
      int rem = 0, left = 0;
      uint32_t mode = 0;
      const int32_t* src = nullptr;
      bool in = false;
      auto seek = [&](bool first, int m) {
        Tiles v(S, flags, digits, L::halves && split ? pass : -1);
        bool more = true;
        if (first) {
          v.start_tile();
          m -= pass * 2 * (v.ce - v.cb) * digits;  // the slots of the earlier passes
        } else {
          v.restore(ws);
          more = next_segment_or_tile(v);
        }
        while (more && m >= 2 * (v.c_end - v.chunk)) {
          m -= 2 * (v.c_end - v.chunk);
          more = next_segment_or_tile(v);
        }
        v.save(ws);
        if (!more) return false;
        const GemmParams& P = v.P();
        const int64_t row = (int64_t)v.ct * N + n, k0 = (int64_t)v.chunk * kChunk + m * kSlotK + 8 * kw;
        in = row < P.rows;
        src = P.x + (in ? row : 0) * P.kred + k0;
        left = (int)(P.kred - k0);
        rem = 2 * (v.c_end - v.chunk) - m;
        mode = ((v.fl & kBounded) ? 1u : 0u) | ((uint32_t)v.d << 1);
        return true;
      };
      bool more = seek(true, (int)it);
      auto issue = [&]() {
        if (more) {
          int4* cell = cells + (issued % kCodeAhead) * 64 * kBWarps;  // two halves of 4 values, 32 kBWarps apart
          if constexpr (VEC) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const bool ok = in && 4 * i < left;
              cp_async16(cell + i * 32 * kBWarps, ok ? src + 4 * i : S.p[0].x, ok);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const bool ok = in && i < left;
              cp_async4(reinterpret_cast<int32_t*>(cell + (i >> 2) * 32 * kBWarps) + (i & 3), ok ? src + i : S.p[0].x, ok);
            }
          }
          const int at = 8 * (int)(issued % kCodeAhead);
          modes = (modes & ~(0xFFu << at)) | (mode << at);
          ++issued;
          rem -= 2;
          if (rem > 0) {
            src += kChunk;
            left -= kChunk;
          } else {
            more = seek(false, -rem);
          }
        }
        cp_async_commit();
      };
#pragma unroll 1
      for (int i = 0; i < kCodeAhead - 1; ++i) issue();
      for (;;) {
        issue();
        if (used == issued) break;
        cp_async_wait<kCodeAhead - 1>();
        const int4* cell = cells + (used % kCodeAhead) * 64 * kBWarps;
        const int4 v0 = cell[0], v1 = cell[32 * kBWarps];
        const uint32_t now = (modes >> (8 * (used % kCodeAhead))) & 0xFFu;
        ++used;
        uint32_t v[8] = {(uint32_t)v0.x, (uint32_t)v0.y, (uint32_t)v0.z, (uint32_t)v0.w,
                         (uint32_t)v1.x, (uint32_t)v1.y, (uint32_t)v1.z, (uint32_t)v1.w};
        if (__builtin_expect(digits > 1, 0)) {
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = pick_digit(v[i], (int)(now >> 1), digits);
        }
        if (!wait(&bars->empty[slot], ring ^ 1u, bars)) break;
        const uint32_t dst = dst0 + slot * L::slot_bytes;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          uint32_t e[4];
          expand_x(v[i], e);
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + i * N * 16), "r"(e[0]), "r"(e[1]),
                       "r"(e[2]), "r"(e[3])
                       : "memory");
        }
        // [buffer][digits, nibbles 3][16-index half][row][16 bytes]
        const uint32_t dd = dig0 + ((it >> 1) & 1) * 3 * L::digit_bytes;
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dd), "r"(digit4(v[0], v[2], v[4], v[6])),
                     "r"(digit4(v[1], v[3], v[5], v[7]))
                     : "memory");
        if (!(now & 1u))
          asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dd + L::digit_bytes), "r"(nibble4(v[0], v[2], v[4], v[6])),
                       "r"(nibble4(v[1], v[3], v[5], v[7]))
                       : "memory");
        tc::fence_smem_async();
        __syncwarp();
        if (lane == 0) arrive(&bars->full[slot]);
        it += 2;
        slot += 2;
        if (slot >= kSlots) {
          slot -= kSlots;
          ring ^= 1u;
        }
      }
    } else if (!SWAP && warp < kMmaWarp) {
      // ---- operand B: three groups of two warps, group g fills ring slot g; a thread decodes 16 codes of one
      // column (NL = 64) or 8 of them (NL = 32) ----
      constexpr int kWords = NL / 32;  // code words of 8 indices
      const int bwarp = warp - kFirstB, tb = (bwarp & 1) * 32 + lane;
      slot = bwarp >> 1;
      if (pass == 0) it = (uint32_t)slot;
      const int col = tb % NL, kw = tb / NL;  // kw: which 8 of the slot's 16 indices (NL = 32)
      const uint32_t lut_a = tc::smem_u32(lut) + (lane & 7) * 16;
      const uint32_t dst0 = tc::smem_u32(bslots) + slot * L::slot_bytes + col * 16 + kw * 8 * NL * 16;
      const uint32_t dig0 = tc::smem_u32(bdigits) + col * 16 + kw * 8;
      // The codes arrive kCodeAhead slots of the group ahead, in a ring of this
      // thread's own words: 16 or 8 codes, sign and non-zero plane.
      uint4* cells = reinterpret_cast<uint4*>(codes) + bwarp * 32 + lane;
      uint32_t issued = 0, used = 0, modes = 0;  // modes, per slot in flight: bounded flag, half of the chunk
      int rem = 0, half = 0;                     // the next load, as in operand A's warps
      uint32_t bounded = 0, in = 0;
      int64_t cols = 0;
      const unsigned char *nsrc = nullptr, *bsrc = nullptr;
      auto seek = [&](bool first, int n) {
        Tiles v(S, flags, digits, L::halves && split ? pass : -1);
        bool more = true;
        if (first) {
          v.start_tile();
          n -= pass * 2 * (v.ce - v.cb) * digits;  // the slots of the earlier passes
        } else {
          v.restore(ws);
          more = next_segment_or_tile(v);
        }
        while (more && n >= 2 * (v.c_end - v.chunk)) {
          n -= 2 * (v.c_end - v.chunk);
          more = next_segment_or_tile(v);
        }
        v.save(ws);
        if (!more) return false;
        const GemmParams& P = v.P();
        const int64_t c = (int64_t)v.ct * N + cta * NL + col;
        cols = P.cols;
        in = c < cols;
        bounded = (v.fl & kBounded) ? 1u : 0u;
        rem = 2 * (v.c_end - v.chunk) - n;
        half = n & 1;
        const int64_t rec = (int64_t)(v.chunk + (n >> 1)) * cols + (in ? c : 0);
        nsrc = P.blob + P.off_nib + rec * 16 + 4 * kw;
        bsrc = P.blob + P.off_bits + rec * 8;
        return true;
      };
      bool more = seek(true, (int)it);
      auto issue = [&]() {
        if (more) {
          unsigned char* cell = reinterpret_cast<unsigned char*>(cells + (issued % kCodeAhead) * 32 * kBWarps);
          if constexpr (kWords == 2)
            cp_async8(cell, in ? nsrc + 8 * half : S.p[0].blob, in);
          else
            cp_async4(cell, in ? nsrc + 8 * half : S.p[0].blob, in);
          cp_async8(cell + 8, in ? bsrc : S.p[0].blob, in);
          const uint32_t m = 1u << (issued % kCodeAhead), hm = m << 8;
          modes = (modes & ~(m | hm)) | (bounded ? m : 0u) | (half ? hm : 0u);
          ++issued;
          rem -= kSlots;
          if (rem > 0) {
            half += kSlots;
            nsrc += (half >> 1) * cols * 16;
            bsrc += (half >> 1) * cols * 8;
            half &= 1;
          } else {
            more = seek(false, -rem);
          }
        }
        cp_async_commit();
      };
#pragma unroll 1
      for (int i = 0; i < kCodeAhead - 1; ++i) issue();
      for (;;) {
        issue();  // into the cell read in the previous turn
        if (used == issued) break;
        cp_async_wait<kCodeAhead - 1>();
        const uint4 cell = cells[(used % kCodeAhead) * 32 * kBWarps];
        const bool bnd = (modes >> (used % kCodeAhead)) & 1u;
        const int h = (modes >> (8 + used % kCodeAhead)) & 1u;
        ++used;
        const uint32_t la = lut_a + (bnd ? 0 : kLutBytes);
        // digit weights: [buffer][hi, lo, n3][16-index half][column][16 bytes]
        const uint32_t dd = dig0 + ((it >> 1) & 1) * 3 * L::digit_bytes + h * NL * 16;
        if (!wait(&bars->empty[slot], ring ^ 1u, bars)) break;
#pragma unroll
        for (int w8 = 0; w8 < kWords; ++w8) {
          const uint32_t nib = w8 ? cell.y : cell.x, b = (uint32_t)(16 * h + 8 * (kw + w8));
          const uint32_t sb = cell.z >> b, zb = ~cell.w >> b;
          const uint32_t ne = ~nib & 0x0F0F0F0Fu, no = ~(nib >> 4) & 0x0F0F0F0Fu;
          const uint32_t se = spread(sb), so = spread(sb >> 1), ze = spread(zb), zo = spread(zb >> 1);
          const uint32_t dst = dst0 + w8 * 8 * NL * 16;
          decode4<2 * NL * 16>(ne, se, ze, la, dst);
          decode4<2 * NL * 16>(no, so, zo, la, dst + NL * 16);
          uint32_t hi[2], lo[2], n3[2];
          digit_weights(ne, se, ze, bnd, hi[0], lo[0], n3[0]);
          digit_weights(no, so, zo, bnd, hi[1], lo[1], n3[1]);
          asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dd + 8 * w8), "r"(hi[0]), "r"(hi[1]) : "memory");
          if (!bnd) {
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dd + 8 * w8 + L::digit_bytes), "r"(lo[0]), "r"(lo[1])
                         : "memory");
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dd + 8 * w8 + 2 * L::digit_bytes), "r"(n3[0]), "r"(n3[1])
                         : "memory");
          }
        }
        tc::fence_smem_async();
        __syncwarp();
        if (lane == 0) arrive(&bars->full[slot]);
        it += kSlots;
        ring ^= 1u;
      }
    } else if (warp == kMmaWarp && cta == 0) {
      // ---- tensor operations (slot: chunks so far mod 3; it: digit buffer; ring: a bit per slot) ----
      Tiles w(S, flags, digits, L::halves && split ? pass : -1);
      w.start_tile();
      const uint64_t b0 = tc::plain_desc(tc::smem_u32(bslots), NL * 16, 128);
      const uint64_t d0 = tc::plain_desc(tc::smem_u32(bdigits), NL * 16, 128);
      bool more = true, dbuf = it != 0;
      while (more) {
        const int b = seg_no % kAccBufs, n = w.c_end - w.chunk;
        const bool bounded = (w.fl & kBounded) != 0;
        if (!wait(&bars->acc_empty[b], ((uint32_t)(seg_no / kAccBufs) & 1u) ^ 1u, bars)) break;
        tc::fence_after();
        const bool ok = kAccBufs == 1 || b == 0
                            ? issue_segment<N, PAIR, SWAP, 0>(bars, b0, d0, n, slot, ring, dbuf, bounded, pair_mask)
                            : issue_segment<N, PAIR, SWAP, kAccBufs - 1>(bars, b0, d0, n, slot, ring, dbuf, bounded, pair_mask);
        if (!ok) break;
        if (tc::elect_one()) tc::commit<PAIR>(&bars->acc_full[b], pair_mask);
        __syncwarp();
        ++seg_no;
        more = next_segment_or_tile(w);
      }
      it = dbuf;
    }

    // The sums left in shared memory (a split tile's partial sums, one set per
    // rank of the cluster, or a convolution's last tile of the CTA): all warps
    // finish them, each rank its share of the columns.
    cg::cluster_group cl = cg::this_cluster();
    cp_async_wait_all();  // none is in flight, unless this thread's role gave up
    tc::fence_before();
    if (split)
      cl.sync();
    else
      __syncthreads();
    tc::fence_after();
    // A CTA that gave up has not made all of its sums: none of the CTAs whose sums
    // meet then writes outputs from them, and no further pass runs (the places of its
    // roles are lost).  Without a split the sums are the CTA's own, and its epilogue
    // gave up if some are missing; the other CTA of the pair is looked at all the same.
    int gone = 0;
    if (CONV || split)
      gone = tc::ld_rank(tc::smem_u32(&bars->abort), min((uint32_t)lane, (uint32_t)(S.splits * kGroupSize - 1)));
    const bool gave_up = __any_sync(0xffffffffu, gone != 0);
    if ((CONV || split) && !gave_up) {
      Tiles v(S, flags, digits, L::halves && split ? pass : -1);
      while (v.t + v.t_step < v.n_tiles) v.t += v.t_step;
      v.start_tile();
      const GemmParams& P = v.P();
      const bool i32 = (v.fl & kInt32) != 0;
      const int per = (!L::halves || i32 ? N : N / 2) / S.splits, c_first = v.rank * per;
      // the tile's accumulator columns are output columns, or rows with swapped roles
      const int64_t col0 = (int64_t)v.ct * N + (!L::halves || i32 ? 0 : (split ? pass : 1) * (N / 2)) + c_first;
      const int64_t row0 = (int64_t)v.rt * (kRows * kGroupSize) + 128 * cta;
      const int nc = (int)min((int64_t)per, (SWAP ? P.rows : P.cols) - col0);
      const int32_t floor_v = (P.flags & DS_RELU) ? 0 : INT32_MIN;
      uint32_t amax_local = 0;
      auto finish = [&](int c, int row, int64_t idx) {
        long long sum = P.bias != nullptr ? __ldg(P.bias + (SWAP ? row0 + row : col0 + c)) : 0;
        const int at = (c_first + c) * kAccStride + row;
        if (i32) {
          uint32_t s32 = reinterpret_cast<uint32_t*>(accs)[at];
          if (split) {
            s32 = 0;
            for (int q = 0; q < S.splits; ++q)
              s32 += *cl.map_shared_rank(reinterpret_cast<uint32_t*>(accs) + at, q * kGroupSize + cta);
          }
          sum = (int32_t)(s32 + (uint32_t)sum);
        } else if (split) {
          for (int q = 0; q < S.splits; ++q)
            sum += *cl.map_shared_rank(reinterpret_cast<long long*>(accs) + at, q * kGroupSize + cta);
          sum = sat32(sum);
        } else {
          sum = sat32(sum + reinterpret_cast<long long*>(accs)[at]);
        }
        int32_t o = (int32_t)sum;
        if (CONV && (P.flags & DS_RESIDUAL)) o = add_sat(o, __ldg(P.residual + idx));
        o = max(o, floor_v);
        amax_local = max(amax_local, uabs(o));
        P.y[idx] = o;
      };
      if constexpr (SWAP) {  // a thread keeps its output column
        constexpr int kRowGroups = kThreads / kRows;
        const int64_t col = row0 + tid % kRows;
        if (col < P.cols && tid < kRowGroups * kRows)
          for (int r = tid / kRows; r < nc; r += kRowGroups) finish(r, tid % kRows, (col0 + r) * P.cols + col);
      } else if constexpr (CONV) {  // a thread keeps its row
        constexpr int kColGroups = kThreads / kRows;
        const int64_t cs = col_stride<true>(P);
        const RowPlace rp = row_place<true>(P, S.info[v.ph], row0 + tid % kRows);
        if (rp.ok && tid < kColGroups * kRows) {
          // Eight outputs of a thread at a time, their loads (bias, residual, the peers'
          // sums) in flight together: one at a time this took 10-17 thousand clocks a tile.
          // place(j, c, row, idx): output j's accumulator column, lane and output element; false if there is none.
          auto finish8 = [&](auto place) {
            int at[8];
            int64_t idx[8];
            int32_t o[8], res[8];
            bool ok[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              int c = 0, row = 0;
              ok[j] = place(j, c, row, idx[j]);
              at[j] = (c_first + c) * kAccStride + row;
              o[j] = ok[j] && P.bias != nullptr ? __ldg(P.bias + col0 + c) : 0;
              res[j] = ok[j] && (P.flags & DS_RESIDUAL) ? __ldg(P.residual + idx[j]) : 0;
              if (!ok[j]) at[j] = 0;
            }
            if (i32) {
              uint32_t* sums = reinterpret_cast<uint32_t*>(accs);
              for (int q = 0; q < S.splits; ++q) {
                const uint32_t* src = split ? cl.map_shared_rank(sums, q * kGroupSize + cta) : sums;
#pragma unroll
                for (int j = 0; j < 8; ++j) o[j] = (int32_t)((uint32_t)o[j] + src[at[j]]);
              }
            } else {
              long long* sums = reinterpret_cast<long long*>(accs);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                long long v = o[j];
                for (int q = 0; q < S.splits; ++q) v += (split ? cl.map_shared_rank(sums, q * kGroupSize + cta) : sums)[at[j]];
                o[j] = sat32(v);
              }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if ((P.flags & DS_RESIDUAL) != 0) o[j] = add_sat(o[j], res[j]);
              o[j] = max(o[j], floor_v);
              if (ok[j]) {
                amax_local = max(amax_local, uabs(o[j]));
                P.y[idx[j]] = o[j];
              }
            }
          };
          for (int b0 = tid / kRows; b0 < nc; b0 += 8 * kColGroups)
            finish8([&](int j, int& c, int& row, int64_t& idx) {
              c = b0 + j * kColGroups;
              row = tid % kRows;
              idx = rp.y0 + (col0 + c) * cs;
              return c < nc;
            });
        }
      } else {  // a warp takes rows, its lanes the columns
        const int nr = (int)min((int64_t)kRows, P.rows - row0);
        for (int row = warp; row < nr; row += kThreads / 32)
          for (int c = lane; c < nc; c += 32) finish(c, row, (row0 + row) * P.cols + col0 + c);
      }
      __syncwarp();
      if (P.amax_out != nullptr) {  // convolutions: one global atomic per CTA instead of one per warp
        amax_local = __reduce_max_sync(0xffffffffu, amax_local);
        if (lane == 0 && amax_local) atomicMax(CONV ? &bars->amax : P.amax_out, amax_local);
      }
    }
    if (split) cl.sync();  // the peers' reads end before this shared memory changes
    if (gave_up) break;
  }

  // every tensor operation has completed, in both CTAs of a pair, before tensor memory is freed
  __syncthreads();
  // a launch that gave up knows no bound of its incomplete outputs
  const uint32_t cta_amax = bars->abort ? 0x80000000u : (CONV ? bars->amax : 0u);
  if (tid == 0 && cta_amax && S.p[0].amax_out != nullptr) atomicMax(S.p[0].amax_out, cta_amax);
  if (warp == kMmaWarp) {
    if (cta == 0 && tc::elect_one()) tc::commit<PAIR>(&bars->done, pair_mask);
    __syncwarp();
    const long long t0 = clock64();
    while (!tc::mbar_try_wait(&bars->done, 0u) && clock64() - t0 < kWaitCycles) {
    }
  }
  if constexpr (PAIR) cg::this_cluster().sync();
  if (warp == kMmaWarp) {
    __syncwarp();
    tc::fence_after();
    tc::tmem_free<PAIR>(tmem, kTmemCols);
  }
}

template <int N, bool PAIR, bool CONV, bool VEC, bool SWAP>
bool set_attributes() {
  // once per process, thread-safe (see conv_direct.cu)
  static const bool ok = [] {
    const bool r = cudaFuncSetAttribute(shift_mma_kernel<N, PAIR, CONV, VEC, SWAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        227 * 1024) == cudaSuccess &&
                   cudaFuncSetAttribute(shift_mma_kernel<N, PAIR, CONV, VEC, SWAP>, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                        1) == cudaSuccess;
    if (!r) (void)cudaGetLastError();
    return r;
  }();
  return ok;
}

// How many clusters of cs CTAs the device holds at once (one CTA per SM), read once per size.
template <int N, bool PAIR, bool CONV, bool VEC, bool SWAP>
int max_clusters(int cs) {
  static int cache[kMaxCluster + 1] = {};
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  if (cache[cs] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cs);
    cfg.blockDim = dim3(cta_threads(SWAP));
    cfg.dynamicSmemBytes = 200 * 1024;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)cs;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, shift_mma_kernel<N, PAIR, CONV, VEC, SWAP>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      n = 0;
    }
    cache[cs] = n > 0 ? n : -1;
  }
  return cache[cs] > 0 ? cache[cs] : 0;
}

template <int N, bool PAIR, bool CONV, bool VEC, bool SWAP>
cudaError_t launch_n(MmaSet& S, int tiles, cudaStream_t st) {
  if (!set_attributes<N, PAIR, CONV, VEC, SWAP>()) return cudaErrorInvalidValue;
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorNoDevice;
  int nch = INT32_MAX;
  for (int i = 0; i < S.n; ++i) nch = (int)std::min<int64_t>(nch, S.p[i].n_chunks);
  // split sizes 1, 2, 4, .. (clusters of at most 16 CTAs): the least waves x
  // chunks of a rank, plus a fixed cost of the cluster reduction
  constexpr int group = PAIR ? 2 : 1;
  const int units = PAIR ? std::max(1, max_clusters<N, PAIR, CONV, VEC, SWAP>(group)) : sms;
  S.splits = 1;
  int64_t best = (int64_t)((tiles + units - 1) / units) * (nch + 4);
  if (tiles < units)
    for (int cs = 2; cs * group <= kMaxCluster && 2 * cs <= nch; cs *= 2) {
      const int n = max_clusters<N, PAIR, CONV, VEC, SWAP>(cs * group);
      if (n <= 0) continue;
      const int64_t cost = (int64_t)((tiles + n - 1) / n) * ((nch + cs - 1) / cs + 6);
      if (cost < best) {
        best = cost;
        S.splits = cs;
      }
    }
  const size_t smem = Layout<N, PAIR>::total(S.table_entries, S.n, CONV);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((S.splits > 1 ? tiles * S.splits : std::min(tiles, units)) * group));
  cfg.blockDim = dim3(cta_threads(SWAP));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)(S.splits * group);
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = S.splits * group > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, shift_mma_kernel<N, PAIR, CONV, VEC, SWAP>, S);
}

template <int N, bool PAIR, bool SWAP = !PAIR>
cudaError_t launch_set(const GemmParams* ps, int n, bool conv, cudaStream_t st) {
  MmaSet S{};
  S.n = n;
  S.wait_cycles = g_wait_cycles.load(std::memory_order_relaxed);
  S.table_entries = 0;
  int64_t tiles = 0;
  int flag_off = 0;
  bool vec = true;
  for (int i = 0; i < n; ++i) {
    const GemmParams& p = ps[i];
    S.p[i] = p;
    PhaseInfo& f = S.info[i];
    f.col_tiles = (int)(((SWAP ? p.rows : p.cols) + N - 1) / N);
    f.ct = make_fastdiv((uint32_t)f.col_tiles);
    f.ohw = make_fastdiv(conv ? (uint32_t)(p.OH * p.OW) : 1u);
    f.ow = make_fastdiv(conv ? (uint32_t)p.OW : 1u);
    constexpr int rows = kRows * (PAIR ? 2 : 1);
    const int64_t row_tiles = ((SWAP ? p.cols : p.rows) + rows - 1) / rows;
    f.flag_off = flag_off;
    f.flag_tiles = SWAP ? (int)row_tiles : f.col_tiles;
    flag_off += f.flag_tiles;
    tiles += row_tiles * f.col_tiles;
    f.tile_end = (int)tiles;
    if (conv) S.table_entries = std::max(S.table_entries, (p.R * p.S + kSlotK + 3) / 4 * 4);
    vec = vec && p.kred % 4 == 0;
  }
  if constexpr (!SWAP) {
    if (conv) return launch_n<N, PAIR, true, false, false>(S, (int)tiles, st);
  }
  return vec ? launch_n<N, PAIR, false, true, SWAP>(S, (int)tiles, st)
             : launch_n<N, PAIR, false, false, SWAP>(S, (int)tiles, st);
}

}  // namespace

// Rules of use, measured against the CUDA-core kernels (us, CUDA cores -> here).  A
// tile's fixed cost (its epilogue, the ring's fill) is that of about 100 reduction
// indices: 1x1 layers of 64 channels and 3x3 layers of 3 ran at 0.5-0.6 of the
// CUDA-core kernels' speed, the 147 indices of a 7x7 layer of 3 channels at 1.2.  A
// launch's fixed cost (setup, ring fill, last tile, teardown) is about 10 us.
// - Convolutions pay from 2^26 terms: 16x60x60 -> 32 3x3 34 -> 31, 512x23x23 -> 64 1x1
//   37 -> 32, and none of the shapes tried there is slower by more than repeated runs
//   differ (128x32x32 -> 128 1x1 28-31 -> 32).  The line at 1024 pixels is not a measured
//   one: 16 images of 512x7x7 -> 512 3x3 (784 pixels) would take 100 for 212.
// - FC pays from 2^27 terms (128 x 2048 x 512 43 -> 35) and 9 rows: up to 8 rows it is bound
//   by its codes, which the cluster kernel reads once (8 x 25088 x 4096: 0.94; 16 rows: 1.8).
// - Without a bound on x (no amax_io) a call needs four digits and 64-bit sums: four
//   walks in tiles of 64 columns or of swapped roles, eight in those of 128 columns.
//   Convolutions take the first then (512x28x28 -> 512 1x1 at 4 images 101 -> 50, CUDA cores
//   84), FC the second up to 64 pair tiles (384 x 10924 x 128 320 -> 100, CUDA cores 177; beyond,
//   384 x 684 x 4096 169 -> 181).  The CUDA cores keep FC of up to 32 rows, where the cluster
//   kernel has small tiles (VGG16 FC1 at 16 rows 539 -> 744, at 64 rows 1162 -> 747), FC of
//   less than 128 indices (1024 x 68 x 4096 82 -> 94), and convolutions of 16 columns and
//   less than 192 indices from 2^27 terms (16x121x121 -> 16 3x3 at 4 images 68 -> 101; of
//   2^26 terms, 16x88x88 at 5 images, 103 -> 60), kernels beyond 3x3 from 2^27.5 (3x119x119 -> 16
//   7x7 at 5 images 189 -> 104, 3x169x169 at 4 images 121 -> 147).
//   With amax_io the digits are known on the device only: VGG16 FC1 at 16 rows takes 337 ->
//   188 up to 2^20, 337 -> 387 up to 2^24, 547 -> 570 up to 2^28 and 547 -> 751 beyond.
// - Columns as lanes: up to 128 rows, as no lane is idle then.  With more rows, where
//   the pairs' tiles are too few: a tile of 256 rows splits over 8 pairs at most, one of
//   64 rows x 128 columns over 16 CTAs (1024 x 1028 x 128: pairs 56, so 31, CUDA cores 35;
//   384 x 1368 x 256: 58, 29, 34; 384 x 10924 x 128: 81, 44, 98).  The lines are at half of
//   the pairs (38 tiles) and 2^29.6 terms (2^29.2 where rows of x are copied word by word,
//   2^28.8 where the small tiles fill half of the chip unsplit): from there on a pair's wider
//   tiles win or come near (129 x 1021 x 4096: pairs 52, so 62; 1024 x 5797 x 128: 72, 80;
//   1024 x 8196 x 128: 75, 89; 256 x 4196 x 1000 still 66, 51).  For tiles of 64 columns,
//   half of whose lanes would be idle, the line is at 384 rows (384 x 7724 x 64: pairs
//   55, so 37, CUDA cores 52; 1024 x 7725 x 48: 58, 99, 103).
int shift_mma_route(const GemmParams* ps, int n, bool conv, bool bound) {
  if (n < 1 || n > kMaxGemmPhases) return DS_ROUTE_CUDA_CORES;
  int64_t tiles = 0, col_tiles = 0;
  double terms = 0.0;
  bool few_columns = true;
  for (int i = 0; i < n; ++i) {
    const GemmParams& p = ps[i];
    if (p.rows > INT32_MAX - kRows || p.n_chunks > INT32_MAX / kChunk) return DS_ROUTE_CUDA_CORES;
    if (conv ? p.kred < 128 || p.rows < 1024 : p.rows <= 8) return DS_ROUTE_CUDA_CORES;
    if (!bound && !conv && (p.kred < 128 || p.rows <= 32)) return DS_ROUTE_CUDA_CORES;
    few_columns = few_columns && p.cols <= 16 && p.kred < 192 && p.R * p.S > 1;
    terms += (double)p.rows * (double)p.kred * (double)p.cols;
    col_tiles += (p.cols + 63) / 64;
    tiles += (p.rows + kRows - 1) / kRows * ((p.cols + 63) / 64);
    if (conv) {
      if (p.R > 16 || p.S > 15 || p.R * p.S > kMaxTaps) return DS_ROUTE_CUDA_CORES;
      // the tap tables' element offsets are 32-bit: 16 indices span up to 17 channels, the tables a few more
      if ((int64_t)(kAGroups * kSlotK + 8) * p.H * p.W + (int64_t)p.R * p.W > INT32_MAX) return DS_ROUTE_CUDA_CORES;
    }
  }
  if (terms < (conv ? 67108864.0 : 134217728.0)) return DS_ROUTE_CUDA_CORES;
  if (col_tiles > kMaxColTiles || tiles > INT32_MAX / kMaxCluster) return DS_ROUTE_CUDA_CORES;
  if (conv && !bound && few_columns && terms >= (ps[0].R * ps[0].S <= 9 ? 134217728.0 : 189812531.0))
    return DS_ROUTE_CUDA_CORES;
  if (conv) return DS_ROUTE_TENSOR_CORES;
  const int64_t rows = ps[0].rows, cols = ps[0].cols;
  const int64_t pair_tiles = (rows + 2 * kRows - 1) / (2 * kRows) * ((cols + 127) / 128);
  const int64_t swap_tiles = (rows + 63) / 64 * ((cols + kRows - 1) / kRows);
  const bool swap = rows <= kRows || (cols <= 64 ? rows <= 3 * kRows
                                      : !bound   ? pair_tiles < 64
                                                 : pair_tiles < 38 && terms < (swap_tiles > 76         ? 469762048.0
                                                                               : ps[0].kred % 4 != 0 ? 603979776.0
                                                                                                     : 805306368.0));
  return swap ? DS_ROUTE_TENSOR_CORES_SWAPPED : DS_ROUTE_TENSOR_CORES;
}

bool shift_mma_preferred(const GemmParams* ps, int n, bool conv) {
  return shift_mma_route(ps, n, conv, ps[0].amax_in != nullptr) != DS_ROUTE_CUDA_CORES;
}

cudaError_t launch_shift_mma(const GemmParams* ps, int n, bool conv, cudaStream_t st) {
  const bool bound = ps[0].amax_in != nullptr;
  if (shift_mma_route(ps, n, conv, bound) == DS_ROUTE_TENSOR_CORES_SWAPPED)
    return launch_set<64, false>(ps, n, false, st);  // columns as lanes
  int64_t cols = 0;
  for (int i = 0; i < n; ++i) cols = std::max(cols, ps[i].cols);
  return cols <= 64 || (conv && !bound) ? launch_set<64, true>(ps, n, conv, st) : launch_set<128, true>(ps, n, conv, st);
}

void set_mma_wait_cycles(long long cycles) {
  g_wait_cycles.store(cycles > 0 ? cycles : kWaitCycles, std::memory_order_relaxed);
}

int read_mma_fault_flag() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_mma_fault, sizeof(int)) != cudaSuccess) return -1;
  const int zero = 0;
  if (v != 0 && cudaMemcpyToSymbol(g_mma_fault, &zero, sizeof(int)) != cudaSuccess) return -1;
  return v;
}

}  // namespace ds
