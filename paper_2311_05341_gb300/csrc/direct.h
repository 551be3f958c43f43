// direct.h -- geometry, tables and launch parameters of the direct tile
// (fwd_direct.cu) for steep plans: more than 5 samples of delay between
// consecutive trial DMs, where the words one trial loads serve no other.
//
// A CTA takes 128 trial DMs x 368 window words of one channel after another:
// every DM adds its own 368 words of the staged window, read at its shift.
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>

#include "fwd_tiled.h"

namespace dd {
namespace dt {

constexpr int kDm = 128;                 // trial DMs per CTA
constexpr int kWarps = 16;
constexpr int kDmWarp = kDm / kWarps;    // 8, in pairs that share a 23rd word
constexpr int kFull = 11;                // words per lane and DM ...
constexpr int kWords = 32 * kFull + 16;  // ... and 16 lanes' more: 368
constexpr int kAcc = 2 * kFull + 1;      // accumulator words per lane and DM pair
constexpr int kMaxNc = 16;               // channels per stage

// Per (block of kDm DMs, channel), 272 bytes (TMA-copyable).
struct Rec {
  int32_t base;        // s(c, first DM of the block)
  int32_t pad[3];
  uint16_t off[kDm];   // window word of each DM: s(c, d) - base + base mod align
};
static_assert(sizeof(Rec) == 272, "Rec must stay 272 bytes");

// Float32 at bin 1 stages its window words (two buffers); the other kinds
// stage raw samples (one buffer) and unpack them into one window buffer.
DD_HOST_DEVICE constexpr bool staged_words(int kind) { return kind == tk::kF32D; }
DD_HOST_DEVICE constexpr int raw_buffers(int kind) { return staged_words(kind) ? 2 : 1; }
DD_HOST_DEVICE constexpr int samples_per_tile(int kind) {
  return kWords * (kind == tk::kU8 ? 2 : 1);
}
// Raw bytes staged per channel for lw window words (uint8 at bin 1 pairs
// samples kWords apart).
DD_HOST_DEVICE constexpr int32_t raw_bytes(int kind, int bin, int32_t lw) {
  return kind == tk::kU8 ? lw + kWords : lw * tk::elem_bytes(kind) * bin;
}
constexpr size_t kRecOff = 128;
DD_HOST_DEVICE constexpr size_t raw_off(int nc) {
  return (kRecOff + 2 * static_cast<size_t>(nc) * sizeof(Rec) + 127) / 128 * 128;
}
inline size_t smem_bytes(int kind, int bin, int nc, int32_t lw) {
  return raw_off(nc) +
         static_cast<size_t>(raw_buffers(kind)) * nc * raw_bytes(kind, bin, lw) +
         (staged_words(kind) ? 0 : static_cast<size_t>(nc) * lw * 4);
}

struct Params {
  const void* x;
  int64_t stride;       // samples per channel row
  int32_t n_chan;
  int32_t n_dm;
  int32_t n_blocks;
  int32_t bin;
  int32_t align;        // window starts: multiples of this many decimated samples
  int32_t nc;           // channels per stage
  int32_t lw;           // window words per channel
  int32_t lraw;         // raw bytes per channel
  int32_t flush;        // channels the 16-bit lanes take between flushes
  const Rec* recs;      // [n_blocks][n_chan]
  int64_t t_begin;      // first output of the launch
  int64_t t_end;
  int64_t out_stride;
  void* out;
  int32_t* err;
  int32_t wait_iters;
  int32_t hold_stage;
};

// Whether the direct tile takes a launch rather than the offset tile of dr DMs
// per lane.  Both run one CTA per SM, so a launch takes whole waves of kSms
// CTAs, and the last one costs as much as the others: waves times the cycles a
// channel takes in each, 368 x 128 words at 27 a cycle here (0.83 to 0.95 us),
// 640 x 12 dr words at 11.75 or 20.6 a cycle on the offset tile of 1 or 2 DMs
// per lane (0.34 to 0.39 us).  Measured over 64 to 1000 DMs x 700 to 131072
// outputs, 5.5 to 26 samples a step, all kinds (2484 launches): never more than
// 2 % slower than the offset tile, 1.06 and 1.31 times its speed on average.
// (Fractions of waves in place of whole ones: up to 0.64 of its speed, 336
// channels x 400 DMs x 16384 outputs in 540 us against 345.)
inline bool faster(int32_t n_dm, int64_t outputs, int kind, int dr) {
  const int per = kind == tk::kU8 ? 2 : 1;
  auto waves = [&](int64_t words, int64_t dms) {
    const int64_t ctas = (outputs + words * per - 1) / (words * per) * ((n_dm + dms - 1) / dms);
    return static_cast<double>((ctas + tk::kSms - 1) / tk::kSms);
  };
  return waves(kWords, kDm) * (kWords * kDm / 27.0) <
         waves(640, 12 * dr) * (640 * 12 * dr / (dr == 1 ? 11.75 : 20.6));
}

}  // namespace dt

// Tables of a range (plan.cpp).
struct DirectTables {
  bool ok = false;
  int32_t kind = 0;     // tk::Kind
  int32_t n_blocks = 0;
  int32_t nc = 0;
  int32_t lw = 0;
  std::vector<unsigned char> bytes;  // dt::Rec [n_blocks][n_chan]
};

}  // namespace dd
