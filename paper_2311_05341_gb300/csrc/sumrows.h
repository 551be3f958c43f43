// sumrows.h -- geometry, device tables and launch parameters of the sum-row
// tile (fwd_sumrows.cu), shared with its planner (plan_sumrows.cpp).
//
// Eq. 3 asks for sum_c X[c][t + s(c, d)].  Over a block of consecutive trial
// DMs the shifts of adjacent channels move almost together: relative to its
// first channel, a group of K adjacent channels takes few distinct vectors of
// shift differences (s(c, d) - s(c_0, d))_c -- about K of them for 128 DMs,
// because each channel changes its difference by one sample at a time.  All
// trial DMs with the same vector need the same time series, moved by
// s(c_0, d).  So the kernel builds each distinct sum over the group once (a
// sum row, in shared memory) and every DM adds one word of its row per output
// word instead of K channel words.
//
// Integer sums are exact in any order, so the outputs equal the direct sum's
// bit for bit; a row is made from the previous one by replacing the words of
// the channels whose difference changed (one subtraction and one addition).
// Float rows could not be made that way (a large or non-finite sample would
// leak into rows that do not hold it), so float32 keeps the pattern tiles.
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>

#include "fwd_tiled.h"

namespace dd {

struct RangePlan;

namespace sr {

constexpr int kDm = 128;             // trial DMs per CTA
constexpr int kMainWarps = 8;        // adding warps, kDmWarp DMs each
constexpr int kDmWarp = kDm / kMainWarps;
constexpr int kBuildGroups = 2;      // row-building warpgroups, taking channel groups in turn
constexpr int kBuildWarps = 4;       // warps of a building warpgroup
constexpr int kThreads = 32 * (kMainWarps + kBuildGroups * kBuildWarps);
// Output words per DM: 11 words per lane for each DM of a pair, and one more
// that the two DMs of the pair share (16 lanes each).  Two such tiles make one
// 736-word time tile of the pattern tiles (32 x 23), whose packed copies (pair
// distance 736) and time-segment boundaries this tile shares.
constexpr int kFull = 11;
constexpr int kWords = 32 * kFull + 16;  // 368
constexpr int kPairWords = 2 * kWords;   // 736: words per pattern time tile, pair distance
constexpr int kAcc = 2 * kFull + 1;      // accumulator words per lane and DM pair
constexpr int kMaxK = 32;                // channels per group
constexpr int kSlots = 3;                // staging slots, row buffers
constexpr int kMaxSteps = 192;           // moves per group
constexpr int kStepPad = 8;              // readable moves past the last one
constexpr int kMaxRec = 16 + kMaxK * 2 + (kMaxSteps + kStepPad) * 4 + kDm * 2 + 16 + kMaxK * 4;

// What the tile stages.  kPairs: 32-bit words of a packed copy (two samples,
// 736 apart, in 16-bit lanes), for decimated uint8.  kBytes, kNibbles: the
// uint8 or 4-bit input itself; a row word pairs samples 368 apart, so a CTA's
// 736 outputs and its staged window are contiguous.  kHalves: the uint16
// input, one sample per 32-bit row word.  kBytes2: the uint8 input decimated by
// 2 as it is read, row words as kBytes (staged samples are the decimated ones).
enum Src : int { kPairs = 0, kBytes = 1, kNibbles = 2, kHalves = 3, kBytes2 = 4 };

struct Format {
  int bits;        // per staged sample (kPairs: per word)
  int align;       // window starts: multiples of this many staged samples (16 bytes or more)
  int build;       // row words per lane of a building warp
  int extra;       // staged samples a lane reads past its last row word's sample
  int raw_bytes;   // staging slot
  int row_words;   // row buffer
  int chain_chan;  // measured cycles of a building warp per channel of a group
  int chain_move;  // and per move (kChainGroup per group besides)
  // A unit's cycles, fitted to measured launches (launch_cycles): unit_fixed,
  // and per group the larger of unit_add and, for each pass of the building
  // warps over its rows, half of unit_group + unit_chan per channel + unit_move
  // per move; unit_flush for each time the 16-bit lanes give up their high bytes.
  int unit_add, unit_group, unit_chan, unit_move, unit_flush, unit_fixed;
  // The same in the persistent kernel, which starts its pipeline anew for every
  // unit and whose adding warps are slower.
  int batch_add, batch_fixed;
};
constexpr int kChainGroup = 900;
constexpr int kAddGroup = 2900;  // cycles of the adding warps per group
// kPairs: five scalar words per lane (an odd lane stride: no bank conflicts),
// 29 KB of staging for 44.5 KB of rows.  The others: four words per lane from
// unaligned bytes (two 32-bit words and a funnel shift), stored 16 bytes at a
// time; a window is less than half as long in bytes, so the rows get more.
DD_HOST_DEVICE constexpr Format format(int src) {
  return src == kPairs ? Format{32, 16, 5, 1, 29696, 11392, 110, 155,
                                1820, 2730, 61, 129, 2040, 28000, 3510, 55000}
         : src == kBytes ? Format{8, 16, 4, kWords + 8, 17408, 14464, 190, 145,
                                  3270, 130, 138, 211, 220, 27000, 4480, 38000}
         : src == kNibbles ? Format{4, 32, 4, kWords + 16, 17408, 14464, 195, 165,
                                    3320, 30, 126, 248, 610, 28500, 4150, 42000}
         : src == kHalves ? Format{16, 16, 4, 4, 17408, 14464, 380, 130,
                                   2870, 80, 89, 193, 0, 13000, 3160, 28000}
                          : Format{16, 16, 4, kWords + 4, 29696, 11392, 300, 200,
                                   3950, 15, 173, 370, 1500, 25000, 4460, 44500};
}
// Output samples of a CTA's words, and of the pattern time tile holding them.
DD_HOST_DEVICE constexpr int pair_dist(int src) { return src == kPairs ? kPairWords : kWords; }
DD_HOST_DEVICE constexpr bool lanes16(int src) { return src != kHalves; }

// One channel group of one DM block.
struct Dir {
  int32_t c0;        // first channel
  uint16_t k;        // channels
  uint16_t lw;       // staged samples per channel (a multiple of 16 bytes)
  uint32_t rec16;    // record offset in the tables, in 16 bytes
  uint16_t rec_n16;  // record length, in 16 bytes
  uint16_t pad;
};
static_assert(sizeof(Dir) == 16, "Dir must stay 16 bytes");

// Record header; then k uint16 staged sample offsets of the first row's
// windows (padded to 8 entries), n_steps moves (padded to a multiple of 4,
// then kStepPad more), kDm uint16 row word offsets (row * stride + the DM's
// shift from the block's first DM), and the directory entry (k == 0: none) and
// kMaxK window starts of the group kSlots later, whose copies are issued while
// this group is added.
struct RecHead {
  uint16_t k;
  uint16_t n_steps;
  uint16_t rs;       // row stride in words (a multiple of Format::build)
  uint16_t flush;    // 1: the 16-bit lanes give up their high bytes after this group
  uint32_t pad[2];
};
static_assert(sizeof(RecHead) == 16, "RecHead must stay 16 bytes");
// A move: staged sample offset (16 bits) of the lower of the channel's two
// windows, whether a row is complete after it, and in the top two bits its
// sign (1 up, -1 down, 0 padding) as a signed number.
constexpr uint32_t kStepEmit = 1u << 17;
constexpr uint32_t kStepUp = 1u << 30;
constexpr uint32_t kStepDown = 3u << 30;
DD_HOST_DEVICE constexpr int rec_steps_off(int k) { return 16 + (k + 7) / 8 * 16; }
DD_HOST_DEVICE constexpr int rec_offs_off(int k, int n_steps) {
  return rec_steps_off(k) + ((n_steps + 3) / 4 * 4 + kStepPad) * 4;
}

// Shared memory: barriers and flags, records, offsets, staging, rows.
constexpr size_t kRecOff = 256;
constexpr size_t kRecBytes = (kMaxRec + 127) / 128 * 128;
constexpr size_t kOffsOff = kRecOff + kSlots * kRecBytes;
// Row addresses, the flush flag, the directory entry and window starts of the
// group kSlots later.
constexpr int kNextDir = kDm + 4;            // in words
constexpr int kNextStart = kNextDir + 4;
constexpr size_t kOffsBytes = (kNextStart + kMaxK) * 4;
constexpr size_t kRawOff = (kOffsOff + kSlots * kOffsBytes + 127) / 128 * 128;
DD_HOST_DEVICE constexpr size_t row_off(int src) {
  return kRawOff + kSlots * static_cast<size_t>(format(src).raw_bytes);
}
DD_HOST_DEVICE constexpr size_t smem_bytes(int src) {
  return row_off(src) + kSlots * static_cast<size_t>(format(src).row_words) * 4;
}
static_assert(smem_bytes(kPairs) <= 227 * 1024 && smem_bytes(kBytes) <= 227 * 1024 &&
                  smem_bytes(kBytes2) <= 227 * 1024,
              "sum-row tile exceeds shared memory");

struct Params {
  const void* x;         // staged rows
  int64_t stride;        // staged samples (kPairs: words) per channel row
  int64_t x_origin;      // staged sample held by element 0 of each row
  int32_t n_chan;
  int32_t n_dm;
  int32_t n_blocks;
  const unsigned char* tables;
  int32_t off_dir;       // byte offsets of the directory and the window starts
  int32_t off_start;
  int64_t half0;         // first half of the launch (half_origin)
  int64_t t_end;         // outputs t >= t_end are not written
  int64_t out_stride;    // elements from output row d to row d + 1
  int32_t* out;
  int32_t* err;
  int32_t wait_iters;
  int32_t hold_stage;    // group whose copies are never issued (timeout test; -1: none)
};

// Persistent batch execution: items (job, DM block, half) over many jobs.
struct BatchArgs {
  const Params* jobs;          // device
  const tk::BatchItem* items;  // device, in execution order (tile: the half)
  int32_t n_items;
  uint32_t* counter;           // device, zero before the launch
};

}  // namespace sr

// Tables of a range (plan_sumrows.cpp): group starts per DM block (int32
// [n_blocks + 1]), directory, window starts (int32 [n_blocks][n_chan]), records.
struct SumTables {
  bool ok = false;
  int32_t src = 0;       // sr::Src
  int32_t n_blocks = 0;
  int32_t off_dir = 0;
  int32_t off_start = 0;
  // What a unit (128 DMs x 368 words) takes, per DM block in ascending order,
  // and in the persistent kernel.
  std::vector<double> unit_cycles;
  std::vector<double> batch_cycles;
  double unit_total = 0.0;  // of unit_cycles
  std::vector<unsigned char> bytes;
};

// Cycles (at about 2 GHz) of a launch of one-CTA-per-SM units, `count` of every
// cost in `sorted` (ascending): whole waves of kSms CTAs of mean cost, the last
// of which starts when as many units as it has are through the wave before (the
// cheapest), and ends with the dearest.  overlapped: among launches that fill
// each other's gaps, for which units count as such, but a launch does not fall
// below half a wave of two in flight.
struct UnitCost {
  double cycles;
  int64_t count;
};
double launch_cycles(const std::vector<UnitCost>& sorted, bool overlapped);
// The units of `outputs` outputs of a range on the sum-row tile, appended, and on
// the pattern kernel `kind` (its tables' kind or the packed copy's).
void add_sum_row_units(const SumTables& t, bool batch, int64_t outputs,
                       std::vector<UnitCost>* units);
UnitCost pattern_units(const RangePlan& rp, int32_t n_chan, bool nibbles, int kind,
                       int64_t outputs);
// Whether the sum-row tile takes the launch.  Its 128-DM units leave more of
// the chip idle than the pattern tile's 64-DM ones where there are few: 150
// channels x 130 DMs x 60000 uint8 outputs make 164 units, 2 waves of 66 us
// together, where 123 of the pattern tile take 58.  Measured over 100 to 3000
// channels, 64 to 1000 DMs, 20000 to 74000 outputs and 0.1 to 2 samples a step,
// every format (1175 launches): never slower than the pattern tile (the sum-row
// tile always: up to 1.21 times its time), and 1.0004 times the better of the
// two on average.
bool sum_rows_faster(const SumTables& t, const RangePlan& rp, int32_t n_chan, bool nibbles,
                     int kind, int64_t outputs, bool overlapped);

// max_sample: the largest (decimated) sample.  ok == false where the tile
// would not be faster than the pattern tile or cannot hold the sums.
void build_sum_tables(const RangePlan& rp, int32_t n_chan, int64_t max_sample, int src,
                      SumTables* out);

}  // namespace dd
