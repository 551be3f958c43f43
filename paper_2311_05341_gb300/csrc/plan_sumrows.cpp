// plan_sumrows.cpp -- host tables of the sum-row tile (sumrows.h): the channel
// groups of every block of 128 trial DMs, the distinct shift-difference
// vectors of each group (its sum rows) and the moves that make one row from
// the next.
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <vector>

#include "dd_internal.h"
#include "host_threads.h"
#include "sumrows.h"

namespace dd {

namespace {

using namespace sr;

// Cost (words_per_channel) per channel and 64 trial DMs x 736 words, half of
// this tile's DMs x twice its words, above which the pattern tile is taken: it
// moves (23 + o_3) words per 4 DMs and 23-word window, about 12000, at 3/4 of
// the pipe's rate.  Measured: 1024 channels, 2048 trials (cost 10800) 3.85 ms
// from packed copies against 5.2 ms, 4.8 against 5.8 ms from the input.  Where
// it first passes as channels grow (1024 DMs x 65536 samples from the input, 0.5
// and 1 sample a step: 192 and 384 channels) it takes 0.81 to 0.88 of the
// pattern tile's time, every format; from 96 to 1280 channels there it is never
// slower.
constexpr double kMaxWordsPerChannel = 13500.0;

// Difference vectors as bit masks: channel i of the group has kLevels bits,
// v_i - min of them set, so that the distance of two vectors in samples is
// the number of differing bits.
constexpr int kLevels = 4;

struct Mask {
  uint64_t w[kMaxK * kLevels / 64] = {};
  int dist(const Mask& o) const {
    int n = 0;
    for (size_t i = 0; i < sizeof(w) / 8; ++i) n += __builtin_popcountll(w[i] ^ o.w[i]);
    return n;
  }
};

struct Group {
  int k = 0;
  int rows = 0;
  int rs = 0;
  int lw = 0;
};

inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Cost of a group of k channels with `rows` rows, in shared-memory words per
// channel (32 words a cycle), of the three that bound it: the shared-memory
// pipe (staging and first row, moves -- their number grows a little faster than
// the rows' -- rows written and the adds' reads, at the 85 % of its rate that it
// gives), the building warps' chain of channels and moves (two warpgroups) and
// the adding warps' time, whose cycles were measured on the device.
double words_per_channel(const Format& f, int k, int rows, int rs) {
  const double moves = rows * (0.75 + k / 40.0);
  const double pipe =
      ((2.0 * k + moves * 1.2 + rows) * rs + static_cast<double>(kDm) * kWords) / 0.85;
  const double chain = 16.0 * (kChainGroup + f.chain_chan * k + f.chain_move * moves);
  const double adds = 32.0 * kAddGroup;
  return std::max({pipe, chain, adds}) / k;
}

template <typename T>
void put(std::vector<unsigned char>& v, const T& x) {
  const size_t n = v.size();
  v.resize(n + sizeof(T));
  std::memcpy(v.data() + n, &x, sizeof(T));
}

// The groups of DM block b: window starts, directory (record offsets from the
// block's first record) and records.  False where the tile cannot serve it.
struct Block {
  std::vector<Dir> dir;
  std::vector<int32_t> start;
  std::vector<unsigned char> recs;
  double words = 0;
  double unit = 0;        // cycles of a unit (Format::unit_add ...)
  double batch_unit = 0;  // in the persistent kernel
};

bool build_block(const RangePlan& rp, int32_t n_chan, int lane_chans, const Format& f, int64_t b,
                 Block* out) {
  std::vector<Dir>& dir = out->dir;
  std::vector<unsigned char>& recs = out->recs;
  out->start.resize(n_chan);
  size_t last_head = 0;  // of the latest group, for the flush flag
  std::vector<int32_t> block(static_cast<size_t>(n_chan) * kDm);  // shifts, DM fastest
  const int n_real = static_cast<int>(std::min<int64_t>(kDm, rp.n_dm - b * kDm));
  for (int d = 0; d < n_real; ++d) {
    const int32_t* row = &rp.shifts[static_cast<size_t>(b * kDm + d) * n_chan];
    for (int32_t c = 0; c < n_chan; ++c) block[static_cast<size_t>(c) * kDm + d] = row[c];
  }
  int32_t c = 0;
  int since = 0;  // channels in the lanes
  out->unit = f.unit_fixed;
  out->batch_unit = f.batch_fixed;
  while (c < n_chan) {
    const int32_t* s0 = &block[static_cast<size_t>(c) * kDm];
    const int rs = round_up(kWords + s0[n_real - 1] - s0[0], f.build);
    if (s0[n_real - 1] < s0[0] || rs > f.row_words) return false;
    // Extend the group channel by channel, splitting the DMs into classes
    // of equal difference vectors, and keep the cheapest size that fits.
    uint8_t cls[kDm] = {};
    int n_cls = 1, reach = 0;
    Group best;
    double best_cost = 1e30;
    uint8_t best_cls[kDm];
    const int kmax = static_cast<int>(std::min<int64_t>({kMaxK, n_chan - c, lane_chans}));
    for (int k = 1; k <= kmax; ++k) {
      const int32_t* s = &block[static_cast<size_t>(c + k - 1) * kDm];
      int lo = s[0] - s0[0], hi = lo;
      for (int d = 1; d < n_real; ++d) {
        lo = std::min(lo, s[d] - s0[d]);
        hi = std::max(hi, s[d] - s0[d]);
      }
      if (hi - lo >= kLevels) break;
      reach = std::max(reach, hi - lo);
      if (hi > lo) {
        uint8_t id[kDm * kLevels];
        std::memset(id, 255, static_cast<size_t>(n_cls) * kLevels);
        int n = 0;
        for (int d = 0; d < n_real; ++d) {
          uint8_t& e = id[cls[d] * kLevels + (s[d] - s0[d] - lo)];
          if (e == 255) e = static_cast<uint8_t>(n++);
          cls[d] = e;
        }
        n_cls = n;
      }
      const int lw = round_up(f.align - 1 + reach + rs + f.extra, 128 / f.bits);
      if (k * lw > 65535 || k * (lw * f.bits / 8) > f.raw_bytes || n_cls * rs > f.row_words) break;
      // The first row adds channels in pairs: only the last group may be odd.
      const double cost = words_per_channel(f, k, n_cls, rs);
      if (cost < best_cost && (k % 2 == 0 || c + k == n_chan || kmax == 1)) {
        best_cost = cost;
        best.k = k;
        best.rows = n_cls;
        best.rs = rs;
        best.lw = lw;
        std::memcpy(best_cls, cls, sizeof(best_cls));
      } else if (cost > 1.25 * best_cost) {
        break;
      }
    }
    if (best.k == 0) return false;

    // The rows' difference vectors, visited nearest first.
    std::vector<int32_t> rel_min(best.k);
    for (int i = 0; i < best.k; ++i) {
      const int32_t* s = &block[static_cast<size_t>(c + i) * kDm];
      int lo = s[0] - s0[0];
      for (int d = 1; d < n_real; ++d) lo = std::min(lo, s[d] - s0[d]);
      rel_min[i] = lo;
    }
    std::vector<Mask> mask(best.rows);
    std::vector<uint8_t> level(static_cast<size_t>(best.rows) * best.k);
    std::vector<char> seen(best.rows, 0);
    for (int d = 0; d < n_real; ++d) {
      const int r = best_cls[d];
      if (seen[r]) continue;
      seen[r] = 1;
      for (int i = 0; i < best.k; ++i) {
        const int v = block[static_cast<size_t>(c + i) * kDm + d] - s0[d] - rel_min[i];
        level[static_cast<size_t>(r) * best.k + i] = static_cast<uint8_t>(v);
        for (int q = 0; q < v; ++q) {
          const int bit = i * kLevels + q;
          mask[r].w[bit / 64] |= uint64_t{1} << (bit % 64);
        }
      }
    }
    std::vector<int> order;
    std::vector<char> used(best.rows, 0);
    int cur = 0;
    const Mask zero;
    for (int r = 1; r < best.rows; ++r)
      if (mask[r].dist(zero) < mask[cur].dist(zero)) cur = r;
    order.push_back(cur);
    used[cur] = 1;
    while (static_cast<int>(order.size()) < best.rows) {
      int nx = -1, nd = 1 << 30;
      for (int r = 0; r < best.rows; ++r) {
        if (used[r]) continue;
        const int dd = mask[cur].dist(mask[r]);
        if (dd < nd) {
          nd = dd;
          nx = r;
        }
      }
      order.push_back(nx);
      used[nx] = 1;
      cur = nx;
    }
    std::vector<int> row_of(best.rows);
    for (int i = 0; i < best.rows; ++i) row_of[order[i]] = i;

    // Window starts, the first row's windows and the moves.
    std::vector<uint16_t> init(round_up(best.k, 8), 0);  // padding: window 0
    std::vector<int32_t> at(best.k);
    for (int i = 0; i < best.k; ++i) {
      const int32_t s = s0[0] + rel_min[i];
      if (s < 0) return false;
      const int32_t m = s % f.align;
      out->start[c + i] = s - m;
      at[i] = i * best.lw + m;
      init[i] = static_cast<uint16_t>(at[i] + level[static_cast<size_t>(order[0]) * best.k + i]);
    }
    std::vector<uint32_t> steps;
    for (int q = 1; q < best.rows; ++q) {
      const uint8_t* from = &level[static_cast<size_t>(order[q - 1]) * best.k];
      const uint8_t* to = &level[static_cast<size_t>(order[q]) * best.k];
      for (int i = 0; i < best.k; ++i) {
        for (int v = from[i]; v < to[i]; ++v)
          steps.push_back(static_cast<uint32_t>(at[i] + v) | kStepUp);
        for (int v = from[i]; v > to[i]; --v)
          steps.push_back(static_cast<uint32_t>(at[i] + v - 1) | kStepDown);
      }
      steps.back() |= kStepEmit;
    }
    if (steps.size() > static_cast<size_t>(kMaxSteps)) return false;

    RecHead h{};
    h.k = static_cast<uint16_t>(best.k);
    h.n_steps = static_cast<uint16_t>(steps.size());
    h.rs = static_cast<uint16_t>(best.rs);
    steps.resize(round_up(static_cast<int>(steps.size()), 4) + kStepPad, 0);
    Dir e{};
    e.c0 = c;
    e.k = h.k;
    e.lw = static_cast<uint16_t>(best.lw);
    e.rec16 = static_cast<uint32_t>(recs.size() / 16);
    const size_t head = recs.size();
    put(recs, h);
    for (uint16_t v : init) put(recs, v);
    for (uint32_t v : steps) put(recs, v);
    for (int d = 0; d < kDm; ++d) {
      const int dr = std::min(d, n_real - 1);
      put(recs, static_cast<uint16_t>(row_of[best_cls[dr]] * best.rs + s0[dr] - s0[0]));
    }
    // The next copies' entry and starts: filled in once they are known.
    recs.resize(round_up(static_cast<int>(recs.size()), 16) + sizeof(Dir) + kMaxK * 4, 0);
    e.rec_n16 = static_cast<uint16_t>(recs.size() / 16 - e.rec16);
    // The lanes give up their high bytes before a group they cannot take.
    if (since + best.k > lane_chans) {
      const uint16_t one = 1;
      std::memcpy(recs.data() + last_head + offsetof(RecHead, flush), &one, 2);
      out->unit += f.unit_flush;
      out->batch_unit += f.unit_flush;
      since = 0;
    }
    since += best.k;
    last_head = head;
    dir.push_back(e);
    out->words += best_cost * best.k;
    const int passes = (best.rs + 32 * f.build * kBuildWarps - 1) / (32 * f.build * kBuildWarps);
    const double building = passes * (f.unit_group + f.unit_chan * best.k +
                                      static_cast<double>(f.unit_move) * h.n_steps) / 2;
    out->unit += std::max<double>(f.unit_add, building);
    out->batch_unit += std::max<double>(f.batch_add, building);
    c += best.k;
    if (recs.size() > (size_t{1} << 30)) return false;
  }
  return true;
}

}  // namespace

namespace {

// launch_cycles of unit(0) .. unit(n_costs - 1).
template <typename Unit>
double launch_cycles_of(int64_t n_costs, Unit unit, bool overlapped) {
  int64_t n = 0;
  double total = 0;
  for (int64_t i = 0; i < n_costs; ++i) {
    const UnitCost u = unit(i);
    n += u.count;
    total += u.cycles * static_cast<double>(u.count);
  }
  if (n == 0) return 0;
  if (overlapped)
    return std::max(static_cast<double>(n) / tk::kSms, 0.5) * total / static_cast<double>(n);
  const int64_t waves = (n + tk::kSms - 1) / tk::kSms;
  if (waves == 1) return unit(n_costs - 1).cycles;
  // The share of the units (by cost) that frees the SMs of the last wave.
  const double share = static_cast<double>(n - (waves - 1) * tk::kSms) / tk::kSms;
  double start = 0, seen = 0;
  for (int64_t i = 0; i < n_costs && seen < share * static_cast<double>(n); ++i) {
    const UnitCost u = unit(i);
    start = u.cycles;
    seen += static_cast<double>(u.count);
  }
  return static_cast<double>(waves - 2) * total / static_cast<double>(n) + start +
         unit(n_costs - 1).cycles;
}

}  // namespace

double launch_cycles(const std::vector<UnitCost>& sorted, bool overlapped) {
  return launch_cycles_of(
      static_cast<int64_t>(sorted.size()), [&](int64_t i) { return sorted[i]; }, overlapped);
}

void add_sum_row_units(const SumTables& t, bool batch, int64_t outputs,
                       std::vector<UnitCost>* units) {
  const int64_t halves = sum_row_halves(t.src, 0, outputs);
  for (double c : batch ? t.batch_cycles : t.unit_cycles) units->push_back({c, halves});
}

UnitCost pattern_units(const RangePlan& rp, int32_t n_chan, bool nibbles, int kind,
                       int64_t outputs) {
  // Cycles of a 64-DM unit, per channel and besides, as measured: one kind and
  // bin each (7 % around them).
  struct {
    double per_chan, fixed;
  } c;
  switch (kind) {
    case tk::kU8: c = {559, 33000}; break;
    case tk::kU4: c = {598, 30000}; break;
    case tk::kU16: c = {536, 13300}; break;
    case tk::kU8W: c = {589, 14000}; break;  // bin 2
    default:                                 // kU8P
      c = {nibbles        ? 475.0
           : rp.r.bin == 1 ? 500.0
           : rp.r.bin == 2 ? 563.0
           : rp.r.bin == 4 ? 672.0
                           : 914.0,
           31000};
  }
  const int ts = tk::pat_tile_samples(kind, rp.tile_h);
  return {c.fixed + c.per_chan * n_chan, (outputs + ts - 1) / ts * rp.tile_n_blocks};
}

bool sum_rows_faster(const SumTables& t, const RangePlan& rp, int32_t n_chan, bool nibbles,
                     int kind, int64_t outputs, bool overlapped) {
  const UnitCost pattern = pattern_units(rp, n_chan, nibbles, kind, outputs);
  const int64_t halves = sum_row_halves(t.src, 0, outputs);
  const int64_t blocks = static_cast<int64_t>(t.unit_cycles.size());
  // From 64 waves on the last one does not tell (and a plan may have millions
  // of blocks): their mean cost.
  const UnitCost mean{t.unit_total / static_cast<double>(blocks), blocks * halves};
  const double sums =
      mean.count >= 64 * tk::kSms
          ? launch_cycles_of(1, [&](int64_t) { return mean; }, overlapped)
          : launch_cycles_of(
                blocks, [&](int64_t i) { return UnitCost{t.unit_cycles[i], halves}; }, overlapped);
  return sums < launch_cycles_of(1, [&](int64_t) { return pattern; }, overlapped);
}

void build_sum_tables(const RangePlan& rp, int32_t n_chan, int64_t max_sample, int src,
                      SumTables* out) {
  *out = SumTables{};
  out->src = src;
  const Format f = format(src);
  const bool lanes16 = sr::lanes16(src);
  // 16-bit lanes: the high bytes carried out of the lanes (TMEM, 16 bits per
  // sample) hold sums below 2^24; 32-bit words hold sums below 2^31.
  const int64_t total = static_cast<int64_t>(n_chan) * max_sample;
  if (total >= (lanes16 ? int64_t{1} << 24 : int64_t{1} << 31)) return;
  // Channels the lanes take on top of the low bytes they keep.
  const int lane_chans = lanes16 ? static_cast<int>(std::min<int64_t>(65280 / max_sample, 1 << 20))
                                 : 1 << 30;
  if (lane_chans < 1) return;
  const int64_t n_blocks = (rp.n_dm + kDm - 1) / kDm;
  // Fewer channels make so few groups that filling the pipeline outweighs the
  // adds saved (48 channels: 3 to 5 us a call slower; 128: none).
  if (n_chan < 96 || n_blocks * n_chan > (int64_t{1} << 28)) return;

  std::vector<Block> blocks(n_blocks);
  if (!parallel_for(n_blocks, 300.0 * n_blocks * n_chan, [&](int64_t b) {
        return build_block(rp, n_chan, lane_chans, f, b, &blocks[b]);
      }))
    return;

  size_t n_dir = 0, n_recs = 0;
  double words = 0;
  for (const Block& b : blocks) {
    n_dir += b.dir.size();
    n_recs += b.recs.size();
    words += b.words;
  }
  const double blocks64 = static_cast<double>((rp.n_dm + 63) / 64);
  if (words > kMaxWordsPerChannel * n_chan * blocks64 / 2.0) return;
  auto pad16 = [](size_t v) { return (v + 15) / 16 * 16; };
  const size_t off_dir = pad16((n_blocks + 1) * sizeof(int32_t));
  const size_t off_start = off_dir + n_dir * sizeof(Dir);
  // Each record ends with the entry and window starts of the group kSlots later.
  const size_t off_rec = pad16(off_start + static_cast<size_t>(n_blocks) * n_chan * 4);
  if (off_rec + n_recs > 0x7fffffffu) return;
  out->bytes.assign(off_rec + n_recs, 0);
  unsigned char* to = out->bytes.data();
  int32_t first = 0;
  size_t at = off_rec;
  for (int64_t b = 0; b < n_blocks; ++b) {
    Block& blk = blocks[b];
    std::memcpy(to + b * 4, &first, 4);
    for (Dir& e : blk.dir) e.rec16 += static_cast<uint32_t>(at / 16);
    for (size_t g = 0; g + kSlots < blk.dir.size(); ++g) {
      const Dir& e = blk.dir[g];
      const Dir& n = blk.dir[g + kSlots];
      unsigned char* tail = blk.recs.data() + (static_cast<size_t>(e.rec16) * 16 - at) +
                            static_cast<size_t>(e.rec_n16) * 16 - sizeof(Dir) - kMaxK * 4;
      std::memcpy(tail, &n, sizeof(Dir));
      std::memcpy(tail + sizeof(Dir), &blk.start[n.c0], n.k * sizeof(int32_t));
    }
    std::memcpy(to + off_dir + first * sizeof(Dir), blk.dir.data(), blk.dir.size() * sizeof(Dir));
    std::memcpy(to + off_start + static_cast<size_t>(b) * n_chan * 4, blk.start.data(),
                static_cast<size_t>(n_chan) * 4);
    std::memcpy(to + at, blk.recs.data(), blk.recs.size());
    at += blk.recs.size();
    first += static_cast<int32_t>(blk.dir.size());
  }
  std::memcpy(to + n_blocks * 4, &first, 4);
  out->n_blocks = static_cast<int32_t>(n_blocks);
  out->off_dir = static_cast<int32_t>(off_dir);
  out->off_start = static_cast<int32_t>(off_start);
  for (const Block& b : blocks) {
    out->unit_total += b.unit;
    out->unit_cycles.push_back(b.unit);
    out->batch_cycles.push_back(b.batch_unit);
  }
  std::sort(out->unit_cycles.begin(), out->unit_cycles.end());
  std::sort(out->batch_cycles.begin(), out->batch_cycles.end());
  out->ok = true;
}

}  // namespace dd
