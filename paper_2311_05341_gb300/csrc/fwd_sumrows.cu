// fwd_sumrows.cu -- the sum-row tile (sumrows.h): Eq. 3 for 128 trial DMs x
// 368 row words per CTA, from integer input or its packed copy: the one-unit
// kernel of dd_run and the persistent kernel of dd_batch_run.
//
// Roles.  Two warpgroups build, taking channel groups in turn: from the staged
// windows of a group of K adjacent channels (one bulk copy per channel, three
// slots) they sum the group's first row, turn each row into the next by
// replacing the windows of the channels whose shift difference changed, and
// store every row to one of three row buffers.  Eight warps add: each owns 16
// DMs x 368 words in 184 accumulator registers per lane and adds, per DM and
// word, one word of the DM's row; they also issue the copies.  Builders and
// adders hand buffers over through mbarriers.  The registers are split
// unevenly (setmaxnreg): 208 per adding thread, 48 per building thread, of the
// 128 x 512 the CTA is launched with.
//
// What bounds it: the shared-memory pipe (128 bytes per clock and SM).  Per
// group and CTA the adders read 128 x 368 words; the builders read about
// (K + 1.2 moves) x W words and write rows x W, W = 368 + the block's delay
// span.  The planner picks K per group to make the whole cheapest: 5300 words
// per channel at 8192 channels and 4096 trials (K = 15, 17 rows, 21 moves on
// average), where the pattern tile moves 12000.  Measured there (262144
// uint8 samples, one launch): 68.4 ms from the packed copy (pattern tile 153.5)
// and 78.5 ms from the input (170.0); uint16, 4096 channels x 65536, 3072
// trials 19.3 ms (29.6).  Per group the adders take 3300 cycles, of which 2400
// are adds against 1472 of the bare reads, 500 the copies' issue and 300 the
// lanes' high bytes; the builders are as long.  One building warpgroup with
// two buffers and groups of 22 channels ran 90 ms: a warp's chain of moves
// (about 150 cycles each behind the adders' reads) was longer than the adds.
// Reading bytes instead of packed words halves the staging but costs the
// builders four funnel shifts and six byte selections per move.
//
// 16-bit lanes (two samples per word): before they can overflow, the adders
// move the lanes' high bytes to tensor memory (16-bit sums of high bytes, 184
// words per thread), so partial sums never leave the SM and every output is
// stored once.
//
// Every mbarrier wait is bounded; a warp that gives one up sets the abort flag,
// which ends the other waits, and on leaving the CTA sets kErrTimeout, waits for
// its copies (drain_copies) and frees its tensor memory.  Lanes of a warp may
// find out one by one, and nothing bounds a warp-wide operation that waits for a
// lane gone ahead, so warps vote on every wait before they go on or leave: the
// building warps in build, the adding warps with the byte counts of the copies
// they issue next (issue_copies).  The votes cost up to 1 % of a launch (8192
// channels: 70.3, now 70.9 ms through the ring, 78.2 and 78.5 ms from the input).
#include <cuda_runtime.h>

#include <cstdint>

#include "dd_internal.h"
#include "sumrows.h"
#include "tile_common.cuh"
#include "tmem.cuh"

namespace dd {
namespace sr {

using tk::bulk_copy;
using tk::mbar_arrive_expect;
using tk::mbar_init;
using tk::smem_u32;

// Shared-memory control block (the first 256 bytes).
struct Ctl {
  uint64_t raw_full[kSlots];    // the slot's copies have landed
  uint64_t rows_full[kSlots];   // the buffer's rows are built
  uint64_t rows_empty[kSlots];  // the adders have read them
  uint32_t tmem;
  volatile int32_t abort;           // a wait gave up: every role leaves
  volatile int32_t issued[kSlots];  // group + 1 whose copies warp 0 last issued into the slot
  volatile int32_t issued_by[kMainWarps];  // groups whose copies each adding warp has issued
};
static_assert(sizeof(Ctl) <= kRecOff, "control block too large");

constexpr int kDrainIters = 1 << 14;  // polls, far longer than a copy takes
// Polls of a shared word: some 40 cycles each, where a poll of an mbarrier
// suspends its warp; a caller's short limit must not end a wait that only the
// adders' work on three groups (10000 cycles) bounds.
constexpr int kIssuePolls = 1 << 16;

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Bounded wait that also ends when the CTA is aborting (a lane's own result).
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, const Ctl* ctl) {
  for (int it = 0; it < tk::kWaitIters; it += 64) {
    if (tk::mbar_wait(bar, parity, 64)) return true;
    if (ctl->abort) return false;
  }
  return false;
}

// Bounded wait for the copies of group g (a lane's own result).  A parity wait
// only tells a phase from the one before it, and the slot's previous group
// belongs to the other warpgroup: the wait starts once the copies of g are
// issued, which follows the end of that group.
__device__ __forceinline__ bool wait_copies(const Params& p, Ctl* ctl, int g) {
  const int slot = g % kSlots, polls = max(p.wait_iters, kIssuePolls);
  for (int it = 0; ctl->issued[slot] <= g; ++it)
    if (it >= polls || ctl->abort) return false;
  return tk::mbar_wait(smem_u32(&ctl->raw_full[slot]), (g / kSlots) & 1, p.wait_iters);
}

// After an abort, every role done: the copies still in flight land before the
// CTA goes on.  The adding warps issue their shares of a group on their own,
// and one that gave up first leaves its share out; a slot's warps are at most
// one group apart (its next group is issued only once all copies of the last
// one have landed).  The arrivals of the warps behind are made here, so that
// the newest group's phase ends with the bytes that were asked for.
__device__ __forceinline__ void drain_copies(const Params& p, const Ctl* ctl) {
#pragma unroll 1
  for (int s = 0; s < kSlots; ++s) {
    int newest = -1;
    uint32_t missing = 0;
#pragma unroll 1
    for (int w = 0; w < kMainWarps; ++w) {
      int g = ctl->issued_by[w] - 1;              // the warp's newest group ...
      g -= (g % kSlots - s + kSlots) % kSlots;    // ... of this slot
      if (g == p.hold_stage) g -= kSlots;         // (never issued)
      missing = g == newest ? missing : g > newest ? w : missing + 1;
      newest = max(newest, g);
    }
    if (newest < 0) continue;
    const uint32_t bar = smem_u32(&ctl->raw_full[s]);
    if (missing > 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(missing)
                   : "memory");
    tk::mbar_wait(bar, (newest / kSlots) & 1, kDrainIters);
  }
}
__device__ __forceinline__ void mbar_inval(uint32_t bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

constexpr int kDmPairs = kDmWarp / 2;
static_assert(kDmPairs * kAcc % 8 == 0, "tensor memory moves 8 words at a time");

// The high bytes of the 16-bit lanes into tensor memory: lane word a becomes
// its low bytes, and the 16-bit sums of high bytes at the word's column grow
// by a >> 8 (below 2^16 while the total is below 2^24).
__device__ __forceinline__ void flush_lanes(uint32_t col, uint32_t (&acc)[kDmPairs][kAcc],
                                            bool first) {
#pragma unroll
  for (int q = 0; q < kDmPairs * kAcc; q += 8) {
    uint32_t v[8] = {};
    if (!first) tmem::load(col + q, v);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      uint32_t& a = acc[(q + e) / kAcc][(q + e) % kAcc];
      v[e] += __byte_perm(a, 0u, 0x4341);
      a &= 0x00ff00ffu;
    }
    tmem::store(col + q, v);
  }
  tmem::wait_stores();
}

__device__ __forceinline__ uint32_t lds(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}

// How a building lane reads its kWindow words of a window and keeps sums.
// offset: staged sample offset (16 bits) of the window in the slot; `first`
// adds the window's words to the sums, `move` replaces them by the next
// sample's (sign 1) or, given the window one sample lower, the other way
// round (sign -1); `words` gives the row words of the sums.
template <int SRC>
struct Lane;

template <>
struct Lane<kPairs> {
  static constexpr int kN = 5, kStep = 5, kLoads = 6, kDepth = 2;
  uint32_t base;  // shared address of the lane's first word at offset 0
  __device__ Lane(uint32_t raw, int k, int) : base(raw + 4u * k) {}
  __device__ void load(uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t a = base + 4u * (offset & 0xffffu);
#pragma unroll
    for (int j = 0; j < kLoads; ++j) x[j] = lds(a + 4 * j);
  }
  __device__ void load_first(uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t a = base + 4u * offset;
#pragma unroll
    for (int j = 0; j < kN; ++j) x[j] = lds(a + 4 * j);
  }
  __device__ void first(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t) const {
#pragma unroll
    for (int j = 0; j < kN; ++j) s[j] += x[j];
  }
  __device__ void move(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t,
                       uint32_t sign) const {
#pragma unroll
    for (int j = 0; j < kN; ++j) s[j] += (x[j + 1] - x[j]) * sign;
  }
  // Five scalar stores, where `on` is not zero (predicated: no branch).
  __device__ static void store(uint32_t a, const uint32_t (&s)[kN], uint32_t on) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %6, 0;\n\t"
        "@p st.shared.u32 [%0], %1;\n\t@p st.shared.u32 [%0+4], %2;\n\t"
        "@p st.shared.u32 [%0+8], %3;\n\t@p st.shared.u32 [%0+12], %4;\n\t"
        "@p st.shared.u32 [%0+16], %5;\n\t}" ::"r"(a),
        "r"(s[0]), "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(on)
        : "memory");
  }
};

__device__ __forceinline__ void store4_if(uint32_t a, uint32_t w0, uint32_t w1, uint32_t w2,
                                          uint32_t w3, uint32_t on) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t"
      "@p st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n\t}" ::"r"(a),
      "r"(w0), "r"(w1), "r"(w2), "r"(w3), "r"(on)
      : "memory");
}

// Sums of uint8 or 4-bit samples k .. k + 3 and those 368 later, as 16-bit
// pairs two samples apart: s[0] = (0, 2), s[1] = (1, 3), s[2], s[3] the later
// ones; a row's words pair a sample with the one 368 later.
struct SplitPairs {
  __device__ static void store(uint32_t a, const uint32_t (&s)[4], uint32_t on) {
    store4_if(a, __byte_perm(s[0], s[2], 0x5410), __byte_perm(s[1], s[3], 0x5410),
              __byte_perm(s[0], s[2], 0x7632), __byte_perm(s[1], s[3], 0x7632), on);
  }
};

template <>
struct Lane<kBytes> : SplitPairs {
  static constexpr int kN = 4, kStep = 4, kLoads = 4, kDepth = 3;
  uint32_t base;
  __device__ Lane(uint32_t raw, int k, int) : base(raw + k) {}  // k a multiple of 4
  __device__ void load_first(uint32_t (&x)[kLoads], uint32_t offset) const { load(x, offset); }
  __device__ void load(uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t a = base + (offset & 0xfffcu);
    x[0] = lds(a);
    x[1] = lds(a + 4);
    x[2] = lds(a + kWords);
    x[3] = lds(a + kWords + 4);
  }
  __device__ void first(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t sh = 8u * (offset & 3u);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t y = __funnelshift_r(x[2 * h], x[2 * h + 1], sh);
      s[2 * h] += y & 0x00ff00ffu;
      s[2 * h + 1] += __byte_perm(y, 0u, 0x4341);
    }
  }
  __device__ void move(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t offset,
                       uint32_t sign) const {
    const uint32_t sh = 8u * (offset & 3u);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t y0 = __funnelshift_r(x[2 * h], x[2 * h + 1], sh);        // samples 0..3
      const uint32_t y1 = __funnelshift_rc(x[2 * h], x[2 * h + 1], sh + 8u);  // samples 1..4
      const uint32_t odd = y1 & 0x00ff00ffu;
      s[2 * h] += (odd - (y0 & 0x00ff00ffu)) * sign;
      s[2 * h + 1] += (__byte_perm(y1, 0u, 0x4341) - odd) * sign;
    }
  }
};

template <>
struct Lane<kNibbles> : SplitPairs {
  static constexpr int kN = 4, kStep = 4, kLoads = 4, kDepth = 3;
  uint32_t raw;
  int k;
  __device__ Lane(uint32_t raw_, int k_, int) : raw(raw_), k(k_) {}
  __device__ void load_first(uint32_t (&x)[kLoads], uint32_t offset) const { load(x, offset); }
  __device__ void load(uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t a = raw + (((offset & 0xffffu) + k) >> 3) * 4u;
    x[0] = lds(a);
    x[1] = lds(a + 4);
    x[2] = lds(a + kWords / 2);
    x[3] = lds(a + kWords / 2 + 4);
  }
  // Samples 0 .. 7 from the lane's first one.
  __device__ uint32_t eight(const uint32_t (&x)[kLoads], int h, uint32_t offset) const {
    return __funnelshift_r(x[2 * h], x[2 * h + 1], 4u * ((offset + k) & 7u));
  }
  __device__ void first(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t offset) const {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t b01 = __byte_perm(eight(x, h, offset), 0u, 0x4140);  // bytes 0 and 1
      s[2 * h] += b01 & 0x000f000fu;
      s[2 * h + 1] += (b01 >> 4) & 0x000f000fu;
    }
  }
  __device__ void move(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t offset,
                       uint32_t sign) const {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t y = eight(x, h, offset);
      const uint32_t b01 = __byte_perm(y, 0u, 0x4140), b12 = __byte_perm(y, 0u, 0x4241);
      const uint32_t odd = (b01 >> 4) & 0x000f000fu;
      s[2 * h] += (odd - (b01 & 0x000f000fu)) * sign;
      s[2 * h + 1] += ((b12 & 0x000f000fu) - odd) * sign;
    }
  }
};

// uint16: four words in a row.  (Two pieces of two words, 64 apart, would load
// without bank conflicts but with four loads for three: 20.7 against 19.2 ms.)
template <>
struct Lane<kHalves> {
  static constexpr int kN = 4, kStep = 4, kLoads = 3, kDepth = 3;
  uint32_t base;
  __device__ Lane(uint32_t raw, int k, int) : base(raw + 2u * k) {}  // k a multiple of 4
  __device__ void load_first(uint32_t (&x)[kLoads], uint32_t offset) const { load(x, offset); }
  __device__ void load(uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t a = base + 2u * (offset & 0xfffeu);
    x[0] = lds(a);
    x[1] = lds(a + 4);
    x[2] = lds(a + 8);
  }
  __device__ void first(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t sh = 16u * (offset & 1u);
    const uint32_t y0 = __funnelshift_r(x[0], x[1], sh), y1 = __funnelshift_r(x[1], x[2], sh);
    s[0] += y0 & 0xffffu;
    s[1] += y0 >> 16;
    s[2] += y1 & 0xffffu;
    s[3] += y1 >> 16;
  }
  __device__ void move(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t offset,
                       uint32_t sign) const {
    const uint32_t sh = 16u * (offset & 1u);
    const uint32_t y0 = __funnelshift_r(x[0], x[1], sh), y1 = __funnelshift_r(x[1], x[2], sh);
    const uint32_t v1 = y0 >> 16, v2 = y1 & 0xffffu, v3 = y1 >> 16;
    s[0] += (v1 - (y0 & 0xffffu)) * sign;
    s[1] += (v2 - v1) * sign;
    s[2] += (v3 - v2) * sign;
    s[3] += (((x[2] >> sh) & 0xffffu) - v3) * sign;
  }
  __device__ static void store(uint32_t a, const uint32_t (&s)[kN], uint32_t on) {
    store4_if(a, s[0], s[1], s[2], s[3], on);
  }
};

// uint8 decimated by 2 from the input: two pieces of two words, 64 words apart
// (the lanes of a load take consecutive 32-bit words): s[0], s[1] the first
// piece's two decimated samples and those 368 later as 16-bit pairs, s[2], s[3]
// the second's.
template <>
struct Lane<kBytes2> {
  static constexpr int kN = 4, kStep = 2, kLoads = 8, kDepth = 2;
  uint32_t base;
  uint32_t d;  // words from the first piece to the second
  __device__ Lane(uint32_t raw, int k, int rs) : base(raw + 2u * k), d(min(64, rs - 2 - k)) {}
  __device__ void load_first(uint32_t (&x)[kLoads], uint32_t offset) const { load(x, offset); }
  __device__ void load(uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t a = base + 2u * (offset & 0xfffeu), b = a + 2u * d;
    x[0] = lds(a);
    x[1] = lds(a + 4);
    x[2] = lds(a + 2 * kWords);
    x[3] = lds(a + 2 * kWords + 4);
    x[4] = lds(b);
    x[5] = lds(b + 4);
    x[6] = lds(b + 2 * kWords);
    x[7] = lds(b + 2 * kWords + 4);
  }
  // Two decimated samples of four bytes, as a 16-bit pair.
  __device__ static uint32_t decimate(uint32_t y) {
    return (y & 0x00ff00ffu) + __byte_perm(y, 0u, 0x4341);
  }
  __device__ void first(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t offset) const {
    const uint32_t sh = 16u * (offset & 1u);
#pragma unroll
    for (int h = 0; h < 4; ++h) s[h] += decimate(__funnelshift_r(x[2 * h], x[2 * h + 1], sh));
  }
  __device__ void move(uint32_t (&s)[kN], const uint32_t (&x)[kLoads], uint32_t offset,
                       uint32_t sign) const {
    const uint32_t sh = 16u * (offset & 1u);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const uint32_t p = decimate(__funnelshift_r(x[2 * h], x[2 * h + 1], sh));
      const uint32_t q = decimate(x[2 * h + 1] >> sh);
      s[h] += (__byte_perm(p, q, 0x5432) - p) * sign;
    }
  }
  __device__ void store(uint32_t a, const uint32_t (&s)[kN], uint32_t on) const {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %6, 0;\n\t"
        "@p st.shared.v2.u32 [%0], {%2, %3};\n\t@p st.shared.v2.u32 [%1], {%4, %5};\n\t}" ::"r"(a),
        "r"(a + 4u * d), "r"(__byte_perm(s[0], s[1], 0x5410)),
        "r"(__byte_perm(s[0], s[1], 0x7632)), "r"(__byte_perm(s[2], s[3], 0x5410)),
        "r"(__byte_perm(s[2], s[3], 0x7632)), "r"(on)
        : "memory");
  }
};

// One group's rows, by warp bw of a building warpgroup: chunks of 32 kN row
// words, lane l's first one kStep l words on; lanes past the row repeat its last
// words.  Loads run a channel pair, then kDepth moves ahead of the sums.
template <int SRC>
__device__ __forceinline__ void build_rows(const unsigned char* rec, uint32_t raw, uint32_t rows,
                                           int bw, int lane) {
  using L = Lane<SRC>;
  constexpr int kN = L::kN, kDepth = L::kDepth;
  static_assert(kN == format(SRC).build && kDepth <= kStepPad / 2, "planner's lane width");
  const RecHead h = *reinterpret_cast<const RecHead*>(rec);
  for (int chunk = bw; chunk * (32 * kN) < h.rs; chunk += kBuildWarps) {
    const int k0 = min(chunk * (32 * kN) + L::kStep * lane, h.rs - L::kStep);
    const L win(raw, k0, h.rs);
    const uint32_t rs4 = 4u * h.rs;
    uint32_t dst = rows + 4u * k0;
    uint32_t s[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j) s[j] = 0u;
    {
      // Channel pairs, the next pair's loads ahead (three-input adds; one
      // channel at a time with loads four ahead ran a quarter slower).
      const uint32_t* pairs = reinterpret_cast<const uint32_t*>(rec + sizeof(RecHead));
      const int np = h.k / 2;
      uint32_t a0[L::kLoads], a1[L::kLoads], b0[L::kLoads], b1[L::kLoads];
      uint32_t oa = pairs[0], ob = pairs[min(1, max(np - 1, 0))];
      win.load_first(a0, oa & 0xffffu);
      win.load_first(a1, oa >> 16);
#pragma unroll 1
      for (int q = 0; q < np; q += 2) {
        win.load_first(b0, ob & 0xffffu);
        win.load_first(b1, ob >> 16);
        const uint32_t na = pairs[min(q + 2, np - 1)], nb = pairs[min(q + 3, np - 1)];
        win.first(s, a0, oa);
        win.first(s, a1, oa >> 16);
        oa = na;
        win.load_first(a0, oa & 0xffffu);
        win.load_first(a1, oa >> 16);
        if (q + 1 < np) {
          win.first(s, b0, ob);
          win.first(s, b1, ob >> 16);
        }
        ob = nb;
      }
      if (h.k & 1) {
        oa = reinterpret_cast<const uint16_t*>(pairs)[h.k - 1];
        win.load_first(a0, oa);
        win.first(s, a0, oa);
      }
    }
    win.store(dst, s, 1u);
    dst += rs4;
    const uint32_t* steps = reinterpret_cast<const uint32_t*>(rec + rec_steps_off(h.k));
    uint32_t x[kDepth][L::kLoads], st[kDepth], nx[kDepth];
#pragma unroll
    for (int e = 0; e < kDepth; ++e) st[e] = steps[e];
#pragma unroll
    for (int e = 0; e < kDepth; ++e) win.load(x[e], st[e]);
#pragma unroll
    for (int e = 0; e < kDepth; ++e) nx[e] = steps[kDepth + e];
#pragma unroll 1
    for (int q = 0; q < h.n_steps; q += kDepth) {
      steps += kDepth;
#pragma unroll
      for (int e = 0; e < kDepth; ++e) {
        win.move(s, x[e], st[e], static_cast<uint32_t>(static_cast<int32_t>(st[e]) >> 30));
        const uint32_t on = st[e] & kStepEmit;
        win.load(x[e], nx[e]);
        st[e] = nx[e];
        nx[e] = steps[kDepth + e];
        win.store(dst, s, on);
        dst += on ? rs4 : 0u;
      }
    }
  }
}

// Copies of group g (directory entry e, this lane's window start) into slot
// g % kSlots, by adding warp w: lane i < 4 the window of channel w + 8 i, warp
// 0 the record too.  A bulk copy takes its warp about 130 cycles whatever its
// size, so the copies are spread over the adding warps.  (8192 channels, from
// the packed copy, before the votes: 67.7 ms; one building warp per warpgroup
// issuing all of them 68.0 ms, half by each 73.1 ms; from the input itself 78.3,
// 85.3 and 85.7 ms.)
// VOTE: also the warp's vote on the wait before it (`ok` of each lane; false
// where any lane gave up, and then nothing is issued).
static_assert(kMaxK <= 4 * kMainWarps, "four channels per adding warp");
template <int SRC, bool VOTE>
__device__ __forceinline__ bool issue_copies(const Params& p, unsigned char* smem, Ctl* ctl,
                                             int64_t w0, int g, const Dir& e, int32_t start,
                                             bool ok = true) {
  if (g == p.hold_stage) return VOTE ? __all_sync(0xffffffffu, ok) : true;
  constexpr int kBits = format(SRC).bits;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, slot = g % kSlots;
  const uint32_t bar = smem_u32(&ctl->raw_full[slot]);
  const int ch = w + kMainWarps * lane;
  const uint32_t row_bytes = static_cast<uint32_t>(e.lw) * kBits / 8;
  const int64_t at = w0 + start - p.x_origin;
  uint32_t bytes = 0;
  if (lane < 4 && ch < e.k && at >= 0 && at < p.stride)
    bytes = static_cast<uint32_t>(
        min(static_cast<int64_t>(row_bytes), (p.stride - at) * kBits / 8));
  constexpr uint32_t kGaveUp = 1u << 24;  // above any sum of bytes, 32 of them below 2^32
  static_assert(format(SRC).raw_bytes < kGaveUp, "byte counts and votes share a word");
  const uint32_t total = __reduce_add_sync(0xffffffffu, VOTE && !ok ? kGaveUp : bytes);
  if (VOTE && total >= kGaveUp) return false;
  // The slot's last readers were ordinary loads.
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (lane == 0) {
    const uint32_t rec = w == 0 ? e.rec_n16 * 16u : 0u;
    mbar_arrive_expect(bar, total + rec);
    if (w == 0) {
      ctl->issued[slot] = g + 1;
      bulk_copy(smem_u32(smem + kRecOff + slot * kRecBytes),
                p.tables + static_cast<size_t>(e.rec16) * 16, rec, bar);
    }
  }
  __syncwarp();
  if (bytes)
    bulk_copy(smem_u32(smem + kRawOff + slot * static_cast<size_t>(format(SRC).raw_bytes)) +
                  ch * row_bytes,
              static_cast<const unsigned char*>(p.x) +
                  (static_cast<int64_t>(e.c0 + ch) * p.stride + at) * kBits / 8,
              bytes, bar);
  return true;
}

// Building warpgroup wg: channel groups wg, wg + 2, ...  Its last warp, which
// has no chunk where rows are at most three chunks long, also prepares what
// the adders need: the DMs' row addresses, the flush flag, the copies to issue.
template <int SRC>
__device__ __forceinline__ void build(const Params& p, unsigned char* smem, Ctl* ctl,
                                      int n_groups) {
  const int wg = (threadIdx.x - 32 * kMainWarps) / (32 * kBuildWarps);
  const int bw = (threadIdx.x >> 5) % kBuildWarps, lane = threadIdx.x & 31;
  constexpr size_t kRows = row_off(SRC), kRowBytes = static_cast<size_t>(format(SRC).row_words) * 4;
  for (int g = wg; g < n_groups; g += kBuildGroups) {
    const int slot = g % kSlots;
    const bool ok = wait_or_abort(smem_u32(&ctl->rows_empty[slot]), ((g / kSlots) & 1) ^ 1, ctl) &&
                    wait_copies(p, ctl, g);
    if (!__all_sync(0xffffffffu, ok)) {
      ctl->abort = 1;
      return;
    }
    const unsigned char* rec = smem + kRecOff + slot * kRecBytes;
    if (bw == kBuildWarps - 1) {
      const RecHead* h = reinterpret_cast<const RecHead*>(rec);
      const uint16_t* offs =
          reinterpret_cast<const uint16_t*>(rec + rec_offs_off(h->k, h->n_steps));
      const uint32_t* next = reinterpret_cast<const uint32_t*>(offs + kDm);
      uint32_t* dst = reinterpret_cast<uint32_t*>(smem + kOffsOff + slot * kOffsBytes);
#pragma unroll
      for (int d = lane; d < kDm; d += 32)
        dst[d] = static_cast<uint32_t>(kRows + slot * kRowBytes) + 4u * offs[d];
      if (lane < 4) dst[kNextDir + lane] = next[lane];
      dst[kNextStart + lane] = next[4 + lane];
      if (lane == 0) dst[kDm] = h->flush;
    }
    build_rows<SRC>(rec,
                    smem_u32(smem + kRawOff + slot * static_cast<size_t>(format(SRC).raw_bytes)),
                    smem_u32(smem + kRows + slot * kRowBytes), bw, lane);
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ctl->rows_full[slot]));
  }
}

// The adding warps: DMs 16 w .. 16 w + 15 of the block.
template <int SRC>
__device__ __forceinline__ void add_and_store(const Params& p, unsigned char* smem, Ctl* ctl,
                                              int blk, int64_t w0, int g0, int n_groups) {
  constexpr bool LANES16 = lanes16(SRC);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t col = LANES16 ? tmem::warp_columns(ctl->tmem, w, 256) : 0u;
  uint32_t acc[kDmPairs][kAcc];
#pragma unroll
  for (int i = 0; i < kDmPairs; ++i)
#pragma unroll
    for (int j = 0; j < kAcc; ++j) acc[i][j] = 0u;
  bool flushed = false;
  const unsigned char* lane_smem = smem + 4 * lane;
  // The word the two DMs of a pair share: lanes below 16 take the first DM's.
  const unsigned char* tail_smem = smem + 4 * (32 * kFull + (lane & 15));
  // The first groups' copies; later ones follow while group g - kSlots is
  // added (its rows are built, so its slot is free).
  {
    const Dir* dir = reinterpret_cast<const Dir*>(p.tables + p.off_dir) + g0;
    const int32_t* starts = reinterpret_cast<const int32_t*>(p.tables + p.off_start) +
                            static_cast<int64_t>(blk) * p.n_chan;
    const int ch = w + kMainWarps * lane;
    for (int g = 0; g < min(kSlots, n_groups); ++g) {
      const int4 v = __ldg(reinterpret_cast<const int4*>(dir + g));
      const Dir e = *reinterpret_cast<const Dir*>(&v);
      issue_copies<SRC, false>(p, smem, ctl, w0, g, e, ch < e.k ? __ldg(starts + e.c0 + ch) : 0);
    }
  }
  for (int g = 0; g < n_groups; ++g) {
    const int slot = g % kSlots;
    bool ok = wait_or_abort(smem_u32(&ctl->rows_full[slot]), (g / kSlots) & 1, ctl);
    const uint32_t* offs = reinterpret_cast<const uint32_t*>(smem + kOffsOff + slot * kOffsBytes);
    const bool flush = LANES16 && offs[kDm] != 0u;
    if (g + kSlots < n_groups) {
      const uint4 v = *reinterpret_cast<const uint4*>(offs + kNextDir);
      const Dir e = *reinterpret_cast<const Dir*>(&v);
      const int ch = min(w + kMainWarps * lane, kMaxK - 1);
      ok = issue_copies<SRC, true>(p, smem, ctl, w0, g + kSlots, e,
                                   static_cast<int32_t>(offs[kNextStart + ch]), ok);
    } else {
      ok = __all_sync(0xffffffffu, ok);
    }
    if (!ok) {
      ctl->issued_by[w] = min(g + kSlots, n_groups);
      ctl->abort = 1;
      return;
    }
#pragma unroll
    for (int i = 0; i < kDmPairs; ++i) {
      const uint2 o = *reinterpret_cast<const uint2*>(offs + kDmWarp * w + 2 * i);
      const uint32_t* a = reinterpret_cast<const uint32_t*>(lane_smem + o.x);
      const uint32_t* b = reinterpret_cast<const uint32_t*>(lane_smem + o.y);
#pragma unroll
      for (int j = 0; j < kFull; ++j) acc[i][j] += a[32 * j];
#pragma unroll
      for (int j = 0; j < kFull; ++j) acc[i][kFull + j] += b[32 * j];
      acc[i][2 * kFull] +=
          *reinterpret_cast<const uint32_t*>(tail_smem + (lane < 16 ? o.x : o.y));
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ctl->rows_empty[slot]));
    if constexpr (LANES16) {
      if (flush) {
        __syncwarp();
        flush_lanes(col, acc, !flushed);
        flushed = true;
      }
    }
  }
  if (lane == 0) ctl->issued_by[w] = n_groups;
  // Word k of the tile holds output w0 + k and, in 16-bit lanes, that plus the
  // pair distance.
  const int64_t lim = p.t_end - w0;
  auto put = [&](int d, int k, uint32_t a, uint32_t hi) {
    const int64_t dm = static_cast<int64_t>(blk) * kDm + d;
    if (dm >= p.n_dm) return;
    int32_t* row = p.out + dm * p.out_stride + w0;
    if constexpr (LANES16) {
      if (k < lim) row[k] = static_cast<int32_t>((a & 0xffffu) + ((hi & 0xffffu) << 8));
      if (k + pair_dist(SRC) < lim)
        row[k + pair_dist(SRC)] = static_cast<int32_t>((a >> 16) + ((hi >> 16) << 8));
    } else {
      if (k < lim) row[k] = static_cast<int32_t>(a);
    }
  };
#pragma unroll
  for (int q = 0; q < kDmPairs * kAcc; q += 8) {
    uint32_t v[8] = {};
    if (LANES16 && flushed) {
      __syncwarp();
      tmem::load(col + q, v);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int i = (q + e) / kAcc, j = (q + e) % kAcc;
      const int d = kDmWarp * w + 2 * i;
      if (j < kFull) put(d, 32 * j + lane, acc[i][j], v[e]);
      else if (j < 2 * kFull) put(d + 1, 32 * (j - kFull) + lane, acc[i][j], v[e]);
      else put(d + (lane >> 4), 32 * kFull + (lane & 15), acc[i][j], v[e]);
    }
  }
}

template <int SRC>
__device__ __forceinline__ void init_barriers(Ctl* ctl) {
  for (int s = 0; s < kSlots; ++s) {
    mbar_init(smem_u32(&ctl->raw_full[s]), kMainWarps);
    mbar_init(smem_u32(&ctl->rows_full[s]), kBuildWarps);
    mbar_init(smem_u32(&ctl->rows_empty[s]), kMainWarps);
    ctl->issued[s] = 0;
  }
  ctl->abort = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// First output sample of half half0 + i (368 words) of the time axis.  Halves
// of packed-copy tiles (736 words, 1472 samples; half0 even) interleave; the
// others are in order.  (32-bit unsigned i: a signed 64-bit division here cost
// the adders' registers, 12 % of the kernel.)
template <int SRC>
__device__ __forceinline__ int64_t half_origin(int64_t half0, uint32_t i) {
  if constexpr (SRC == kPairs)
    return half0 * kPairWords + static_cast<int64_t>(i / 2) * (2 * kPairWords) + (i % 2) * kWords;
  else return (half0 + i) * (lanes16(SRC) ? 2 * kWords : kWords);
}

template <int SRC>
__global__ void __launch_bounds__(kThreads, 1) sum_row_kernel(const __grid_constant__ Params p) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr bool LANES16 = lanes16(SRC);
  Ctl* ctl = reinterpret_cast<Ctl*>(smem);
  if (threadIdx.x == 0) init_barriers<SRC>(ctl);
  if constexpr (LANES16) {
    if (threadIdx.x < 32) tmem::alloc(smem_u32(&ctl->tmem));
    tmem::fence_before();
  }
  __syncthreads();
  if constexpr (LANES16) tmem::fence_after();
  const int blk = blockIdx.x % static_cast<uint32_t>(p.n_blocks);
  const int64_t w0 = half_origin<SRC>(p.half0, blockIdx.x / static_cast<uint32_t>(p.n_blocks));
  const int32_t* first = reinterpret_cast<const int32_t*>(p.tables);
  const int g0 = first[blk], n_groups = first[blk + 1] - g0;
  // 256 x 208 + 256 x 48 registers: the 512 x 128 of the launch.
  if (threadIdx.x >= 32 * kMainWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
    build<SRC>(p, smem, ctl, n_groups);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    add_and_store<SRC>(p, smem, ctl, blk, w0, g0, n_groups);
  }
  if constexpr (LANES16) tmem::fence_before();
  __syncthreads();
  if (ctl->abort && threadIdx.x == 0) {
    atomicOr(p.err, tk::kErrTimeout);
    drain_copies(p, ctl);
  }
  if constexpr (LANES16) {
    tmem::fence_after();
    __syncwarp();
    if (threadIdx.x < 32) tmem::dealloc(ctl->tmem);
  }
}

// All threads of the CTA, from either role.
__device__ __forceinline__ void cta_sync() {
  asm volatile("barrier.cta.sync 0, %0;" ::"n"(kThreads) : "memory");
}

// Persistent kernel: the CTAs take (job, DM block, half) items from a counter;
// the job's parameters are copied into shared memory and the barriers made
// anew for every item.
struct BatchCtl {
  Ctl ctl;
  int32_t item;
  Params p;
};
static_assert(sizeof(BatchCtl) <= kRecOff, "control block too large");

template <int SRC>
__global__ void __launch_bounds__(kThreads, 1) sum_row_batch_kernel(const BatchArgs b) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr bool LANES16 = lanes16(SRC);
  BatchCtl* bc = reinterpret_cast<BatchCtl*>(smem);
  Ctl* ctl = &bc->ctl;
  if constexpr (LANES16) {
    if (threadIdx.x < 32) tmem::alloc(smem_u32(&ctl->tmem));
    tmem::fence_before();
  }
  // The next item, or false: none is left or the last one was given up.
  bool fresh = true;
  auto next_item = [&]() {
    cta_sync();  // the previous item is done (and, the first time, tensor memory allocated)
    const bool aborted = !fresh && ctl->abort;
    if (threadIdx.x == 0) {
      if (!fresh) {
        if (aborted) {
          atomicOr(bc->p.err, tk::kErrTimeout);
          drain_copies(bc->p, ctl);
        }
        for (int s = 0; s < kSlots; ++s) {
          mbar_inval(smem_u32(&ctl->raw_full[s]));
          mbar_inval(smem_u32(&ctl->rows_full[s]));
          mbar_inval(smem_u32(&ctl->rows_empty[s]));
        }
      }
      const int it = aborted ? b.n_items : static_cast<int>(atomicAdd(b.counter, 1u));
      bc->item = it;
      if (it < b.n_items) bc->p = b.jobs[b.items[it].job];
    }
    cta_sync();  // every thread has read the abort flag; the item is known
    if (threadIdx.x == 0) init_barriers<SRC>(ctl);
    cta_sync();
    fresh = false;
    return bc->item < b.n_items;
  };
  auto unit = [&](int* blk, int64_t* w0, int* g0, int* n_groups) {
    const tk::BatchItem item = b.items[bc->item];
    const int32_t* first = reinterpret_cast<const int32_t*>(bc->p.tables);
    *blk = item.blk;
    *w0 = half_origin<SRC>(bc->p.half0, static_cast<uint32_t>(item.tile));
    *g0 = first[item.blk];
    *n_groups = first[item.blk + 1] - *g0;
  };
  int blk, g0, n_groups;
  int64_t w0;
  if (threadIdx.x >= 32 * kMainWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
    while (next_item()) {
      unit(&blk, &w0, &g0, &n_groups);
      build<SRC>(bc->p, smem, ctl, n_groups);
      __syncwarp();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    while (next_item()) {
      if constexpr (LANES16) tmem::fence_after();
      unit(&blk, &w0, &g0, &n_groups);
      add_and_store<SRC>(bc->p, smem, ctl, blk, w0, g0, n_groups);
      __syncwarp();
    }
  }
  if constexpr (LANES16) {
    tmem::fence_before();
    __syncthreads();
    tmem::fence_after();
    __syncwarp();
    if (threadIdx.x < 32) tmem::dealloc(ctl->tmem);
  }
}

template <int SRC>
int launch(const Params& prm, int64_t grid, cudaStream_t st) {
  auto kern = sum_row_kernel<SRC>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem_bytes(SRC)));
  if (e != cudaSuccess) return static_cast<int>(e);
  kern<<<static_cast<unsigned>(grid), kThreads, smem_bytes(SRC), st>>>(prm);
  return static_cast<int>(cudaGetLastError());
}

template <int SRC>
int launch_batch(const BatchArgs& args, int32_t grid, cudaStream_t st) {
  auto kern = sum_row_batch_kernel<SRC>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem_bytes(SRC)));
  if (e != cudaSuccess) return static_cast<int>(e);
  kern<<<static_cast<unsigned>(grid), kThreads, smem_bytes(SRC), st>>>(args);
  return static_cast<int>(cudaGetLastError());
}

}  // namespace sr

sr::Params sum_row_params(const dd_plan_s* p, const RangePlan& rp, const SumTables& sums,
                          const void* tables, int32_t* err, const void* d_rows, int64_t stride,
                          void* d_out, int64_t t_end, int64_t out_stride) {
  sr::Params prm{};
  prm.x = d_rows;
  // In staged samples: the decimated ones of a row (a partial one at its end
  // holds no output's sample).
  prm.stride = sums.src == sr::kBytes2 ? stride / 2 : stride;
  prm.n_chan = p->n_chan;
  prm.n_dm = static_cast<int32_t>(rp.n_dm);
  prm.n_blocks = sums.n_blocks;
  prm.tables = static_cast<const unsigned char*>(tables);
  prm.off_dir = sums.off_dir;
  prm.off_start = sums.off_start;
  prm.t_end = t_end;
  prm.out_stride = out_stride;
  prm.out = static_cast<int32_t*>(d_out);
  prm.err = err;
  prm.wait_iters = p->wait_iters;
  prm.hold_stage = p->hold_stage;
  return prm;
}

int64_t sum_row_halves(int src, int64_t t_begin, int64_t t_end) {
  const int64_t half = sr::kWords * (sr::lanes16(src) ? 2 : 1);
  if (src != sr::kPairs) return (t_end + half - 1) / half - t_begin / half;
  // A half of a packed-copy tile holds its first 368 samples and those 736
  // later: the last tile's second half only counts where the tile has more
  // than 368 outputs.
  const int64_t ts = 2 * half, whole = t_end / ts - t_begin / ts, rest = t_end % ts;
  return 2 * whole + (rest > sr::kWords ? 2 : rest > 0 ? 1 : 0);
}

int launch_sum_row_batch(int src, const sr::BatchArgs& args, int32_t grid, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  switch (src) {
    case sr::kPairs: return sr::launch_batch<sr::kPairs>(args, grid, st);
    case sr::kBytes: return sr::launch_batch<sr::kBytes>(args, grid, st);
    case sr::kNibbles: return sr::launch_batch<sr::kNibbles>(args, grid, st);
    case sr::kHalves: return sr::launch_batch<sr::kHalves>(args, grid, st);
    case sr::kBytes2: return sr::launch_batch<sr::kBytes2>(args, grid, st);
  }
  return static_cast<int>(cudaErrorInvalidValue);
}

int launch_forward_sum_rows(const dd_plan_s* p, const RangePlan& rp, const SumTables& sums,
                            const void* tables, int32_t* err, const void* d_rows, int64_t stride, void* d_out,
                            int64_t t_begin, int64_t t_end, void* stream, int64_t out_stride,
                            int64_t x_origin) {
  const int src = sums.src;
  const int64_t half = sr::kWords * (sr::lanes16(src) ? 2 : 1);
  if (x_origin < 0 || x_origin % sr::format(src).align != 0 || t_begin < 0 ||
      t_begin % (src == sr::kPairs ? 2 * half : half) != 0 || t_end <= t_begin)
    return static_cast<int>(cudaErrorInvalidValue);
  sr::Params prm =
      sum_row_params(p, rp, sums, tables, err, d_rows, stride, d_out, t_end, out_stride);
  prm.x_origin = x_origin;
  prm.half0 = t_begin / half;
  const int64_t halves = sum_row_halves(src, t_begin, t_end);
  const int64_t grid = halves * prm.n_blocks;
  if (grid <= 0 || grid > 0x7fffffffLL) return static_cast<int>(cudaErrorInvalidConfiguration);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  switch (src) {
    case sr::kPairs: return sr::launch<sr::kPairs>(prm, grid, st);
    case sr::kBytes: return sr::launch<sr::kBytes>(prm, grid, st);
    case sr::kNibbles: return sr::launch<sr::kNibbles>(prm, grid, st);
    case sr::kHalves: return sr::launch<sr::kHalves>(prm, grid, st);
    case sr::kBytes2: return sr::launch<sr::kBytes2>(prm, grid, st);
  }
  return static_cast<int>(cudaErrorInvalidValue);
}

}  // namespace dd
