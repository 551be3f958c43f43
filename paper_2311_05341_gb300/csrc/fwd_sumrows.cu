// fwd_sumrows.cu -- the sum-row tile (sumrows.h): Eq. 3 for 128 trial DMs x
// 368 packed words per CTA, from a packed copy of integer input.
//
// Roles.  Two warpgroups build, taking channel groups in turn: they stage the
// windows of a group of K adjacent channels (one bulk copy per channel, three
// slots), sum them into the group's first row, turn each row into the next by
// replacing the windows of the channels whose shift difference changed, and
// store every row to one of three row buffers.  Eight warps add: each owns 16
// DMs x 368 words in 184 accumulator registers per lane and adds, per DM and
// word, one word of the DM's row.  Builders and adders hand buffers over
// through mbarriers.  The registers are split unevenly (setmaxnreg): 208 per
// adding thread, 48 per building thread, of the 128 x 512 the CTA is launched
// with.
//
// What bounds it: the shared-memory pipe (128 bytes per clock and SM).  Per
// group and CTA the adders read 128 x 368 words; the builders read about
// (K + 1.2 moves) x W words and write rows x W, W = 368 + the block's delay
// span.  The planner picks K per group to make the sum per channel smallest:
// 5200 words at 8192 channels and 4096 trials (K = 15, 18 rows, 22 moves on
// average), where the pattern tile moves 12000.  Measured there: 68.0 ms per
// launch against 153.5 ms (uint8, 262144 samples); per group 3600 cycles, of
// which the adders wait 890.  One building warpgroup with two buffers and
// groups of 22 channels ran 90 ms: a warp's chain of moves (about 130 cycles
// each, shared-memory latency behind the adders' loads) was longer than the
// adders' work.
//
// 16-bit lanes (two samples per word): before they can overflow, the adders
// move the lanes' high bytes to tensor memory (16-bit sums of high bytes, 184
// words per thread), so partial sums never leave the SM and every output is
// stored once.
//
// Every mbarrier wait is bounded; on timeout the CTA sets kErrTimeout, waits
// for its copies, frees its tensor memory and stores nothing.
#include <cuda_runtime.h>

#include <cstdint>

#include "dd_internal.h"
#include "sumrows.h"
#include "tile_common.cuh"

namespace dd {
namespace sr {

using tk::bulk_copy;
using tk::mbar_arrive_expect;
using tk::mbar_init;
using tk::smem_u32;

// Shared-memory control block (the first 256 bytes).
struct Ctl {
  uint64_t raw_full[kSlots];    // the slot's copies have landed
  uint64_t raw_empty[kSlots];   // its builders have read them
  uint64_t rows_full[kSlots];   // the buffer's rows are built
  uint64_t rows_empty[kSlots];  // the adders have read them
  uint32_t tmem;
  volatile int32_t abort;           // a wait gave up: every role leaves
  volatile int32_t issued[kSlots];  // group + 1 whose copies were last issued into the slot
};
static_assert(sizeof(Ctl) <= kRecOff, "control block too large");

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Bounded wait that also ends when the CTA is aborting.
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, const Ctl* ctl) {
  for (int it = 0; it < tk::kWaitIters; it += 64) {
    if (tk::mbar_wait(bar, parity, 64)) return true;
    if (ctl->abort) return false;
  }
  return false;
}

// Bounded wait for the copies of group g.  A parity wait only tells a phase
// from the one before it, and the slot's previous group belongs to the other
// warpgroup: the wait starts once the copies of g are issued, which follows
// the end of that group.
__device__ __forceinline__ bool wait_copies(const Params& p, Ctl* ctl, int g) {
  const int slot = g % kSlots;
  for (int it = 0; ctl->issued[slot] <= g; ++it)
    if (it >= p.wait_iters || ctl->abort) return false;
  return tk::mbar_wait(smem_u32(&ctl->raw_full[slot]), (g / kSlots) & 1, p.wait_iters);
}

// Tensor memory: all 512 columns (the tile's shared memory admits one CTA per
// SM); thread t of a warp reaches lane 32 (warp % 4) + t.
__device__ __forceinline__ void tmem_alloc(uint32_t dst) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(dst)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t addr) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_load8(uint32_t addr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                 "=r"(v[6]), "=r"(v[7])
               : "r"(addr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_store8(uint32_t addr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(
                   addr),
               "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]),
               "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_stores() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

constexpr int kPairs = kDmWarp / 2;
static_assert(kPairs * kAcc % 8 == 0, "tensor memory moves 8 words at a time");

// The high bytes of the 16-bit lanes into tensor memory: lane word a becomes
// its low bytes, and the 16-bit sums of high bytes at the word's column grow
// by a >> 8 (below 2^16 while the total is below 2^24).
__device__ __forceinline__ void flush_lanes(uint32_t col, uint32_t (&acc)[kPairs][kAcc],
                                            bool first) {
#pragma unroll
  for (int q = 0; q < kPairs * kAcc; q += 8) {
    uint32_t v[8] = {};
    if (!first) tmem_load8(col + q, v);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      uint32_t& a = acc[(q + e) / kAcc][(q + e) % kAcc];
      v[e] += __byte_perm(a, 0u, 0x4341);
      a &= 0x00ff00ffu;
    }
    tmem_store8(col + q, v);
  }
  tmem_wait_stores();
}

__device__ __forceinline__ uint32_t lds(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}

// kBuild words of a row, where `on` is not zero (predicated: no branch).
__device__ __forceinline__ void store_row_if(uint32_t a, const uint32_t (&s)[kBuild],
                                             uint32_t on) {
  static_assert(kBuild == 5, "five words per lane");
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %6, 0;\n\t"
      "@p st.shared.u32 [%0], %1;\n\t@p st.shared.u32 [%0+4], %2;\n\t"
      "@p st.shared.u32 [%0+8], %3;\n\t@p st.shared.u32 [%0+12], %4;\n\t"
      "@p st.shared.u32 [%0+16], %5;\n\t}" ::"r"(a),
      "r"(s[0]), "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(on)
      : "memory");
}

template <int N>
__device__ __forceinline__ void load_words(uint32_t (&x)[N], uint32_t a) {
#pragma unroll
  for (int j = 0; j < N; ++j) x[j] = lds(a + 4 * j);
}

// One group's rows, by warp bw of a building warpgroup: chunks of 160 row
// words, lane l words 5 l .. 5 l + 4 (scalar accesses at an odd lane stride:
// no bank conflicts).  Lanes past the row repeat its last five words.  Loads
// run one channel pair, then kDepth moves ahead of the sums.
__device__ __forceinline__ void build_rows(const unsigned char* rec, uint32_t raw, uint32_t rows,
                                           int bw, int lane) {
  constexpr int kDepth = 2;
  const RecHead h = *reinterpret_cast<const RecHead*>(rec);
  for (int chunk = bw; chunk * kChunk < h.rs; chunk += kBuildWarps) {
    const uint32_t w0 = 4u * min(chunk * kChunk + kBuild * lane, h.rs - kBuild);
    const uint32_t src = raw + w0, rs4 = 4u * h.rs;
    uint32_t dst = rows + w0;
    uint32_t s[kBuild];
#pragma unroll
    for (int j = 0; j < kBuild; ++j) s[j] = 0u;
    const uint32_t* steps = reinterpret_cast<const uint32_t*>(rec + rec_steps_off(h.k));
    {
      const uint32_t* pairs = reinterpret_cast<const uint32_t*>(rec + sizeof(RecHead));
      const int np = h.k / 2;
      uint32_t a0[kBuild], a1[kBuild], b0[kBuild], b1[kBuild];
      uint32_t o = pairs[0];
      load_words(a0, src + (o & 0xffffu));
      load_words(a1, src + (o >> 16));
      o = pairs[1];  // past the last pair: padding (window 0) or the moves
#pragma unroll 1
      for (int q = 0; q < np; q += 2) {
        const bool two = q + 1 < np;
        const uint32_t ob = two ? o : 0u;
        load_words(b0, src + (ob & 0xffffu));
        load_words(b1, src + (ob >> 16));
        o = pairs[min(q + 2, np - 1)];
#pragma unroll
        for (int j = 0; j < kBuild; ++j) s[j] += a0[j] + a1[j];
        load_words(a0, src + (o & 0xffffu));
        load_words(a1, src + (o >> 16));
        o = pairs[min(q + 3, np - 1)];
        if (two) {
#pragma unroll
          for (int j = 0; j < kBuild; ++j) s[j] += b0[j] + b1[j];
        }
      }
      if (h.k & 1) {
        load_words(a0, src + reinterpret_cast<const uint16_t*>(pairs)[h.k - 1]);
#pragma unroll
        for (int j = 0; j < kBuild; ++j) s[j] += a0[j];
      }
    }
    store_row_if(dst, s, 1u);
    dst += rs4;
    uint32_t x[kDepth][kBuild + 1], st[kDepth], nx[kDepth];
#pragma unroll
    for (int e = 0; e < kDepth; ++e) st[e] = steps[e];
#pragma unroll
    for (int e = 0; e < kDepth; ++e) load_words(x[e], src + (st[e] & 0xffffu));
#pragma unroll
    for (int e = 0; e < kDepth; ++e) nx[e] = steps[kDepth + e];
#pragma unroll 1
    for (int q = 0; q < h.n_steps; q += kDepth) {
      steps += kDepth;
#pragma unroll
      for (int e = 0; e < kDepth; ++e) {
        const uint32_t sign = static_cast<uint32_t>(static_cast<int32_t>(st[e]) >> 30);
#pragma unroll
        for (int j = 0; j < kBuild; ++j) s[j] += (x[e][j + 1] - x[e][j]) * sign;
        const uint32_t on = st[e] & kStepEmit;
        load_words(x[e], src + (nx[e] & 0xffffu));
        st[e] = nx[e];
        nx[e] = steps[kDepth + e];
        store_row_if(dst, s, on);
        dst += on ? rs4 : 0u;
      }
    }
  }
}

// Building warpgroup wg: channel groups wg, wg + 2, ...  Its last warp also
// issues the copies and writes the DMs' row addresses: it only builds where
// rows are longer than three chunks.
__device__ __forceinline__ void build(const Params& p, unsigned char* smem, Ctl* ctl, int blk,
                                      int64_t w0, int g0, int n_groups) {
  const int wg = (threadIdx.x - 32 * kMainWarps) / (32 * kBuildWarps);
  const int bw = (threadIdx.x >> 5) % kBuildWarps, lane = threadIdx.x & 31;
  const bool feeder = bw == kBuildWarps - 1;
  const Dir* dir = reinterpret_cast<const Dir*>(p.tables + p.off_dir) + g0;
  const int32_t* starts = reinterpret_cast<const int32_t*>(p.tables + p.off_start) +
                          static_cast<int64_t>(blk) * p.n_chan;
  // Copies of group g into slot g % kSlots: lane i < K the window of channel
  // i, lane 0 the record too.
  static_assert(kMaxK <= 32, "one lane per channel");
  auto issue = [&](int g) {
    if (g >= n_groups || g == p.hold_stage) return;
    const int slot = g % kSlots;
    const uint32_t bar = smem_u32(&ctl->raw_full[slot]);
    const int4 v = __ldg(reinterpret_cast<const int4*>(dir + g));
    const Dir e = *reinterpret_cast<const Dir*>(&v);
    uint32_t bytes = 0;
    int64_t at = 0;
    if (lane < e.k) {
      at = w0 + __ldg(starts + e.c0 + lane) - p.x_origin;
      if (at >= 0 && at < p.stride)
        bytes = static_cast<uint32_t>(min(static_cast<int64_t>(e.lw), p.stride - at)) * 4u;
      at += static_cast<int64_t>(e.c0 + lane) * p.stride;
    }
    const uint32_t total = __reduce_add_sync(0xffffffffu, bytes) + e.rec_n16 * 16u;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (lane == 0) {
      mbar_arrive_expect(bar, total);
      ctl->issued[slot] = g + 1;
      bulk_copy(smem_u32(smem + kRecOff + slot * kRecBytes),
                p.tables + static_cast<size_t>(e.rec16) * 16, e.rec_n16 * 16u, bar);
    }
    __syncwarp();
    const uint32_t dst = smem_u32(smem + kRawOff + slot * (size_t{kRawWords} * 4));
    if (bytes) bulk_copy(dst + lane * (e.lw * 4u), p.x + at, bytes, bar);
  };
  if (feeder)
    for (int g = wg; g < kSlots; g += kBuildGroups) issue(g);
  for (int g = wg; g < n_groups; g += kBuildGroups) {
    const int slot = g % kSlots;
    const uint32_t parity = (g / kSlots) & 1;
    if (!wait_copies(p, ctl, g) ||
        !wait_or_abort(smem_u32(&ctl->rows_empty[slot]), parity ^ 1, ctl)) {
      if (lane == 0) {
        atomicOr(p.err, tk::kErrTimeout);
        ctl->abort = 1;
      }
      return;
    }
    const unsigned char* rec = smem + kRecOff + slot * kRecBytes;
    if (feeder) {
      // Row addresses of the DMs (bytes from the start of shared memory) and
      // the flush flag.
      const RecHead* h = reinterpret_cast<const RecHead*>(rec);
      const uint16_t* offs =
          reinterpret_cast<const uint16_t*>(rec + rec_offs_off(h->k, h->n_steps));
      uint32_t* dst = reinterpret_cast<uint32_t*>(smem + kOffsOff + slot * kOffsBytes);
#pragma unroll
      for (int d = lane; d < kDm; d += 32)
        dst[d] = static_cast<uint32_t>(kRowOff + slot * (size_t{kRowWords} * 4)) + 4u * offs[d];
      if (lane == 0) dst[kDm] = h->flush;
    }
    build_rows(rec, smem_u32(smem + kRawOff + slot * (size_t{kRawWords} * 4)),
               smem_u32(smem + kRowOff + slot * (size_t{kRowWords} * 4)), bw, lane);
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(smem_u32(&ctl->rows_full[slot]));
      mbar_arrive(smem_u32(&ctl->raw_empty[slot]));
    }
    if (feeder && g + kSlots < n_groups) {
      if (!wait_or_abort(smem_u32(&ctl->raw_empty[slot]), parity, ctl)) {
        if (lane == 0) {
          atomicOr(p.err, tk::kErrTimeout);
          ctl->abort = 1;
        }
        return;
      }
      issue(g + kSlots);
    }
  }
}

// The adding warps: DMs 16 w .. 16 w + 15 of the block.
template <bool LANES16>
__device__ __forceinline__ void add_and_store(const Params& p, unsigned char* smem, Ctl* ctl,
                                              int blk, int64_t w0, int n_groups) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t col =
      LANES16 ? ctl->tmem + (static_cast<uint32_t>(32 * (w & 3)) << 16) + 256u * (w >> 2) : 0u;
  uint32_t acc[kPairs][kAcc];
#pragma unroll
  for (int i = 0; i < kPairs; ++i)
#pragma unroll
    for (int j = 0; j < kAcc; ++j) acc[i][j] = 0u;
  bool flushed = false;
  const unsigned char* lane_smem = smem + 4 * lane;
  // The word the two DMs of a pair share: lanes below 16 take the first DM's.
  const unsigned char* tail_smem = smem + 4 * (32 * kFull + (lane & 15));
  for (int g = 0; g < n_groups; ++g) {
    const int slot = g % kSlots;
    if (!wait_or_abort(smem_u32(&ctl->rows_full[slot]), (g / kSlots) & 1, ctl)) {
      if (lane == 0) {
        atomicOr(p.err, tk::kErrTimeout);
        ctl->abort = 1;
      }
      return;
    }
    const uint32_t* offs = reinterpret_cast<const uint32_t*>(smem + kOffsOff + slot * kOffsBytes);
    const bool flush = LANES16 && offs[kDm] != 0u;
#pragma unroll
    for (int i = 0; i < kPairs; ++i) {
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
  // Word k of the tile holds output t0 + k and, in 16-bit lanes, that + 736.
  const int64_t lim = p.t_end - w0;
  auto put = [&](int d, int k, uint32_t a, uint32_t hi) {
    const int64_t dm = static_cast<int64_t>(blk) * kDm + d;
    if (dm >= p.n_dm) return;
    int32_t* row = p.out + dm * p.out_stride + w0;
    if constexpr (LANES16) {
      if (k < lim) row[k] = static_cast<int32_t>((a & 0xffffu) + ((hi & 0xffffu) << 8));
      if (k + kPairWords < lim)
        row[k + kPairWords] = static_cast<int32_t>((a >> 16) + ((hi >> 16) << 8));
    } else {
      if (k < lim) row[k] = static_cast<int32_t>(a);
    }
  };
#pragma unroll
  for (int q = 0; q < kPairs * kAcc; q += 8) {
    uint32_t v[8] = {};
    if (LANES16 && flushed) {
      __syncwarp();
      tmem_load8(col + q, v);
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

template <bool LANES16>
__global__ void __launch_bounds__(kThreads, 1) sum_row_kernel(const __grid_constant__ Params p) {
  extern __shared__ __align__(128) unsigned char smem[];
  Ctl* ctl = reinterpret_cast<Ctl*>(smem);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(smem_u32(&ctl->raw_full[s]), 1);
      mbar_init(smem_u32(&ctl->raw_empty[s]), kBuildWarps);
      mbar_init(smem_u32(&ctl->rows_full[s]), kBuildWarps);
      mbar_init(smem_u32(&ctl->rows_empty[s]), kMainWarps);
      ctl->issued[s] = 0;
    }
    ctl->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if constexpr (LANES16) {
    if (threadIdx.x < 32) tmem_alloc(smem_u32(&ctl->tmem));
    tmem_fence_before();
  }
  __syncthreads();
  if constexpr (LANES16) tmem_fence_after();
  const int blk = blockIdx.x % p.n_blocks;
  const int64_t half = blockIdx.x / p.n_blocks;  // 368-word halves of the time tiles
  constexpr int kTile = kPairWords * (LANES16 ? 2 : 1);
  const int64_t w0 = (p.tile0 + half / 2) * kTile + (half % 2) * kWords;
  const int32_t* first = reinterpret_cast<const int32_t*>(p.tables);
  const int g0 = first[blk], n_groups = first[blk + 1] - g0;
  // 256 x 208 + 256 x 48 registers: the 512 x 128 of the launch.
  if (threadIdx.x >= 32 * kMainWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
    build(p, smem, ctl, blk, w0, g0, n_groups);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    add_and_store<LANES16>(p, smem, ctl, blk, w0, n_groups);
  }
  if constexpr (LANES16) tmem_fence_before();
  __syncthreads();
  if (ctl->abort && threadIdx.x == 0) {
    // Copies still in flight land before the CTA exits (bounded).
    for (int s = 0; s < kSlots; ++s)
      if (ctl->issued[s] > 0)
        tk::mbar_wait(smem_u32(&ctl->raw_full[s]), ((ctl->issued[s] - 1) / kSlots) & 1);
  }
  if constexpr (LANES16) {
    tmem_fence_after();
    __syncwarp();
    if (threadIdx.x < 32) tmem_dealloc(ctl->tmem);
  }
}

}  // namespace sr

int launch_forward_sum_rows(const dd_plan_s* p, const RangePlan& rp, const void* tables,
                            int32_t* err, const void* d_words, int64_t stride, void* d_out,
                            int64_t t_begin, int64_t t_end, void* stream, int64_t out_stride,
                            int kind, int64_t x_origin) {
  const bool lanes16 = tk::packed_pairs(kind);
  const int64_t ts = sr::kPairWords * (lanes16 ? 2 : 1);
  if (x_origin < 0 || x_origin % sr::kAlign != 0 || t_begin % ts != 0 || t_begin < 0 ||
      t_end <= t_begin)
    return static_cast<int>(cudaErrorInvalidValue);
  sr::Params prm{};
  prm.x = static_cast<const uint32_t*>(d_words);
  prm.stride = stride;
  prm.x_origin = x_origin;
  prm.n_chan = p->n_chan;
  prm.n_dm = static_cast<int32_t>(rp.n_dm);
  prm.n_blocks = rp.sums.n_blocks;
  prm.tables = static_cast<const unsigned char*>(tables);
  prm.off_dir = rp.sums.off_dir;
  prm.off_start = rp.sums.off_start;
  prm.tile0 = t_begin / ts;
  prm.t_end = t_end;
  prm.out_stride = out_stride;
  prm.out = static_cast<int32_t*>(d_out);
  prm.err = err;
  prm.wait_iters = p->wait_iters;
  prm.hold_stage = p->hold_stage;
  // Halves of time tiles; the last tile's second half only where it has outputs.
  const int64_t whole = t_end / ts - prm.tile0, rest = t_end % ts;
  const int64_t halves = 2 * whole + (rest > sr::kWords ? 2 : rest > 0 ? 1 : 0);
  const int64_t grid = halves * prm.n_blocks;
  if (grid <= 0 || grid > 0x7fffffffLL) return static_cast<int>(cudaErrorInvalidConfiguration);
  auto kern = lanes16 ? sr::sum_row_kernel<true> : sr::sum_row_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sr::kSmemBytes));
  if (e != cudaSuccess) return static_cast<int>(e);
  kern<<<static_cast<unsigned>(grid), sr::kThreads, sr::kSmemBytes,
         static_cast<cudaStream_t>(stream)>>>(prm);
  return static_cast<int>(cudaGetLastError());
}

}  // namespace dd
