// fwd_direct.cu -- the direct tile (direct.h): Eq. 3 for 128 trial DMs x 368
// window words per CTA on plans too steep for the pattern tiles.
//
// Sixteen warps of 8 DMs each; a lane holds 11 words of every DM and one more
// that the two DMs of a pair share (16 lanes each): 92 accumulators.  Lanes
// take consecutive words, so every read is conflict-free at any shift and the
// output rows are stored straight from the registers.
//
// What bounds it: shared-memory reads, one word per added word (32 a clock and
// SM: 10e12 float32 or 20e12 uint8 sample-adds/s); the staging is a tenth of
// that.  The offset tile reads 36-word windows for 20 words of one or two DMs
// with vector loads and an indexed branch per DM; on 336 channels x 32768
// float32 samples, 1024 DMs at up to 12 samples a step, it
// took 2.03 ms, this tile 0.82 ms (8.5e12 adds/s, 0.84 of the pipe).
//
// Every mbarrier wait is bounded; on timeout the CTA sets kErrTimeout, waits
// for its copies and stores nothing.
#include <cuda_runtime.h>

#include <cstdint>

#include "dd_internal.h"
#include "direct.h"
#include "tile_common.cuh"
#include "tmem.cuh"

namespace dd {
namespace dt {

using tk::smem_u32;

struct Ctl {
  uint64_t bar[2];
  uint32_t tmem;
};

template <int KIND>
using Acc = std::conditional_t<tk::float_kind(KIND), float, uint32_t>;

constexpr int kPairs = kDmWarp / 2;
static_assert(kPairs * kAcc % 4 == 0, "tensor memory moves 4 words at a time");

template <int KIND>
__global__ void __launch_bounds__(32 * kWarps, 1) direct_kernel(const __grid_constant__ Params p) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr bool kLanes16 = KIND == tk::kU8;
  constexpr bool kStaged = staged_words(KIND);
  Ctl* ctl = reinterpret_cast<Ctl*>(smem);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    tk::mbar_init(smem_u32(&ctl->bar[0]), p.nc + 1);
    tk::mbar_init(smem_u32(&ctl->bar[1]), p.nc + 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if constexpr (kLanes16) {
    if (tid < 32) tmem::alloc(smem_u32(&ctl->tmem));
    tmem::fence_before();
  }
  __syncthreads();
  if constexpr (kLanes16) tmem::fence_after();
  const uint32_t col = kLanes16 ? tmem::warp_columns(ctl->tmem, w, 128) : 0u;

  const int blk = blockIdx.x % p.n_blocks;
  const int64_t t0 =
      p.t_begin + static_cast<int64_t>(blockIdx.x / p.n_blocks) * samples_per_tile(KIND);
  const int n_st = (p.n_chan + p.nc - 1) / p.nc;
  const Rec* my_recs = p.recs + static_cast<int64_t>(blk) * p.n_chan;
  Rec* recs = reinterpret_cast<Rec*>(smem + kRecOff);                // [2][nc]
  uint8_t* raw = smem + raw_off(p.nc);                               // [1 or 2][nc][lraw]
  uint32_t* words = reinterpret_cast<uint32_t*>(raw + static_cast<size_t>(p.nc) * p.lraw);

  auto base_of = [&](int st) -> int32_t {
    const int c = st * p.nc + tid;
    return tid < p.nc && c < p.n_chan ? __ldg(&my_recs[c].base) : 0;
  };
  // Copies of stage st: thread i < nc the window of channel i, thread nc the
  // records (none of them for the withheld stage of the timeout test).
  auto issue = [&](int st, int32_t base) {
    if (tid > p.nc || st == p.hold_stage) return;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    const uint32_t bar = smem_u32(&ctl->bar[kStaged ? st & 1 : 0]);
    const int c = st * p.nc + tid;
    uint32_t bytes = 0;
    const void* src = nullptr;
    void* dst = nullptr;
    if (tid == p.nc) {
      bytes = static_cast<uint32_t>(min(p.nc, p.n_chan - st * p.nc) * sizeof(Rec));
      src = my_recs + st * p.nc;
      dst = recs + (st & 1) * p.nc;
    } else if (c < p.n_chan) {
      // Window start: 16-byte aligned raw samples at or before t0 + base,
      // clipped at the end of the row.
      const int64_t at = ((t0 + base) & ~static_cast<int64_t>(p.align - 1)) * p.bin;
      if (at < p.stride)
        bytes = static_cast<uint32_t>(min(static_cast<int64_t>(p.lraw),
                                          tk::sample_bytes(KIND, p.stride - at)));
      src = static_cast<const uint8_t*>(p.x) +
            tk::sample_bytes(KIND, static_cast<int64_t>(c) * p.stride + at);
      dst = raw + (static_cast<size_t>(kStaged ? st & 1 : 0) * p.nc + tid) * p.lraw;
    }
    tk::mbar_arrive_expect(bar, bytes);
    if (bytes) tk::bulk_copy(smem_u32(dst), src, bytes, bar);
  };

  Acc<KIND> acc[kPairs][kAcc];
#pragma unroll
  for (int i = 0; i < kPairs; ++i)
#pragma unroll
    for (int j = 0; j < kAcc; ++j) acc[i][j] = Acc<KIND>(0);
  bool flushed = false;
  int since = 0;
  issue(0, base_of(0));
  int32_t next_base = base_of(1);
  bool gave_up = false;
  for (int st = 0; st < n_st; ++st) {
    const int nc = min(p.nc, p.n_chan - st * p.nc);
    const int buf = kStaged ? st & 1 : 0;
    // Two buffers: the next stage's copies start now (its buffer was read in
    // stage st - 1, which ended with a barrier).
    if (kStaged && st + 1 < n_st) {
      issue(st + 1, next_base);
      next_base = base_of(st + 2);
    }
    const bool ok = tk::mbar_wait(smem_u32(&ctl->bar[buf]), kStaged ? (st >> 1) & 1 : st & 1,
                                  p.wait_iters);
    if constexpr (!kStaged) {
      if (ok) {
        // Warp w unpacks channels w, w + 16; lanes consecutive 4-word units.
        for (int ch = w; ch < nc; ch += kWarps) {
          const uint8_t* r = raw + static_cast<size_t>(ch) * p.lraw;
          uint32_t* dst = words + static_cast<size_t>(ch) * p.lw;
          for (int q = lane; q < p.lw / 4; q += 32)
            *reinterpret_cast<uint4*>(dst + 4 * q) = tk::unpack_unit<KIND, kWords>(r, q, p.bin);
        }
      }
    }
    if (__syncthreads_or(!ok)) {
      if (tid == 0) {
        atomicOr(p.err, tk::kErrTimeout);
        // Copies still in flight land before the CTA exits (bounded).
        for (int q = st; q < min(st + (kStaged ? 2 : 1), n_st); ++q)
          if (q != p.hold_stage)
            tk::mbar_wait(smem_u32(&ctl->bar[kStaged ? q & 1 : 0]),
                          kStaged ? (q >> 1) & 1 : q & 1);
      }
      gave_up = true;
      break;
    }
    if (!kStaged && st + 1 < n_st) {
      issue(st + 1, next_base);
      next_base = base_of(st + 2);
    }
    if constexpr (kLanes16) {
      if (since + nc > p.flush) {
        __syncwarp();
#pragma unroll
        for (int q = 0; q < kPairs * kAcc; q += 4) {
          uint32_t v[4] = {};
          if (flushed) tmem::load(col + q, v);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            uint32_t& a = acc[(q + e) / kAcc][(q + e) % kAcc];
            v[e] += __byte_perm(a, 0u, 0x4341);
            a &= 0x00ff00ffu;
          }
          tmem::store(col + q, v);
        }
        tmem::wait_stores();
        flushed = true;
        since = 0;
      }
      since += nc;
    }
    const Rec* rs = recs + (st & 1) * p.nc;
    const uint32_t* win =
        kStaged ? reinterpret_cast<const uint32_t*>(raw + static_cast<size_t>(buf) * p.nc * p.lraw)
                : words;
    auto word = [](const uint32_t* a) {
      if constexpr (tk::float_kind(KIND)) return __uint_as_float(*a);
      else return *a;
    };
#pragma unroll 1
    for (int ch = 0; ch < nc; ++ch, win += p.lw) {
      const uint4 o4 = *reinterpret_cast<const uint4*>(&rs[ch].off[kDmWarp * w]);
      const uint32_t o[kPairs] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
      for (int i = 0; i < kPairs; ++i) {
        const uint32_t oa = o[i] & 0xffffu, ob = o[i] >> 16;
        const uint32_t* a = win + oa + lane;
        const uint32_t* b = win + ob + lane;
#pragma unroll
        for (int j = 0; j < kFull; ++j) acc[i][j] += word(a + 32 * j);
#pragma unroll
        for (int j = 0; j < kFull; ++j) acc[i][kFull + j] += word(b + 32 * j);
        acc[i][2 * kFull] +=
            word(win + (lane < 16 ? oa : ob) + 32 * kFull + (lane & 15));
      }
    }
    __syncthreads();  // the window (and record) buffers are free
  }

  if (!gave_up) {
    const int64_t lim = p.t_end - t0;
    auto put = [&](int d, int k, Acc<KIND> a, uint32_t hi) {
      const int64_t dm = static_cast<int64_t>(blk) * kDm + d;
      if (dm >= p.n_dm) return;
      tk::OutT<KIND>* row = static_cast<tk::OutT<KIND>*>(p.out) + dm * p.out_stride + t0;
      if constexpr (kLanes16) {
        if (k < lim) row[k] = static_cast<int32_t>((a & 0xffffu) + ((hi & 0xffffu) << 8));
        if (k + kWords < lim)
          row[k + kWords] = static_cast<int32_t>((a >> 16) + ((hi >> 16) << 8));
      } else {
        if (k < lim) row[k] = static_cast<tk::OutT<KIND>>(a);
      }
    };
#pragma unroll
    for (int q = 0; q < kPairs * kAcc; q += 4) {
      uint32_t v[4] = {};
      if (kLanes16 && flushed) {
        __syncwarp();
        tmem::load(col + q, v);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int i = (q + e) / kAcc, j = (q + e) % kAcc;
        const int d = kDmWarp * w + 2 * i;
        if (j < kFull) put(d, 32 * j + lane, acc[i][j], v[e]);
        else if (j < 2 * kFull) put(d + 1, 32 * (j - kFull) + lane, acc[i][j], v[e]);
        else put(d + (lane >> 4), 32 * kFull + (lane & 15), acc[i][j], v[e]);
      }
    }
  }
  if constexpr (kLanes16) {
    tmem::fence_before();
    __syncthreads();
    tmem::fence_after();
    __syncwarp();
    if (tid < 32) tmem::dealloc(ctl->tmem);
  }
}

template <int KIND>
int launch(const Params& prm, int64_t grid, size_t smem, cudaStream_t st) {
  auto kern = direct_kernel<KIND>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return static_cast<int>(e);
  kern<<<static_cast<unsigned>(grid), 32 * kWarps, smem, st>>>(prm);
  return static_cast<int>(cudaGetLastError());
}

}  // namespace dt

int launch_forward_direct(const dd_plan_s* p, const RangePlan& rp, const void* recs, int32_t* err,
                          const void* d_in, int64_t stride, int64_t n_out, void* d_out,
                          int64_t t_begin, int64_t t_end, void* stream) {
  const DirectTables& t = rp.direct;
  dt::Params prm{};
  prm.x = d_in;
  prm.stride = stride;
  prm.n_chan = p->n_chan;
  prm.n_dm = static_cast<int32_t>(rp.n_dm);
  prm.n_blocks = t.n_blocks;
  prm.bin = rp.r.bin;
  prm.align = tk::align_samples(t.kind, rp.r.bin);
  prm.nc = t.nc;
  prm.lw = t.lw;
  prm.lraw = dt::raw_bytes(t.kind, rp.r.bin, t.lw);
  prm.flush = 256;  // 255 kept + 256 x 255 fill a 16-bit lane
  prm.recs = static_cast<const dt::Rec*>(recs);
  prm.t_begin = t_begin;
  prm.t_end = t_end;
  prm.out_stride = n_out;
  prm.out = d_out;
  prm.err = err;
  prm.wait_iters = p->wait_iters;
  prm.hold_stage = p->hold_stage;
  if (t_begin < 0 || t_begin % 16 != 0 || t_end > n_out || t_end <= t_begin)
    return static_cast<int>(cudaErrorInvalidValue);
  const int ts = dt::samples_per_tile(t.kind);
  const int64_t grid = (t_end - t_begin + ts - 1) / ts * prm.n_blocks;
  if (grid > 0x7fffffffLL) return static_cast<int>(cudaErrorInvalidConfiguration);
  const size_t smem = dt::smem_bytes(t.kind, rp.r.bin, t.nc, t.lw);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  switch (t.kind) {
    case tk::kU8: return dt::launch<tk::kU8>(prm, grid, smem, st);
    case tk::kU8W: return dt::launch<tk::kU8W>(prm, grid, smem, st);
    case tk::kU16: return dt::launch<tk::kU16>(prm, grid, smem, st);
    case tk::kF32D: return dt::launch<tk::kF32D>(prm, grid, smem, st);
  }
  return static_cast<int>(cudaErrorInvalidValue);
}

}  // namespace dd
