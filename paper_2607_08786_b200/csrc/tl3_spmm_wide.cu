// SpMM for more than 64 columns (a prompt, a wide batch), sm_100a: W is streamed and decoded once for
// up to 256 columns.
//
// The pieces are those of tl3_spmm.cu (bulk copies of the packed blocks, Algorithm 1 by decode warps
// into a second 2:4 operand W_r, tcgen05.mma.sp on W_t and W_r into one fp32 accumulator, split-K over
// contiguous tile ranges with one reduction at the end), arranged for an accumulator of up to 256
// columns:
//   * the blocks and X have rings of their own: X arrives in slices of 64 k-values x n_pad columns
//     (one TMA box when X is [batch, hidden], one per 64 columns when it is [hidden, batch]) that are
//     given back half a tile at a time, so that shared memory holds more of the blocks;
//   * one launch covers all columns: a row-tile is worked on once per group of n_pad columns, the
//     groups of a row-tile directly after one another (its blocks then come from L2);
//   * two accumulators while they fit tensor memory beside the metadata, else one;
//   * above 128 columns, and above 64 in long launches, two CTAs of a cluster work on two row-tiles as one tcgen05.mma of 256 rows: each
//     decodes its own blocks and loads half of the columns of X.
// What bounds it at 256 columns (20480 x 5120, N = 512: 110 us at 1965 MHz, 135 at the clock that the power cap leaves): without
// decode 97, without MMAs 87, without either 80, which is 61 for the bytes from L2 (53 KB a tile and CTA at 77
// GB/s) and the ends of the launch; 11 pass while the one accumulator is written out.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include <cstdint>
#include <mutex>
#include <vector>

#include "tl3_device.cuh"
#include "tl3_internal.h"

namespace tl3 {
namespace {

constexpr int kProducerWarp = 0;          // packed blocks
constexpr int kMmaWarp = 1;
constexpr int kClearWarp = 2;             // clears W_r; owns the tensor-memory allocation
constexpr int kXWarp = 3;                 // X slices
constexpr int kDecodeWarp0 = 4;
// Decode groups of four warps.  A pair has shared memory for a fourth block in flight and wins 4-8 % by
// decoding four at a time; alone, a fourth group brings nothing where there is no buffer for it, and
// costs the epilogue its registers (80 instead of 96 a thread: 700 x 700, N = 70 takes 10.4 us, not 9).
template <int S> constexpr int kGroupsOf = S == 1 ? 3 : 4;
template <int S> constexpr int kThreadsOf = (kDecodeWarp0 + 4 * kGroupsOf<S> + 4) * 32;
constexpr int kEpilogueBarrier = 1;
constexpr int kMaxRing = 8;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColMetaT = 480;       // + 4 * (W_r buffer)
constexpr uint32_t kColMetaR = 496;
constexpr uint32_t kSlack = 1024u + 4u * kTurnBytes + 1024u;   // barriers, the epilogue warps' turning areas, alignment

struct WideArgs {
  const uint8_t* blob;
  const DirEntry* dir;
  uint32_t tiles_m, tiles_k;              // tiles of W
  int M, N;
  int n_pad[2];                           // columns of a pass; above 128 also: in a workspace with room for no more than that
  uint32_t chunks[2];                     // groups of so many columns
  const unsigned char* room;              // columns of partial sums per CTA that the workspace holds, / kRoomUnit
  long long ldy;
  __half* Y;
  const __half* bias;
  int act;
  float* partials;                        // [gridDim.x][n_pad][128]
  unsigned int* flags;                    // [gridDim.x]
  unsigned int* status;
  uint32_t block_area, x_bytes;           // of a block, of a slice of X: multiples of 1024
  int n_w, n_x, n_wr;                     // ring sizes: blocks (>= n_wr), X slices, W_r buffers
  int n_acc;
};

// ---- What differs between a CTA alone (S = 1) and a pair (S = 2, a cluster).  Both CTAs of a pair lay
// their shared memory out alike, so that an address of one names the same thing in the other.
template <int S>
__device__ __forceinline__ uint32_t leader_address(uint32_t addr) {   // of shared memory in the CTA of rank 0
  if constexpr (S == 1) return addr;
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
// (No release at cluster scope, which cost a decode warp 0.6 us: what the arrival announces was
// written to this SM's own shared and tensor memory and is read there by its tensor core, ordered by
// the proxy and tcgen05 fences in front of the arrival.)
template <int S>
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {
  if constexpr (S == 1) mbar_arrive(bar);
  else asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(leader_address<S>(bar)) : "memory");
}
template <int S>
__device__ __forceinline__ bool mbar_try_wait_unit(uint32_t bar, uint32_t parity) {
  if constexpr (S == 1) return mbar_try_wait(bar, parity);
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(done) : "r"(bar), "r"(parity), "r"(kTryWaitHintNs) : "memory");
  return done != 0;
}
// mbar_wait() for barriers on which the other CTA, or the pair's tensor cores, arrive
template <int S>
__device__ __forceinline__ bool mbar_wait_unit(uint32_t bar, uint32_t parity, const WaitCtx& w, uint32_t code) {
  unsigned long long t_slow = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait_unit<S>(bar, parity)) return true;
    if ((it & 15u) == 15u) {
      if (*w.abort_flag) return false;
      const unsigned long long now = global_timer();
      if (t_slow == 0) t_slow = now;
      if (now - t_slow > kWaitLimitNs) {
        atomicCAS(w.status, 0u, code);
        *w.abort_flag = 1;
        return false;
      }
    }
  }
}
template <int S>
__device__ __forceinline__ void sync_all() {                        // every thread of the CTA, or of the pair
  if constexpr (S == 1) {
    __syncthreads();
  } else {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}
// a load into this CTA's shared memory that reports to a barrier of the leader
template <int S>
__device__ __forceinline__ void tma_load_x(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t leader_bar) {
  if constexpr (S == 1) tma_load_2d(dst, map, c0, c1, leader_bar);
  else asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                    ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(leader_bar) : "memory");
}
// umma_sp_f16(); on a pair 256 rows, each CTA with 128 of them (its own A, metadata and accumulator)
// and with half of B's columns
template <int S>
__device__ __forceinline__ void umma_sp_f16_unit(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                                 uint32_t e_tmem, uint32_t idesc, uint32_t accumulate) {
  if constexpr (S == 1) {
    umma_sp_f16(d_tmem, a_lo, a_hi, b_lo, b_hi, e_tmem, idesc, accumulate);
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %7, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.sp.cta_group::2.kind::f16 [%0], da, db, [%5], %6, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(e_tmem), "r"(idesc), "r"(accumulate) : "memory");
  }
}
template <int S>
__device__ __forceinline__ void umma_commit_unit(uint32_t bar) {     // arrives in both CTAs of a pair
  if constexpr (S == 1) umma_commit(bar);
  else asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                    ::"r"(bar), "h"(static_cast<uint16_t>(3)) : "memory");
}
template <int S>
__device__ __forceinline__ void tmem_alloc(uint32_t slot) {
  if constexpr (S == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
}
template <int S>
__device__ __forceinline__ void tmem_dealloc(uint32_t base) {
  if constexpr (S == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(kTmemCols) : "memory");
  else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(kTmemCols) : "memory");
}

// barriers, one 64-bit word each; Dec, XFull and AccEmpty are used in the leader, by both CTAs
enum : uint32_t {
  kBarFull = 0, kBarDone = 8, kBarDec = 16, kBarXFull = 24, kBarHalf = 32, kBarWrReady = 40,
  kBarAccFull = 48, kBarReduce = 50, kBarAccEmpty = 51, kBarCount = 53, kTmemSlot = 53, kAbort = 54
};

// Columns c_begin, c_begin + c_step, ... (16 at a time) of one row of a row-tile: accumulator (+ the
// partial sums of the n_others CTAs after this one, in ascending order whatever the order they came
// in), bias, activation, rounding, Y.  Executed by whole warps, `et` is the row, 32 * (warp % 4) + lane.
// `turn`: kTurnBytes of shared memory of the warp's own.  A thread holds a row, so rows of Y that
// 16-byte stores do not fit are turned there first: stored by their rows' threads, two bytes each a
// row pitch apart, they took 6 us of 25 on 4096 x 4096, N = 65.
template <bool XT, int S, bool kShared>
__device__ __noinline__ void write_columns(const WideArgs& a, int less, uint32_t acc_tmem, int et, uint32_t vrow, int c_begin, int c_step, int n_others,
                                           uint32_t turn) {
  constexpr int CH = 16;
  const int n_pad = S == 1 ? a.n_pad[0] : a.n_pad[less];
  const uint32_t chunks = S == 1 ? a.chunks[0] : a.chunks[less];
  const int row = static_cast<int>(S * (vrow / chunks) + blockIdx.x % S) * kTileM + et;
  const int n0 = static_cast<int>(vrow % chunks) * n_pad;
  const int cols = a.N - n0 < n_pad ? a.N - n0 : n_pad;
  const bool plain = a.bias == nullptr && a.act == TL3_ACT_NONE;
  const float bias = a.bias != nullptr && row < a.M ? __half2float(__ldg(a.bias + row)) : 0.f;
  const bool vec_ok = !XT && (a.ldy & 7) == 0 && (reinterpret_cast<uintptr_t>(a.Y) & 15) == 0;
  const size_t slot = static_cast<size_t>(n_pad) * 128;
  const int lane = et & 31;
  // XT: four lanes hand each other their values, so that a thread stores four rows of one column
  const bool quads = XT && row - lane + 32 <= a.M && (a.ldy & 3) == 0 && (reinterpret_cast<uintptr_t>(a.Y) & 7) == 0;
  // A CTA alone reads a row-tile of its own one step ahead (4096 x 4096, N = 100 19.6 us, without 19.9).  In pairs the
  // registers for it cost more than the wait (20000 x 256, N = 500 29.1 and 27.7, 20480 x 5120, N = 512 111.1 and 109.7,
  // 5120 x 5120, N = 256 29.4 and 28.9), and a row-tile that others contribute to keeps them for
  // their partial sums, two slots' loads in flight.
  constexpr bool kAhead = !kShared && S == 1;
  uint32_t next[CH];
  if constexpr (kAhead) TmemLd<CH>::ld(acc_tmem + c_begin, next);
#pragma unroll 1
  for (int c0 = c_begin; c0 < cols; c0 += c_step) {
    uint32_t v[CH];
    if constexpr (kAhead) {
      tmem_wait_ld<CH>(next);
#pragma unroll
      for (int c = 0; c < CH; ++c) v[c] = next[c];
      if (c0 + c_step < cols) TmemLd<CH>::ld(acc_tmem + c0 + c_step, next);
    } else {
      TmemLd<CH>::ld(acc_tmem + c0, v);
      tmem_wait_ld<CH>(v);
    }
    if constexpr (kShared) {
      const float* p = a.partials + slot * (blockIdx.x + S) + c0 * 128 + et;   // the next CTA, or the same one of the next pair
      for (int k = 0; k < n_others; k += 2, p += 2 * S * slot) {
        float p0[CH], p1[CH];
        const bool second = k + 1 < n_others;
#pragma unroll
        for (int c = 0; c < CH; ++c) { p0[c] = __ldcg(p + c * 128); p1[c] = second ? __ldcg(p + S * slot + c * 128) : 0.f; }
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          float x = __uint_as_float(v[c]) + p0[c];
          if (second) x += p1[c];
          v[c] = __float_as_uint(x);
        }
      }
    }
    if (!plain) apply_epilogue<CH>(v, bias, a.act, row < a.M ? cols - c0 : 0);
    uint32_t o[CH / 2];
#pragma unroll
    for (int c = 0; c < CH / 2; ++c) {
      const __half2 h = __floats2half2_rn(__uint_as_float(v[2 * c]), __uint_as_float(v[2 * c + 1]));
      o[c] = *reinterpret_cast<const uint32_t*>(&h);
    }
    if constexpr (XT) {
      if (quads) {
        // lane 4 r + j ends with column 4 q + j of rows 4 r .. 4 r + 3 (two exchanges of what the
        // other lane keeps), q = 0 .. 3
        __half* y = a.Y + static_cast<long long>(n0 + c0 + (lane & 3)) * a.ldy + (row - (lane & 3));
        const bool odd = (lane & 1) != 0, high = (lane & 2) != 0;
#pragma unroll
        for (int q = 0; q < CH / 4; ++q) {
          // columns 4 q, 4 q + 1 and 4 q + 2, 4 q + 3 of this row -> two rows of one column of either pair
          const uint32_t e0 = __shfl_xor_sync(0xFFFFFFFFu, o[2 * q], 1), e1 = __shfl_xor_sync(0xFFFFFFFFu, o[2 * q + 1], 1);
          const uint32_t f0 = odd ? __byte_perm(e0, o[2 * q], 0x7632u) : __byte_perm(o[2 * q], e0, 0x5410u);
          const uint32_t f1 = odd ? __byte_perm(e1, o[2 * q + 1], 0x7632u) : __byte_perm(o[2 * q + 1], e1, 0x5410u);
          // f0: column 4 q + odd, f1: column 4 q + 2 + odd, rows (lane & ~1), + 1 -> four rows of column 4 q + (lane & 3)
          const uint32_t g = __shfl_xor_sync(0xFFFFFFFFu, high ? f0 : f1, 2);
          if (c0 + 4 * q + (lane & 3) < cols)
            *reinterpret_cast<uint2*>(y + static_cast<long long>(4 * q) * a.ldy) = high ? make_uint2(g, f1) : make_uint2(f0, g);
        }
      } else if (row < a.M) {
        uint16_t* y = reinterpret_cast<uint16_t*>(a.Y) + static_cast<long long>(n0 + c0) * a.ldy + row;
#pragma unroll
        for (int c = 0; c < CH; ++c, y += a.ldy)
          if (c0 + c < cols) *y = static_cast<uint16_t>(o[c / 2] >> (16 * (c & 1)));
      }
    } else if (vec_ok && c0 + CH <= cols) {
      // two lanes hand each other half of their row, so that a store covers 32 bytes of each row
      uint32_t other[4];
      const bool odd = (lane & 1) != 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) other[i] = __shfl_xor_sync(0xFFFFFFFFu, odd ? o[i] : o[4 + i], 1);
      const int r0 = row - (odd ? 1 : 0);                          // the pair's first row
      __half* y = a.Y + static_cast<long long>(r0) * a.ldy + n0 + c0 + (odd ? 8 : 0);
      if (r0 < a.M)
        *reinterpret_cast<uint4*>(y) = odd ? make_uint4(other[0], other[1], other[2], other[3]) : make_uint4(o[0], o[1], o[2], o[3]);
      if (r0 + 1 < a.M)
        *reinterpret_cast<uint4*>(y + a.ldy) = odd ? make_uint4(o[4], o[5], o[6], o[7]) : make_uint4(other[0], other[1], other[2], other[3]);
    } else if (vec_ok && cols - c0 == 8) {
      // half a step at the end (20480 x 128, N = 72 turned 9.5 us, so 8.2; 20480 x 5120, N = 88 46.2 and 45.0)
      if (row < a.M) *reinterpret_cast<uint4*>(a.Y + static_cast<long long>(row) * a.ldy + n0 + c0) = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
      const int col = lane & 15;
      __syncwarp();
#pragma unroll
      for (int c = 0; c < CH / 2; ++c) sts_u32(turn + static_cast<uint32_t>(lane) * kTurnPitch + 4u * c, o[c]);
      __syncwarp();
      const int row0 = row - lane + (lane >> 4);                   // half a warp writes one row
      __half* y = a.Y + static_cast<long long>(row0) * a.ldy + n0 + c0 + col;
#pragma unroll 4
      for (int i = 0; i < 16; ++i, y += 2 * a.ldy) {
        const uint32_t h = lds_u16(turn + static_cast<uint32_t>(2 * i + (lane >> 4)) * kTurnPitch + 2u * col);
        if (row0 + 2 * i < a.M && c0 + col < cols) *reinterpret_cast<uint16_t*>(y) = static_cast<uint16_t>(h);
      }
    }
  }
}

// XT as in tl3_spmm.cu: activations and result transposed ([batch, hidden]).
// S: CTAs that work together, 1 or 2 (a cluster).
// kLongRes: see scatter_residual().
template <bool XT, int S, bool kLongRes>
__global__ void __launch_bounds__(kThreadsOf<S>, 1)
tl3_spmm_wide_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ WideArgs a) {
  constexpr int kGroups = kGroupsOf<S>, kEpilogueWarp0 = kDecodeWarp0 + 4 * kGroups;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t w_base = smem_u32(smem);
  const uint32_t x_base = w_base + static_cast<uint32_t>(a.n_w) * a.block_area;
  const uint32_t wr_base = x_base + static_cast<uint32_t>(a.n_x) * a.x_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (wr_base - w_base) + static_cast<uint32_t>(a.n_wr) * kWrBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto bar = [&](uint32_t which, int i) -> uint32_t { return bar0 + 8u * (which + static_cast<uint32_t>(i)); };
  // The MMAs of tile i, or of its first half, are done: rings of eight barriers (no ring below holds more
  // than eight tiles, so nobody who waits here is more than one phase behind).
  auto wait_done = [&](int i, const WaitCtx& w, uint32_t code) -> bool { return mbar_wait_unit<S>(bar(kBarDone, i & 7), (i >> 3) & 1, w, code); };
  auto wait_half = [&](int i, const WaitCtx& w, uint32_t code) -> bool { return mbar_wait_unit<S>(bar(kBarHalf, i & 7), (i >> 3) & 1, w, code); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kTmemSlot);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + kAbort);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // Tile v of the launch: rows v / tiles_k of ceil(tiles_m / S) * chunks (S row-tiles, one per CTA; column
  // group minor), k-tile v % tiles_k.  An odd last row-tile is done by both CTAs of a pair (the second
  // one's rows lie beyond M and are not stored).
  const uint32_t rank = blockIdx.x % S, unit = blockIdx.x / S;
  // The partial sums of a pair are up to 256 columns per CTA.  Above 128, a workspace made for fewer, which
  // tl3_workspace_init() recorded in it, gets passes of half the columns: the slices of X are then loaded
  // as wide as ever and used in part.  (The record is older than anything a kernel before this one does:
  // no wait for it.)
  const int less = S == 2 && static_cast<int>(__ldcg(a.room)) * kRoomUnit < a.n_pad[0] ? 1 : 0;
  const uint32_t TK = a.tiles_k, T = (a.tiles_m + S - 1) / S * a.chunks[less] * TK, G = gridDim.x / S;
  const uint32_t t_begin = range_begin(unit, T, G), t_end = range_begin(unit + 1, T, G);
  const int n_tiles = static_cast<int>(t_end - t_begin);
  const uint32_t kt_begin = t_begin % TK, vrow_begin = t_begin / TK;
  const int AG = a.n_wr < kGroups ? a.n_wr : kGroups;   // decode groups in use: see the waits of the decode warps

  if (warp == kProducerWarp) {
    if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&x_map) : "memory");
    for (int i = lane; i < static_cast<int>(kBarCount); i += 32) {
      const uint32_t u = static_cast<uint32_t>(i);
      const uint32_t count = (u >= kBarDec && u < kBarXFull) || u >= kBarAccEmpty ? 128u * S : (u >= kBarWrReady && u < kBarAccFull) ? 32u : 1u;
      mbar_init(bar0 + 8u * u, count);
    }
    if (lane == 0) *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kClearWarp) {
    tmem_alloc<S>(smem_u32(tmem_slot));
  }
  tc_fence_before();
  sync_all<S>();                               // (the other CTA uses this one's barriers, too)
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const WaitCtx wctx{abort_flag, a.status};
  pdl_launch_dependents();

  if (warp == kProducerWarp) {
    // ------------------------------------------------------------------ packed blocks
    // (never written by the kernel before this one: no wait for it)
    int issued = 0, s = 0;
    uint32_t kt = kt_begin, vrow = vrow_begin;
    bool alive = true;
    for (int base = 0; base < n_tiles && alive; base += 32) {
      // directory entries of the next 32 tiles, one per lane
      uint4 mine = make_uint4(0, 0, 0, 0);
      if (base + lane < n_tiles) {
        uint32_t k = kt + static_cast<uint32_t>(lane), v = vrow;
        while (k >= TK) { k -= TK; ++v; }
        const uint32_t mt = S * (v / a.chunks[less]) + rank;
        mine = __ldg(reinterpret_cast<const uint4*>(a.dir + static_cast<size_t>(mt < a.tiles_m ? mt : a.tiles_m - 1) * TK + k));
      }
      const int cnt = n_tiles - base < 32 ? n_tiles - base : 32;
      for (int j = 0; j < cnt; ++j) {
        const uint32_t off16 = __shfl_sync(0xFFFFFFFFu, mine.x, j), bytes = __shfl_sync(0xFFFFFFFFu, mine.y, j);
        if (base + j >= a.n_w) alive = __all_sync(0xFFFFFFFFu, wait_done(base + j - a.n_w, wctx, kStProducer));
        if (!alive) break;
        if (elect_one()) {
          mbar_arrive_expect_tx(bar(kBarFull, s), bytes);
          bulk_copy_g2s(w_base + static_cast<uint32_t>(s) * a.block_area, a.blob + static_cast<size_t>(off16) * 16, bytes, bar(kBarFull, s));
        }
        __syncwarp();
        issued = base + j + 1;
        if (++s == a.n_w) s = 0;
        if (++kt == TK) { kt = 0; ++vrow; }
      }
    }
    if (lane == 0 && *abort_flag) {
      // let the copies still in flight land before the CTA goes away
      for (int i = issued > a.n_w ? issued - a.n_w : 0; i < issued; ++i) {
        const unsigned long long t1 = global_timer();
        while (!mbar_try_wait(bar(kBarFull, i % a.n_w), (i / a.n_w) & 1)) {
          if (global_timer() - t1 > kWaitLimitNs / 4) { atomicCAS(a.status, 0u, (uint32_t)kStDrain); break; }
        }
      }
    }
  } else if (warp == kXWarp) {
    // ------------------------------------------------------------------ X slices (64 k-values), two per tile
    int s = 0;
    uint32_t kt = kt_begin, vrow = vrow_begin;
    pdl_wait();                                                    // the kernel before this one may have written X
    for (int j = 0; j < 2 * n_tiles; ++j) {
      const int n0 = static_cast<int>(vrow % a.chunks[less]) * a.n_pad[less] + static_cast<int>(rank) * (a.n_pad[less] / S);
      const int last = j - a.n_x;                                  // the slice that was here before
      if (last >= 0 && !__all_sync(0xFFFFFFFFu, (last & 1) ? wait_done(last >> 1, wctx, kStProducer) : wait_half(last >> 1, wctx, kStProducer))) break;
      if (elect_one()) {
        const uint32_t full = leader_address<S>(bar(kBarXFull, s)), dst = x_base + static_cast<uint32_t>(s) * a.x_bytes;
        const int k0 = static_cast<int>(kt) * kTileK + 64 * (j & 1);
        if (rank == 0) mbar_arrive_expect_tx(bar(kBarXFull, s), S * a.x_bytes);   // both CTAs' (the other one's may be there first)
        if (XT) {
          tma_load_x<S>(dst, &x_map, k0, n0, full);
        } else {
          for (uint32_t c = 0; c * 8192u < a.x_bytes; ++c) tma_load_x<S>(dst + c * 8192u, &x_map, n0 + static_cast<int>(64u * c), k0, full);
        }
      }
      __syncwarp();
      if (++s == a.n_x) s = 0;
      if ((j & 1) && ++kt == TK) { kt = 0; ++vrow; }
    }
    // (Giving up takes two seconds without progress in one of the CTAs: copies in flight have long landed,
    // and neither CTA goes before the other.)
  } else if (warp == kClearWarp) {
    // ------------------------------------------------------------------ W_r clearing
    int wb = 0;
    for (int i = 0; i < n_tiles; ++i) {
      if (i >= a.n_wr && !__all_sync(0xFFFFFFFFu, wait_done(i - a.n_wr, wctx, kStClearWrFree))) break;
      const uint32_t wr = wr_base + static_cast<uint32_t>(wb) * kWrBytes;
#pragma unroll
      for (int c = 0; c < 32; ++c) sts_zero16B(wr + (c * 32 + lane) * 16);
      fence_proxy_async_smem();
      mbar_arrive(bar(kBarWrReady, wb));
      if (++wb == a.n_wr) wb = 0;
    }
  } else if (warp == kMmaWarp && rank == 0) {
    // ------------------------------------------------------------------ MMA issuer, for the pair
    // Descriptors as in tl3_spmm.cu.  B: with XT n_pad rows x 128 bytes, K-major, 8-row groups 1024 B
    // apart, a k-block is 64 bytes of a row; otherwise blocks of 64 k-rows x 128 bytes (64 columns),
    // MN-major, 8-row groups 1024 B apart (stride field), the blocks 8192 B (leading-offset field), a
    // k-block is 32 rows.
    const uint32_t idesc = (1u << 2) | (1u << 4) | (XT ? 0u : (1u << 16)) | (static_cast<uint32_t>(a.n_pad[less] >> 3) << 17) | (8u * S << 24);
    constexpr uint32_t kHi = (1024u >> 4) | (1u << 14) | (2u << 29);
    constexpr uint32_t kLboA = 1u << 16, kLboB = XT ? (1u << 16) : ((8192u >> 4) << 16);
    constexpr uint32_t kBStep = (XT ? 64u : 4096u) >> 4;
    int seg = 0, s = 0, sx = 0, wb = 0;
    uint32_t ph = 0, phx = 0, kt = kt_begin;
    bool ok = true;
    for (int i = 0; i < n_tiles && ok; ++i) {
      const bool first_of_seg = (i == 0) || (kt == 0);
      const bool last_of_seg = (i == n_tiles - 1) || (kt == TK - 1);
      const int b = a.n_acc == 2 ? seg & 1 : 0, b_use = a.n_acc == 2 ? seg >> 1 : seg;
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(b * a.n_pad[less]);
      const uint32_t e_t = tmem_base + kColMetaT + 4 * wb, e_r = tmem_base + kColMetaR;
      const uint32_t a_lo = ((w_base + static_cast<uint32_t>(s) * a.block_area) >> 4) | kLboA;
      const uint32_t r_lo = ((wr_base + static_cast<uint32_t>(wb) * kWrBytes) >> 4) | kLboA;
      const uint32_t done = bar(kBarDone, i & 7), half = bar(kBarHalf, i & 7), acc = bar(kBarAccFull, b);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h == 0) {
          if (first_of_seg && b_use >= 1) ok = mbar_wait_unit<S>(bar(kBarAccEmpty, b), (b_use - 1) & 1, wctx, kStMmaAccEmpty);
          ok = ok && mbar_wait_unit<S>(bar(kBarDec, s), ph, wctx, kStMmaDecoded);
        }
        ok = ok && mbar_wait_unit<S>(bar(kBarXFull, sx), phx, wctx, kStMmaX);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        tc_fence_after();
        const uint32_t b_lo = ((x_base + static_cast<uint32_t>(sx) * a.x_bytes) >> 4) | kLboB;
        if (elect_one()) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const uint32_t kb = 2u * h + q, id = idesc | static_cast<uint32_t>(q);
            umma_sp_f16_unit<S>(d_tmem, a_lo + kb * 2u, kHi, b_lo + q * kBStep, kHi, e_t + 2u * h, id, (first_of_seg && kb == 0) ? 0u : 1u);
            umma_sp_f16_unit<S>(d_tmem, r_lo + kb * 2u, kHi, b_lo + q * kBStep, kHi, e_r, id, 1u);
          }
          umma_commit_unit<S>(h ? done : half);
          if (h == 1 && last_of_seg) umma_commit_unit<S>(acc);
        }
        __syncwarp();
        if (++sx == a.n_x) { sx = 0; phx ^= 1u; }
      }
      if (last_of_seg) ++seg;
      if (++s == a.n_w) { s = 0; ph ^= 1u; }
      if (++kt == TK) kt = 0;
      if (++wb == a.n_wr) wb = 0;
    }
  } else if (warp >= kDecodeWarp0 && warp < kEpilogueWarp0) {
    // ------------------------------------------------------------------ decode (Algorithm 1)
    const int g = (warp - kDecodeWarp0) >> 2;
    const int r = tid - (kDecodeWarp0 + 4 * g) * 32;            // chain / row / tensor-memory lane 0..127
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    if (g == 0) {   // constant metadata of W_r: every window selects in-window positions {2, 3}
      asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};"
                   ::"r"(tmem_base + lane_base + kColMetaR), "r"(0xEEEEEEEEu), "r"(0xEEEEEEEEu) : "memory");
    }
    // Tile i goes to group i % AG, W_r buffer i % n_wr, block stage i % n_w, AG <= n_wr <= n_w.  Parity
    // waits cannot tell phases two apart; here they need not: when tile i is waited for, this group
    // has finished tile i - AG, whose buffer was opened after that of tile i - n_wr (they open in
    // order), so the buffer is at most one phase behind; and once it is open the MMAs of tile
    // i - n_wr are done, so the stage's last user i - n_w has been loaded and consumed.
    int wb = g, use = 0;
    int s = g;
    uint32_t ph = 0;
    for (int i = g, j = 0; g < AG && i < n_tiles; i += AG, ++j) {
      const int cr = (r + 32 * (j & 3)) & 127;                  // chain handled by this thread (lengths differ by warp: rotated)
      const uint32_t wr = wr_base + static_cast<uint32_t>(wb) * kWrBytes;
      bool ok = mbar_wait(bar(kBarWrReady, wb), use & 1, wctx, kStDecodeWrReady);
      ok = ok && mbar_wait(bar(kBarFull, s), ph, wctx, kStDecodeFull);
      const uint32_t stage = w_base + static_cast<uint32_t>(s) * a.block_area;
      uint32_t m0 = 0, m1 = 0, m2 = 0, m3 = 0, n_words = 0, hdr = 0xFFFFFFFFu, pdd_len = 0, res_cnt = 0;
      if (ok) {
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(m0), "=r"(m1), "=r"(m2), "=r"(m3) : "r"(stage + kMetaOff + r * 16));
        n_words = lds_u32(stage + kInfoOff + 8);
        hdr = lds_u32(stage + kHdrOff + cr * 4);
        pdd_len = lds_u32(stage + kInfoOff);
        res_cnt = lds_u32(stage + kInfoOff + 4);
      }
      if (!__all_sync(0xFFFFFFFFu, ok)) break;
      asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                   ::"r"(tmem_base + lane_base + kColMetaT + 4 * wb), "r"(m0), "r"(m1), "r"(m2), "r"(m3) : "memory");
      uint32_t bad = 0;
      const uint32_t room = a.block_area - kPddOff;             // bytes a block may use after its fixed part
      const bool lens_ok = pdd_len <= room && res_cnt <= room / 4 && ((pdd_len + 3u) & ~3u) + 4u * res_cnt <= room &&
                           n_words <= 3u && pdd_len == n_words * 512u;
      if (lens_ok) decode_chain(stage, wr, hdr, stage + kPddOff + cr * 4, n_words, &bad);
      else bad = 3u;
      __syncwarp();
      if (lens_ok) {                                              // Residual layer: (position, value) entries go to W_r too
        scatter_residual<kLongRes>(stage + kPddOff + ((pdd_len + 3u) & ~3u), wr, r, res_cnt, &bad);
      }
      if (bad) atomicCAS(a.status, 0u, kStBadBlock | (bad << 8) | (static_cast<uint32_t>(i) << 12));
      fence_proxy_async_smem();                                   // generic-proxy writes -> MMA reads
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      mbar_arrive_leader<S>(bar(kBarDec, s));
      s += AG;
      while (s >= a.n_w) { s -= a.n_w; ph ^= 1u; }
      wb += AG;
      while (wb >= a.n_wr) { wb -= a.n_wr; ++use; }
    }
    // The last row-tile of this CTA's range, if other CTAs finish it: the decode warps, idle by now, read
    // the partial sums together with the epilogue warps (an accumulator is as wide as 256 columns, and
    // four warps alone had 16 us of loads in a row in front of them on 4096 x 4096, N = 128).
    const uint32_t vrow = (t_end - 1) / TK;
    if (vrow * TK >= t_begin && (vrow + 1) * TK > t_end) {
      if (__all_sync(0xFFFFFFFFu, mbar_wait(bar(kBarReduce, 0), 0, wctx, kStEpilogueTail, kHandOverLimitNs))) {
        tc_fence_after();
        __threadfence();
        const int last_seg = static_cast<int>(vrow - vrow_begin);
        const uint32_t acc = tmem_base + lane_base + static_cast<uint32_t>((a.n_acc == 2 ? last_seg & 1 : 0) * a.n_pad[less]);
        write_columns<XT, S, true>(a, less, acc, r, vrow, 16 * (g + 1), 16 * (kGroups + 1), owner_of((vrow + 1) * TK - 1, T, G) - static_cast<int>(unit),
                          wr_base + static_cast<uint32_t>(warp - kDecodeWarp0) * kTurnBytes);   // (the W_r buffers are idle too)
      }
    }
  } else if (warp >= kEpilogueWarp0) {
    // ------------------------------------------------------------------ epilogue
    const int et = tid - kEpilogueWarp0 * 32;                    // row of the tile = tensor-memory lane
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    int seg = 0;
    uint32_t t = t_begin;
    pdl_wait();   // Y, the partial sums and their flags may still be in use by the previous kernel
    while (t < t_end) {
      const uint32_t vrow = t / TK;
      const uint32_t row_begin = vrow * TK, row_end = row_begin + TK;
      const uint32_t seg_end = row_end < t_end ? row_end : t_end;
      const bool complete = (t == row_begin) && (seg_end == row_end);
      const int b = a.n_acc == 2 ? seg & 1 : 0, b_use = a.n_acc == 2 ? seg >> 1 : seg;
      const int c_first = owner_of(row_begin, T, G), c_last = owner_of(row_end - 1, T, G);
      // A shared row-tile is finished by the CTA that owns its first tile; for that CTA it is the last segment.
      const bool reducer = !complete && static_cast<int>(unit) == c_first;
      const int n_others = c_last - c_first;
      if (!named_bar_all(kEpilogueBarrier, 128, mbar_wait_unit<S>(bar(kBarAccFull, b), b_use & 1, wctx, kStEpilogueAccFull))) break;
      tc_fence_after();
      const uint32_t acc_tmem = tmem_base + lane_base + static_cast<uint32_t>(b * a.n_pad[less]);
      bool ready = true;
      if (reducer) {
        // The contributors (the CTAs after this one, or its counterparts in the pairs after this one) store their partial sums and raise their flags;
        // the sum runs in ascending CTA order, so the result does not depend on timing.  Every
        // contributor holds an SM or gets one without waiting for this CTA; the wait is bounded.
        bool ok = true;
        if (et < 32) {
          for (int base = 0; base < n_others && ok; base += 32) {
            bool pending = base + et < n_others;
            const int c_id = S * (c_first + 1 + base + et) + static_cast<int>(rank);
            unsigned long long t_slow = 0;
            for (uint32_t it = 0; __any_sync(0xFFFFFFFFu, pending); ++it) {
              if (pending) {
                unsigned int up;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(up) : "l"(a.flags + c_id) : "memory");
                if (up != 0u) {
                  pending = false;
                  a.flags[c_id] = 0u;                             // leave the workspace cleared
                }
              }
              if ((it & 15u) == 15u) {
                const unsigned long long now = global_timer();
                if (t_slow == 0) t_slow = now;
                const bool out = *abort_flag != 0 || now - t_slow > kWaitLimitNs;
                if (__any_sync(0xFFFFFFFFu, out)) {
                  if (et == 0) { atomicCAS(a.status, 0u, static_cast<uint32_t>(kStEpilogueFlags)); *abort_flag = 1; }
                  ok = false;
                  break;
                }
              }
            }
          }
          __syncwarp();
        }
        if (et == 0 && ok) mbar_arrive(bar(kBarReduce, 0));       // the decode warps take part
        ready = named_bar_all(kEpilogueBarrier, 128, ok);
        __threadfence();                                          // the others' partial sums, after their flags
      }
      if (ready) {
        const uint32_t turn = bar0 + 1024u + static_cast<uint32_t>(warp & 3) * kTurnBytes;
        if (complete) {
          write_columns<XT, S, false>(a, less, acc_tmem, et, vrow, 0, 16, 0, turn);
        } else if (reducer) {
          write_columns<XT, S, true>(a, less, acc_tmem, et, vrow, 0, 16 * (kGroups + 1), n_others, turn);
        } else {
          float* mine = a.partials + static_cast<size_t>(a.n_pad[less]) * 128 * blockIdx.x + et;
#pragma unroll 1
          for (int c0 = 0; c0 < a.n_pad[less]; c0 += 16) {
            uint32_t v[16];
            TmemLd<16>::ld(acc_tmem + c0, v);
            tmem_wait_ld<16>(v);
#pragma unroll
            for (int c = 0; c < 16; ++c) __stcg(mine + (c0 + c) * 128, __uint_as_float(v[c]));
          }
        }
      }
      tc_fence_before();
      mbar_arrive_leader<S>(bar(kBarAccEmpty, b));
      if (!complete && !reducer) {
        __threadfence();                                          // the partial sums, before the flag
        named_bar_sync(kEpilogueBarrier, 128);
        if (et == 0) asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(a.flags + blockIdx.x), "r"(1u) : "memory");
      }
      ++seg;
      t = seg_end;
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  sync_all<S>();                               // (neither CTA goes while the other may still arrive on its barriers)
  if (warp == kClearWarp) {
    tc_fence_after();
    tmem_dealloc<S>(tmem_base);
  }
}

template <bool XT, int S, bool kLongRes>
int launch_wide_kernel(const CUtensorMap& map, const WideArgs& args, int grid, uint32_t smem_bytes, cudaStream_t stream) {
  {
    int dev = 0;
    TL3_CUDA(cudaGetDevice(&dev));
    static std::mutex mu;
    static std::vector<char> configured;                          // per device, as in tl3_spmm.cu
    std::lock_guard<std::mutex> lock(mu);
    if (static_cast<size_t>(dev) >= configured.size()) configured.resize(dev + 1, 0);
    if (!configured[dev]) {
      TL3_CUDA(cudaFuncSetAttribute(tl3_spmm_wide_kernel<XT, S, kLongRes>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemLimit)));
      configured[dev] = 1;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreadsOf<S>);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see pdl_wait() in the kernel
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = S;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = S == 1 ? 1 : 2;
  TL3_CUDA(cudaLaunchKernelEx(&cfg, tl3_spmm_wide_kernel<XT, S, kLongRes>, map, args));
  TL3_CUDA(cudaGetLastError());
  return TL3_OK;
}

template <bool XT, int S>
int launch_wide(const CUtensorMap& map, const WideArgs& args, bool long_res, int grid, uint32_t smem_bytes, cudaStream_t stream) {
  return long_res ? launch_wide_kernel<XT, S, true>(map, args, grid, smem_bytes, stream) : launch_wide_kernel<XT, S, false>(map, args, grid, smem_bytes, stream);
}

}  // namespace

// Columns per pass, and whether CTAs work in pairs.  More columns decode W less often, fewer give a small
// matrix more row-tiles to share out and less to add up at the end.  The estimate of a launch, in us, from
// measured launches: a tile costs 0.45 (its decode) + 0.0036 per column for a CTA alone, 0.8 + 0.0014 for a
// pair, which is the way above 128 columns: half of X per CTA leaves room for more blocks in flight and
// halves what the tensor cores read of it (20480 x 5120, N = 512: 110 us, alone 123; 5120 x 20480, N = 200:
// 56 and 66), while up to 128 columns a cluster's start costs a short launch more than that gains (1024 x 1024, N = 128:
// 11.3 us, alone 9.5; 5120 x 5120, N = 160: 23.6, alone 23.7).  Passes of up to 128 columns are priced as a CTA alone
// also where ctas_together() then takes pairs for them: those differ by a few per cent, passes by tens.  The CTAs that share a row-tile hand over n_pad columns each at
// 0.008 per column and CTA.  (1024 x 1024, N = 500: 23 us in 2 passes, 17 in 3, 13 in 4; 20480 x 5120, N = 512:
// 125 in 2, 142 in 3, 160 in 4, all with one CTA per tile.)
constexpr int kAloneColumns = 128;

// Long launches of 65 to 128 columns go in pairs as well: from 32 tiles per CTA on what a tile saves by half of X
// outweighs the cluster's start and the columns that a multiple of 32 adds.  (us alone / in pairs, N = 128, X [batch, hidden] and
// [hidden, batch]: 20480 x 5120, 43 tiles, 45.0 / 42.2 and 46.2 / 43.8; 33 tiles, 8704 x 9216, 37.7 / 36.4 and 39.0 / 38.7, 20480 x
// 3840 35.7 / 33.8 and 36.2 / 35.2; 36864 x 9216 127 / 118.  With 19 to 20 tiles 0.94 to 1.05 of alone, N = 112 on 7000 x 7000
// 27.9 / 28.6; 4096 x 4096, 7 tiles, 17.1 / 19.1.)  Up to 64 columns a CTA alone is never
// slower (1000 x 20000, N = 128 in passes of 64 23.4 / 24.4).
// Few row-tiles are shared by many CTAs, and pairs take longer to hand over the partial sums (and do an odd last row-tile
// twice): above 80 columns they lose there.  (N = 128, the same two layouts: 9 row-tiles 47.1 / 47.9 and 49.9 / 56.4, 15
// 43.1 / 44.7 and 45.5 / 49.8, 29 40.3 / 39.7 and 42.0 / 43.0, 37 38.3 / 38.4 and 40.1 / 41.3, 45 39.3 / 38.3 and 40.7 / 40.9, 61
// 40.2 / 38.7 and 41.8 / 41.7; N = 96 and 112 as N = 128.)  Up to 80 they win from two on (N = 80, 5 row-tiles 49.6 / 47.3, 15 39.2 / 38.8,
// 29 37.0 / 36.0; 1 row-tile 73.7 / 74.7).  One rule for both layouts, so that they give the same bits.
constexpr int kPairTiles = 32, kPairRowTiles = 36;
static int ctas_together(const tl3_matrix* m, int N, int n_pad, int sm_count) {
  if (n_pad > kAloneColumns) return 2;
  const int64_t tiles = m->n_tiles * ((N + n_pad - 1) / n_pad);
  return n_pad > kAloneColumns / 2 && tiles >= static_cast<int64_t>(kPairTiles) * sm_count && m->tiles_m >= (n_pad > 80 ? kPairRowTiles : 2) ? 2 : 1;
}

static int wide_columns(const tl3_matrix* m, int N, int sm_count) {
  double best = 0;
  int best_n = 0;
  for (int passes = (N + kWideColumns - 1) / kWideColumns; passes <= (N + 63) / 64; ++passes) {
    const int each = (N + passes - 1) / passes;
    const int n_pad = each <= kAloneColumns ? (each + 15) / 16 * 16 : (each + 31) / 32 * 32;
    const double rows = static_cast<double>(m->tiles_m) * ((N + n_pad - 1) / n_pad);
    const double per_cta = rows * m->tiles_k / sm_count;
    const double ctas = per_cta < 1 ? static_cast<double>(m->tiles_k) : sm_count / rows;   // that share a row-tile
    const double tile = n_pad <= kAloneColumns ? 0.45 + 0.0036 * n_pad : 0.8 + 0.0014 * n_pad;
    const double t = (per_cta < 1 ? 1.0 : per_cta) * tile + 0.008 * n_pad * (ctas > 1 ? ctas : 1.0);
    if (best_n == 0 || t < best) { best = t; best_n = n_pad; }
  }
  return best_n;
}

int spmm_wide(const tl3_matrix* m, const void* X, int64_t ldx, void* Y, int64_t ldy, int N, const tl3_epilogue* ep, bool xt,
              void* workspace, void* stream) {
  if ((ldx & 7) != 0 || (reinterpret_cast<uintptr_t>(X) & 15) != 0 || (reinterpret_cast<uintptr_t>(Y) & 1) != 0 ||
      (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return TL3_ERR_INVALID_ARG;
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  if (di.cc_major != 10) return TL3_ERR_UNSUPPORTED;

  WideArgs a{};
  int n_pad = wide_columns(m, N, di.sm_count);
  const int S = ctas_together(m, N, n_pad, di.sm_count);
  if (S == 2) n_pad = (n_pad + 31) / 32 * 32;                       // (an MMA of 256 rows takes multiples of 32)
  a.block_area = (m->max_block_bytes + 1023u) / 1024u * 1024u;
  a.n_pad[0] = n_pad;
  // (The smallest workspace that serves any N has room for 128 columns: only wider passes are ever halved.  20480 x 5120, N = 128
  // with memory that was only zeroed: in one pass 42.5 us, in two 69.7.)
  a.n_pad[1] = n_pad <= kAloneColumns ? n_pad : (n_pad / 2 + 31) / 32 * 32;
  for (int i = 0; i < 2; ++i) a.chunks[i] = static_cast<uint32_t>((N + a.n_pad[i] - 1) / a.n_pad[i]);
  a.x_bytes = xt ? static_cast<uint32_t>(n_pad / S) * 128u : static_cast<uint32_t>((n_pad / S + 63) / 64) * 8192u;   // per CTA
  a.n_acc = 2 * n_pad <= static_cast<int>(kColMetaT) ? 2 : 1;
  {
    // A W_r buffer per decode group (with two of them instead of three 20480 x 5120, N = 512 took 131 us, not
    // 122, with three instead of four, in pairs, 113, not 108), at least as many blocks, and four X slices, three
    // for a CTA alone; with large blocks less, down to two of each; with small ones what is left goes to
    // blocks (five are enough), then to X.
    const uint32_t room = kSmemLimit - kSlack;
    auto blocks = [&]() -> int {
      const uint32_t fixed = a.n_wr * kWrBytes + a.n_x * a.x_bytes;
      return fixed < room ? static_cast<int>((room - fixed) / a.block_area) : 0;
    };
    a.n_wr = S == 1 ? kGroupsOf<1> : kGroupsOf<2>;
    a.n_x = S == 1 ? 3 : 4;
    while (blocks() < a.n_wr && a.n_x > 3) --a.n_x;
    while (blocks() < a.n_wr && a.n_wr > 3) --a.n_wr;
    while (blocks() < a.n_wr && a.n_x > 2) --a.n_x;
    while (blocks() < a.n_wr && a.n_wr > 2) --a.n_wr;
    while (a.n_x < kMaxRing) {
      ++a.n_x;
      if (blocks() < 5) { --a.n_x; break; }
    }
    a.n_w = blocks();
    if (a.n_w > kMaxRing) a.n_w = kMaxRing;
    if (a.n_w < a.n_wr) return kWideNoPlan;                       // (blocks of more Residual entries than a tile has windows: none that an encoder makes)
  }
  const uint32_t smem_bytes = a.n_w * a.block_area + a.n_x * a.x_bytes + a.n_wr * kWrBytes + kSlack;

  EncodeTiledFn encode = encode_tiled_fn();
  if (!encode) return TL3_ERR_UNSUPPORTED;
  CUtensorMap map;
  // dims {N, K}, box {64 columns, 64 k}; transposed: dims {K, N}, box {64 k, n_pad / S rows}.  What lies beyond reads as zero.
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(xt ? m->K : N), static_cast<cuuint64_t>(xt ? N : m->K)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(ldx) * 2};
  const cuuint32_t box[2] = {64, static_cast<cuuint32_t>(xt ? n_pad / S : 64)};
  const cuuint32_t elem_strides[2] = {1, 1};
  const CUresult cr = encode(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(X), dims, strides, box, elem_strides,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS) { set_cuda_error(static_cast<int>(cr)); return TL3_ERR_CUDA; }

  const unsigned long long total = static_cast<unsigned long long>((m->tiles_m + S - 1) / S) * m->tiles_k * a.chunks[0];
  const int units = static_cast<int>(total < static_cast<unsigned long long>(di.sm_count / S) ? total : di.sm_count / S);
  // the kernel splits the tiles in 32-bit arithmetic, whichever the columns of a pass
  const unsigned long long most = total / a.chunks[0] * a.chunks[1];
  if (most * static_cast<unsigned long long>(units + 1) >= (1ull << 32)) return kWideNoPlan;
  const int grid = S * units;
  const WorkspaceLayout wl = workspace_layout(N, di.sm_count);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  a.blob = static_cast<const uint8_t*>(m->dptr);
  a.dir = reinterpret_cast<const DirEntry*>(a.blob + m->dir_offset);
  a.tiles_m = static_cast<uint32_t>(m->tiles_m);
  a.tiles_k = static_cast<uint32_t>(m->tiles_k);
  a.M = static_cast<int>(m->M);
  a.N = N;
  a.ldy = ldy;
  a.Y = static_cast<__half*>(Y);
  a.bias = ep ? static_cast<const __half*>(ep->bias) : nullptr;
  a.act = ep ? ep->activation : TL3_ACT_NONE;
  a.partials = reinterpret_cast<float*>(ws + wl.partials_off);
  a.flags = reinterpret_cast<unsigned int*>(ws + wl.flags_off);
  a.status = reinterpret_cast<unsigned int*>(ws + wl.status_off);
  a.room = ws + wl.room_off;
  m->last_ctas = grid; m->last_stages = a.n_w; m->last_smem = static_cast<int>(smem_bytes);
  m->last_pass.store(n_pad | S << 16 | a.n_acc << 24, std::memory_order_relaxed);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (S == 2) return xt ? launch_wide<true, 2>(map, a, long_residual(m), grid, smem_bytes, st) : launch_wide<false, 2>(map, a, long_residual(m), grid, smem_bytes, st);
  return xt ? launch_wide<true, 1>(map, a, long_residual(m), grid, smem_bytes, st) : launch_wide<false, 1>(map, a, long_residual(m), grid, smem_bytes, st);
}

}  // namespace tl3
