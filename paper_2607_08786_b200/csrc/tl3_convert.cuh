// What the encoder, the packer and the converter on the GPU share: scans over the CTA, the classification of
// a window, the pairs of a tile, the coordinates of the device image, and the packer's steps from the sets of
// empty slots and surplus weights to the finished block (tl3_pack.cpp has the reasoning behind that layout).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "tl3_internal.h"

namespace tl3 {
namespace {

constexpr int kTileThreads = 256;          // one CTA per tile
constexpr uint32_t kMaxd = 15;
constexpr int kChainCap = 255;
constexpr int kSlots = kTileM * kH;        // 8192
constexpr int kChains = 128;               // of the device image
constexpr int kFlagWords = kSlots / 32;    // 256: one per thread
constexpr uint32_t kHeadBytes = kPddOff - kInfoOff;               // info words and chain starts of a block
constexpr uint32_t kMaxHead = kHeadBytes + 3u * 4u * kChains;     // ... and its code words

__device__ __forceinline__ uint32_t u_of_pos(uint32_t pos) {
  const uint32_t r = pos >> 6, q = (pos >> 1) & 31u, s = pos & 1u;
  const uint32_t bank = (((q >> 2) ^ (r & 7u)) << 2) | (q & 3u);
  return (bank << 8) | (s << 7) | r;
}
__device__ __forceinline__ uint32_t pos_of_u(uint32_t u) {
  const uint32_t r = u & 127u, s = (u >> 7) & 1u, bank = u >> 8;
  const uint32_t q = (((bank >> 2) ^ (r & 7u)) << 2) | (bank & 3u);
  return r * 64u + 2u * q + s;
}
__device__ __forceinline__ uint32_t delta_bytes(uint32_t gt, uint32_t gr) { return (gt - 1) / 15 + (gr - 1) / 15 + 1; }
__device__ __forceinline__ uint32_t align_up_d(uint32_t x, uint32_t a) { return (x + a - 1) / a * a; }

// exclusive scan over the threads of the CTA (two 16-bit sums per word where a caller packs them); *total
// gets the sum in every thread
__device__ __forceinline__ uint32_t scan_cta(uint32_t v, uint32_t* s_warp, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  uint32_t base = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kTileThreads / 32; ++w) {
    base += w < warp ? s_warp[w] : 0u;
    all += s_warp[w];
  }
  *total = all;
  __syncthreads();
  return base + x - v;
}

// dummy points in front of a pair that lies gt slots and gr positions behind the one before it
__device__ __forceinline__ uint32_t dummies(uint32_t gt, uint32_t gr) {
  return (gt > kMaxd ? (gt - 1) / kMaxd : 0u) + (gr > kMaxd ? (gr - 1) / kMaxd : 0u);
}

// One window of four consecutive weights (Sec. 3.2, Sparse-TC layer): the first two non-zeros stay;
// a window short of two completes its index pair with the lowest unused positions (those slots are
// empty); the third and fourth non-zero are surplus and always sit at in-window index 2 or 3.
// Entry p of the table, for non-zeros at the positions set in p: x = byte selector that puts the two
// weights of the index pair into one word | metadata nibble << 16, y = mask of the occupied slots.
__device__ __forceinline__ uint2 window_entry(uint32_t p) {
  const uint32_t first = __ffs(p) - 1u, second = __ffs(p & (p - 1u)) - 1u;
  uint32_t i0 = 0, i1 = 1, mask = 0;
  if (__popc(p) >= 2) { i0 = first; i1 = second; mask = 0xFFFFFFFFu; }
  else if (p == 1u) mask = 0x0000FFFFu;
  else if (p != 0u) { i1 = first; mask = 0xFFFF0000u; }
  return make_uint2((0x10u + 0x22u * i0) | (0x10u + 0x22u * i1) << 8 | (i0 | i1 << 2) << 16, mask);
}

// The dense matrix that a tile is read from.
struct DenseView {
  const uint16_t* W;            // device, row-major, leading dimension ldw
  long long M, K, ldw;
  int vec;                      // windows may be loaded as 8 bytes (base and row pitch are multiples of 8 bytes)
};
inline DenseView dense_view(const void* W, long long M, long long K, long long ldw) {
  return {static_cast<const uint16_t*>(W), M, K, ldw, (reinterpret_cast<uintptr_t>(W) & 7) == 0 && (ldw & 3) == 0};
}

// Shared memory SM of the two functions below: nz[4][128] (non-zeros of a row by in-window index, one bit per window),
// vals (image of W_t: kept values, zero where a slot is empty), high (weights 2 and 3 of every window: the
// surplus value at position rho is half-word rho), nib (metadata of every window), window (window_entry()).
// Lane q holds window q of the warp's rows; four votes make a row's masks.  A barrier is left to the caller.
template <class SM>
__device__ __forceinline__ void classify_tile(const DenseView& a, long long tm, long long tk, SM& sm, bool values) {
  constexpr int kRows = kTileM / (kTileThreads / 32);   // rows per warp
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 16) sm.window[tid] = window_entry(static_cast<uint32_t>(tid));
  uint2 w[kRows];
  {
    const int row0 = warp * kRows;
    const long long left_m = a.M - tm * kTileM - row0, left_k = a.K - tk * kTileK - 4 * lane;
    const int rows = left_m < kRows ? static_cast<int>(left_m) : kRows;                // (may be negative)
    const int cols = left_k < 4 ? static_cast<int>(left_k) : 4;
    const uint16_t* src = a.W + (tm * kTileM + row0) * a.ldw + tk * kTileK + 4 * lane;
    if (a.vec && rows == kRows && cols == 4) {
#pragma unroll
      for (int k = 0; k < kRows; ++k, src += a.ldw) w[k] = __ldg(reinterpret_cast<const uint2*>(src));
    } else {
#pragma unroll
      for (int k = 0; k < kRows; ++k, src += a.ldw) {
        uint32_t h[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = k < rows && i < cols ? src[i] : 0u;
        w[k] = make_uint2(h[0] | h[1] << 16, h[2] | h[3] << 16);
      }
    }
  }
  __syncthreads();                             // (the window table)
  uint32_t mine[4] = {0u, 0u, 0u, 0u};         // lane k: masks of the warp's row k
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    // a half-word without its sign is non-zero if adding 0x7FFF carries into its top bit
    const uint32_t x = (w[k].x & 0x7FFF7FFFu) + 0x7FFF7FFFu, y = (w[k].y & 0x7FFF7FFFu) + 0x7FFF7FFFu;
    const uint32_t m0 = __ballot_sync(0xFFFFFFFFu, (x & 0x8000u) != 0), m1 = __ballot_sync(0xFFFFFFFFu, static_cast<int>(x) < 0);
    const uint32_t m2 = __ballot_sync(0xFFFFFFFFu, (y & 0x8000u) != 0), m3 = __ballot_sync(0xFFFFFFFFu, static_cast<int>(y) < 0);
    if (lane == k) { mine[0] = m0; mine[1] = m1; mine[2] = m2; mine[3] = m3; }
    if (values) {
      const int at = (warp * kRows + k) * 32 + lane;
      const uint32_t bits = ((x >> 15) & 0x00010001u) | ((y >> 13) & 0x00040004u);
      const uint2 e = sm.window[(bits | bits >> 15) & 15u];
      reinterpret_cast<uint32_t*>(sm.vals)[at] = __byte_perm(w[k].x, w[k].y, e.x) & e.y;
      sm.high[at] = w[k].y;
      sm.nib[at] = static_cast<uint8_t>(e.x >> 16);
    }
  }
  if (lane < kRows) {
#pragma unroll
    for (int i = 0; i < 4; ++i) sm.nz[i][warp * kRows + lane] = mine[i];
  }
}

// Eight windows of metadata (`nib` of two words), the even one in the low nibble of its byte.
__device__ __forceinline__ uint32_t meta_word(uint2 v) { return __byte_perm(v.x | v.x >> 4, v.y | v.y >> 4, 0x6420u); }

// Entry L of a block's metadata, in tensor-memory lane order, from the metadata of its two rows (L & 7) + 16 (L >> 4) and
// eight below: two bytes (four windows) of every word.
__device__ __forceinline__ uint4 meta_entry(uint4 lo, uint4 hi, int half) {
  const uint32_t sel = half ? 0x7632u : 0x5410u;
  return make_uint4(__byte_perm(lo.x, hi.x, sel), __byte_perm(lo.y, hi.y, sel), __byte_perm(lo.z, hi.z, sel), __byte_perm(lo.w, hi.w, sel));
}

// The empty slots and surplus weights of a classified tile, and their pairs: the i-th surplus weight is parked in the
// i-th empty slot.  A thread takes a run of consecutive pairs and a scan over the threads gives every pair
// the place of its delta bytes: the chains of a tile (one per row) follow each other in the order of the pairs.
// Only a tile with a chain of more than 255 bytes, which is cut there, walks rows one by one.
struct TilePairs {
  uint32_t lo, hi;              // thread r < 128: windows of row r whose slot 0 / 1 is empty; 128 + r: whose weight 2 / 3 is surplus
  uint32_t count;               // of those
  int my_first;                 // (threads >= 128) index of the row's first surplus weight
  int totS, totE, P;            // surplus weights, empty slots, pairs
  int tot_cut;                  // pairs that cut chains have lost
  uint32_t tot_len;             // delta bytes of the tile
  int p0, p1;                   // this thread's pairs
  uint32_t tau_before, rho_before;   // the pair in front of them
  uint32_t pre;                 // delta bytes before them
  int chains;                   // chains that begin among them
  bool has_chain;               // (threads >= 128) row r has a chain, of len delta bytes
  int len;
};
// SM: list (empty slots ascending, then surplus positions ascending: a window has empty slots or surplus weights, not
// both, and never more than two of them), first / last (delta bytes before the first and after the last pair of a
// row), parked_end (first pair of a row that is not parked any more), moved (delta bytes that cut chains before a
// row have lost), warp_tmp, nnz (0).  cut(rho, i0, i1, before): the pairs that a cut chain leaves to the Residual
// layer, their positions in rho, `before` of them in rows above.
template <class SM, class Cut>
__device__ __forceinline__ TilePairs find_pairs(SM& sm, const Cut& cut) {
  TilePairs t;
  const int tid = threadIdx.x, lane = tid & 31;
  // ---- lists: threads 0..127 the empty slots of row tid, threads 128..255 the surplus weights of row tid - 128
  const int row = tid & (kTileM - 1);
  const bool surplus = tid >= kTileM;
  {
    const uint32_t n0 = sm.nz[0][row], n1 = sm.nz[1][row], n2 = sm.nz[2][row], n3 = sm.nz[3][row];
    const uint32_t two = (n0 & n1) | ((n0 | n1) & (n2 | n3)) | (n2 & n3);          // at least two non-zeros
    if (surplus) {
      t.lo = n0 & n1 & n2;                                                          // the weight at index 2 is a third one
      t.hi = n3 & ((n0 & n1) | ((n0 | n1) & n2));                                   // the weight at index 3 is a third or fourth
    } else {
      t.lo = ~two & ~n0;                                                            // slot 0 (index 0) is empty
      t.hi = ~two & ~(n1 | n2 | n3);                                                // slot 1 is empty
      const int n = __popc(n0) + __popc(n1) + __popc(n2) + __popc(n3);
      const int sum = __reduce_add_sync(0xFFFFFFFFu, n);
      if (lane == 0) atomicAdd(&sm.nnz, sum);
    }
  }
  t.count = static_cast<uint32_t>(__popc(t.lo) + __popc(t.hi));
  uint32_t tot = 0;
  uint32_t at = scan_cta(t.count | (surplus ? t.count << 16 : 0u), sm.warp_tmp, &tot);   // low half: both kinds, high half: surplus
  t.totS = static_cast<int>(tot >> 16);
  t.totE = static_cast<int>(tot & 0xFFFFu) - t.totS;
  t.P = t.totS < t.totE ? t.totS : t.totE;
  t.my_first = static_cast<int>(at >> 16);
  at &= 0xFFFFu;
  for (uint32_t any = t.lo | t.hi; any; any &= any - 1u) {
    const uint32_t bit = any & (0u - any), pos = static_cast<uint32_t>(row * kH) + 2u * (31u - __clz(bit));
    if (t.lo & bit) sm.list[at++] = static_cast<uint16_t>(pos);
    if (t.hi & bit) sm.list[at++] = static_cast<uint16_t>(pos + 1);
  }
  if (surplus) {
    const int end = t.my_first + static_cast<int>(t.count);
    sm.parked_end[row] = static_cast<uint16_t>(end < t.P ? end : t.P);
    sm.moved[row] = 0;
  }
  __syncthreads();

  // ---- pairs: thread t takes pairs [t * run, (t + 1) * run).  A pair that is the first of its row
  //      (rho in another row than the one before) starts a chain and has no delta byte.
  const uint16_t* const tau_list = sm.list;
  const uint16_t* const rho_list = sm.list + t.totE;
  const int run = (t.P + kTileThreads - 1) / kTileThreads;
  t.p0 = tid * run < t.P ? tid * run : t.P;
  t.p1 = t.p0 + run < t.P ? t.p0 + run : t.P;
  uint32_t bytes = 0;
  t.chains = 0;
  t.tau_before = 0;
  t.rho_before = 0xFFFFFFFFu;
  if (t.p0 > 0 && t.p0 < t.p1) { t.tau_before = tau_list[t.p0 - 1]; t.rho_before = rho_list[t.p0 - 1]; }
  {
    uint32_t tau = t.tau_before, rho = t.rho_before;
    for (int i = t.p0; i < t.p1; ++i) {
      const uint32_t nt = tau_list[i], nr = rho_list[i];
      if (nr / kH == rho / kH) bytes += 1u + dummies(nt - tau, nr - rho);
      else ++t.chains;
      tau = nt;
      rho = nr;
    }
  }
  t.tot_len = 0;
  t.pre = scan_cta(bytes, sm.warp_tmp, &t.tot_len);                                  // delta bytes before this run (at most 4096 pairs + 2 * 546 dummies)
  t.tot_cut = 0;
  {
    // where every row's chain begins and ends: the run has to be walked again for it, by the few
    // threads that hold the first or last pair of a row
    uint32_t tau = t.tau_before, rho = t.rho_before, at_byte = t.pre;
    for (int i = t.p0; i < t.p1; ++i) {
      const uint32_t nt = tau_list[i], nr = rho_list[i];
      if (nr / kH == rho / kH) at_byte += 1u + dummies(nt - tau, nr - rho);
      else sm.first[nr / kH] = static_cast<uint16_t>(at_byte);
      if (i + 1 == t.P || rho_list[i + 1] / kH != nr / kH) sm.last[nr / kH] = static_cast<uint16_t>(at_byte);
      tau = nt;
      rho = nr;
    }
  }
  __syncthreads();
  t.has_chain = surplus && t.my_first < t.P && t.count > 0;
  t.len = t.has_chain ? sm.last[row] - sm.first[row] : 0;
  if (__syncthreads_or(t.len > kChainCap)) {
    // ---- a chain is cut: its row is walked for the last pair that fits, what follows is Residual
    int n_cut = 0, lost = 0;
    if (t.len > kChainCap) {
      const int end = sm.parked_end[row];
      int i = t.my_first + 1, fit = 0;
      for (; i < end; ++i) {
        const int need = 1 + static_cast<int>(dummies(tau_list[i] - tau_list[i - 1], rho_list[i] - rho_list[i - 1]));
        if (fit + need > kChainCap) break;
        fit += need;
      }
      n_cut = end - i;
      lost = t.len - fit;
      t.len = fit;
      sm.parked_end[row] = static_cast<uint16_t>(i);
    }
    uint32_t t2 = 0;
    const uint32_t before = scan_cta(static_cast<uint32_t>(lost) | static_cast<uint32_t>(n_cut) << 16, sm.warp_tmp, &t2);
    if (surplus) sm.moved[row] = static_cast<uint16_t>(before & 0xFFFFu);
    t.tot_cut = static_cast<int>(t2 >> 16);
    t.tot_len -= t2 & 0xFFFFu;
    if (n_cut) {
      const int end = t.my_first + static_cast<int>(t.count) < t.P ? t.my_first + static_cast<int>(t.count) : t.P;
      cut(rho_list, end - n_cut, end, before >> 16);
    }
    __syncthreads();
  }
  return t;
}

// Layer statistics (Sec. 3.2 quotes their shares): counter `which` of nnz, n_tc, n_sf, n_res, n_dummy, n_slots_unused.  Every
// parked weight that does not start a chain has one byte, the other bytes are dummy points.
__device__ __forceinline__ int tile_statistic(int which, const TilePairs& t, int nnz, int n_chains) {
  const int n_sf = t.P - t.tot_cut;
  return which == 0 ? nnz : which == 1 ? nnz - t.totS : which == 2 ? n_sf : which == 3 ? t.tot_cut + t.totS - t.P
       : which == 4 ? static_cast<int>(t.tot_len) - (n_sf - n_chains) : t.totE - n_sf;
}

// shared memory of pack_block() beside the tile's arrays
struct PackWork {
  uint32_t flag[kFlagWords];     // bit u set: a surplus weight sits at u
  uint32_t empty[kFlagWords];    // bit u set: slot u is empty
  uint32_t bank_cand[33];        // empty slots before bank b
  int beyond[4];
  int real_bytes[4];
  uint32_t warp_tmp[kTileThreads / 32];
  int carry[kChains];            // parked elements that run i hands on to the next
  int len[kChains];              // delta bytes of device chain c
};

// From the bitmaps of `sm` (and beyond, real_bytes = 0; a barrier behind all of it) to the block:
//   vals      value slots of the tile by row-major position, the empty ones zero; parked values are put there
//   cand, sur room for the positions u of the empty slots and of the surplus weights, ascending (sur
//             begins where cand ends if sur_behind)
//   head      kMaxHead bytes for info words, chain starts and code words
//   value(u)  the surplus weight at u
//   place()   told the block's sizes, answers where it goes (null: nowhere, return)
//   meta(L)   entry L of the metadata;  extra(j)  canonical Residual entry j as position and value
template <class Value, class Place, class Meta, class Extra>
__device__ __forceinline__ void pack_block(PackWork& sm, uint16_t* vals, uint16_t* cand, uint16_t* sur, bool sur_behind, uint8_t* head_bytes,
                                           uint32_t n_extra, const Value& value, const Place& place, const Meta& meta, const Extra& extra) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t tot = 0;
  int n_cand = 0, n_pairs = 0;
  {
    uint32_t e = sm.empty[tid], f = sm.flag[tid];
    const uint32_t off = scan_cta(static_cast<uint32_t>(__popc(e)) | static_cast<uint32_t>(__popc(f)) << 16, sm.warp_tmp, &tot);
    n_cand = static_cast<int>(tot & 0xFFFFu);
    n_pairs = static_cast<int>(tot >> 16);
    if (sur_behind) sur = cand + n_cand;
    uint32_t oc = off & 0xFFFFu, os = off >> 16;
    if ((tid & 7) == 0) sm.bank_cand[tid >> 3] = oc;
    if (tid == 0) sm.bank_cand[32] = static_cast<uint32_t>(n_cand);
    for (; e; e &= e - 1u) cand[oc++] = static_cast<uint16_t>(tid * 32 + __ffs(e) - 1);
    for (; f; f &= f - 1u) sur[os++] = static_cast<uint16_t>(tid * 32 + __ffs(f) - 1);
  }
  __syncthreads();

  // (4) every bank gets a share of the parked elements proportional to its empty slots; its empty
  //     slots are cut into four runs of equal count and run q uses its first slots.  What a run
  //     cannot take is carried to the next: with d = wanted - size of a run, S its inclusive prefix
  //     sum, the carry out of run i is S_i - min(0, S_0 .. S_i), two scans over the 128 runs.
  int my_take = 0, my_src = 0;
  {
    int want = 0, size = 0;
    if (tid < kChains) {
      const uint32_t b = static_cast<uint32_t>(tid) >> 2, q = tid & 3u;
      const uint32_t c0 = sm.bank_cand[b], c1 = sm.bank_cand[b + 1], N_b = c1 - c0;
      const uint32_t lo = n_cand ? c0 * n_pairs / n_cand : 0u, hi = n_cand ? c1 * n_pairs / n_cand : 0u;   // (<= 8192^2)
      const uint32_t n_b = hi - lo, first = N_b * q / 4;
      size = static_cast<int>(N_b * (q + 1) / 4 - first);
      want = static_cast<int>(n_b * (q + 1) / 4 - n_b * q / 4);
      my_src = static_cast<int>(c0 + first);
    }
    const int d = want - size;
    int S = d;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, S, k);
      if (lane >= k) S += y;
    }
    if (lane == 31) sm.warp_tmp[warp] = static_cast<uint32_t>(S);
    __syncthreads();
    for (int w = 0; w < warp && w < 4; ++w) S += static_cast<int>(sm.warp_tmp[w]);
    __syncthreads();
    int low = S < 0 ? S : 0;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, low, k);
      if (lane >= k && y < low) low = y;
    }
    if (lane == 31) sm.warp_tmp[warp] = static_cast<uint32_t>(low);
    __syncthreads();
    for (int w = 0; w < warp && w < 4; ++w) { const int y = static_cast<int>(sm.warp_tmp[w]); low = y < low ? y : low; }
    if (tid < kChains) sm.carry[tid] = S - low;
    __syncthreads();
    if (tid < kChains) my_take = want + (tid ? sm.carry[tid - 1] : 0) - sm.carry[tid];
  }
  uint32_t n_sel = 0;
  const int i0 = static_cast<int>(scan_cta(static_cast<uint32_t>(my_take), sm.warp_tmp, &n_sel));   // (n_sel <= n_pairs)
  const uint16_t* const sel = cand + my_src;                // this thread's run of empty slots

  // (5) device chain c = the pairs [i0, i1) of run c.  One walk: for a chain of at most 0, 4, 8 and
  //     12 delta bytes, how many bytes it has, how many entries move a value, how many are cut off.
  int by[4] = {0, 0, 0, 0}, end_at[4] = {0, 0, 0, 0};
  {
    int end = 0;
    for (int i = 1; i < my_take; ++i) {
      end += static_cast<int>(delta_bytes(static_cast<uint32_t>(sel[i] - sel[i - 1]), static_cast<uint32_t>(sur[i0 + i] - sur[i0 + i - 1])));
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        if (end > 4 * w) ++by[w];
        else end_at[w] = end;
      }
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int sum = __reduce_add_sync(0xFFFFFFFFu, by[w]);
      const int real = __reduce_add_sync(0xFFFFFFFFu, my_take > 1 ? my_take - 1 - by[w] : 0);
      if (lane == 0 && sum) atomicAdd(&sm.beyond[w], sum);
      if (lane == 0 && real) atomicAdd(&sm.real_bytes[w], real);
    }
  }
  __syncthreads();
  uint32_t n_words = 0;
  for (uint32_t w = 1; w < 4; ++w)
    if (512u * w + 4u * sm.beyond[w] < 512u * n_words + 4u * sm.beyond[n_words]) n_words = w;
  const int n_tail = n_words == 0 ? by[0] : n_words == 1 ? by[1] : n_words == 2 ? by[2] : by[3];
  const int n_bytes = n_words == 0 ? end_at[0] : n_words == 1 ? end_at[1] : n_words == 2 ? end_at[2] : end_at[3];
  const uint32_t tot_tail = static_cast<uint32_t>(sm.beyond[n_words]);
  const uint32_t pdd_len = n_words * 4u * kChains;
  const uint32_t n_left = static_cast<uint32_t>(n_pairs) - n_sel;
  const uint32_t res_cnt = tot_tail + n_left + n_extra;
  const uint32_t block_bytes = align_up_d(kPddOff + pdd_len + 4u * res_cnt, 16);
  uint8_t* const blk = place(pdd_len, res_cnt, static_cast<uint32_t>(sm.real_bytes[n_words]), block_bytes);
  if (!blk) return;
  if (tid < kChains) sm.len[tid] = n_bytes;
  const uint32_t off_tail = scan_cta(static_cast<uint32_t>(n_tail), sm.warp_tmp, &tot);

  // (7) the block.  Info words, chain starts and code words are put together in shared memory.
  const uint32_t head_words = (kHeadBytes + pdd_len) / 4;
  uint32_t* head = reinterpret_cast<uint32_t*>(head_bytes);
  for (uint32_t i = tid; i < head_words; i += kTileThreads) head[i] = 0u;      // (padding of short chains)
  __syncthreads();
  uint32_t* res = reinterpret_cast<uint32_t*>(blk + kPddOff + pdd_len);
  if (tid < kChains) {
    // chain slot w * 32 + l holds the w-th longest of the four chains of bank l (ties: lower chain first)
    const int b = tid >> 2;
    int w = 0;
    for (int c = 4 * b; c < 4 * b + 4; ++c)
      if (sm.len[c] > n_bytes || (sm.len[c] == n_bytes && c < tid)) ++w;
    const uint32_t slot = static_cast<uint32_t>(w * 32 + b);
    uint32_t hdr = 0xFFFFFFFFu;
    uint8_t* code = head_bytes + kHeadBytes + slot * 4u;
    uint32_t at = 0;
    const int kept = my_take - n_tail;
    uint32_t u0 = 0, r0 = 0;
    for (int i = 0; i < kept; ++i) {
      const uint32_t u = sel[i], r_u = sur[i0 + i];
      if (i == 0) {
        hdr = u | r_u << 16;
      } else {
        uint32_t gt = u - u0, gr = r_u - r0;
        auto put = [&](uint8_t v) { code[(at >> 2) * (4u * kChains) + (at & 3u)] = v; ++at; };
        while (gt > 15) { put(0x0F); gt -= 15; }           // dummy points (a zero nibble moves nothing)
        while (gr > 15) { put(0xF0); gr -= 15; }
        put(static_cast<uint8_t>(gt | gr << 4));
      }
      u0 = u;
      r0 = r_u;
      vals[pos_of_u(u)] = value(r_u);     // the value is parked in its new slot
    }
    head[4 + slot] = hdr;
    for (int i = kept; i < my_take; ++i) {     // the chain is full: the rest of its run goes to the Residual list
      const uint32_t r_u = sur[i0 + i];
      res[off_tail + static_cast<uint32_t>(i - kept)] = r_u | static_cast<uint32_t>(value(r_u)) << 16;
    }
  } else {
    // meanwhile the other warps: metadata in tensor-memory lane order ...
    reinterpret_cast<uint4*>(blk + kMetaOff)[tid - kChains] = meta(tid - kChains);
    // ... and surplus weights beyond the selected empty slots, the canonical Residual entries, the padding
    const uint32_t j0 = static_cast<uint32_t>(tid - kChains);
    for (uint32_t i = n_sel + j0; i < static_cast<uint32_t>(n_pairs); i += kTileThreads - kChains)
      res[tot_tail + (i - n_sel)] = sur[i] | static_cast<uint32_t>(value(sur[i])) << 16;
    for (uint32_t j = j0; j < n_extra; j += kTileThreads - kChains) {
      const uint2 e = extra(j);
      res[tot_tail + n_left + j] = u_of_pos(e.x) | e.y << 16;
    }
    const uint32_t n_pad = (align_up_d(block_bytes, kBlockAlign) - (kPddOff + pdd_len + 4u * res_cnt)) / 4;
    if (j0 < n_pad) res[res_cnt + j0] = 0u;
  }
  if (tid == 0) {
    head[0] = pdd_len;
    head[1] = res_cnt;
    head[2] = n_words;
  }
  __syncthreads();
  // values: row r of the K-major 128-byte-swizzled image; word `bank` of the row holds both slots of one window
#pragma unroll
  for (int i = tid; i < kSlots / 8; i += kTileThreads)
    reinterpret_cast<uint4*>(blk)[i] = reinterpret_cast<const uint4*>(vals)[i ^ ((i >> 3) & 7)];
  for (uint32_t i = tid; i < head_words / 4; i += kTileThreads) reinterpret_cast<uint4*>(blk + kInfoOff)[i] = reinterpret_cast<const uint4*>(head)[i];
}

}  // namespace
}  // namespace tl3
