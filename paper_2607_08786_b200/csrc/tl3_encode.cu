// Format conversion on the GPU: dense masked fp16 W (device) -> the canonical three-layer container
// of Sec. 3.2, byte for byte what tl3_encode() builds on the host.  (The paper converts on the CPU,
// 41-93 s per model, Sec. 5.3 "Storage Format Conversion".)
//
// Tiles are independent, so one CTA of eight warps takes one 128 x 128 tile.
//   classify a lane loads one window of four weights, a warp one row at a time (a coalesced 256-byte
//            load); four votes turn the row's non-zeros into four 32-bit masks, one per in-window
//            index, and from there on a row is classified with a few bit operations on its masks
//            (which two weights stay, which slots are empty, which weights are surplus);
//   lists    one thread per row and kind writes the positions of the row's empty slots and of its
//            surplus weights into shared memory at their scanned places, sorted by construction;
//   pairs    the i-th surplus weight is parked in the i-th empty slot.  A thread takes a run of
//            consecutive pairs and a scan over the threads gives every pair the place of its delta
//            bytes: the chains of a tile (one per row: 16-bit starts, 4-bit delta pairs, dummy points
//            for spans above the 4-bit range) follow each other in the order of the pairs.  Only a
//            tile with a chain of more than 255 bytes, which is cut there, walks rows one by one;
//   residual what found no empty slot (and what a cut chain left over) goes to the Residual list.
// The kernel runs twice: first it only counts the PDD bytes and Residual entries of every tile,
// a one-block scan turns the counts into the offsets of the tile directory, then it runs again
// and writes the bytes where they belong.
// What bounds it is the number of instructions it issues (its memory traffic, W once per pass and the
// container once, is a few microseconds).  Two passes on 5120 x 5120 at 50 % sparsity: 31 + 52 us.
// A thread per row, two-byte accesses a row pitch apart and 512 atomics per tile on four
// addresses took 351 + 898 us; coalesced rows that every lane classified for itself, with chains
// walked by a thread per row, 57 + 89 us.
#include <cuda_runtime.h>

#include <cstdint>
#include <new>
#include <vector>

#include "tl3_internal.h"

namespace tl3 {

void set_cuda_error(int e);

#define TL3_ENC_CUDA(expr)                                    \
  do {                                                        \
    cudaError_t e_ = (expr);                                  \
    if (e_ != cudaSuccess) {                                  \
      tl3::set_cuda_error(static_cast<int>(e_));              \
      rc = TL3_ERR_CUDA;                                      \
      goto done;                                              \
    }                                                         \
  } while (0)

namespace {

constexpr int kEncThreads = 256;
constexpr int kEncRows = kTileM / (kEncThreads / 32);   // rows per warp
constexpr uint32_t kMaxd = 15;
constexpr int kChainCap = 255;

struct EncodeArgs {
  const uint16_t* W;            // device, row-major, leading dimension ldw
  long long M, K, ldw;
  long long K_pad;
  int tiles_k;
  int vec;                      // windows may be loaded as 8 bytes (base and row pitch are multiples of 8 bytes)
  uint16_t* tc_vals;            // [M_pad][K_pad / 2]
  uint8_t* tc_meta;             // [M_pad][K_pad / 8]
  uint16_t* chain_tau0;         // [tiles][128]
  uint16_t* chain_rho0;
  uint8_t* chain_len;
  uint32_t* tile_dir;           // [tiles][4]: pdd_off, pdd_len, res_off, res_cnt
  uint8_t* pdd_bytes;           // emit pass only
  uint16_t* res_rho;
  uint16_t* res_val;
  unsigned long long* stats;    // nnz, n_tc, n_sf, n_res, n_dummy, n_slots_unused
  int emit;                     // 0: count pass (fills pdd_len and res_cnt of the directory), 1: write everything
};

// exclusive scan over the threads of the CTA; *total gets the sum in every thread
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
  for (int w = 0; w < kEncThreads / 32; ++w) {
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

struct EncodeSmem {
  uint16_t vals[kTileM * kH];   // image of W_t (kept values, then the parked ones too)
  uint32_t high[kTileM * 32];   // weights 2 and 3 of every window: the surplus value at position rho is half-word rho
  uint16_t list[kTileM * kH];   // empty slots ascending, then surplus positions ascending: a window has empty slots
                                // or surplus weights, not both, and never more than two of them
  uint8_t nib[kTileM * 32];     // metadata of every window; later the code bytes of the tile, while they fit
  uint32_t nz[4][kTileM];       // non-zeros of a row by in-window index, one bit per window
  uint2 window[16];
  uint16_t first[kTileM];       // delta bytes before the first pair of the row
  uint16_t last[kTileM];        // ... and after its last pair
  uint16_t parked_end[kTileM];  // first pair of the row that is not parked any more
  uint16_t moved[kTileM];       // delta bytes that cut chains before this row have lost
  uint32_t warp_tmp[kEncThreads / 32];
  int nnz, n_chains;
};
constexpr int kCodeStage = kTileM * 32;       // a tile has 1.5-2 KB of code bytes as a rule

__global__ void __launch_bounds__(kEncThreads, 4)
tl3_encode_kernel(const EncodeArgs a) {
  extern __shared__ __align__(16) uint8_t encode_smem_raw[];
  EncodeSmem& sm = *reinterpret_cast<EncodeSmem*>(encode_smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long tile = blockIdx.x;
  const long long tm = tile / a.tiles_k, tk = tile % a.tiles_k;
  const long long half_ld = a.K_pad / 2, meta_ld = a.K_pad / 8;
  if (tid < 16) sm.window[tid] = window_entry(static_cast<uint32_t>(tid));
  if (tid == 16) { sm.nnz = 0; sm.n_chains = 0; }

  // ---- classify: lane q holds window q of the warp's rows
  uint2 w[kEncRows];
  {
    const int row0 = warp * kEncRows;
    const long long left_m = a.M - tm * kTileM - row0, left_k = a.K - tk * kTileK - 4 * lane;
    const int rows = left_m < kEncRows ? static_cast<int>(left_m) : kEncRows;          // (may be negative)
    const int cols = left_k < 4 ? static_cast<int>(left_k) : 4;
    const uint16_t* src = a.W + (tm * kTileM + row0) * a.ldw + tk * kTileK + 4 * lane;
    if (a.vec && rows == kEncRows && cols == 4) {
#pragma unroll
      for (int k = 0; k < kEncRows; ++k, src += a.ldw) w[k] = __ldg(reinterpret_cast<const uint2*>(src));
    } else {
#pragma unroll
      for (int k = 0; k < kEncRows; ++k, src += a.ldw) {
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
  for (int k = 0; k < kEncRows; ++k) {
    // a half-word without its sign is non-zero if adding 0x7FFF carries into its top bit
    const uint32_t x = (w[k].x & 0x7FFF7FFFu) + 0x7FFF7FFFu, y = (w[k].y & 0x7FFF7FFFu) + 0x7FFF7FFFu;
    const uint32_t m0 = __ballot_sync(0xFFFFFFFFu, (x & 0x8000u) != 0), m1 = __ballot_sync(0xFFFFFFFFu, static_cast<int>(x) < 0);
    const uint32_t m2 = __ballot_sync(0xFFFFFFFFu, (y & 0x8000u) != 0), m3 = __ballot_sync(0xFFFFFFFFu, static_cast<int>(y) < 0);
    if (lane == k) { mine[0] = m0; mine[1] = m1; mine[2] = m2; mine[3] = m3; }
    if (a.emit) {
      const int at = (warp * kEncRows + k) * 32 + lane;
      const uint32_t bits = ((x >> 15) & 0x00010001u) | ((y >> 13) & 0x00040004u);
      const uint2 e = sm.window[(bits | bits >> 15) & 15u];
      reinterpret_cast<uint32_t*>(sm.vals)[at] = __byte_perm(w[k].x, w[k].y, e.x) & e.y;
      sm.high[at] = w[k].y;
      sm.nib[at] = static_cast<uint8_t>(e.x >> 16);
    }
  }
  if (lane < kEncRows) {
#pragma unroll
    for (int i = 0; i < 4; ++i) sm.nz[i][warp * kEncRows + lane] = mine[i];
  }
  __syncthreads();

  // ---- lists: threads 0..127 the empty slots of row tid, threads 128..255 the surplus weights of row tid - 128
  const int row = tid & (kTileM - 1);
  const bool surplus = tid >= kTileM;
  uint32_t lo, hi;                             // windows whose even / odd position is listed
  {
    const uint32_t n0 = sm.nz[0][row], n1 = sm.nz[1][row], n2 = sm.nz[2][row], n3 = sm.nz[3][row];
    const uint32_t two = (n0 & n1) | ((n0 | n1) & (n2 | n3)) | (n2 & n3);          // at least two non-zeros
    if (surplus) {
      lo = n0 & n1 & n2;                                                            // the weight at index 2 is a third one
      hi = n3 & ((n0 & n1) | ((n0 | n1) & n2));                                     // the weight at index 3 is a third or fourth
    } else {
      lo = ~two & ~n0;                                                              // slot 0 (index 0) is empty
      hi = ~two & ~(n1 | n2 | n3);                                                  // slot 1 is empty
      const int n = __popc(n0) + __popc(n1) + __popc(n2) + __popc(n3);
      const int sum = __reduce_add_sync(0xFFFFFFFFu, n);
      if (lane == 0) atomicAdd(&sm.nnz, sum);
    }
  }
  const uint32_t count = static_cast<uint32_t>(__popc(lo) + __popc(hi));
  uint32_t tot = 0;
  uint32_t at = scan_cta(count | (surplus ? count << 16 : 0u), sm.warp_tmp, &tot);   // low half: both kinds, high half: surplus
  const int totS = static_cast<int>(tot >> 16), totE = static_cast<int>(tot & 0xFFFFu) - totS;
  const int P = totS < totE ? totS : totE;     // pairs: the i-th surplus weight goes to the i-th empty slot
  const int my_first = static_cast<int>(at >> 16);                                   // (surplus threads: index of the row's first surplus weight)
  at &= 0xFFFFu;
  for (uint32_t any = lo | hi; any; any &= any - 1u) {
    const uint32_t bit = any & (0u - any), pos = static_cast<uint32_t>(row * kH) + 2u * (31u - __clz(bit));
    if (lo & bit) sm.list[at++] = static_cast<uint16_t>(pos);
    if (hi & bit) sm.list[at++] = static_cast<uint16_t>(pos + 1);
  }
  if (surplus) {
    const int end = my_first + static_cast<int>(count);
    sm.parked_end[row] = static_cast<uint16_t>(end < P ? end : P);
    sm.moved[row] = 0;
  }
  if (a.emit) {
    // metadata: eight windows per word, the even one in the low nibble of its byte
#pragma unroll
    for (int i = tid; i < kTileM * 4; i += kEncThreads) {
      const uint2 v = reinterpret_cast<const uint2*>(sm.nib)[i];
      const uint32_t x = v.x | v.x >> 4, y = v.y | v.y >> 4;
      *reinterpret_cast<uint32_t*>(a.tc_meta + (tm * kTileM + (i >> 2)) * meta_ld + tk * (kTileK / 8) + (i & 3) * 4) = __byte_perm(x, y, 0x6420u);
    }
  }
  __syncthreads();

  // ---- pairs: thread t takes pairs [t * run, (t + 1) * run).  A pair that is the first of its row
  //      (rho in another row than the one before) starts a chain and has no delta byte.
  const uint16_t* const tau_list = sm.list;
  const uint16_t* const rho_list = sm.list + totE;
  const int run = (P + kEncThreads - 1) / kEncThreads;
  const int p0 = tid * run < P ? tid * run : P, p1 = p0 + run < P ? p0 + run : P;
  uint32_t bytes = 0;
  int chains = 0;
  uint32_t tau_before = 0, rho_before = 0xFFFFFFFFu;                                 // of the pair in front of this run
  if (p0 > 0 && p0 < p1) { tau_before = tau_list[p0 - 1]; rho_before = rho_list[p0 - 1]; }
  {
    uint32_t tau = tau_before, rho = rho_before;
    for (int i = p0; i < p1; ++i) {
      const uint32_t nt = tau_list[i], nr = rho_list[i];
      if (nr / kH == rho / kH) bytes += 1u + dummies(nt - tau, nr - rho);
      else ++chains;
      tau = nt;
      rho = nr;
    }
  }
  uint32_t tot_len = 0;
  uint32_t pre = scan_cta(bytes, sm.warp_tmp, &tot_len);                             // delta bytes before this run (at most 4096 pairs + 2 * 546 dummies)
  int tot_cut = 0;
  {
    // where every row's chain begins and ends: the run has to be walked again for it, by the few
    // threads that hold the first or last pair of a row
    uint32_t tau = tau_before, rho = rho_before, at_byte = pre;
    for (int i = p0; i < p1; ++i) {
      const uint32_t nt = tau_list[i], nr = rho_list[i];
      if (nr / kH == rho / kH) at_byte += 1u + dummies(nt - tau, nr - rho);
      else sm.first[nr / kH] = static_cast<uint16_t>(at_byte);
      if (i + 1 == P || rho_list[i + 1] / kH != nr / kH) sm.last[nr / kH] = static_cast<uint16_t>(at_byte);
      tau = nt;
      rho = nr;
    }
  }
  __syncthreads();
  const bool has_chain = surplus && my_first < P && count > 0;
  int len = has_chain ? sm.last[row] - sm.first[row] : 0;
  if (__syncthreads_or(len > kChainCap)) {
    // ---- a chain is cut: its row is walked for the last pair that fits, what follows is Residual
    int n_cut = 0, lost = 0;
    if (len > kChainCap) {
      const int end = sm.parked_end[row];
      int i = my_first + 1, fit = 0;
      for (; i < end; ++i) {
        const int need = 1 + static_cast<int>(dummies(tau_list[i] - tau_list[i - 1], rho_list[i] - rho_list[i - 1]));
        if (fit + need > kChainCap) break;
        fit += need;
      }
      n_cut = end - i;
      lost = len - fit;
      len = fit;
      sm.parked_end[row] = static_cast<uint16_t>(i);
    }
    uint32_t t2 = 0;
    const uint32_t before = scan_cta(static_cast<uint32_t>(lost) | static_cast<uint32_t>(n_cut) << 16, sm.warp_tmp, &t2);
    if (surplus) sm.moved[row] = static_cast<uint16_t>(before & 0xFFFFu);
    tot_cut = static_cast<int>(t2 >> 16);
    tot_len -= t2 & 0xFFFFu;
    if (a.emit && n_cut) {
      uint32_t to = a.tile_dir[tile * 4 + 2] + (before >> 16);
      const int end = my_first + static_cast<int>(count) < P ? my_first + static_cast<int>(count) : P;
      for (int i = end - n_cut; i < end; ++i, ++to) {
        a.res_rho[to] = rho_list[i];
        a.res_val[to] = reinterpret_cast<const uint16_t*>(sm.high)[rho_list[i]];
      }
    }
    __syncthreads();
  }
  const int n_beyond = totS - P;               // surplus weights that found no empty slot
  if (!a.emit) {
    if (tid == 0) {
      a.tile_dir[tile * 4 + 1] = tot_len;
      a.tile_dir[tile * 4 + 3] = static_cast<uint32_t>(tot_cut + n_beyond);
    }
    return;
  }

  // ---- the code bytes (dummy points: a zero nibble moves nothing), the parked values, the chain starts
  const uint32_t pdd_off = a.tile_dir[tile * 4 + 0], res_off = a.tile_dir[tile * 4 + 2];
  const bool staged = tot_len <= static_cast<uint32_t>(kCodeStage);                  // (the metadata in that place has left)
  uint8_t* const code = staged ? sm.nib : a.pdd_bytes + pdd_off;
  const uint16_t* const high = reinterpret_cast<const uint16_t*>(sm.high);
  {
    uint32_t tau = tau_before, rho = rho_before;
    for (int i = p0; i < p1; ++i) {
      const uint32_t nt = tau_list[i], nr = rho_list[i], r = nr / kH;
      const bool parked = i < sm.parked_end[r];
      if (r == rho / kH) {
        uint32_t gt = nt - tau, gr = nr - rho;
        if (parked) {
          uint8_t* c = code + (pre - sm.moved[r]);
          pre += 1u + dummies(gt, gr);
          while (gt > kMaxd) { *c++ = static_cast<uint8_t>(kMaxd); gt -= kMaxd; }
          while (gr > kMaxd) { *c++ = static_cast<uint8_t>(kMaxd << 4); gr -= kMaxd; }
          *c = static_cast<uint8_t>(gt | gr << 4);
        } else {
          pre += 1u + dummies(gt, gr);
        }
      }
      if (parked) sm.vals[nt] = high[nr];
      tau = nt;
      rho = nr;
    }
  }
  if (surplus) {
    const long long ch = tile * kTileM + row;
    a.chain_tau0[ch] = has_chain ? tau_list[my_first] : uint16_t{0xFFFFu};
    a.chain_rho0[ch] = has_chain ? rho_list[my_first] : uint16_t{0xFFFFu};
    a.chain_len[ch] = static_cast<uint8_t>(len);
  }
  // surplus weights beyond the number of empty slots: Residual entries after the cut leftovers
  for (int i = P + tid; i < totS; i += kEncThreads) {
    const uint32_t to = res_off + static_cast<uint32_t>(tot_cut + (i - P)), rho = rho_list[i];
    a.res_rho[to] = static_cast<uint16_t>(rho);
    a.res_val[to] = high[rho];
  }
  chains = __reduce_add_sync(0xFFFFFFFFu, chains);
  if (lane == 0 && chains) atomicAdd(&sm.n_chains, chains);
  __syncthreads();
  // ---- the tile leaves: 128 bytes of values per row, and the code bytes
#pragma unroll
  for (int i = tid; i < kTileM * kH / 8; i += kEncThreads)
    *reinterpret_cast<uint4*>(a.tc_vals + (tm * kTileM + (i >> 3)) * half_ld + tk * kH + (i & 7) * 8) = reinterpret_cast<const uint4*>(sm.vals)[i];
  if (staged)
    for (uint32_t i = tid; i < tot_len; i += kEncThreads) a.pdd_bytes[pdd_off + i] = sm.nib[i];
  // layer statistics (Sec. 3.2 quotes their shares): one addition per tile and counter.  Every parked
  // weight that does not start a chain has one byte, the other bytes are dummy points.
  if (tid < 6) {
    const int n_sf = P - tot_cut;
    const int v = tid == 0 ? sm.nnz : tid == 1 ? sm.nnz - totS : tid == 2 ? n_sf : tid == 3 ? tot_cut + n_beyond
                : tid == 4 ? static_cast<int>(tot_len) - (n_sf - sm.n_chains) : totE - n_sf;
    if (v) atomicAdd(a.stats + tid, static_cast<unsigned long long>(v));
  }
}

// Exclusive scan of the per-tile byte and entry counts into the offsets of the tile directory: one
// CTA, each thread sums a run of consecutive tiles, so that there is one scan however many tiles
// there are.
__global__ void __launch_bounds__(1024)
tl3_encode_scan_kernel(uint32_t* tile_dir, long long n_tiles, unsigned long long* totals) {
  __shared__ unsigned long long s_part[2][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long per = (n_tiles + 1023) / 1024;
  const long long t0 = per * tid < n_tiles ? per * tid : n_tiles, t1 = t0 + per < n_tiles ? t0 + per : n_tiles;
  uint4* dir = reinterpret_cast<uint4*>(tile_dir);
  unsigned long long v[2] = {0, 0};
  for (long long t = t0; t < t1; ++t) {
    const uint4 d = dir[t];
    v[0] += d.y;
    v[1] += d.w;
  }
  unsigned long long x[2] = {v[0], v[1]};
#pragma unroll
  for (int k = 0; k < 2; ++k) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, x[k], d);
      if (lane >= d) x[k] += y;
    }
    if (lane == 31) s_part[k][warp] = x[k];
  }
  __syncthreads();
  unsigned long long at[2] = {x[0] - v[0], x[1] - v[1]};
  for (int w = 0; w < warp; ++w) { at[0] += s_part[0][w]; at[1] += s_part[1][w]; }
  if (tid == 1023) { totals[0] = at[0] + v[0]; totals[1] = at[1] + v[1]; }
  for (long long t = t0; t < t1; ++t) {
    uint4 d = dir[t];
    d.x = static_cast<uint32_t>(at[0]);
    d.z = static_cast<uint32_t>(at[1]);
    dir[t] = d;
    at[0] += d.y;
    at[1] += d.w;
  }
}

}  // namespace
}  // namespace tl3

namespace tl3 {
namespace {
// More than 48 KB of dynamic shared memory is opted into.  On every call, like the packer's (a microsecond
// of a millisecond): an opt-in that is remembered per device does not outlive a cudaDeviceReset().
cudaError_t configure_encode_kernel() {
  return cudaFuncSetAttribute(tl3_encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sizeof(EncodeSmem)));
}

void release_encoded(void* p) {
  DeviceCanon* c = static_cast<DeviceCanon*>(p);
  if (!c) return;
  for (void* a : c->alloc) if (a) cudaFree(a);
  delete c;
}
}  // namespace
}  // namespace tl3

extern "C" int tl3_plan_device(tl3_matrix* m, void* stream);

// keep_on_device: leave the container where the kernels wrote it (for tl3_upload_device) and make
// no host copies of it.
static int encode_device_impl(const void* dW, int64_t M, int64_t K, int64_t ldw, void* stream, bool keep_on_device, tl3_matrix** out) {
  using namespace tl3;
  if (!dW || !out || M <= 0 || K <= 0 || ldw < K || M > (int64_t{1} << 31) || K > (int64_t{1} << 31)) return TL3_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  tl3_matrix* m = new (std::nothrow) tl3_matrix();
  if (!m) return TL3_ERR_NO_MEMORY;
  m->M = M; m->K = K; m->p = tl3_params{kTileM, kTileK, kMaxd};
  m->tiles_m = (M + kTileM - 1) / kTileM;
  m->tiles_k = (K + kTileK - 1) / kTileK;
  m->M_pad = m->tiles_m * kTileM;
  m->K_pad = m->tiles_k * kTileK;
  m->n_tiles = m->tiles_m * m->tiles_k;
  if (m->n_tiles > 0x7FFFFFFF) { delete m; return TL3_ERR_UNSUPPORTED; }
  const size_t n_vals = static_cast<size_t>(m->M_pad) * m->K_pad / 2, n_meta = n_vals / 4;
  const size_t n_chain = static_cast<size_t>(m->n_tiles) * kTileM, n_dir = static_cast<size_t>(m->n_tiles) * 4;

  int rc = TL3_OK;
  uint8_t* scratch = nullptr;               // everything the kernels write, in one allocation
  uint8_t* extra = nullptr;                 // PDD bytes and Residual entries that do not fit it
  unsigned long long totals[2] = {0, 0}, stats[6] = {0, 0, 0, 0, 0, 0};
  // layout of `scratch` (every part 256-byte aligned)
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  // One allocation serves the whole conversion (cudaMalloc and cudaFree of more than 2 MB take 0.35 ms
  // each, whatever the size: more than all kernels of a 5120 x 5120 matrix): the arrays of known size,
  // the packer's scratch, and a guess at the PDD bytes and Residual entries that holds down to 40 %
  // sparsity; only a matrix that needs more has them allocated when their sizes are known.
  const size_t o_vals = 0, o_meta = o_vals + up(n_vals * 2), o_tau = o_meta + up(n_meta), o_rho = o_tau + up(n_chain * 2),
               o_len = o_rho + up(n_chain * 2), o_dir = o_len + up(n_chain), o_stats = o_dir + up(n_dir * 4), o_pack = o_stats + 256,
               o_var = o_pack + up(pack_scratch_bytes(m->n_tiles));
  size_t guess = static_cast<size_t>(m->n_tiles) * 10240;
  EncodeArgs a{};
  {
    cudaError_t got = cudaMalloc(reinterpret_cast<void**>(&scratch), o_var + guess);
    if (got == cudaErrorMemoryAllocation) {                         // a device that is nearly full: without the guess, which is twice
      cudaGetLastError();                                           // to five times what a matrix needs
      guess = 0;
      got = cudaMalloc(reinterpret_cast<void**>(&scratch), o_var);
    }
    TL3_ENC_CUDA(got);
    TL3_ENC_CUDA(cudaMemsetAsync(scratch + o_stats, 0, 256, st));
    a.W = static_cast<const uint16_t*>(dW);
    a.M = M; a.K = K; a.ldw = ldw; a.K_pad = m->K_pad; a.tiles_k = static_cast<int>(m->tiles_k);
    a.tc_vals = reinterpret_cast<uint16_t*>(scratch + o_vals);
    a.tc_meta = scratch + o_meta;
    a.chain_tau0 = reinterpret_cast<uint16_t*>(scratch + o_tau);
    a.chain_rho0 = reinterpret_cast<uint16_t*>(scratch + o_rho);
    a.chain_len = scratch + o_len;
    a.tile_dir = reinterpret_cast<uint32_t*>(scratch + o_dir);
    a.stats = reinterpret_cast<unsigned long long*>(scratch + o_stats);
    a.vec = (reinterpret_cast<uintptr_t>(dW) & 7) == 0 && (ldw & 3) == 0;
    a.emit = 0;
    TL3_ENC_CUDA(configure_encode_kernel());
    tl3_encode_kernel<<<static_cast<unsigned>(m->n_tiles), kEncThreads, sizeof(EncodeSmem), st>>>(a);
    tl3_encode_scan_kernel<<<1, 1024, 0, st>>>(a.tile_dir, m->n_tiles, a.stats + 8);
    TL3_ENC_CUDA(cudaGetLastError());
    TL3_ENC_CUDA(cudaMemcpyAsync(totals, a.stats + 8, sizeof(totals), cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaStreamSynchronize(st));
    if (totals[0] > 0xFFFFFFFFull || totals[1] > 0xFFFFFFFFull) { rc = TL3_ERR_UNSUPPORTED; goto done; }   // 32-bit directory offsets
    const size_t o_res_rho = up(totals[0]), o_res_val = o_res_rho + up(totals[1] * 2), var_total = o_res_val + up(totals[1] * 2) + 256;
    uint8_t* var = scratch + o_var;
    if (var_total > guess) {
      TL3_ENC_CUDA(cudaMalloc(reinterpret_cast<void**>(&extra), var_total));
      var = extra;
    }
    a.pdd_bytes = var;
    a.res_rho = reinterpret_cast<uint16_t*>(var + o_res_rho);
    a.res_val = reinterpret_cast<uint16_t*>(var + o_res_val);
    a.emit = 1;
    tl3_encode_kernel<<<static_cast<unsigned>(m->n_tiles), kEncThreads, sizeof(EncodeSmem), st>>>(a);
    TL3_ENC_CUDA(cudaGetLastError());
    if (keep_on_device) {
      TL3_ENC_CUDA(cudaMemcpyAsync(stats, a.stats, sizeof(stats), cudaMemcpyDeviceToHost, st));
      TL3_ENC_CUDA(cudaStreamSynchronize(st));
      m->nnz = static_cast<int64_t>(stats[0]); m->n_tc = static_cast<int64_t>(stats[1]); m->n_sf = static_cast<int64_t>(stats[2]);
      m->n_res = static_cast<int64_t>(stats[3]); m->n_dummy = static_cast<int64_t>(stats[4]); m->n_slots_unused = static_cast<int64_t>(stats[5]);
      DeviceCanon* c = new (std::nothrow) DeviceCanon();
      if (!c) { rc = TL3_ERR_NO_MEMORY; goto done; }
      *c = DeviceCanon{a.tc_vals, a.tc_meta, a.chain_tau0, a.chain_rho0, a.chain_len, a.pdd_bytes, a.tile_dir, a.res_rho, a.res_val, scratch + o_pack, {scratch, extra}};
      m->device_canon = c;
      m->release_device_canon = release_encoded;
      m->host_arrays = false;
      m->canon_bytes = static_cast<int64_t>(n_vals * 2 + n_meta + n_chain * 5 + n_dir * 4 + totals[0] + totals[1] * 4);
      scratch = nullptr;                                            // owned by the handle from here on
      extra = nullptr;
      goto done;
    }
    try {
      m->tc_vals.resize(n_vals); m->tc_meta.resize(n_meta);
      m->chain_tau0.resize(n_chain); m->chain_rho0.resize(n_chain); m->chain_len.resize(n_chain);
      m->tile_dir.resize(n_dir);
      m->pdd_bytes.resize(totals[0]); m->res_rho.resize(totals[1]); m->res_val.resize(totals[1]);
    } catch (const std::bad_alloc&) { rc = TL3_ERR_NO_MEMORY; goto done; }
    prefault(m->tc_vals.data(), n_vals * 2);                       // while the kernel runs
    prefault(m->tc_meta.data(), n_meta);
    TL3_ENC_CUDA(cudaMemcpyAsync(m->tc_vals.data(), a.tc_vals, n_vals * 2, cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaMemcpyAsync(m->tc_meta.data(), a.tc_meta, n_meta, cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaMemcpyAsync(m->chain_tau0.data(), a.chain_tau0, n_chain * 2, cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaMemcpyAsync(m->chain_rho0.data(), a.chain_rho0, n_chain * 2, cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaMemcpyAsync(m->chain_len.data(), a.chain_len, n_chain, cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaMemcpyAsync(m->tile_dir.data(), a.tile_dir, n_dir * 4, cudaMemcpyDeviceToHost, st));
    if (totals[0]) TL3_ENC_CUDA(cudaMemcpyAsync(m->pdd_bytes.data(), a.pdd_bytes, totals[0], cudaMemcpyDeviceToHost, st));
    if (totals[1]) {
      TL3_ENC_CUDA(cudaMemcpyAsync(m->res_rho.data(), a.res_rho, totals[1] * 2, cudaMemcpyDeviceToHost, st));
      TL3_ENC_CUDA(cudaMemcpyAsync(m->res_val.data(), a.res_val, totals[1] * 2, cudaMemcpyDeviceToHost, st));
    }
    TL3_ENC_CUDA(cudaMemcpyAsync(stats, a.stats, sizeof(stats), cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaStreamSynchronize(st));
    m->nnz = static_cast<int64_t>(stats[0]); m->n_tc = static_cast<int64_t>(stats[1]); m->n_sf = static_cast<int64_t>(stats[2]);
    m->n_res = static_cast<int64_t>(stats[3]); m->n_dummy = static_cast<int64_t>(stats[4]); m->n_slots_unused = static_cast<int64_t>(stats[5]);
  }
done:
  if (scratch) cudaFree(scratch);
  if (extra) cudaFree(extra);
  if (rc == TL3_OK && keep_on_device) rc = tl3_plan_device(m, stream);   // sizes of the packed blocks: tl3_device_bytes() is valid on return
  if (rc != TL3_OK) { tl3_free(m); return rc; }
  *out = m;
  return TL3_OK;
}

extern "C" int tl3_encode_device(const void* dW, int64_t M, int64_t K, int64_t ldw, void* stream, tl3_matrix** out) {
  return encode_device_impl(dW, M, K, ldw, stream, false, out);
}

extern "C" int tl3_encode_device_only(const void* dW, int64_t M, int64_t K, int64_t ldw, void* stream, tl3_matrix** out) {
  return encode_device_impl(dW, M, K, ldw, stream, true, out);
}
