// Format conversion that never leaves the GPU: dense masked fp16 W (device) -> the packed blocks that the
// SpMM kernel streams, without the canonical container in between.
//
// One CTA of eight warps takes one 128 x 128 tile and holds all of its way in shared memory: the encoder's
// classification and pairs (they decide which weights are parked and which are Residual, and give the layer
// statistics), the sets of empty slots and parked weights turned to bank-major order (bit matrices of 32
// rows by 32 windows, transposed by five exchanges each), and the packer's steps from there.  A block's
// place in the image is taken from a counter when its size is known, so one pass over W is enough; the
// image is put in order when the caller says where the blob is to lie.
// What bounds it is instructions (62 % of the issue slots) and barriers in front of the threads that walk a tile's lists and
// chains, four tiles per SM (56 KB each) at once; DRAM is at 9 %.
// 5120 x 5120 at 50 % sparsity: 73 us, and 9 to put the image in order; the encoder's two passes, its scan between them and
// the packer's two, with the container written and read in between, take 30 + 5 + 51 + 55 + 75 us.
#include <cuda_runtime.h>

#include <cstdint>
#include <new>
#include <vector>

#include "tl3_convert.cuh"
#include "tl3_internal.h"

namespace tl3 {
namespace {

struct ConvertArgs {
  DenseView dense;
  int tiles_k;
  int again;                            // second pass: only the tiles whose blocks have not been made yet
  uint8_t* image;
  unsigned long long capacity;          // bytes of `image`
  uint32_t* sizes;                      // per tile: {pdd_len, res_cnt, real delta bytes} of its block
  uint8_t** where;                      // per tile: its block; null: no room for it
  unsigned long long* counters;
};
// the six layer statistics, delta bytes of the container; bytes of all blocks, and of those that found no room
enum { kCountStats = 0, kCountRes = 3, kCountPdd = 6, kCountImage = 7, kCountBeyond = 8, kCounters = 9 };

struct ConvertSmem {
  uint16_t vals[kSlots];                // image of W_t
  uint32_t high[kTileM * 32];           // weights 2 and 3 of every window
  uint16_t list[kSlots];                // empty slots and surplus weights, row-major; then empty slots, parked weights
                                        // (both bank-major) and canonical Residual entries
  uint8_t nib[kTileM * 32];             // metadata; later entries that cut chains leave, then the head of the block
  union {
    struct {
      uint32_t nz[4][kTileM];
      uint32_t unused[49];
      uint16_t first[kTileM], last[kTileM], parked_end[kTileM], moved[kTileM];
    };
    PackWork work;
  };
  uint2 window[16];
  uint32_t warp_tmp[kTileThreads / 32];
  unsigned long long place;
  int nnz, n_chains;
};
static_assert(sizeof(PackWork) == 4 * (512 + 49) + 8 * kTileM, "sets over the masks, runs over the rows");
static_assert(4 * (sizeof(ConvertSmem) + 1024) <= 233472, "four tiles per SM");
static_assert(sizeof(ConvertSmem::nib) >= kMaxHead, "the head of a block fits");

// bit c of lane r -> bit r of lane c: the transposition by halves of halves in Warren, "Hacker's Delight", 7-3, a lane per row
__device__ __forceinline__ uint32_t transpose_bits(uint32_t x, int lane) {
  uint32_t m = 0x0000FFFFu;
#pragma unroll
  for (int j = 16; j; j >>= 1, m ^= m << j) {
    const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, j);
    x = (lane & j) ? (x & ~m) | ((y >> j) & m) : (x & m) | ((y << j) & ~m);
  }
  return x;
}

// windows of row r -> banks: bank = ((window >> 2) ^ (r & 7)) << 2 | (window & 3)
__device__ __forceinline__ uint32_t to_banks(uint32_t x, int r) {
  if (r & 1) x = ((x >> 4) & 0x0F0F0F0Fu) | ((x & 0x0F0F0F0Fu) << 4);
  if (r & 2) x = ((x >> 8) & 0x00FF00FFu) | ((x & 0x00FF00FFu) << 8);
  if (r & 4) x = x >> 16 | x << 16;
  return x;
}

__global__ void __launch_bounds__(kTileThreads, 4)
tl3_convert_kernel(const ConvertArgs a) {
  extern __shared__ __align__(16) uint8_t convert_smem_raw[];
  ConvertSmem& sm = *reinterpret_cast<ConvertSmem*>(convert_smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long tile = blockIdx.x;
  const long long tm = tile / a.tiles_k, tk = tile % a.tiles_k;
  if (a.again && a.where[tile]) return;
  if (tid == 16) { sm.nnz = 0; sm.n_chains = 0; }
  classify_tile(a.dense, tm, tk, sm, true);
  __syncthreads();
  const int row = tid & (kTileM - 1);
  const bool surplus = tid >= kTileM;
  uint4 meta = make_uint4(0, 0, 0, 0);          // threads >= 128: entry `row` of the block's metadata
  if (surplus) {
    uint4 m[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint4* n = reinterpret_cast<const uint4*>(sm.nib) + ((row & 7) + 16 * (row >> 4) + 8 * h) * 2;
      const uint4 x = n[0], y = n[1];
      m[h] = make_uint4(meta_word(make_uint2(x.x, x.y)), meta_word(make_uint2(x.z, x.w)), meta_word(make_uint2(y.x, y.y)), meta_word(make_uint2(y.z, y.w)));
    }
    meta = meta_entry(m[0], m[1], (row >> 3) & 1);
  }
  uint16_t* const leftover = reinterpret_cast<uint16_t*>(sm.nib);
  // (rows whose chain is cut have 193 dummy points and more, a tile has 1092 at most: five rows, 315 entries)
  const TilePairs t = find_pairs(sm, [&](const uint16_t* rho, int i0, int i1, uint32_t before) {
    for (int i = i0; i < i1; ++i, ++before)
      if (before < sizeof(sm.nib) / 2) leftover[before] = rho[i];
  });
  const int n_parked = t.P - t.tot_cut;
  uint32_t lo = t.lo, hi = t.hi;
  if (surplus) {
    // only what is parked: the row's first ones
    int left = static_cast<int>(sm.parked_end[row]) - t.my_first;
    if (left < static_cast<int>(t.count)) {
      uint32_t kept_lo = 0, kept_hi = 0;
      for (uint32_t any = lo | hi; any && left > 0; any &= any - 1u) {
        const uint32_t bit = any & (0u - any);
        if (lo & bit) { kept_lo |= bit; --left; }
        if ((hi & bit) && left > 0) { kept_hi |= bit; --left; }
      }
      lo = kept_lo;
      hi = kept_hi;
    }
  }
  const int chains = __reduce_add_sync(0xFFFFFFFFu, t.chains);
  if (lane == 0 && chains) atomicAdd(&sm.n_chains, chains);
  lo = transpose_bits(to_banks(lo, row), lane);                   // lane b: bank b, a bit per row
  hi = transpose_bits(to_banks(hi, row), lane);
  __syncthreads();                                                // everybody has read lists and rows
  {
    uint32_t* set = surplus ? sm.work.flag : sm.work.empty;
    set[lane * 8 + (warp & 3)] = lo;
    set[lane * 8 + 4 + (warp & 3)] = hi;
    if (tid < 4) { sm.work.beyond[tid] = 0; sm.work.real_bytes[tid] = 0; }
    for (int i = tid; i < t.tot_cut; i += kTileThreads) sm.list[t.totE + n_parked + i] = leftover[i];
    if (tid < 6) {
      const int v = tile_statistic(tid, t, sm.nnz, sm.n_chains);
      if (v) atomicAdd(a.counters + kCountStats + tid, static_cast<unsigned long long>(v));
    } else if (tid == 6 && t.tot_len) {
      atomicAdd(a.counters + kCountPdd, static_cast<unsigned long long>(t.tot_len));
    }
  }
  __syncthreads();
  const uint16_t* const high = reinterpret_cast<const uint16_t*>(sm.high);
  const uint16_t* const residual = sm.list + t.totE + n_parked;   // what cut chains left, then what found no empty slot
  pack_block(sm.work, sm.vals, sm.list, sm.list, true, sm.nib, static_cast<uint32_t>(t.totS - n_parked),
    [&](uint32_t u) { return high[pos_of_u(u)]; },
    [&](uint32_t pdd_len, uint32_t res_cnt, uint32_t real_bytes, uint32_t block_bytes) -> uint8_t* {
      const unsigned long long bytes = align_up_d(block_bytes, kBlockAlign);
      if (tid == 0) {
        a.sizes[tile * 3 + 0] = pdd_len;
        a.sizes[tile * 3 + 1] = res_cnt;
        a.sizes[tile * 3 + 2] = real_bytes;
        const unsigned long long at = sm.place = atomicAdd(a.counters + kCountImage, bytes);
        if (at + bytes <= a.capacity) a.where[tile] = a.image + at;
        else atomicAdd(a.counters + kCountBeyond, bytes);
      }
      __syncthreads();
      return sm.place + bytes <= a.capacity ? a.image + sm.place : nullptr;
    },
    [&](int) { return meta; },
    [&](uint32_t j) { return make_uint2(residual[j], high[residual[j]]); });
}

// The blocks to their places in the blob, and the tile directory.
__global__ void __launch_bounds__(256)
tl3_place_kernel(const uint8_t* const* where, const unsigned long long* block_off, uint8_t* blob, unsigned long long dir_offset) {
  const long long t = blockIdx.x;
  const uint8_t* src = where[t];
  const unsigned long long off = block_off[t];
  const uint2 info = *reinterpret_cast<const uint2*>(src + kInfoOff);             // pdd_len, res_cnt
  const uint32_t bytes = align_up_d(kPddOff + info.x + 4u * info.y, 16);
  const uint32_t n = align_up_d(bytes, kBlockAlign) / 16;
  const uint4* from = reinterpret_cast<const uint4*>(src);
  uint4* to = reinterpret_cast<uint4*>(blob + off);
  for (uint32_t i = threadIdx.x; i < n; i += 256) to[i] = __ldcs(from + i);
  if (threadIdx.x == 0)
    reinterpret_cast<DirEntry*>(blob + dir_offset)[t] = DirEntry{static_cast<uint32_t>(off / 16), bytes, info.x, info.y};
}

void release_image(void* p) {
  DeviceCanon* c = static_cast<DeviceCanon*>(p);
  if (!c) return;
  for (void* a : c->alloc) if (a) cudaFree(a);
  delete c;
}

}  // namespace

cudaError_t place_image(const DeviceCanon& c, const unsigned long long* d_block_off, uint8_t* blob, size_t dir_offset, int64_t n_tiles, cudaStream_t st) {
  tl3_place_kernel<<<static_cast<unsigned>(n_tiles), 256, 0, st>>>(c.where, d_block_off, blob, dir_offset);
  return cudaGetLastError();
}

}  // namespace tl3

extern "C" int tl3_encode_device_only(const void* dW, int64_t M, int64_t K, int64_t ldw, void* stream, tl3_matrix** out) {
  using namespace tl3;
  if (!dW || !out || M <= 0 || K <= 0 || ldw < K || M > (int64_t{1} << 31) || K > (int64_t{1} << 31)) return TL3_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  tl3_matrix* m = new_device_matrix(M, K);
  if (!m) return TL3_ERR_NO_MEMORY;
  if (m->n_tiles > 0x7FFFFFFF) { tl3_free(m); return TL3_ERR_UNSUPPORTED; }
  const size_t tiles = static_cast<size_t>(m->n_tiles);
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t o_where = up(pack_scratch_bytes(m->n_tiles)), o_counters = o_where + up(tiles * 8), o_image = o_counters + 256;
  // One allocation (cudaMalloc takes 0.33 ms and cudaFree 0.29, from a megabyte on whatever the size: more than the
  // kernels of a 5120 x 5120 matrix) with 29.25 KB a tile for the blocks, which holds down to 35.5 % sparsity.  Blocks that find no room
  // there get a second allocation and a second pass over their tiles.  (5120 x 5120, whole conversions: at
  // 36 % 800 us, at 30 % 1390; 2110 and 2140 with 28 KB a tile, given up for one allocation of the blocks' size where that was too little.)  Where the device has no memory for that, the
  // first pass writes no blocks and the second one all, into exactly what they need.
  uint8_t *scratch = nullptr, *image = nullptr;
  unsigned long long got[kCounters] = {};
  std::vector<uint32_t> sizes;
  ConvertArgs a{};
  a.dense = dense_view(dW, M, K, ldw);
  a.tiles_k = static_cast<int>(m->tiles_k);
  int rc = TL3_OK;
  cudaError_t e = cudaSuccess;
  auto pass = [&](bool again, uint8_t* to, size_t capacity) {
    a.again = again;
    a.sizes = reinterpret_cast<uint32_t*>(scratch);
    a.where = reinterpret_cast<uint8_t**>(scratch + o_where);
    a.counters = reinterpret_cast<unsigned long long*>(scratch + o_counters) + (again ? 16 : 0);   // (a tile made again counts once)
    a.image = to;
    a.capacity = capacity;
    e = again ? cudaSuccess : cudaMemsetAsync(scratch + o_where, 0, o_image - o_where, st);
    if (e == cudaSuccess) {
      tl3_convert_kernel<<<static_cast<unsigned>(tiles), kTileThreads, sizeof(ConvertSmem), st>>>(a);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess && !again) e = cudaMemcpyAsync(got, a.counters, sizeof(got), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && !again) e = cudaMemcpyAsync(sizes.data(), a.sizes, tiles * 12, cudaMemcpyDeviceToHost, st);
    const cudaError_t done = cudaStreamSynchronize(st);             // (also when something failed: nothing of it may still run)
    if (e == cudaSuccess) e = done;
    return e == cudaSuccess;
  };
  DeviceCanon* c = new (std::nothrow) DeviceCanon();
  try { sizes.resize(tiles * 3); } catch (const std::bad_alloc&) { rc = TL3_ERR_NO_MEMORY; }
  if (!c) rc = TL3_ERR_NO_MEMORY;
  if (rc == TL3_OK) {
    // (on every call, like the packer's: an opt-in that is remembered does not outlive a cudaDeviceReset())
    e = cudaFuncSetAttribute(tl3_convert_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sizeof(ConvertSmem)));
    for (const size_t room : {tiles * 29952 + 32768, size_t{0}}) {
      if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&scratch), o_image + room);
      if (e == cudaSuccess && pass(false, scratch + o_image, room) && got[kCountBeyond]) {
        e = cudaMalloc(reinterpret_cast<void**>(&image), got[kCountBeyond]);
        if (e == cudaSuccess) pass(true, image, got[kCountBeyond]);
      }
      if (e != cudaErrorMemoryAllocation || room == 0) break;
      cudaGetLastError();
      if (scratch) cudaFree(scratch);
      scratch = image = nullptr;
      e = cudaSuccess;
    }
    if (e != cudaSuccess) { set_cuda_error(static_cast<int>(e)); rc = TL3_ERR_CUDA; }
    else if (got[kCountPdd] > 0xFFFFFFFFull || got[kCountRes] > 0xFFFFFFFFull) rc = TL3_ERR_UNSUPPORTED;   // 32-bit offsets of the container's directory
  }
  if (rc == TL3_OK) {
    m->nnz = static_cast<int64_t>(got[0]); m->n_tc = static_cast<int64_t>(got[1]); m->n_sf = static_cast<int64_t>(got[2]);
    m->n_res = static_cast<int64_t>(got[3]); m->n_dummy = static_cast<int64_t>(got[4]); m->n_slots_unused = static_cast<int64_t>(got[5]);
    try { set_device_layout(m, sizes.data()); } catch (const std::bad_alloc&) { rc = TL3_ERR_NO_MEMORY; }   // (counts with them)
  }
  if (rc != TL3_OK) {
    if (scratch) cudaFree(scratch);
    if (image) cudaFree(image);
    delete c;
    tl3_free(m);
    return rc;
  }
  const size_t n_vals = static_cast<size_t>(m->M_pad) * m->K_pad / 2;
  m->canon_bytes = static_cast<int64_t>(n_vals * 2 + n_vals / 4 + tiles * kTileM * 5 + tiles * 16 + got[kCountPdd] + got[kCountRes] * 4);
  c->where = a.where;
  c->pack_scratch = scratch;
  c->alloc[0] = scratch;
  c->alloc[1] = image;
  m->device_canon = c;
  m->release_device_canon = release_image;
  m->host_arrays = false;
  *out = m;
  return TL3_OK;
}
