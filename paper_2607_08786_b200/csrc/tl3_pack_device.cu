// The device packer on the GPU: canonical container -> the blob of per-tile blocks that the SpMM
// kernel streams, byte for byte what tl3_pack() / tl3_upload() build on the host (tl3_pack.cpp has
// the reasoning behind the layout: bank-major re-pairing of the Slot-Filling layer, four equal
// chains per bank, the same number of transposed code words for every chain of a tile, the tails
// as Residual entries).
//
// One CTA of 256 threads per 128 x 128 tile.  In turn a thread is the owner of canonical chain r (to
// lift the parked values out of the value array), of row r of a quarter of the value array (to mark
// the empty slots), of 32 consecutive bank-major slot coordinates (to list the empty slots and the
// surplus weights in that order), and of device chain c (bank c / 4, run c % 4).  The sets are
// bitmaps over the bank-major coordinate -- a warp's ballot over 32 rows is one word of it -- so the
// listing costs one step per set bit.  The kernel runs twice: a count pass that yields every tile's
// number of code words and Residual entries, from which the host lays the blocks out exactly as
// plan_device_layout() does, and an emit pass that writes the blocks.
// What bounds it is the latency of a tile's serial steps (the chains), hidden by three tiles per SM.
// With two-byte copies, a thread per 64 coordinates tested one by one and one thread sharing out the
// banks, the two passes took 181 + 247 us on 5120 x 5120 at 50 % sparsity; now 57 + 77 us.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

#include "tl3_internal.h"

namespace tl3 {

void set_cuda_error(int e);

namespace {

constexpr int kSlots = kTileM * kH;        // 8192
constexpr int kChains = 128;
constexpr int kPackThreads = 256;
constexpr int kFlagWords = kSlots / 32;    // 256: one per thread
constexpr int kStagedPdd = 4096;           // canonical PDD bytes staged in shared memory (a tile has 1.5-2 KB as a rule)

struct PackArgs {
  // canonical container (device copies)
  const uint16_t* tc_vals;
  const uint8_t* tc_meta;
  const uint16_t* chain_tau0;
  const uint16_t* chain_rho0;
  const uint8_t* chain_len;
  const uint8_t* pdd_bytes;
  const uint32_t* tile_dir;
  const uint16_t* res_rho;
  const uint16_t* res_val;
  long long K_pad;
  int tiles_k;
  // count pass: per tile {pdd_len, res_cnt, real delta bytes}
  uint32_t* sizes;
  // emit pass
  uint8_t* blob;
  const unsigned long long* block_off;     // byte offset of every tile's block in the blob
  unsigned long long dir_offset;
  int emit;
};

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

// exclusive scan over the threads of the CTA (two 16-bit sums per word where a caller packs them)
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
  for (int w = 0; w < kPackThreads / 32; ++w) {
    base += w < warp ? s_warp[w] : 0u;
    all += s_warp[w];
  }
  *total = all;
  __syncthreads();
  return base + x - v;
}

// dynamic shared memory of the pack kernel
struct PackSmem {
  uint16_t vals[kSlots];         // value slots of the tile by row-major position; parked values lifted out, later re-parked
  uint16_t sval[kSlots];         // value of the surplus weight at bank-major coordinate u
  uint16_t cand[kSlots];         // empty slots, ascending u
  uint16_t sur[kSlots];          // surplus weights, ascending u
  uint32_t flag[kFlagWords];     // bit u set: a surplus weight sits at u
  uint32_t empty[kFlagWords];    // bit u set: slot u is empty
  uint8_t pdd[kStagedPdd];       // canonical code bytes; later the chain starts and code words of the block
  uint32_t bank_cand[33];        // empty slots before bank b
  int carry[kChains];            // parked elements that run i hands on to the next
  int len[kChains];              // delta bytes of device chain c
  int beyond[4];
  int real_bytes[4];
  uint32_t warp_tmp[kPackThreads / 32];
};
static_assert(kStagedPdd >= 16 + 4 * kChains + 3 * 4 * kChains, "the block's info words, chain starts and code words fit the staging area");

__global__ void __launch_bounds__(kPackThreads, 3)
tl3_pack_kernel(const PackArgs a) {
  extern __shared__ __align__(16) uint8_t pack_smem_raw[];
  PackSmem& sm = *reinterpret_cast<PackSmem*>(pack_smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long t = blockIdx.x;
  const long long tm = t / a.tiles_k, tk = t % a.tiles_k;
  const long long half_ld = a.K_pad / 2, meta_ld = a.K_pad / 8;
  const uint4 dir = *reinterpret_cast<const uint4*>(a.tile_dir + t * 4);       // pdd_off, pdd_len, res_off, res_cnt

  // (1) the tile's value slots and code bytes
#pragma unroll
  for (int i = tid; i < kSlots / 8; i += kPackThreads)
    reinterpret_cast<uint4*>(sm.vals)[i] = *reinterpret_cast<const uint4*>(a.tc_vals + (tm * kTileM + (i >> 3)) * half_ld + tk * kH + (i & 7) * 8);
  const bool staged = dir.y <= static_cast<uint32_t>(kStagedPdd);
  if (staged)
    for (uint32_t i = tid; i < dir.y; i += kPackThreads) sm.pdd[i] = a.pdd_bytes[dir.x + i];
  sm.flag[tid] = 0u;
  if (tid < 4) { sm.beyond[tid] = 0; sm.real_bytes[tid] = 0; }
  const int canon_len = tid < kChains ? a.chain_len[t * kTileM + tid] : 0;
  uint32_t tot = 0;
  const uint32_t at0 = scan_cta(static_cast<uint32_t>(canon_len), sm.warp_tmp, &tot);

  // (2) Algorithm 1 over the canonical chains (one per tile row): lift every parked value out of
  //     its slot and note it at the bank-major coordinate of the position it belongs to
  if (tid < kChains) {
    uint32_t tau = a.chain_tau0[t * kTileM + tid], rho = a.chain_rho0[t * kTileM + tid];
    auto lift = [&](uint32_t ta, uint32_t rh) {
      const uint32_t ur = u_of_pos(rh);
      sm.sval[ur] = sm.vals[ta];
      atomicOr(&sm.flag[ur >> 5], 1u << (ur & 31u));
      sm.vals[ta] = 0;
    };
    if (tau != 0xFFFFu) {
      lift(tau, rho);
      const uint8_t* code = staged ? sm.pdd + at0 : a.pdd_bytes + dir.x + at0;
      for (int k = 0; k < canon_len; ++k) {
        const uint32_t b = code[k], dt = b & 15u, dr = b >> 4;
        tau += dt;
        rho += dr;
        if (dt && dr) lift(tau, rho);
      }
    }
  }
  __syncthreads();

  // (3) empty slots and surplus weights in bank-major order.  A lane looks at one row: four of its
  //     eight 16-byte chunks (warps 0-3 the first four bank groups, warps 4-7 the others), in the
  //     order in which chunk j of row r holds the banks 4 (j ^ (r & 7)) ...: the lanes' accesses
  //     then spread over all shared-memory banks.
  {
    const int row = (warp & 3) * 32 + lane;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int b4 = (warp >> 2) * 4 + g;
      const uint4 v = reinterpret_cast<const uint4*>(sm.vals)[row * 8 + (b4 ^ (row & 7))];
      const uint32_t word[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t e0 = __ballot_sync(0xFFFFFFFFu, (word[i] & 0x7FFFu) == 0), e1 = __ballot_sync(0xFFFFFFFFu, (word[i] & 0x7FFF0000u) == 0);
        if (lane == 2 * i) sm.empty[(4 * b4 + i) * 8 + (warp & 3)] = e0;
        if (lane == 2 * i + 1) sm.empty[(4 * b4 + i) * 8 + 4 + (warp & 3)] = e1;
      }
    }
  }
  __syncthreads();
  int n_cand = 0, n_pairs = 0;
  {
    uint32_t e = sm.empty[tid], f = sm.flag[tid];
    const uint32_t off = scan_cta(static_cast<uint32_t>(__popc(e)) | static_cast<uint32_t>(__popc(f)) << 16, sm.warp_tmp, &tot);
    n_cand = static_cast<int>(tot & 0xFFFFu);
    n_pairs = static_cast<int>(tot >> 16);
    uint32_t oc = off & 0xFFFFu, os = off >> 16;
    if ((tid & 7) == 0) sm.bank_cand[tid >> 3] = oc;
    if (tid == 0) sm.bank_cand[32] = static_cast<uint32_t>(n_cand);
    for (; e; e &= e - 1u) sm.cand[oc++] = static_cast<uint16_t>(tid * 32 + __ffs(e) - 1);
    for (; f; f &= f - 1u) sm.sur[os++] = static_cast<uint16_t>(tid * 32 + __ffs(f) - 1);
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
  const uint16_t* const sel = sm.cand + my_src;                // this thread's run of empty slots

  // (5) device chain c = the pairs [i0, i1) of run c.  One walk: for a chain of at most 0, 4, 8 and
  //     12 delta bytes, how many bytes it has, how many entries move a value, how many are cut off.
  int by[4] = {0, 0, 0, 0}, end_at[4] = {0, 0, 0, 0};
  {
    int end = 0;
    for (int i = 1; i < my_take; ++i) {
      end += static_cast<int>(delta_bytes(static_cast<uint32_t>(sel[i] - sel[i - 1]), static_cast<uint32_t>(sm.sur[i0 + i] - sm.sur[i0 + i - 1])));
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
  const uint32_t res_cnt = tot_tail + n_left + dir.w;
  if (!a.emit) {
    if (tid == 0) {
      a.sizes[t * 3 + 0] = pdd_len;
      a.sizes[t * 3 + 1] = res_cnt;
      a.sizes[t * 3 + 2] = static_cast<uint32_t>(sm.real_bytes[n_words]);
    }
    return;
  }
  if (tid < kChains) sm.len[tid] = n_bytes;
  const uint32_t off_tail = scan_cta(static_cast<uint32_t>(n_tail), sm.warp_tmp, &tot);

  // (7) the block.  Info words, chain starts and code words are put together in shared memory.
  uint8_t* blk = a.blob + a.block_off[t];
  const uint32_t block_bytes = align_up_d(kPddOff + pdd_len + 4u * res_cnt, 16);
  constexpr uint32_t kHead = kPddOff - kInfoOff;               // info words and chain starts
  const uint32_t head_words = (kHead + pdd_len) / 4;
  uint32_t* head = reinterpret_cast<uint32_t*>(sm.pdd);
  for (uint32_t i = tid; i < head_words; i += kPackThreads) head[i] = 0u;      // (padding of short chains)
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
    uint8_t* code = sm.pdd + kHead + slot * 4u;
    uint32_t at = 0;
    const int kept = my_take - n_tail;
    uint32_t u0 = 0, r0 = 0;
    for (int i = 0; i < kept; ++i) {
      const uint32_t u = sel[i], r_u = sm.sur[i0 + i];
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
      sm.vals[pos_of_u(u)] = sm.sval[r_u];     // the value is parked in its new slot
    }
    head[4 + slot] = hdr;
    for (int i = kept; i < my_take; ++i) {     // the chain is full: the rest of its run goes to the Residual list
      const uint32_t r_u = sm.sur[i0 + i];
      res[off_tail + static_cast<uint32_t>(i - kept)] = r_u | static_cast<uint32_t>(sm.sval[r_u]) << 16;
    }
  } else {
    // meanwhile the other warps: metadata in tensor-memory lane order ...
    {
      const int L = tid - kChains, mrow = (L & 7) + 16 * (L >> 4), half = (L >> 3) & 1;
      const uint8_t* m0 = a.tc_meta + (tm * kTileM + mrow) * meta_ld + tk * (kTileK / 8);
      const uint4 lo = *reinterpret_cast<const uint4*>(m0), hi = *reinterpret_cast<const uint4*>(m0 + 8 * meta_ld);
      const uint32_t sel2 = half ? 0x7632u : 0x5410u;           // this half's two bytes of either word
      reinterpret_cast<uint4*>(blk + kMetaOff)[L] = make_uint4(__byte_perm(lo.x, hi.x, sel2), __byte_perm(lo.y, hi.y, sel2),
                                                               __byte_perm(lo.z, hi.z, sel2), __byte_perm(lo.w, hi.w, sel2));
    }
    // ... and surplus weights beyond the selected empty slots, the canonical Residual entries, the padding
    const uint32_t j0 = static_cast<uint32_t>(tid - kChains);
    for (uint32_t i = n_sel + j0; i < static_cast<uint32_t>(n_pairs); i += kPackThreads - kChains)
      res[tot_tail + (i - n_sel)] = sm.sur[i] | static_cast<uint32_t>(sm.sval[sm.sur[i]]) << 16;
    for (uint32_t j = j0; j < dir.w; j += kPackThreads - kChains)
      res[tot_tail + n_left + j] = u_of_pos(a.res_rho[dir.z + j]) | static_cast<uint32_t>(a.res_val[dir.z + j]) << 16;
    const uint32_t n_pad = (align_up_d(block_bytes, kBlockAlign) - (kPddOff + pdd_len + 4u * res_cnt)) / 4;
    if (j0 < n_pad) res[res_cnt + j0] = 0u;
  }
  if (tid == 0) {
    head[0] = pdd_len;
    head[1] = res_cnt;
    head[2] = n_words;
    DirEntry* out = reinterpret_cast<DirEntry*>(a.blob + a.dir_offset);
    out[t] = DirEntry{static_cast<uint32_t>(a.block_off[t] / 16), block_bytes, pdd_len, res_cnt};
  }
  __syncthreads();
  // values: row r of the K-major 128-byte-swizzled image; word `bank` of the row holds both slots of one window
#pragma unroll
  for (int i = tid; i < kSlots / 8; i += kPackThreads)
    reinterpret_cast<uint4*>(blk)[i] = reinterpret_cast<const uint4*>(sm.vals)[i ^ ((i >> 3) & 7)];
  for (uint32_t i = tid; i < head_words / 4; i += kPackThreads) reinterpret_cast<uint4*>(blk + kInfoOff)[i] = reinterpret_cast<const uint4*>(head)[i];
}

}  // namespace
}  // namespace tl3

namespace tl3 {
namespace {

struct CanonOnDevice {
  uint8_t* base = nullptr;
  PackArgs args{};
};

void release_canon(void* p) {
  DeviceCanon* c = static_cast<DeviceCanon*>(p);
  if (!c) return;
  for (void* a : c->alloc) if (a) cudaFree(a);
  delete c;
}

#define TL3_PK_CUDA(expr)                                     \
  do {                                                        \
    cudaError_t e_ = (expr);                                  \
    if (e_ != cudaSuccess) {                                  \
      tl3::set_cuda_error(static_cast<int>(e_));              \
      return TL3_ERR_CUDA;                                    \
    }                                                         \
  } while (0)

struct HostPiece {
  void* dst;
  const void* src;
  size_t bytes;
};

// The pinned memory of copy_from_host(): 6 MB that stay between calls (pinning them costs more than a copy
// of 100 MB) until tl3_trim(), for one caller at a time.  Somebody's cudaDeviceReset() takes such memory
// away, and its address may then be another allocation's: what is kept is used only while the driver
// still knows it by the number that it gave it.
constexpr int kRingSlots = 6;
constexpr size_t kRingSlotBytes = size_t{1} << 20;

template <class Fn> Fn driver_entry(const char* name) {
  void* f = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint(name, &f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) return nullptr;
  return reinterpret_cast<Fn>(f);
}

unsigned long long buffer_id(const void* p) {                    // 0: not an allocation of the driver's
  static const auto fn = driver_entry<CUresult (*)(void*, CUpointer_attribute, CUdeviceptr)>("cuPointerGetAttribute");
  unsigned long long id = 0;
  if (!fn || !p || fn(&id, CU_POINTER_ATTRIBUTE_BUFFER_ID, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS) return 0;
  return id;
}

struct PinnedRing {
  std::mutex mu;
  uint8_t* base = nullptr;
  unsigned long long id = 0;

  uint8_t* get() {                                               // (mu held) the memory, or null
    if (base && buffer_id(base) == id) return base;
    void* p = nullptr;
    base = nullptr;
    if (cudaHostAlloc(&p, kRingSlots * kRingSlotBytes, cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    id = buffer_id(p);
    if (id == 0) { cudaFreeHost(p); return nullptr; }
    return base = static_cast<uint8_t*>(p);
  }
  cudaError_t release() {                                        // (mu held)
    const bool there = base && buffer_id(base) == id;
    uint8_t* p = base;
    base = nullptr;
    return there ? cudaFreeHost(p) : cudaSuccess;
  }
};
PinnedRing& ring_of_process() {
  static PinnedRing* r = new PinnedRing();                       // (never destroyed: a thread may still copy while the process exits)
  return *r;
}

// Pageable host memory to the device, complete on return.  The runtime's own copy moves 11 GB/s, one
// thread of its filling one staging buffer; here six threads fill a pinned megabyte each (one caller at a
// time; another one that comes meanwhile takes the runtime's way).  132 MB: 12.2 -> 5 ms.
cudaError_t copy_from_host(const std::vector<HostPiece>& arrays, cudaStream_t st) {
  size_t total = 0;
  for (const HostPiece& p : arrays) total += p.bytes;
  PinnedRing& pinned = ring_of_process();
  std::unique_lock<std::mutex> lock(pinned.mu, std::defer_lock);
  cudaStream_t own = nullptr;
  // the caller's context, which need not be its device's primary one, for the threads
  static const auto get_context = driver_entry<CUresult (*)(CUcontext*)>("cuCtxGetCurrent");
  static const auto set_context = driver_entry<CUresult (*)(CUcontext)>("cuCtxSetCurrent");
  CUcontext context = nullptr;
  uint8_t* ring = nullptr;
  bool staged = total >= (size_t{8} << 20) && get_context && set_context && lock.try_lock() && (ring = pinned.get()) != nullptr &&
                get_context(&context) == CUDA_SUCCESS && context;
  // (a stream of its own: the caller's may be one that means another stream in another thread)
  if (staged && cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking) != cudaSuccess) { staged = false; cudaGetLastError(); }
  if (!staged) {
    for (const HostPiece& p : arrays) {
      if (!p.bytes) continue;
      if (cudaError_t e = cudaMemcpyAsync(p.dst, p.src, p.bytes, cudaMemcpyHostToDevice, st)) return e;
    }
    return cudaStreamSynchronize(st);
  }
  std::vector<HostPiece> pieces;
  std::vector<std::thread> pool;
  std::atomic<size_t> next{0};
  std::atomic<int> failed{cudaSuccess};
  auto worker = [&](int slot) {
    uint8_t* buf = ring + static_cast<size_t>(slot) * kRingSlotBytes;
    cudaEvent_t done = nullptr;
    cudaError_t e = set_context(context) == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&done, cudaEventDisableTiming);
    bool busy = false;
    while (e == cudaSuccess && failed.load(std::memory_order_relaxed) == cudaSuccess) {
      const size_t i = next.fetch_add(1);
      if (i >= pieces.size()) break;
      if (busy) e = cudaEventSynchronize(done);
      if (e != cudaSuccess) break;
      std::memcpy(buf, pieces[i].src, pieces[i].bytes);
      e = cudaMemcpyAsync(pieces[i].dst, buf, pieces[i].bytes, cudaMemcpyHostToDevice, own);
      if (e == cudaSuccess) e = cudaEventRecord(done, own);
      busy = true;
    }
    if (done) cudaEventDestroy(done);
    if (e != cudaSuccess) failed.store(e, std::memory_order_relaxed);
  };
  bool listed = false;
  try {
    for (const HostPiece& p : arrays)
      for (size_t at = 0; at < p.bytes; at += kRingSlotBytes)
        pieces.push_back({static_cast<uint8_t*>(p.dst) + at, static_cast<const uint8_t*>(p.src) + at, std::min(kRingSlotBytes, p.bytes - at)});
    listed = true;
    for (int t = 1; t < kRingSlots; ++t) pool.emplace_back(worker, t);
  } catch (const std::exception&) {                              // fewer threads, or no list at all
  }
  if (!listed) failed.store(cudaErrorMemoryAllocation);
  worker(0);
  for (auto& th : pool) th.join();
  const cudaError_t e = cudaStreamSynchronize(own);              // the ring is free again, whatever happened
  cudaStreamDestroy(own);
  return failed.load() != cudaSuccess ? static_cast<cudaError_t>(failed.load()) : e;
}

// Copies the canonical arrays of the handle to the device (one allocation, kept in the handle) and
// fills the kernel arguments that point into it.
int canon_to_device(tl3_matrix* m, cudaStream_t st, PackArgs* out) {
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t sz[9] = {m->tc_vals.size() * 2, m->tc_meta.size(), m->chain_tau0.size() * 2, m->chain_rho0.size() * 2, m->chain_len.size(),
                        m->pdd_bytes.size(), m->tile_dir.size() * 4, m->res_rho.size() * 2, m->res_val.size() * 2};
  const void* src[9] = {m->tc_vals.data(), m->tc_meta.data(), m->chain_tau0.data(), m->chain_rho0.data(), m->chain_len.data(),
                        m->pdd_bytes.data(), m->tile_dir.data(), m->res_rho.data(), m->res_val.data()};
  size_t off[10];
  off[0] = 0;
  for (int i = 0; i < 9; ++i) off[i + 1] = off[i] + up(sz[i] + 16);
  const size_t o_pack = off[9];
  if (!m->device_canon) {
    if (!m->host_arrays) return TL3_ERR_UNSUPPORTED;           // a device-only handle whose container has been packed and released
    void* p = nullptr;
    TL3_PK_CUDA(cudaMalloc(&p, o_pack + pack_scratch_bytes(m->n_tiles)));
    DeviceCanon* c = new (std::nothrow) DeviceCanon();
    if (!c) { cudaFree(p); return TL3_ERR_NO_MEMORY; }
    uint8_t* b = static_cast<uint8_t*>(p);
    *c = DeviceCanon{reinterpret_cast<const uint16_t*>(b + off[0]), b + off[1], reinterpret_cast<const uint16_t*>(b + off[2]),
                     reinterpret_cast<const uint16_t*>(b + off[3]), b + off[4], b + off[5], reinterpret_cast<const uint32_t*>(b + off[6]),
                     reinterpret_cast<const uint16_t*>(b + off[7]), reinterpret_cast<const uint16_t*>(b + off[8]), b + o_pack, {p, nullptr}};
    m->device_canon = c;
    m->release_device_canon = release_canon;
    std::vector<HostPiece> arrays;
    cudaError_t e = cudaErrorMemoryAllocation;
    try {
      for (int i = 0; i < 9; ++i) arrays.push_back({b + off[i], src[i], sz[i]});
      e = copy_from_host(arrays, st);
    } catch (const std::bad_alloc&) {
    }
    if (e != cudaSuccess) {                                        // nothing half-copied stays with the handle
      m->device_canon = nullptr;
      release_canon(c);
      set_cuda_error(static_cast<int>(e));
      return TL3_ERR_CUDA;
    }
  }
  const DeviceCanon* c = static_cast<const DeviceCanon*>(m->device_canon);
  PackArgs a{};
  a.tc_vals = c->tc_vals;
  a.tc_meta = c->tc_meta;
  a.chain_tau0 = c->chain_tau0;
  a.chain_rho0 = c->chain_rho0;
  a.chain_len = c->chain_len;
  a.pdd_bytes = c->pdd_bytes;
  a.tile_dir = c->tile_dir;
  a.res_rho = c->res_rho;
  a.res_val = c->res_val;
  a.K_pad = m->K_pad;
  a.tiles_k = static_cast<int>(m->tiles_k);
  *out = a;
  return TL3_OK;
}

int configure_pack_kernel() {
  TL3_PK_CUDA(cudaFuncSetAttribute(tl3_pack_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sizeof(PackSmem))));
  return TL3_OK;
}

}  // namespace
}  // namespace tl3

extern "C" int tl3_plan_device(tl3_matrix* m, void* stream) {
  using namespace tl3;
  if (!m) return TL3_ERR_INVALID_ARG;
  if (m->p.tile_m != kTileM || m->p.tile_k != kTileK) return TL3_ERR_UNSUPPORTED;
  if (m->layout_ready.load(std::memory_order_acquire)) return TL3_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (int rc = configure_pack_kernel()) return rc;
  PackArgs a{};
  if (int rc = canon_to_device(m, st, &a)) return rc;
  a.sizes = static_cast<uint32_t*>(static_cast<DeviceCanon*>(m->device_canon)->pack_scratch);
  a.emit = 0;
  tl3_pack_kernel<<<static_cast<unsigned>(m->n_tiles), kPackThreads, sizeof(PackSmem), st>>>(a);
  std::vector<uint32_t> sizes;
  int rc = TL3_OK;
  try { sizes.resize(static_cast<size_t>(m->n_tiles) * 3); } catch (const std::bad_alloc&) { rc = TL3_ERR_NO_MEMORY; }
  cudaError_t e = cudaGetLastError();
  if (rc == TL3_OK && e == cudaSuccess) e = cudaMemcpyAsync(sizes.data(), a.sizes, sizes.size() * 4, cudaMemcpyDeviceToHost, st);
  if (rc == TL3_OK && e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (rc != TL3_OK) return rc;
  if (e != cudaSuccess) { set_cuda_error(static_cast<int>(e)); return TL3_ERR_CUDA; }
  set_device_layout(m, sizes.data());
  return TL3_OK;
}

extern "C" int tl3_upload_device(tl3_matrix* m, void* dptr, void* stream) {
  using namespace tl3;
  if (!m || !dptr || (reinterpret_cast<uintptr_t>(dptr) & 255) != 0) return TL3_ERR_INVALID_ARG;
  if (m->p.tile_m != kTileM || m->p.tile_k != kTileK) return TL3_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (int rc = tl3_plan_device(m, stream)) return rc;          // no-op when the layout is known already
  if (int rc = configure_pack_kernel()) return rc;
  PackArgs a{};
  if (int rc = canon_to_device(m, st, &a)) return rc;
  uint8_t header[256];
  std::vector<unsigned long long> block_off;
  try { blob_header_and_offsets(m, header, &block_off); } catch (const std::bad_alloc&) { return TL3_ERR_NO_MEMORY; }
  unsigned long long* d_off = static_cast<unsigned long long*>(static_cast<DeviceCanon*>(m->device_canon)->pack_scratch);
  cudaError_t e = cudaMemcpyAsync(d_off, block_off.data(), block_off.size() * 8, cudaMemcpyHostToDevice, st);
  // zeros where no block is: before the first and behind the last (a block's padding is the kernel's)
  const size_t blocks_end = block_off.back();
  if (e == cudaSuccess) e = cudaMemsetAsync(dptr, 0, m->blocks_offset, st);
  if (e == cudaSuccess && blocks_end < m->device_bytes)
    e = cudaMemsetAsync(static_cast<uint8_t*>(dptr) + blocks_end, 0, m->device_bytes - blocks_end, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(dptr, header, 256, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    a.blob = static_cast<uint8_t*>(dptr);
    a.block_off = d_off;
    a.dir_offset = m->dir_offset;
    a.emit = 1;
    tl3_pack_kernel<<<static_cast<unsigned>(m->n_tiles), kPackThreads, sizeof(PackSmem), st>>>(a);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);          // header, offsets and the canonical copies are released below
  if (m->device_canon) { release_canon(m->device_canon); m->device_canon = nullptr; }
  if (e != cudaSuccess) { set_cuda_error(static_cast<int>(e)); return TL3_ERR_CUDA; }
  m->dptr = dptr;
  return TL3_OK;
}

extern "C" int tl3_trim(void) {
  using namespace tl3;
  PinnedRing& pinned = ring_of_process();
  std::lock_guard<std::mutex> lock(pinned.mu);                   // (waits for a copy under way)
  TL3_PK_CUDA(pinned.release());
  return TL3_OK;
}
