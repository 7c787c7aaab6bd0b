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
// banks, the two passes took 181 + 247 us on 5120 x 5120 at 50 % sparsity; now 55 + 75 us.
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

#include "tl3_convert.cuh"
#include "tl3_internal.h"

namespace tl3 {

namespace {

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

// dynamic shared memory of the pack kernel
struct PackSmem {
  uint16_t vals[kSlots];         // value slots of the tile by row-major position; parked values lifted out, later re-parked
  uint16_t sval[kSlots];         // value of the surplus weight at bank-major coordinate u
  uint16_t cand[kSlots];         // empty slots, ascending u
  uint16_t sur[kSlots];          // surplus weights, ascending u
  uint8_t pdd[kStagedPdd];       // canonical code bytes; later the head of the block
  PackWork work;
};
static_assert(kStagedPdd >= kMaxHead, "the head of a block fits the staging area");

__global__ void __launch_bounds__(kTileThreads, 3)
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
  for (int i = tid; i < kSlots / 8; i += kTileThreads)
    reinterpret_cast<uint4*>(sm.vals)[i] = *reinterpret_cast<const uint4*>(a.tc_vals + (tm * kTileM + (i >> 3)) * half_ld + tk * kH + (i & 7) * 8);
  const bool staged = dir.y <= static_cast<uint32_t>(kStagedPdd);
  if (staged)
    for (uint32_t i = tid; i < dir.y; i += kTileThreads) sm.pdd[i] = a.pdd_bytes[dir.x + i];
  sm.work.flag[tid] = 0u;
  if (tid < 4) { sm.work.beyond[tid] = 0; sm.work.real_bytes[tid] = 0; }
  const int canon_len = tid < kChains ? a.chain_len[t * kTileM + tid] : 0;
  uint32_t tot = 0;
  const uint32_t at0 = scan_cta(static_cast<uint32_t>(canon_len), sm.work.warp_tmp, &tot);

  // (2) Algorithm 1 over the canonical chains (one per tile row): lift every parked value out of
  //     its slot and note it at the bank-major coordinate of the position it belongs to
  if (tid < kChains) {
    uint32_t tau = a.chain_tau0[t * kTileM + tid], rho = a.chain_rho0[t * kTileM + tid];
    auto lift = [&](uint32_t ta, uint32_t rh) {
      const uint32_t ur = u_of_pos(rh);
      sm.sval[ur] = sm.vals[ta];
      atomicOr(&sm.work.flag[ur >> 5], 1u << (ur & 31u));
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
        if (lane == 2 * i) sm.work.empty[(4 * b4 + i) * 8 + (warp & 3)] = e0;
        if (lane == 2 * i + 1) sm.work.empty[(4 * b4 + i) * 8 + 4 + (warp & 3)] = e1;
      }
    }
  }
  __syncthreads();

  // (4) to (7)
  pack_block(sm.work, sm.vals, sm.cand, sm.sur, false, sm.pdd, dir.w,
    [&](uint32_t u) { return sm.sval[u]; },
    [&](uint32_t pdd_len, uint32_t res_cnt, uint32_t real_bytes, uint32_t block_bytes) -> uint8_t* {
      if (!a.emit) {
        if (tid == 0) {
          a.sizes[t * 3 + 0] = pdd_len;
          a.sizes[t * 3 + 1] = res_cnt;
          a.sizes[t * 3 + 2] = real_bytes;
        }
        return nullptr;
      }
      if (tid == 0) {
        DirEntry* out = reinterpret_cast<DirEntry*>(a.blob + a.dir_offset);
        out[t] = DirEntry{static_cast<uint32_t>(a.block_off[t] / 16), block_bytes, pdd_len, res_cnt};
      }
      return a.blob + a.block_off[t];
    },
    [&](int L) {
      const int mrow = (L & 7) + 16 * (L >> 4), half = (L >> 3) & 1;
      const uint8_t* m0 = a.tc_meta + (tm * kTileM + mrow) * meta_ld + tk * (kTileK / 8);
      return meta_entry(*reinterpret_cast<const uint4*>(m0), *reinterpret_cast<const uint4*>(m0 + 8 * meta_ld), half);
    },
    [&](uint32_t j) { return make_uint2(a.res_rho[dir.z + j], a.res_val[dir.z + j]); });
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

// The pinned memory of copy_pieces(): 12 MB that stay between calls (pinning them costs more than a copy
// of 100 MB) until tl3_trim(), for one caller at a time.  Somebody's cudaDeviceReset() takes such memory
// away, and its address may then be another allocation's: what is kept is used only while the driver
// still knows it by the number that it gave it.
constexpr int kRingThreads = 6;
constexpr int kRingSlots = 2 * kRingThreads;
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

}  // namespace

// Pageable host memory to or from the device, complete on return.  What comes down is read behind what is on `st`.  What goes up is
// not ordered behind it (a stream of its own carries it): its destination has to be memory that nothing on `st` uses
// any more, such as a fresh allocation.  The runtime's own copy moves
// 11 GB/s, one thread of its filling or emptying one staging buffer; here six threads do that with two
// pinned megabytes each, one of them under way while the other is worked on (one caller at a
// time; another one that comes meanwhile takes the runtime's way).  132 MB up: 12.2 ms the runtime's way, 5.9 with one megabyte per thread, 4.7
// with two (5.9 with two halves, 4.5 with two of two); 55 MB down 5.0 and 2.0.
cudaError_t copy_pieces(const std::vector<HostPiece>& arrays, cudaMemcpyKind kind, cudaStream_t st) {
  const bool up = kind == cudaMemcpyHostToDevice;
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
      if (!up) prefault(p.dst, p.bytes);
      if (cudaError_t e = cudaMemcpyAsync(p.dst, p.src, p.bytes, kind, st)) return e;
    }
    return cudaStreamSynchronize(st);
  }
  std::vector<HostPiece> pieces;
  std::vector<std::thread> pool;
  std::atomic<size_t> next{0};
  std::atomic<int> failed{cudaSuccess};
  auto worker = [&](int thread) {
    uint8_t* buf[2];
    cudaEvent_t done[2] = {nullptr, nullptr};
    const HostPiece* under_way[2] = {nullptr, nullptr};
    cudaError_t e = set_context(context) == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
    for (int k = 0; k < 2; ++k) {
      buf[k] = ring + static_cast<size_t>(2 * thread + k) * kRingSlotBytes;
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&done[k], cudaEventDisableTiming);
    }
    auto finish = [&](int k) {                                     // the slot's copy is through; what came down goes to its place
      if (e != cudaSuccess || !under_way[k]) return;
      e = cudaEventSynchronize(done[k]);
      if (e == cudaSuccess && !up) std::memcpy(under_way[k]->dst, buf[k], under_way[k]->bytes);
      under_way[k] = nullptr;
    };
    for (int k = 0; e == cudaSuccess && failed.load(std::memory_order_relaxed) == cudaSuccess; k ^= 1) {
      const size_t i = next.fetch_add(1);
      finish(k);
      if (i >= pieces.size() || e != cudaSuccess) break;
      const HostPiece& p = pieces[i];
      if (up) std::memcpy(buf[k], p.src, p.bytes);
      e = up ? cudaMemcpyAsync(p.dst, buf[k], p.bytes, kind, own) : cudaMemcpyAsync(buf[k], p.src, p.bytes, kind, own);
      if (e == cudaSuccess) e = cudaEventRecord(done[k], own);
      under_way[k] = &p;
    }
    finish(0);
    finish(1);
    for (int k = 0; k < 2; ++k)
      if (done[k]) cudaEventDestroy(done[k]);
    if (e != cudaSuccess) failed.store(e, std::memory_order_relaxed);
  };
  if (!up) failed.store(cudaStreamSynchronize(st));                // (what comes down has been written)
  bool listed = false;
  try {
    for (const HostPiece& p : arrays)
      for (size_t at = 0; at < p.bytes; at += kRingSlotBytes)
        pieces.push_back({static_cast<uint8_t*>(p.dst) + at, static_cast<const uint8_t*>(p.src) + at, std::min(kRingSlotBytes, p.bytes - at)});
    listed = true;
    for (int t = 1; t < kRingThreads; ++t) pool.emplace_back(worker, t);
  } catch (const std::exception&) {                              // fewer threads, or no list at all
  }
  if (!listed) failed.store(cudaErrorMemoryAllocation);
  worker(0);
  for (auto& th : pool) th.join();
  const cudaError_t e = cudaStreamSynchronize(own);              // the ring is free again, whatever happened
  cudaStreamDestroy(own);
  return failed.load() != cudaSuccess ? static_cast<cudaError_t>(failed.load()) : e;
}

namespace {

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
    *c = DeviceCanon{nullptr, reinterpret_cast<const uint16_t*>(b + off[0]), b + off[1], reinterpret_cast<const uint16_t*>(b + off[2]),
                     reinterpret_cast<const uint16_t*>(b + off[3]), b + off[4], b + off[5], reinterpret_cast<const uint32_t*>(b + off[6]),
                     reinterpret_cast<const uint16_t*>(b + off[7]), reinterpret_cast<const uint16_t*>(b + off[8]), b + o_pack, {p, nullptr}};
    m->device_canon = c;
    m->release_device_canon = release_canon;
    std::vector<HostPiece> arrays;
    cudaError_t e = cudaErrorMemoryAllocation;
    try {
      for (int i = 0; i < 9; ++i) arrays.push_back({b + off[i], src[i], sz[i]});
      e = copy_pieces(arrays, cudaMemcpyHostToDevice, st);
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
  tl3_pack_kernel<<<static_cast<unsigned>(m->n_tiles), kTileThreads, sizeof(PackSmem), st>>>(a);
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
    const DeviceCanon& c = *static_cast<const DeviceCanon*>(m->device_canon);
    if (c.where) {
      e = place_image(c, d_off, a.blob, a.dir_offset, m->n_tiles, st);
    } else {
      tl3_pack_kernel<<<static_cast<unsigned>(m->n_tiles), kTileThreads, sizeof(PackSmem), st>>>(a);
      e = cudaGetLastError();
    }
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
