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
// container once, is a few microseconds).  Two passes on 5120 x 5120 at 50 % sparsity: 30 + 51 us.
// A thread per row, two-byte accesses a row pitch apart and 512 atomics per tile on four
// addresses took 351 + 898 us; coalesced rows that every lane classified for itself, with chains
// walked by a thread per row, 57 + 89 us.
#include <cuda_runtime.h>

#include <cstdint>
#include <new>
#include <vector>

#include "tl3_convert.cuh"
#include "tl3_internal.h"

namespace tl3 {

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

struct EncodeArgs {
  DenseView dense;
  long long K_pad;
  int tiles_k;
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
  uint32_t warp_tmp[kTileThreads / 32];
  int nnz, n_chains;
};
constexpr int kCodeStage = kTileM * 32;       // a tile has 1.5-2 KB of code bytes as a rule

__global__ void __launch_bounds__(kTileThreads, 4)
tl3_encode_kernel(const EncodeArgs a) {
  extern __shared__ __align__(16) uint8_t encode_smem_raw[];
  EncodeSmem& sm = *reinterpret_cast<EncodeSmem*>(encode_smem_raw);
  const int tid = threadIdx.x, lane = tid & 31;
  const long long tile = blockIdx.x;
  const long long tm = tile / a.tiles_k, tk = tile % a.tiles_k;
  const long long half_ld = a.K_pad / 2, meta_ld = a.K_pad / 8;
  if (tid == 16) { sm.nnz = 0; sm.n_chains = 0; }
  classify_tile(a.dense, tm, tk, sm, a.emit != 0);
  __syncthreads();
  if (a.emit) {
#pragma unroll
    for (int i = tid; i < kTileM * 4; i += kTileThreads)
      *reinterpret_cast<uint32_t*>(a.tc_meta + (tm * kTileM + (i >> 2)) * meta_ld + tk * (kTileK / 8) + (i & 3) * 4) = meta_word(reinterpret_cast<const uint2*>(sm.nib)[i]);
  }
  const uint16_t* const high = reinterpret_cast<const uint16_t*>(sm.high);
  const TilePairs t = find_pairs(sm, [&](const uint16_t* rho, int i0, int i1, uint32_t before) {
    if (!a.emit) return;
    uint32_t to = a.tile_dir[tile * 4 + 2] + before;
    for (int i = i0; i < i1; ++i, ++to) {
      a.res_rho[to] = rho[i];
      a.res_val[to] = high[rho[i]];
    }
  });
  const int row = tid & (kTileM - 1);
  const bool surplus = tid >= kTileM;
  const uint16_t* const tau_list = sm.list;
  const uint16_t* const rho_list = sm.list + t.totE;
  const int n_beyond = t.totS - t.P;           // surplus weights that found no empty slot
  if (!a.emit) {
    if (tid == 0) {
      a.tile_dir[tile * 4 + 1] = t.tot_len;
      a.tile_dir[tile * 4 + 3] = static_cast<uint32_t>(t.tot_cut + n_beyond);
    }
    return;
  }

  // ---- the code bytes (dummy points: a zero nibble moves nothing), the parked values, the chain starts
  const uint32_t pdd_off = a.tile_dir[tile * 4 + 0], res_off = a.tile_dir[tile * 4 + 2];
  const bool staged = t.tot_len <= static_cast<uint32_t>(kCodeStage);                  // (the metadata in that place has left)
  uint8_t* const code = staged ? sm.nib : a.pdd_bytes + pdd_off;
  {
    uint32_t tau = t.tau_before, rho = t.rho_before, pre = t.pre;
    for (int i = t.p0; i < t.p1; ++i) {
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
    a.chain_tau0[ch] = t.has_chain ? tau_list[t.my_first] : uint16_t{0xFFFFu};
    a.chain_rho0[ch] = t.has_chain ? rho_list[t.my_first] : uint16_t{0xFFFFu};
    a.chain_len[ch] = static_cast<uint8_t>(t.len);
  }
  // surplus weights beyond the number of empty slots: Residual entries after the cut leftovers
  for (int i = t.P + tid; i < t.totS; i += kTileThreads) {
    const uint32_t to = res_off + static_cast<uint32_t>(t.tot_cut + (i - t.P)), rho = rho_list[i];
    a.res_rho[to] = static_cast<uint16_t>(rho);
    a.res_val[to] = high[rho];
  }
  const int chains = __reduce_add_sync(0xFFFFFFFFu, t.chains);
  if (lane == 0 && chains) atomicAdd(&sm.n_chains, chains);
  __syncthreads();
  // ---- the tile leaves: 128 bytes of values per row, and the code bytes
#pragma unroll
  for (int i = tid; i < kTileM * kH / 8; i += kTileThreads)
    *reinterpret_cast<uint4*>(a.tc_vals + (tm * kTileM + (i >> 3)) * half_ld + tk * kH + (i & 7) * 8) = reinterpret_cast<const uint4*>(sm.vals)[i];
  if (staged)
    for (uint32_t i = tid; i < t.tot_len; i += kTileThreads) a.pdd_bytes[pdd_off + i] = sm.nib[i];
  // one addition per tile and counter
  if (tid < 6) {
    const int v = tile_statistic(tid, t, sm.nnz, sm.n_chains);
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
}  // namespace
}  // namespace tl3

extern "C" int tl3_encode_device(const void* dW, int64_t M, int64_t K, int64_t ldw, void* stream, tl3_matrix** out) {
  using namespace tl3;
  if (!dW || !out || M <= 0 || K <= 0 || ldw < K || M > (int64_t{1} << 31) || K > (int64_t{1} << 31)) return TL3_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  tl3_matrix* m = new_device_matrix(M, K);
  if (!m) return TL3_ERR_NO_MEMORY;
  if (m->n_tiles > 0x7FFFFFFF) { tl3_free(m); return TL3_ERR_UNSUPPORTED; }
  const size_t n_vals = static_cast<size_t>(m->M_pad) * m->K_pad / 2, n_meta = n_vals / 4;
  const size_t n_chain = static_cast<size_t>(m->n_tiles) * kTileM, n_dir = static_cast<size_t>(m->n_tiles) * 4;

  int rc = TL3_OK;
  uint8_t* scratch = nullptr;               // everything the kernels write, in one allocation
  uint8_t* extra = nullptr;                 // PDD bytes and Residual entries that do not fit it
  unsigned long long totals[2] = {0, 0}, stats[6] = {0, 0, 0, 0, 0, 0};
  // layout of `scratch` (every part 256-byte aligned)
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  // One allocation serves the whole conversion (cudaMalloc and cudaFree of more than 2 MB take 0.35 ms
  // each, whatever the size: more than all kernels of a 5120 x 5120 matrix): the arrays of known size
  // and a guess at the PDD bytes and Residual entries that holds down to 40 %
  // sparsity; only a matrix that needs more has them allocated when their sizes are known.
  const size_t o_vals = 0, o_meta = o_vals + up(n_vals * 2), o_tau = o_meta + up(n_meta), o_rho = o_tau + up(n_chain * 2),
               o_len = o_rho + up(n_chain * 2), o_dir = o_len + up(n_chain), o_stats = o_dir + up(n_dir * 4), o_var = o_stats + 256;
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
    a.dense = dense_view(dW, M, K, ldw);
    a.K_pad = m->K_pad; a.tiles_k = static_cast<int>(m->tiles_k);
    a.tc_vals = reinterpret_cast<uint16_t*>(scratch + o_vals);
    a.tc_meta = scratch + o_meta;
    a.chain_tau0 = reinterpret_cast<uint16_t*>(scratch + o_tau);
    a.chain_rho0 = reinterpret_cast<uint16_t*>(scratch + o_rho);
    a.chain_len = scratch + o_len;
    a.tile_dir = reinterpret_cast<uint32_t*>(scratch + o_dir);
    a.stats = reinterpret_cast<unsigned long long*>(scratch + o_stats);
    a.emit = 0;
    TL3_ENC_CUDA(configure_encode_kernel());
    tl3_encode_kernel<<<static_cast<unsigned>(m->n_tiles), kTileThreads, sizeof(EncodeSmem), st>>>(a);
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
    tl3_encode_kernel<<<static_cast<unsigned>(m->n_tiles), kTileThreads, sizeof(EncodeSmem), st>>>(a);
    TL3_ENC_CUDA(cudaGetLastError());
    std::vector<HostPiece> arrays;
    try {
      m->tc_vals.resize(n_vals); m->tc_meta.resize(n_meta);
      m->chain_tau0.resize(n_chain); m->chain_rho0.resize(n_chain); m->chain_len.resize(n_chain);
      m->tile_dir.resize(n_dir);
      m->pdd_bytes.resize(totals[0]); m->res_rho.resize(totals[1]); m->res_val.resize(totals[1]);
      arrays = {
        {m->tc_vals.data(), a.tc_vals, n_vals * 2}, {m->tc_meta.data(), a.tc_meta, n_meta},
        {m->chain_tau0.data(), a.chain_tau0, n_chain * 2}, {m->chain_rho0.data(), a.chain_rho0, n_chain * 2},
        {m->chain_len.data(), a.chain_len, n_chain}, {m->tile_dir.data(), a.tile_dir, n_dir * 4},
        {m->pdd_bytes.data(), a.pdd_bytes, totals[0]}, {m->res_rho.data(), a.res_rho, totals[1] * 2}, {m->res_val.data(), a.res_val, totals[1] * 2}};
    } catch (const std::bad_alloc&) { rc = TL3_ERR_NO_MEMORY; goto done; }
    TL3_ENC_CUDA(copy_pieces(arrays, cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaMemcpyAsync(stats, a.stats, sizeof(stats), cudaMemcpyDeviceToHost, st));
    TL3_ENC_CUDA(cudaStreamSynchronize(st));
    m->nnz = static_cast<int64_t>(stats[0]); m->n_tc = static_cast<int64_t>(stats[1]); m->n_sf = static_cast<int64_t>(stats[2]);
    m->n_res = static_cast<int64_t>(stats[3]); m->n_dummy = static_cast<int64_t>(stats[4]); m->n_slots_unused = static_cast<int64_t>(stats[5]);
  }
done:
  if (scratch) cudaFree(scratch);
  if (extra) cudaFree(extra);
  if (rc != TL3_OK) { tl3_free(m); return rc; }
  *out = m;
  return TL3_OK;
}
