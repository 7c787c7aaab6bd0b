// What the two SpMM kernels (tl3_spmm.cu: up to 64 columns a launch; tl3_spmm_wide.cu: more) share:
// PTX wrappers, the bounded wait, Algorithm 1 for one chain, the split of the tiles over the CTAs, and
// the host-side pieces of a launch.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include <cstdint>

#include "tl3_internal.h"

namespace tl3 {

#define TL3_CUDA(expr)                                        \
  do {                                                        \
    cudaError_t e_ = (expr);                                  \
    if (e_ != cudaSuccess) {                                  \
      tl3::set_cuda_error(static_cast<int>(e_));              \
      return TL3_ERR_CUDA;                                    \
    }                                                         \
  } while (0)

constexpr uint32_t kWrBytes = 16384;      // one W_r buffer
constexpr uint32_t kSmemLimit = 232448;   // 227 KB
constexpr uint32_t kTurnPitch = 36;       // bytes per row of a warp's turning area (16 halves, odd number of words)
constexpr uint32_t kTurnBytes = 32u * kTurnPitch;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // 2 s without progress, per wait
// A wait behind several others of the same CTA, each with its own 2 s (the last MMAs, an accumulator, the
// contributors' flags): one that gives up raises the abort flag, this one ends with it and reports nothing.
constexpr unsigned long long kHandOverLimitNs = 4 * kWaitLimitNs;
#ifndef TL3_TRYWAIT_HINT_NS
#define TL3_TRYWAIT_HINT_NS 20000u
#endif
constexpr uint32_t kTryWaitHintNs = TL3_TRYWAIT_HINT_NS;     // how long one barrier probe may park the thread

// status codes written to the workspace status word (0 = ok)
enum : uint32_t {
  kStProducer = 1, kStDecodeFull = 2, kStDecodeWrFree = 3, kStMmaDecoded = 4, kStMmaAccEmpty = 5,
  kStEpilogueAccFull = 6, kStDrain = 7, kStClearWrFree = 8, kStDecodeWrReady = 9, kStEpilogueTail = 10, kStEpilogueFlags = 11, kStMmaX = 12,
  kStBadBlock = 16           // a block's lengths or a decoded position were out of range (+ detail in bits 8..)
};

// ---------------------------------------------------------------------------------------------
// PTX helpers
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ unsigned long long global_timer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {   // more bytes to come, no arrival
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// One probe of the barrier phase.  The hint lets the hardware park the thread (up to that many
// nanoseconds, or until the phase completes) instead of spinning, so waiting warps do not take
// issue slots from the warps that have work.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(done) : "r"(bar), "r"(parity), "r"(kTryWaitHintNs) : "memory");
  return done != 0;
}

// Shared state every wait looks at: the abort flag (set by whoever gives up first) and the
// status word in global memory.
struct WaitCtx {
  volatile int* abort_flag;
  unsigned int* status;
};

// Bounded wait.  Returns false if the CTA is aborting (this or another waiter ran out of time).
// The limit runs from the moment THIS wait began to look slow (its sixteenth unsuccessful probe), not
// from the start of the kernel: a wait that completes is progress, so a long launch, or one whose
// context was switched out for a while earlier on, does not use up the allowance of later waits.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const WaitCtx& w, uint32_t code, unsigned long long limit = kWaitLimitNs) {
  unsigned long long t_slow = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 15u) == 15u) {
      if (*w.abort_flag) return false;
      const unsigned long long now = global_timer();
      if (t_slow == 0) t_slow = now;
      if (now - t_slow > limit) {
        atomicCAS(w.status, 0u, code);
        *w.abort_flag = 1;
        return false;
      }
    }
  }
}

__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void named_bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// barrier + AND-reduction of a predicate over the `threads` threads that use barrier `id`
__device__ __forceinline__ bool named_bar_all(int id, int threads, bool pred) {
  uint32_t out;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %3, 0;\n\t"
      "bar.red.and.pred p, %1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(out) : "r"(id), "r"(threads), "r"(static_cast<uint32_t>(pred)) : "memory");
  return out != 0;
}

// The weight blocks are read once: they are marked evict-first in L2 so that what is read again
// (X, the kernel's own code, partial sums) is not pushed out by the stream.
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar) : "memory");
}

// Programmatic dependent launch: the next kernel on the stream may be scheduled as soon as every
// CTA of this one has said so (it still cannot take an SM before a CTA here exits), and a kernel
// must call pdl_wait() before it reads what its predecessor wrote or writes what its
// predecessor may still read.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One lane of a converged warp; the caller keeps every operand warp-uniform so that the
// single-thread instructions (bulk copies, MMAs, commits) take uniform registers directly.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}

// D[tmem] (+)= A_sparse[smem] * B[smem] with the 2-bit metadata at e_tmem.  The shared-memory
// descriptors are passed as their low words (start address field) and one common high word each.
__device__ __forceinline__ void umma_sp_f16(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                            uint32_t e_tmem, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %7, 0;\n\t"
      "mov.b64 da, {%1, %2};\n\t"
      "mov.b64 db, {%3, %4};\n\t"
      "tcgen05.mma.sp.cta_group::1.kind::f16 [%0], da, db, [%5], %6, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(e_tmem), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Positions in a block are bank-major slot coordinates u = bank << 8 | slot-in-window << 7 | row,
// where bank is the 32-bit word of the 128-byte (swizzled) row that holds the slot's window.  The
// byte offset of slot u inside the 128 x 128-byte K-major image is therefore a bit-field move:
// row * 128 + bank * 4 + slot-in-window * 2.  The packer orders both PDD streams by u and gives
// lane l of a decode warp a chain whose empty slots all lie in bank l.
__device__ __forceinline__ uint32_t swizzled_offset(uint32_t u) { return ((u & 0x7Fu) << 7) | ((u >> 6) & 0x7Eu); }

// SiLU or GELU of sum + bias, in fp32, before the rounding to fp16, four columns at a time.  A real call,
// not inlined: it is used from many unrolled places, and a kernel image that grows by tens of kilobytes
// costs every launch time at its start.  Four at a time because a call per element left a reducer's tail
// waiting for one chain of dependent instructions after another (5120 x 5120, N = 64 with GELU 20.2 -> 17.4 us).
static __device__ __noinline__ float4 activate4(float4 v, float bias, int act) {
  float x[4] = {v.x + bias, v.y + bias, v.z + bias, v.w + bias};
  if (act == TL3_ACT_SILU) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = x[i] / (1.f + __expf(-x[i]));
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = 0.5f * x[i] * (1.f + tanhf(0.7978845608f * (x[i] + 0.044715f * x[i] * x[i] * x[i])));
  }
  return make_float4(x[0], x[1], x[2], x[3]);
}

// Epilogue of tl3_spmm_ex for the first `cols` of n sums of a row (what lies beyond may change or not; 0 for a
// row that is not stored: its zeros would take the slow way through SiLU's division): bias and ReLU in
// place, the functions by call.
template <int n>
__device__ __forceinline__ void apply_epilogue(uint32_t* v, float bias, int act, int cols) {
  if (act <= TL3_ACT_RELU) {
#pragma unroll
    for (int c = 0; c < n; ++c) v[c] = __float_as_uint(__uint_as_float(v[c]) + bias);
    if (act == TL3_ACT_RELU) {
#pragma unroll
      for (int c = 0; c < n; ++c) v[c] = __float_as_uint(fmaxf(__uint_as_float(v[c]), 0.f));
    }
    return;
  }
#pragma unroll
  for (int c = 0; c < n; c += 4) {
    if (c >= cols) continue;
    const float4 x = activate4(make_float4(__uint_as_float(v[c]), __uint_as_float(v[c + 1]), __uint_as_float(v[c + 2]), __uint_as_float(v[c + 3])), bias, act);
    v[c] = __float_as_uint(x.x); v[c + 1] = __float_as_uint(x.y); v[c + 2] = __float_as_uint(x.z); v[c + 3] = __float_as_uint(x.w);
  }
}

template <int NPAD> struct TmemLd;
template <> struct TmemLd<16> {
  static __device__ __forceinline__ void ld(uint32_t taddr, uint32_t* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(taddr) : "memory");
  }
};
template <> struct TmemLd<32> {
  static __device__ __forceinline__ void ld(uint32_t taddr, uint32_t* v) {
    TmemLd<16>::ld(taddr, v);
    TmemLd<16>::ld(taddr + 16, v + 16);
  }
};
template <> struct TmemLd<64> {
  static __device__ __forceinline__ void ld(uint32_t taddr, uint32_t* v) {
    TmemLd<32>::ld(taddr, v);
    TmemLd<32>::ld(taddr + 32, v + 32);
  }
};

// The wait for TmemLd<n>::ld(.., v).  It names the registers that the load fills: to the compiler they are
// ready when the load has been issued, and it might copy or read them in front of a wait that does not.
template <int n>
__device__ __forceinline__ void tmem_wait_ld(uint32_t* v) {
  static_assert(n == 16 || n == 32, "columns of one step of an epilogue");
  if constexpr (n == 16) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]) :: "memory");
  } else {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                   "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                   "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31]) :: "memory");
  }
}

// CTA c of G owns tiles [c*T/G, (c+1)*T/G); the CTA that owns tile t.  In 32 bits: the launcher
// refuses matrices with (G + 1) * T >= 2^32 (hundreds of gigabytes), and a 64-bit division costs a
// CTA 0.15 us each at its cold start, where there are three of them.
__device__ __forceinline__ uint32_t range_begin(uint32_t c, uint32_t T, uint32_t G) { return c * T / G; }
__host__ __device__ __forceinline__ int owner_of(uint32_t t, uint32_t T, uint32_t G) { return static_cast<int>(((t + 1u) * G - 1u) / T); }

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_u16(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(static_cast<uint16_t>(v)) : "memory");
}
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_zero16B(uint32_t addr) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0u) : "memory");
}

// Algorithm 1 for one chain, one code word (four delta bytes) at a time.  `pos` carries offset_t in
// its low and offset_r in its high 16 bits (both as bank-major coordinates u), so one add advances
// both cursors and two shift/mask pairs form both byte offsets.  Within a round all positions are
// formed first, then all W_t loads are issued, then all stores, so that the shared-memory round
// trips of different entries overlap.  (Rounds of two code words, and a software-pipelined loop
// that issues the next round's loads before this round's stores, both measured slower.)

// packed byte offsets (W_t offset low, W_r offset high) of the packed positions `pos`
__device__ __forceinline__ uint32_t swizzled_offset2(uint32_t pos) { return ((pos & 0x007F007Fu) << 7) | ((pos >> 6) & 0x007E007Eu); }

// Positions are checked (< 8192 slots per tile) before they become addresses; a violation is
// reported in *bad and the entry is skipped.  The code words of a tile are stored transposed
// (word k of chain slot j at (k * 128 + j) * 4) and every chain has `n_words` of them (<= 3, padded
// with zero bytes = dummy points), so the loads are conflict free and the loop is warp-uniform.
__device__ __forceinline__ void decode_chain(uint32_t stage, uint32_t wr, uint32_t hdr, uint32_t code_addr, uint32_t n_words, uint32_t* bad) {
  if (hdr == 0xFFFFFFFFu) return;                       // empty chain
  if (hdr & 0xE000E000u) { *bad = 1u; return; }
  uint32_t pos = hdr;
  uint32_t w[3] = {0u, 0u, 0u};
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (static_cast<uint32_t>(k) < n_words) w[k] = lds_u32(code_addr + k * 512);
  {                                                     // first pair: absolute 16-bit positions
    const uint32_t off2 = swizzled_offset2(pos);
    const uint32_t at = stage + (off2 & 0xFFFFu);
    const uint32_t v = lds_u16(at);
    sts_u16(at, 0);                                     // the slot it was parked in is empty again
    sts_u16(wr + (off2 >> 16), v);                      // the value goes to its own position in W_r
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {                         // one code word = four delta bytes
    if (static_cast<uint32_t>(k) >= n_words) break;
    const uint32_t bytes = w[k];
    uint32_t off2[4], val[4];
    bool real[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t bt = __byte_perm(bytes, 0u, 0x4440u + q);    // delta byte q
      const uint32_t delta = (bt * 0x1001u) & 0x000F000Fu;        // t delta | r delta << 16
      pos += delta;
      real[q] = ((delta - 0x00010001u) & 0x80008000u) == 0u;      // both nibbles non-zero (else a dummy point)
      off2[q] = swizzled_offset2(pos);
    }
    // both cursors only grow, so the last position of the round bounds them all
    if (pos & 0xE000E000u) {
      *bad = 2u;
#pragma unroll
      for (int q = 0; q < 4; ++q) real[q] = false;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (real[q]) val[q] = lds_u16(stage + (off2[q] & 0xFFFFu));
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (real[q]) { sts_u16(stage + (off2[q] & 0xFFFFu), 0); sts_u16(wr + (off2[q] >> 16), val[q]); }
  }
}

// Residual layer of a tile for thread r of a decode group: (position, value) entries go to W_r.  Tiles with many (kLong)
// take four at a time, loads before stores: one after another, 13 per thread at 40 % sparsity, their round
// trips stood in the decode's way (11008 x 4096 at 40 %, N = 24 23.2 -> 22.2 us, N = 16 18.9 -> 18.2; 20480 x 5120 at 40 %, N = 128
// 49.4 -> 46.8).  A kernel of its own, because tiles with one or two per thread only lose by the longer code
// (9216 x 9216, N = 64 30.5 -> 30.8).
template <bool kLong>
__device__ __forceinline__ void scatter_residual(uint32_t res, uint32_t wr, uint32_t r, uint32_t res_cnt, uint32_t* bad) {
  uint32_t k = r;
  if constexpr (kLong) {
    for (uint32_t left = res_cnt; left >= 512u; left -= 512u, k += 512u) {
      uint32_t rv[4], any = 0u;
#pragma unroll
      for (int q = 0; q < 4; ++q) { rv[q] = lds_u32(res + 4 * (k + 128u * q)); any |= rv[q]; }
      if (any & 0xE000u) { *bad = 4u; return; }
#pragma unroll
      for (int q = 0; q < 4; ++q) sts_u16(wr + swizzled_offset(rv[q] & 0xFFFFu), rv[q] >> 16);
    }
  }
  for (; k < res_cnt; k += 128) {
    const uint32_t rv = lds_u32(res + 4 * k);
    if ((rv & 0xFFFFu) < 8192u) sts_u16(wr + swizzled_offset(rv & 0xFFFFu), rv >> 16);
    else *bad = 4u;
  }
}

// ---------------------------------------------------------------------------------------------
// Host side, in tl3_spmm.cu
// ---------------------------------------------------------------------------------------------
struct DeviceInfo {
  int sm_count = 0;
  int cc_major = 0;
  bool ok = false;
};
int device_info(DeviceInfo* out);

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn();

// whether a matrix's tiles have so many Residual entries that scatter_residual<true> pays: one batch of four per thread
// on average, which leaves out 48 % sparsity and more and takes in 46 %.  (us short / long: 656 entries a tile, 46 %, 11008 x 4096, N =
// 16, 24, 64, 128 17.3 / 17.1, 18.5 / 18.2, 21.2 / 20.9, 26.6 / 26.0, 9216 x 9216 26.7 / 26.3, 28.4 / 28.1, 32.7 / 32.3, 39.0 / 39.0; 491, 47 %,
// 17.1 / 16.9, 18.1 / 17.8, 20.9 / 20.7, 26.4 / 26.0, but 26.3 / 26.7, 28.1 / 28.4, 32.1 / 32.5, 38.6 / 39.1; 328, 48 %, level; 164, 49 %,
// 16.1 / 16.2, 17.4 / 17.4, 19.9 / 20.0, 25.8 / 25.9.)
inline bool long_residual(const tl3_matrix* m) { return m->dev_n_res >= 512 * m->n_tiles; }

struct WorkspaceLayout {
  size_t status_off = 0, flags_off = 256, room_off = 0, partials_off = 0, total = 0;
};
WorkspaceLayout workspace_layout(int N, int sm_count);

// ---- tl3_spmm_wide.cu: N > 64 columns in one launch
constexpr int kWideColumns = 256;                               // most columns of one pass over W
constexpr int kRoomUnit = 16;                                   // unit of the workspace's record of its size, in columns per CTA
int spmm_wide(const tl3_matrix* m, const void* X, int64_t ldx, void* Y, int64_t ldy, int N, const tl3_epilogue* ep, bool xt,
              void* workspace, void* stream);                   // kWideNoPlan: blocks too large for it, or 2^32 / (CTAs + 1) tiles and more

constexpr int kWideNoPlan = 1;

}  // namespace tl3
