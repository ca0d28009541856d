// tcgen05 helpers (sm_103a): shared-memory and instruction descriptors for
// kind::tf32 with K-major, non-swizzled operands, TMEM allocation, MMA issue,
// commit to an mbarrier and bounded waits.
//
// Operand layout in shared memory ("canonical K-major, no swizzle"): an R x K
// fp32 matrix is stored as core matrices of 8 rows x 4 values (16 bytes per
// row, 128 bytes per core matrix); element (r, k) sits at float offset
//   ((k/4) * (R/8) + r/8) * 32 + (r%8) * 4 + (k%4),
// so core matrices adjacent along M/N are 128 B apart (stride byte offset) and
// adjacent along K are (R/8)*128 B apart (leading byte offset).  One
// kind::tf32 MMA consumes K = 8 (two core matrices along K).
// Accumulator layout in TMEM: M = 128 puts row r in lane r; M = 64 puts rows
// 16w..16w+15 in lanes 32w..32w+15 (w = 0..3); column j of D is TMEM column j.
#pragma once
#include <cstdint>
#include <utility>

namespace adg {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__host__ __device__ __forceinline__ int canon(int r, int k, int R) {
  return ((k >> 2) * (R >> 3) + (r >> 3)) * 32 + (r & 7) * 4 + (k & 3);
}

__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version
  return d;
}

// instruction descriptor: D f32, A and B tf32, both K-major, dense
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// round-toward-zero to tf32 (keep sign, exponent and 10 mantissa bits)
__host__ __device__ __forceinline__ float tf32_trunc(float x) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
#else
  uint32_t u;
  __builtin_memcpy(&u, &x, 4);
  u &= 0xFFFFE000u;
  __builtin_memcpy(&x, &u, 4);
  return x;
#endif
}

// MMA with the A operand in TMEM (lane = row, one tf32 per column)
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(db), "r"(idesc), "r"(acc));
}

// 3xTF32 product chain into d (M = 128): A in TMEM (hi at column ah, lo at
// al) times B^T, B canonical K-major N x K in shared memory (hi at byte
// address bh, lo at bl); K / 8 steps of A_hi B_hi + A_hi B_lo + A_lo B_hi.
// The descriptors are built once; a step advances their start address.
template <int N, int K>
__device__ __forceinline__ void mma3_ts(uint32_t d, uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl,
                                        bool acc_first) {
  constexpr uint32_t idesc = idesc_tf32(128, N);
  constexpr uint32_t lbo = (N / 8) * 128;
  const uint64_t dh0 = sdesc(bh, lbo, 128), dl0 = sdesc(bl, lbo, 128);
#pragma unroll
  for (int kk = 0; kk < K / 8; ++kk) {
    const uint64_t step = (uint64_t)((kk * 2 * lbo) >> 4);
    mma_ts(d, ah + 8 * kk, dh0 + step, idesc, (kk > 0 || acc_first) ? 1u : 0u);
    mma_ts(d, ah + 8 * kk, dl0 + step, idesc, 1u);
    mma_ts(d, al + 8 * kk, dh0 + step, idesc, 1u);
  }
}

__device__ __forceinline__ void commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar)));
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count));
  asm volatile("fence.mbarrier_init.release.cluster;");
}

// one thread's arrival on the mbarrier, announcing `bytes` of asynchronous copies
__device__ __forceinline__ void mbar_expect_tx(uint64_t* mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes)
               : "memory");
}
// bulk copy (TMA engine, non-tensor) global -> this CTA's shared memory, both
// 16-byte aligned, bytes a multiple of 16; completes on the mbarrier
__device__ __forceinline__ void bulk_load(void* sm, const void* g, uint32_t bytes, uint64_t* mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(sm)),
               "l"(g), "r"(bytes), "r"(smem_u32(mbar))
               : "memory");
}
// thread 0 of the CTA: `bytes` from global to shared memory in bulk copies of
// at most 32 KB, all completing on `mbar` (initialised, phase 0)
__device__ __forceinline__ void bulk_load_all(void* sm, const void* g, uint32_t bytes, uint64_t* mbar) {
  mbar_expect_tx(mbar, bytes);
  for (uint32_t o = 0; o < bytes; o += 32768u)
    bulk_load(static_cast<char*>(sm) + o, static_cast<const char*>(g) + o, bytes - o < 32768u ? bytes - o : 32768u,
              mbar);
}

// wait for phase `parity` of the mbarrier; false if the bound ran out
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t parity, int max_iter) {
  for (int it = 0; it < max_iter; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(mbar)), "r"(parity));
    if (ok) return true;
  }
  return false;
}

// bring [p, p + bytes) into L2 ahead of use (16-byte aligned, bytes a multiple
// of 16), in pieces of at most 8 KB
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  const char* c = static_cast<const char*>(p);
  for (uint32_t o = 0; o < bytes; o += 8192u) {
    const uint32_t n = bytes - o < 8192u ? bytes - o : 8192u;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(c + o), "r"(n) : "memory");
  }
}

// asynchronous 4-byte copy global -> shared (cp.async; committed and waited
// for with cp.async.commit_group / cp.async.wait_group)
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
// ... and of 16 bytes (both 16-byte aligned)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int NPEND>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(NPEND) : "memory"); }

// the same for any span: only its 16-byte aligned interior (a hint; the
// bytes at either end that share a 16-byte unit with the span's neighbours
// are left out)
__device__ __forceinline__ void prefetch_l2_inner(const void* p, uint32_t bytes) {
  const uintptr_t a0 = ((uintptr_t)p + 15) & ~(uintptr_t)15, a1 = ((uintptr_t)p + bytes) & ~(uintptr_t)15;
  if (a1 > a0) prefetch_l2(reinterpret_cast<const void*>(a0), (uint32_t)(a1 - a0));
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;"); }

template <int NCOLS>
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "n"(NCOLS));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
template <int NCOLS>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "n"(NCOLS));
}

// 8 C consecutive fp32 columns of this warp's lanes (one wait)
template <int C>
__device__ __forceinline__ void ld8s(uint32_t t, float* o) {
  uint32_t r[8 * C];
#pragma unroll
  for (int c = 0; c < C; ++c)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[8 * c]), "=r"(r[8 * c + 1]), "=r"(r[8 * c + 2]), "=r"(r[8 * c + 3]), "=r"(r[8 * c + 4]),
                   "=r"(r[8 * c + 5]), "=r"(r[8 * c + 6]), "=r"(r[8 * c + 7])
                 : "r"(t + 8 * c));
  // (the wait ties every loaded register: none may be read before it)
#pragma unroll
  for (int c = 0; c < C; ++c) {
    if (c == 0)
      asm volatile("tcgen05.wait::ld.sync.aligned;"
                   : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]));
    else
      asm volatile("" : "+r"(r[8 * c]), "+r"(r[8 * c + 1]), "+r"(r[8 * c + 2]), "+r"(r[8 * c + 3]),
                   "+r"(r[8 * c + 4]), "+r"(r[8 * c + 5]), "+r"(r[8 * c + 6]), "+r"(r[8 * c + 7]));
  }
#pragma unroll
  for (int k = 0; k < 8 * C; ++k) o[k] = __uint_as_float(r[k]);
}

// 8 values of this lane's row -> tf32 hi at column th, lo (the remainder) at column tl
__device__ __forceinline__ void st_split8(uint32_t th, uint32_t tl, const float x[8]) {
  uint32_t h[8], l[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float hh = tf32_trunc(x[j]);
    h[j] = __float_as_uint(hh);
    l[j] = __float_as_uint(x[j] - hh);
  }
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(th), "r"(h[0]),
               "r"(h[1]), "r"(h[2]), "r"(h[3]), "r"(h[4]), "r"(h[5]), "r"(h[6]), "r"(h[7]));
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(tl), "r"(l[0]),
               "r"(l[1]), "r"(l[2]), "r"(l[3]), "r"(l[4]), "r"(l[5]), "r"(l[6]), "r"(l[7]));
}

__host__ __device__ constexpr int up8(int x) { return (x + 7) / 8 * 8; }
__host__ __device__ constexpr int up16(int x) { return (x + 15) / 16 * 16; }

// C chunks of 8 columns of this lane's A row, value k from f(integral_constant<k>)
template <int C, class F, int... I>
__device__ __forceinline__ void put_chunk(uint32_t th, uint32_t tl, F&& f, std::integer_sequence<int, I...>) {
  const float x[8] = {f(std::integral_constant<int, 8 * C + I>{})...};
  st_split8(th + 8 * C, tl + 8 * C, x);
}
template <class F, int... C>
__device__ __forceinline__ void put_chunks(uint32_t th, uint32_t tl, F&& f, std::integer_sequence<int, C...>) {
  (put_chunk<C>(th, tl, f, std::make_integer_sequence<int, 8>{}), ...);
}
template <int C, class F>
__device__ __forceinline__ void put_row(uint32_t th, uint32_t tl, F&& f) {
  put_chunks(th, tl, f, std::make_integer_sequence<int, C>{});
}

constexpr int kWaitIters = 1 << 22;
// the 128 threads of a slot (one tile in flight): named barrier slot + 1
__device__ __forceinline__ void slot_bar(int slot) { asm volatile("bar.sync %0, 128;" ::"r"(slot + 1) : "memory"); }

// The tensor-core products of one slot.  issue(f): the A columns that the
// slot's threads wrote made visible, then f's MMAs by one thread.  done(): the
// products complete; one lane per warp waits (more waiting lanes take issue
// slots from the other slots' warps).  A wait that runs out is reported and the
// slot goes on to the end of its tile, where it leaves together.
struct SlotMma {
  uint64_t* mbar;
  int* abort;
  unsigned int* err;
  int slot, t, lane;
  uint32_t phase;
  // (by the first thread of warp `who`: the rounds of a tile take turns, a thread's
  // MMA instructions would make one warp of the slot late)
  template <class F>
  __device__ __forceinline__ void issue(int who, F&& f) {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    fence_before();
    slot_bar(slot);
    fence_after();
    if (t == 32 * who) {
      f();
      commit(mbar);
    }
  }
  __device__ __forceinline__ void done() {
    if (lane == 0 && !mbar_wait(mbar, phase, *(volatile int*)abort ? 1 : kWaitIters)) {
      atomicOr(err, 2u /* ERR_TIMEOUT */);
      *(volatile int*)abort = 1;
    }
    __syncwarp();
    mbar_wait(mbar, phase, 1);  // every thread observes the completed phase
    phase ^= 1u;
    fence_after();
  }
};


// The tiles of a slot.  Its first one is fixed (slot `me` of `slots` over all
// CTAs), later ones come from a counter in global memory, `chunk` consecutive
// tiles at a time, so that CTAs that start late (the kernels of a phase run side
// by side and share the SMs) or meet slow tiles take fewer.  One thread of the slot asks for the tile
// after the next at the start of a tile; the slot reads the answer after the
// barrier at its end.  The last CTA to leave resets the counter for the next
// launch.
struct TileFeed {
  int* counter;  // [0] units handed out, [1] CTAs that have left
  int* box;      // shared, [2] of this slot
  int slots, chunk;
  int64_t n;
  __device__ __forceinline__ int64_t after(int64_t tile) const {  // (by one thread)
    if (chunk > 1 && ((int)tile + 1) % chunk) return tile + 1;
    return tile < n ? ((int64_t)slots + atomicAdd(counter, 1)) * chunk : n;
  }
  __device__ __forceinline__ int64_t first(int me) const { return (int64_t)me * chunk; }
  // one thread of the CTA, when its slots are done
  __device__ __forceinline__ void leave() const {
    __threadfence();
    if (atomicAdd(counter + 1, 1) == (int)gridDim.x - 1) {
      counter[0] = 0;
      counter[1] = 0;
    }
  }
};


}  // namespace tc
}  // namespace adg
