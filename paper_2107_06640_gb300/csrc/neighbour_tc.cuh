// Neighbour kernel on the tensor cores (tcgen05, 3xTF32), degrees 5 and 4,
// FP32 dofs: face fluxes of Sec. 4.2 (Eq. numerical-flux), formed as in the row
// kernel (row_neighbour.cuh), and their lift as a tensor-core product.
//
// A tile is 12 (virtual) elements x 9 quantities = 128 TMEM lanes: warp w of a
// slot holds elements 3w..3w+2, lane 9j+p = element 3w+j, quantity p (lanes
// 27..31 idle).  A CTA of 512 threads keeps four tiles in flight, one per slot
// of 128 threads and 128 TMEM columns; the warps of a slot meet only where an
// operand of the lift is complete.  A warp forms, face by face,
// the flux rows of row_flux.cuh; lane (element, quantity) then takes its row.
// The lift Q[l] -= sum_f sum_r R_f[r][l] G_f[r] is one product per face (A in
// TMEM, one face after another in the same 48 columns), which runs while the
// next face is worked on, so that a thread holds one flux row at a time and 128
// registers suffice for four tiles.  (Faces 0 and 1 through their sum and
// difference and the parities of faces 2 and 3 apart take half the tensor
// work, but hold two more rows: three tiles of 168 registers, 483 us on the
// 183,456-tet degree-5 box where this form takes 378; the nodal kernel before,
// nine quantities staged and two tiles in flight, took 652.)
//
// What bounds it: shared-memory traffic (L1 / shared-memory pipe 81 % busy) and
// instruction issue (52 %); DRAM 50 % busy (374,400 tets; 0.66 of the copy
// bandwidth in needed bytes at 1,497,600).  The 128 registers spill 36 bytes at
// degree 5, up to 148 with LTS faces, none at degree 4.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "func_attr.hpp"
#include "kernels.cuh"
#include "row_flux.cuh"
#include "sparse_ops.cuh"
#include "tc_common.cuh"

namespace adg {

namespace {

constexpr int TE = kTileElems;
constexpr int kSlotsN = 4, kThreadsN = 128 * kSlotsN;
using tc::kWaitIters;

using sp::count_par;
using sp::par_index;
using tc::up16;
using tc::up8;

template <int N>
struct NImg {
  static constexpr int B = nb3(N), BF = nb2(N), FS = face_block(N);
  static constexpr int NE = up16(count_par(B, 0)), NO = up16(count_par(B, 1));    // outputs: even, odd l
  static constexpr int KS = up8(BF), NL = NE + NO;
  // lift operands (floats): per face, hi block then lo block; rows: even l, then odd l from NE
  static constexpr int sF = NL * KS, image = 4 * 2 * sF;
  using F = FaceSmem<float, N>;
  static constexpr int oPV = image;
  static constexpr int oW = oPV + (F::table + 3) / 4 * 4;   // per warp: two stage buffers, the flux rows
  static constexpr int sW = 2 * F::stage + F::rows;
  static_assert(F::stage + F::rows >= 27 * B, "the lifted rows take the second stage buffer and the flux rows");
  static_assert(oW % 4 == 0 && F::stage % 4 == 0 && sW % 4 == 0, "16-byte aligned buffers");
  static constexpr int bytes = (oW + 4 * kSlotsN * sW) * 4;
  static constexpr int cAl = 24, cAcc = 48;  // TMEM columns: A hi 0, A lo, accumulator
  static_assert(KS <= 24 && cAcc + NL <= 128, "TMEM columns of a slot");
  static_assert(bytes + 256 <= 232448, "neighbour tensor-core kernel exceeds the shared memory of one CTA");
};

// kOne: one scenario (S = 1), where a virtual element is its element and the
// 64-bit divisions by S drop out; kLts: the launch's elements may have a
// neighbour in another cluster or a gravitational face (without, that code
// stays out of the kernel)
template <int N, bool kOne, bool kLts>
__global__ void __launch_bounds__(kThreadsN, 1) neighbour_tc_kernel(StepArgs a, const __grid_constant__ Segs g) {
  using NI = NImg<N>;
  using F = FaceSmem<float, N>;
  constexpr int B = NI::B, BF = NI::BF, FS = NI::FS;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  float* const sm = reinterpret_cast<float*>(smem_raw);
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t mbar[kSlotsN], s_img;
  __shared__ int s_abort[kSlotsN], s_next[kSlotsN][2];

  const int tid = threadIdx.x, slot = tid >> 7, t = tid & 127, w = t >> 5, lane = tid & 31;
  if (tid == 0) {
    tc::mbar_init(&s_img, 1);
    tc::bulk_load_all(sm, a.tc_lift, NI::image * 4, &s_img);
  }
  reorient_table<float, N>(sm + NI::oPV, reinterpret_cast<const float*>(a.reorient), tid, kThreadsN);
  if (tid < kSlotsN) {
    tc::mbar_init(&mbar[tid], 1);
    s_abort[tid] = 0;
  }
  const int64_t ntiles = g.first[g.n];
  const int slots = (int)gridDim.x * kSlotsN, me = slot * (int)gridDim.x + (int)blockIdx.x;
  const tc::TileFeed feed{a.tiles, s_next[slot], slots, g.chunk, ntiles};
  int64_t tile = feed.first(me);
  if (t == 32) s_next[slot][1] = (int)feed.after(tile);
  if (tid < 32) tc::tmem_alloc<512>(&tmem_base);
  __syncthreads();  // (the image barrier is initialised)
  const bool img_ok = tc::mbar_wait(&s_img, 0, kWaitIters);
  tc::fence_async_smem();
  tc::fence_before();
  const bool all_ok = __syncthreads_and(img_ok);
  tc::fence_after();
  if (!all_ok) {
    // the operands did not arrive within the bound: report, give the copies a
    // bounded chance to finish, free the columns and leave
    if (tid == 0) {
      atomicOr(a.err, ERR_TIMEOUT);
      tc::mbar_wait(&s_img, 0, kWaitIters);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid < 32) tc::tmem_dealloc<512>(tmem_base);
    if (tid == 0) feed.leave();
    return;
  }

  const uint32_t tbase = tmem_base + (uint32_t)slot * 128u, trow = tbase + ((uint32_t)(32 * w) << 16);
  const uint32_t sL = tc::smem_u32(sm);
  float* const sStage = sm + NI::oW + (slot * 4 + w) * NI::sW;
  float* const sG = sStage + 2 * F::stage;
  float* const sRows = sStage + F::stage;  // the lifted rows at a tile's end
  const float* const trace = reinterpret_cast<const float*>(a.trace);
  auto elem = [&](int64_t vv) -> int64_t { return kOne ? vv : elem_of(vv, a.S); };
  // this warp's part of tile tl: first virtual element, elements (<= 3, may be 0), segment
  using Part = TilePart;
  auto part_of = [&](int64_t tl) { return tile_part<TE, 3>(g, tl, w); };
  // lane 4 j + f (< 12): face f of the part's element j
  auto faces_of = [&](const Part& p, int& info, int& nbr) {
    info = 0;
    nbr = 0;
    if (lane < 4 * p.nE) {
      const int64_t ef = elem(p.v0 + (lane >> 2)) * 4 + (lane & 3);
      info = a.ninfo[ef];
      nbr = a.nbr[ef];
    }
  };
  auto stage = [&](const Part& p, int info, int nbr, int f, int buf) {
    face_stage<float, N, kOne>(a, sStage + buf * F::stage, p.v0, p.nE, info, nbr, f, lane);
  };

  float bad = 0.f;  // stays 0 while every updated dof is finite (x * 0 is NaN for x = inf, NaN)
  tc::SlotMma mma{&mbar[slot], &s_abort[slot], a.err, slot, t, lane, 0};
  // an operand row (zero past `cnt`) into the A columns
  auto put = [&](const auto& x, auto cc) {
    constexpr int cnt = decltype(cc)::value;
    tc::put_row<up8(cnt) / 8>(trow, trow + NI::cAl, [&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (k < cnt) return x[k]; else return 0.f;
    });
  };

  int it = 0;
  Part p{0, 0, 0};
  int info = 0, nbr = 0;
  if (tile < ntiles) {
    p = part_of(tile);
    faces_of(p, info, nbr);
    stage(p, info, nbr, 0, 0);
  }
  for (int64_t next = s_next[slot][1]; tile < ntiles;) {
    // the tile after the next, asked for now and handed to the slot at the end
    const int64_t after = t == 32 ? feed.after(next) : 0;
    Part pn{0, 0, 0};
    int info_n = 0, nbr_n = 0;
    if (next < ntiles) {
      pn = part_of(next);
      faces_of(pn, info_n, nbr_n);
      // the next tile's dofs and own face blocks into L2
      if (lane == 0 && pn.nE > 0) {
        tc::prefetch_l2_inner(reinterpret_cast<const float*>(a.Q) + pn.v0 * 9 * B, (uint32_t)(pn.nE * 9 * B * 4));
        tc::prefetch_l2(trace + pn.v0 * 4 * FS, (uint32_t)(pn.nE * 4 * FS * 4));
      }
    }
    const bool valid = lane < 9 * p.nE;
    // some face's neighbour is in another cluster
    const bool lts = kLts && __any_sync(0xffffffffu, ((info >> 5) & 7) == NK_COARSE || ((info >> 5) & 7) == NK_FINE);

    // the faces one after another (one copy of the code): the flux row x of
    // this lane's element and quantity, then what the lift does with it
    constexpr int VW = B % 4 == 0 ? 4 : 1;
    constexpr int nV = 27 * B / VW;
    struct alignas(4 * VW) V {
      float x[VW];
    };
    float* const Q = reinterpret_cast<float*>(a.Q) + p.v0 * 9 * B;
    const int cnt = p.nE * 9 * B / VW;
#pragma unroll 1
    for (int f = 0; f < 4; ++f) {
      tc::cp_async_wait<0>();
      __syncwarp();
      if (f < 3)
        stage(p, info, nbr, f + 1, (f + 1) & 1);
      else if (next < ntiles)
        stage(pn, info_n, nbr_n, 0, 0);
      float* const st = sStage + (f & 1) * F::stage;
      if (lts) {
        face_lts<float, N>(a, g.s[p.seg], st, p.v0, p.nE, info, nbr, f, lane);
        __syncwarp();
      }
      face_items<float, N, kLts>(a, st, sm + NI::oPV, sG, p.v0, p.nE, info, f, lane);
      __syncwarp();
      float x[BF];
      face_row<float, N>(sG, lane < 27 ? lane : 0, x);
      // (rows past the part's elements hold anything: no other row reads them)
      if (f > 0) mma.done();  // the face before has been lifted: its columns are free
      put(x, std::integral_constant<int, BF>{});
      mma.issue(f, [&] {
        const uint32_t b = sL + 4 * f * 2 * NI::sF;
        tc::mma3_ts<NI::NL, NI::KS>(tbase + NI::cAcc, tbase, tbase + NI::cAl, b, b + 4 * NI::sF, f > 0);
      });
    }
    // the dofs of this warp's part, as they lie in memory, requested before the last product is waited for
    V q[(nV + 31) / 32];
#pragma unroll
    for (int k = 0; k < (nV + 31) / 32; ++k)
      if (lane + 32 * k < cnt) q[k] = reinterpret_cast<const V*>(Q)[lane + 32 * k];
    mma.done();
    // ---- Q -= lift: the rows through shared memory, laid out as in memory
    {
      constexpr int CE = (count_par(B, 0) + 7) / 8, CO = (count_par(B, 1) + 7) / 8;
      float x[8 * (CE + CO)];
      tc::ld8s<CE>(trow + NI::cAcc, x);
      tc::ld8s<CO>(trow + NI::cAcc + NI::NE, x + 8 * CE);
      if (valid) {
        float* const r = sRows + lane * B;
        sp::each<B / VW>([&](auto cc) {
          constexpr int c = decltype(cc)::value;
          V v;
          sp::each<VW>([&](auto kc) {
            constexpr int l = c * VW + decltype(kc)::value;
            v.x[decltype(kc)::value] = x[(sp::parity(l) ? 8 * CE : 0) + par_index(l)];
          });
          reinterpret_cast<V*>(r)[c] = v;
        });
      }
      tc::fence_before();
      __syncwarp();
#pragma unroll
      for (int k = 0; k < (nV + 31) / 32; ++k) {
        if (lane + 32 * k < cnt) {
          const V y = reinterpret_cast<const V*>(sRows)[lane + 32 * k];
#pragma unroll
          for (int d = 0; d < VW; ++d) {
            q[k].x[d] -= y.x[d];
            bad = fmaf(q[k].x[d], 0.f, bad);
          }
          reinterpret_cast<V*>(Q)[lane + 32 * k] = q[k];
        }
      }
      __syncwarp();  // the rows are read before the next tile's fluxes overwrite them
    }
    if (t == 32) s_next[slot][it & 1] = (int)after;
    tc::slot_bar(slot);
    if (*(volatile int*)&s_abort[slot]) break;
    tile = next;
    next = s_next[slot][it & 1];
    ++it;
    p = pn;
    info = info_n;
    nbr = nbr_n;
  }
  if (__any_sync(0xffffffffu, bad != 0.f) && lane == 0) atomicOr(a.err, ERR_NAN);
  tc::cp_async_wait<0>();  // no copy into shared memory outlives the loop
  // after a timed-out wait, give this slot's products in flight a bounded chance to finish
  if (t == 0 && s_abort[slot]) tc::mbar_wait(&mbar[slot], mma.phase ^ 1u, kWaitIters);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (tid < 32) tc::tmem_dealloc<512>(tmem_base);
  if (tid == 0) feed.leave();
}

}  // namespace

// The launcher of degree N (the kernel table of that degree's translation unit).
template <int N>
int launch_neighbour_tc_deg(const StepArgs& a, const Segs& g, int n_sms, void* stream, bool lts) {
  using K = void (*)(StepArgs, Segs);
  // [S == 1][lts]
  static const K kern[2][2] = {{neighbour_tc_kernel<N, false, false>, neighbour_tc_kernel<N, false, true>},
                               {neighbour_tc_kernel<N, true, false>, neighbour_tc_kernel<N, true, true>}};
  const int rc = configure_on_device((const void*)kern[0][0], [] {
    cudaError_t ce = cudaSuccess;
    for (int i = 0; i < 4; ++i)
      if (ce == cudaSuccess)
        ce = cudaFuncSetAttribute((const void*)kern[i / 2][i % 2], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  NImg<N>::bytes);
    return ce;
  });
  if (rc) return rc;
  const int64_t ntiles = g.n ? g.first[g.n] : 0;
  if (ntiles <= 0) return 0;
  const int64_t units = (ntiles + g.chunk - 1) / g.chunk;
  const unsigned grid = (unsigned)(units < n_sms ? units : n_sms);
  StepArgs b = a;
  b.tiles = a.tiles + 2 * TILES_NEIGHBOUR;
  kern[a.S == 1 ? 1 : 0][lts ? 1 : 0]<<<grid, kThreadsN, NImg<N>::bytes, (cudaStream_t)stream>>>(b, g);
  return (int)cudaGetLastError();
}

// Host-side B operands of the lift of degree N: rfc[f][l][r], the face modes of
// phi_l, split into tf32 hi / lo, canonical K-major layout.
template <int N>
void pack_lift_tc_deg(const double* rfc, float* out) {
  using NI = NImg<N>;
  constexpr int B = NI::B, BF = NI::BF;
  for (int i = 0; i < NI::image; ++i) out[i] = 0.f;
  for (int f = 0; f < 4; ++f)
    for (int l = 0; l < B; ++l)
      for (int r = 0; r < BF; ++r) {
        const float xf = (float)rfc[((size_t)f * B + l) * BF + r], hi = tc::tf32_trunc(xf);
        const int o = f * 2 * NI::sF + tc::canon((sp::parity(l) ? NI::NE : 0) + par_index(l), r, NI::NL);
        out[o] = hi;
        out[o + NI::sF] = xf - hi;
      }
}

}  // namespace adg
