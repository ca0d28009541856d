// Local element kernel on the tensor cores (tcgen05, 3xTF32), degrees 5 and 4,
// FP32 dofs: Cauchy-Kovalewski predictor, time integral, modal face traces and
// volume term of Sec. 4.1 for elements without fault faces or two or more
// gravitational faces (those take the row kernel, row_local.cuh).
//
// A tile is 12 (virtual) elements x 9 quantities = the 128 rows of the MMAs,
// one row per TMEM lane and thread: warp w of a slot holds elements
// 3w..3w+2, lane 9j+p = quantity p of its j-th element (lanes 27..31 idle), as
// in the row kernel, with which this one shares everything but its three
// large products.  Those run on the tensor cores, rows (A, in TMEM, split into
// tf32 hi + lo by the row's thread) times reference matrices (B, in shared
// memory, hi and lo): the first predictor level, the face projections and the
// volume term.  All three are split by the parity of i (sparse_ops.inc), even
// and odd input modes apart: 10,368 multiplications per row at degree 5 where
// the dense products take 19,264, and an 81 KB operand image.  The other
// predictor levels (35 rows and fewer) are sparse FMAs on the thread's own
// registers: two MMA rounds less per tile, each of which cost a barrier, the
// split of an operand and two TMEM round trips.
//
// A CTA keeps two tiles in flight, one per slot of 128 threads and 256 TMEM
// columns (512 are what TMEM holds: the limit); the slot's warps meet only at
// its three MMA rounds.  The dofs rows of the next tile are requested with
// cp.async at the start of a tile; the row update happens in shared memory.
// The trace products' results leave while the volume product runs.
//
// Acoustic ocean (Sec. 4.1: the fluid is the elastic system with mu = 0;
// stress -p I): the fluid instantiation works on the 4 quantities (p, v) only,
// stored as the sigma_xx row (sigma_yy = sigma_zz = sigma_xx, no shear) and the
// velocity rows; a tile is 32 elements x 4 quantities (warp w: elements
// 8w..8w+7, lane 4j+p).  Face blocks are those of every other element.
//
// kSpec: elements with one gravitational face or a finer LTS neighbour, with
// row_local.cuh's SpecLevels between the levels (one buffer of dofs rows: the
// room goes to the surfaces' modes).
//
// What bounds it: the latency of a warp's own instruction stream (eight warps
// per SM, 0.40 instructions per clock and scheduler), not a roof: DRAM 28 % busy
// (0.32 of the copy bandwidth in needed bytes at 1,497,600 tets), tensor pipe
// active 19 % of the time (374,400 tets, elastic launch).  Local phase of the
// 183,456-tet degree-5 coupled box (all kinds): 788 us with 256 threads per
// tile, five dense MMA rounds and nodal nine-quantity faces, 594 us now; plain
// elastic launch of its 93,600-tet version 392 -> 266 us.  Degree 4: 593 -> 435 us;
// 81,600 acoustic tets at degree 4: 101 us (161 with the faces' normals read from
// global memory where they are used), 0.29 of the HBM bandwidth.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "func_attr.hpp"
#include "kernels.cuh"
#include "row_local.cuh"
#include "tc_common.cuh"

namespace adg {

namespace {

using sp::count_fpar;
using sp::count_par;
using sp::fpar_index;
using sp::fparity;
using sp::par_index;
using sp::par_mode;
using sp::parity;
using tc::kWaitIters;
using tc::up16;
using tc::up8;

// The medium of an instantiation: quantities per element, elements per warp
// and per tile, and the dofs row of quantity p.
struct Elastic {
  static constexpr bool fluid = false;
  static constexpr int Q = 9, EW = 3, TE = kTileElems;
};
struct Acoustic {
  static constexpr bool fluid = true;
  static constexpr int Q = 4, EW = row::EWF, TE = kTileElemsFluid;
};
static_assert(Elastic::TE == 4 * Elastic::EW && Acoustic::TE == 4 * Acoustic::EW, "tile of 4 warps");

// Operands (floats): for each product the even-input and the odd-input matrix,
// hi block then lo block, canonical K-major.  Output columns:
//   level 0   even inputs: KY of the even rows, KZ of the even rows, KX of the
//             odd rows; odd inputs: KY odd, KZ odd, KX even (rows below B1)
//   traces    even inputs: R0, then the even modes of R2 and of R3; odd inputs
//             the same with the odd modes (face 0 = even + odd sums, face 1 =
//             their difference)
//   volume    as level 0 with the transposes (rows below B, inputs below B1)
template <int N>
struct LImg {
  static constexpr int B = nb3(N), B1 = nb3(N - 1), BF = nb2(N);
  static constexpr int BE = count_par(B, 0), BO = count_par(B, 1), ME = count_par(B1, 0), MO = count_par(B1, 1);
  static constexpr int FE = count_fpar(BF, 0), FO = count_fpar(BF, 1);
  static constexpr int KE = up8(BE), KO = up8(BO), VE = up8(ME), VO = up8(MO);  // K of the products
  static constexpr int nPE = up16(2 * ME + MO), nPO = up16(2 * MO + ME);
  static constexpr int nTE = up16(BF + 2 * FE), nTO = up16(BF + 2 * FO);
  static constexpr int nVE = up16(2 * BE + BO), nVO = up16(2 * BO + BE);
  static constexpr int sPE = nPE * KE, sPO = nPO * KO, sTE = nTE * KE, sTO = nTO * KO, sVE = nVE * VE, sVO = nVO * VO;
  static constexpr int oPE = 0, oPO = oPE + 2 * sPE, oTE = oPO + 2 * sPO, oTO = oTE + 2 * sTE, oVE = oTO + 2 * sTO,
                       oVO = oVE + 2 * sVE, floats = oVO + 2 * sVO;
  // TMEM columns of a slot: A hi (even, odd) at 0, lo at cL, accumulators from cD; the volume product's at cVL, cV
  static constexpr int cL = KE + KO, cD = 2 * cL, cVL = VE + VO, cV = 2 * cVL;
  static_assert(cD + nPE + nPO <= 256 && cD + nTE + nTO <= 256 && cV + nVE + nVO <= 256, "TMEM columns of a slot");
};

// Shared memory of one warp (floats): two buffers of dofs rows, the element
// parameters, the faces' normals, the modes of
// two faces' rows (acoustic: of one, there are more rows), with kSpec the modes
// of the gravitational faces.
template <int N, class M, bool kSpec>
struct LSmem {
  using S = row::Shape<float, N>;
  static constexpr int rowsN = M::Q * M::EW;
  static constexpr int nQ = (rowsN * S::SB + 3) / 4 * 4, nT = ((M::fluid ? 1 : 2) * rowsN * S::Bf + 3) / 4 * 4;
  static constexpr int nD = kSpec ? row::SpecLevels<float, N, true>::values : 0;
  static constexpr int nP = M::EW * PAR, nN = M::fluid ? 0 : row::LocalSmem<float, N, kSpec>::nN;
  static constexpr int bufs = kSpec ? 1 : 2;
  static constexpr int oP = bufs * nQ, oN = oP + nP, oT = oN + nN, oD = oT + nT, warp = (oD + nD + 3) / 4 * 4;
  static constexpr int slots = 2, threads = 128 * slots;
  static constexpr int bytes = (LImg<N>::floats + 4 * slots * warp) * 4;
  static_assert(bytes + 256 <= 232448, "local tensor-core kernel exceeds the shared memory of one CTA");
};

// the dofs rows of a warp's nE elements into shared memory (row stride SB),
// asynchronously; acoustic: rows sigma_xx and v of each element
template <int N, class M>
__device__ __forceinline__ void rows_request(float* sQ, const float* Q, int nE, int lane) {
  using S = row::Shape<float, N>;
  constexpr int C = S::B / S::VW;
#pragma unroll
  for (int k = 0; k < (M::Q * M::EW * C + 31) / 32; ++k) {
    const int i = lane + 32 * k, r = i / C, c = (i - r * C) * S::VW;
    if (r >= M::Q * nE) continue;
    const int gr = M::fluid ? row::fluid_row(r) : r;
    if constexpr (S::VW == 4)
      tc::cp_async16(sQ + r * S::SB + c, Q + gr * S::B + c);
    else
      tc::cp_async4(sQ + r * S::SB + c, Q + gr * S::B + c);
  }
}
// ... and back; acoustic: the normal stress as sigma_xx, sigma_yy and sigma_zz
template <int N, class M>
__device__ __forceinline__ void rows_back(const float* sQ, float* Q, int nE, int lane) {
  using S = row::Shape<float, N>;
  if constexpr (M::fluid)
    row::fluid_rows_out<float, N>(sQ, Q, nE, lane);
  else
    row::rows_out_v<float, N, S::VW>(sQ, Q, nE, lane);
}

// kBuf: some elements of the launch have an LTS buffer (a coarser neighbour)
template <int N, class M, bool kBuf, bool kSpec>
__global__ void __launch_bounds__(LSmem<N, M, kSpec>::threads, 1)
    local_tc_kernel(StepArgs a, const __grid_constant__ Segs g) {
  using I_ = LImg<N>;
  using SM = LSmem<N, M, kSpec>;
  using S = row::Shape<float, N>;
  constexpr int B = I_::B, BF = I_::BF, B1 = I_::B1, kSlots = SM::slots, VW = S::VW;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  float* const sm = reinterpret_cast<float*>(smem_raw);
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t mbar[kSlots], s_img;
  __shared__ int s_abort[kSlots], s_next[kSlots][2];

  const int tid = threadIdx.x, slot = tid >> 7, t = tid & 127, w = t >> 5, lane = tid & 31;
  // the operand image into shared memory by the TMA engine, while the threads set up the rest
  if (tid == 0) {
    tc::mbar_init(&s_img, 1);
    tc::bulk_load_all(sm, a.tc_local, I_::floats * 4, &s_img);
  }
  if (tid < kSlots) {
    tc::mbar_init(&mbar[tid], 1);
    s_abort[tid] = 0;
  }
  if (tid < 32) tc::tmem_alloc<256 * kSlots>(&tmem_base);

  // this warp's part of tile tl: first virtual element, elements (may be 0), segment
  const int64_t ntiles = g.first[g.n];
  const int slots = (int)gridDim.x * kSlots, me = slot * (int)gridDim.x + (int)blockIdx.x;
  using Part = TilePart;
  auto part_of = [&](int64_t tl) { return tile_part<M::TE, M::EW>(g, tl, w); };
  float* const sW = sm + I_::floats + (slot * 4 + w) * SM::warp;
  float* const Qg = reinterpret_cast<float*>(a.Q);
  const tc::TileFeed feed{a.tiles, s_next[slot], slots, g.chunk, ntiles};
  int it = 0;
  int64_t tile = feed.first(me);
  if (t == 32) s_next[slot][1] = (int)feed.after(tile);
  Part p{0, 0, 0};
  // a part's dofs rows (buffer b) and element parameters
  auto request = [&](const Part& q, int b) {
    rows_request<N, M>(sW + b * SM::nQ, Qg + q.v0 * 9 * B, q.nE, lane);
    if (lane < 4 * q.nE)
      tc::cp_async16(sW + SM::oP + 4 * lane,
                     reinterpret_cast<const float*>(a.par) + elem_of(q.v0 + (lane >> 2), a.S) * PAR + 4 * (lane & 3));
  };
  if (tile < ntiles) {
    p = part_of(tile);
    request(p, 0);
  }
  tc::cp_async_commit();

  __syncthreads();  // (the image barrier is initialised)
  const bool img_ok = tc::mbar_wait(&s_img, 0, kWaitIters);
  tc::fence_async_smem();
  tc::fence_before();
  const bool all_ok = __syncthreads_and(img_ok);
  tc::fence_after();
  if (!all_ok) {
    // the image did not arrive within the bound: report, give the copies a
    // bounded chance to finish, free the columns and leave
    if (tid == 0) {
      atomicOr(a.err, ERR_TIMEOUT);
      tc::mbar_wait(&s_img, 0, kWaitIters);
    }
    tc::cp_async_wait<0>();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid < 32) tc::tmem_dealloc<256 * kSlots>(tmem_base);
    if (tid == 0) feed.leave();
    return;
  }

  const uint32_t tbase = tmem_base + (uint32_t)slot * 256u, trow = tbase + ((uint32_t)(32 * w) << 16);
  const uint32_t sB = tc::smem_u32(sm);
  tc::SlotMma mma{&mbar[slot], &s_abort[slot], a.err, slot, t, lane, 0};
  float* const sT = sW + SM::oT;
  const int j = lane / M::Q;
  // a row's modes (of the first LIM) into the A columns, even then odd ones
  auto put = [&](const float* x, auto ke, auto ko, auto lim, uint32_t lo) {
    constexpr int KE = decltype(ke)::value, KO = decltype(ko)::value, LIM = decltype(lim)::value;
    tc::put_row<KE / 8>(trow, trow + lo, [&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (k < count_par(LIM, 0)) return x[par_mode(0, k)]; else return 0.f;
    });
    tc::put_row<KO / 8>(trow + KE, trow + lo + KE, [&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (k < count_par(LIM, 1)) return x[par_mode(1, k)]; else return 0.f;
    });
  };

  for (int64_t next = s_next[slot][1]; tile < ntiles;) {
    // the tile after the next, asked for now and handed to the slot at the end
    const int64_t after = t == 32 ? feed.after(next) : 0;
    const Seg& sg = g.s[p.seg];
    float* const sQ = sW + (SM::bufs > 1 ? it & 1 : 0) * SM::nQ;
    tc::cp_async_wait<0>();  // this tile's rows and parameters
    __syncwarp();
    const bool valid = lane < M::Q * p.nE;
    row::RowStar<float> st;
    {
      const float* const par = sW + SM::oP + (valid ? j : 0) * PAR;
      if constexpr (M::fluid)
        st.setup_acoustic(lane, valid, par);
      else
        st.setup(lane, valid, par);
    }
    __syncwarp();
    Part pn{0, 0, 0};
    if (next < ntiles) {
      pn = part_of(next);
      if constexpr (SM::bufs > 1) request(pn, (it + 1) & 1);
    }
    if constexpr (!M::fluid) row::normals_request(a, sW + SM::oN, p.v0, p.nE, lane);
    tc::cp_async_commit();
    float* const rowp = sQ + (valid ? lane : 0) * S::SB;
    std::conditional_t<kSpec, row::SpecLevels<float, N, true>, row::NoLevels> lev = [&] {
      if constexpr (kSpec) {
        tc::cp_async_wait<0>();
        __syncwarp();  // the normals
        return row::SpecLevels<float, N, true>(a, valid, sT, sW + SM::oD, sW + SM::oN, p.v0, p.nE, lane);
      } else {
        return row::NoLevels{};
      }
    }();

    // ---- level 0 on the tensor cores: D^1 from D^0 = the dofs row
    float I[B];
    auto load_row = [&] {
#pragma unroll
      for (int c = 0; c < B / VW; ++c) {
        const row::Vec<float, VW> x = *reinterpret_cast<const row::Vec<float, VW>*>(rowp + c * VW);
#pragma unroll
        for (int k = 0; k < VW; ++k) I[c * VW + k] = x.x[k];
      }
    };
    load_row();
    put(I, std::integral_constant<int, I_::KE>{}, std::integral_constant<int, I_::KO>{},
        std::integral_constant<int, B>{}, I_::cL);
    mma.issue(0, [&] {
      tc::mma3_ts<I_::nPE, I_::KE>(tbase + I_::cD, tbase, tbase + I_::cL, sB + 4 * I_::oPE,
                                   sB + 4 * (I_::oPE + I_::sPE), false);
      tc::mma3_ts<I_::nPO, I_::KO>(tbase + I_::cD + I_::nPE, tbase + I_::KE, tbase + I_::cL + I_::KE,
                                   sB + 4 * I_::oPO, sB + 4 * (I_::oPO + I_::sPO), false);
    });
    lev(std::integral_constant<int, 0>{}, I);  // (while the product runs)
    mma.done();
    {
      float D1[B1];
      {
        constexpr int ME = I_::ME, MO = I_::MO;
        float ye[I_::nPE], yo[I_::nPO];
        tc::ld8s<I_::nPE / 8>(trow + I_::cD, ye);
        tc::ld8s<I_::nPO / 8>(trow + I_::cD + I_::nPE, yo);
        // (pairs of equal parity: their values lie side by side)
        sp::each<2>([&](auto pc) {
          constexpr int par = decltype(pc)::value, n = par ? MO : ME;
          float d[n];
          row::star_rows<n>(st, d, [&](auto bc, auto kc) {
            constexpr int b = decltype(bc)::value, k = decltype(kc)::value;
            if constexpr (b == 0) return par ? ye[2 * ME + k] : yo[2 * MO + k];
            else return par ? yo[(b - 1) * MO + k] : ye[(b - 1) * ME + k];
          });
          sp::each<n>([&](auto kc) { D1[par_mode(par, decltype(kc)::value)] = d[decltype(kc)::value]; });
        });
      }
      // ---- I = dt D^0 + dt^2/2 D^1 + ..., the other levels on this thread's registers
      load_row();
      const float c0 = seg_tcoef<float>(sg, 0), c1 = seg_tcoef<float>(sg, 1);
#pragma unroll
      for (int l = 0; l < B; ++l) I[l] *= c0;
#pragma unroll
      for (int m = 0; m < B1; ++m) I[m] = fmaf(c1, D1[m], I[m]);
      lev(std::integral_constant<int, 1>{}, D1);
      row::predict<float, N, 1>(D1, I, st, sg, lev);
    }
    // ---- modal face traces
    put(I, std::integral_constant<int, I_::KE>{}, std::integral_constant<int, I_::KO>{},
        std::integral_constant<int, B>{}, I_::cL);
    mma.issue(1, [&] {
      tc::mma3_ts<I_::nTE, I_::KE>(tbase + I_::cD, tbase, tbase + I_::cL, sB + 4 * I_::oTE,
                                   sB + 4 * (I_::oTE + I_::sTE), false);
      tc::mma3_ts<I_::nTO, I_::KO>(tbase + I_::cD + I_::nTE, tbase + I_::KE, tbase + I_::cL + I_::KE,
                                   sB + 4 * I_::oTO, sB + 4 * (I_::oTO + I_::sTO), false);
    });
    [[maybe_unused]] float nrm[3];  // (acoustic; requested while the product runs)
    if constexpr (M::fluid) row::fluid_normal(a, p.v0, p.nE, lane, nrm);
    mma.done();
    {
      float te[I_::nTE], to[I_::nTO];
      tc::ld8s<I_::nTE / 8>(trow + I_::cD, te);
      tc::ld8s<I_::nTO / 8>(trow + I_::cD + I_::nTE, to);
      // ---- the volume product runs while the traces leave
      put(I, std::integral_constant<int, I_::VE>{}, std::integral_constant<int, I_::VO>{},
          std::integral_constant<int, B1>{}, I_::cVL);
      mma.issue(2, [&] {
        tc::mma3_ts<I_::nVE, I_::VE>(tbase + I_::cV, tbase, tbase + I_::cVL, sB + 4 * I_::oVE,
                                     sB + 4 * (I_::oVE + I_::sVE), false);
        tc::mma3_ts<I_::nVO, I_::VO>(tbase + I_::cV + I_::nVE, tbase + I_::VE, tbase + I_::cVL + I_::VE,
                                     sB + 4 * I_::oVO, sB + 4 * (I_::oVO + I_::sVO), false);
      });
      tc::cp_async_wait<0>();  // the normals (and the next tile's rows, by now)
      float* const s0 = sT + (valid ? lane : 0) * BF;
      // mode r of face f from the even and odd sums
      auto mode = [&](auto fc, auto rc) {
        constexpr int f = decltype(fc)::value, r = decltype(rc)::value;
        constexpr int k = BF + fpar_index(r) + (f == 3 ? (fparity(r) ? I_::FO : I_::FE) : 0);
        if constexpr (f == 0) return te[r] + to[r];
        else if constexpr (f == 1) return te[r] - to[r];
        else if constexpr (fparity(r) == 0) return te[k];
        else return to[k];
      };
      // (acoustic: one face at a time through the buffer, else two)
      constexpr int NF = M::fluid ? 1 : 2;
      sp::each<4 / NF>([&](auto gc) {
        constexpr int f0 = decltype(gc)::value * NF;
        if (valid) {
          sp::each<NF>([&](auto kc) {
            sp::each<BF>([&](auto rc) {
              s0[decltype(kc)::value * SM::rowsN * BF + decltype(rc)::value] =
                  mode(std::integral_constant<int, f0 + decltype(kc)::value>{}, rc);
            });
          });
        }
        __syncwarp();
        if constexpr (M::fluid)
          row::fluid_face_out<float, N>(a, p.v0, p.nE, f0, sT, nrm, lane);
        else
          row::faces_out<float, N, kBuf>(a, sg, p.v0, p.nE, f0, sT, sW + SM::oN, lane);
        __syncwarp();
      });
    }
    mma.done();
    // ---- Q += volume term (face terms follow in the neighbour kernel)
    {
      constexpr int BE = I_::BE, BO = I_::BO;
      float ye[I_::nVE], yo[I_::nVO];
      tc::ld8s<I_::nVE / 8>(trow + I_::cV, ye);
      tc::ld8s<I_::nVO / 8>(trow + I_::cV + I_::nVE, yo);
      tc::fence_before();
      float x[B];
      sp::each<2>([&](auto pc) {
        constexpr int par = decltype(pc)::value, n = par ? BO : BE;
        float d[n];
        row::star_rows<n>(st, d, [&](auto bc, auto kc) {
          constexpr int b = decltype(bc)::value, k = decltype(kc)::value;
          if constexpr (b == 0) return par ? ye[2 * BE + k] : yo[2 * BO + k];
          else return par ? yo[(b - 1) * BO + k] : ye[(b - 1) * BE + k];
        });
        sp::each<n>([&](auto kc) { x[par_mode(par, decltype(kc)::value)] = d[decltype(kc)::value]; });
      });
      if (valid) {
#pragma unroll
        for (int c = 0; c < B / VW; ++c) {
          row::Vec<float, VW> q = *reinterpret_cast<const row::Vec<float, VW>*>(rowp + c * VW);
#pragma unroll
          for (int k = 0; k < VW; ++k) q.x[k] -= x[c * VW + k];
          *reinterpret_cast<row::Vec<float, VW>*>(rowp + c * VW) = q;
        }
      }
    }
    __syncwarp();
    rows_back<N, M>(sQ, Qg + p.v0 * 9 * B, p.nE, lane);
    if constexpr (kSpec) {
      lev.surface(sg);
      __syncwarp();  // the rows have left: the next tile's take their place
      if (next < ntiles) request(pn, 0);
      tc::cp_async_commit();
    }
    if (t == 32) s_next[slot][it & 1] = (int)after;
    tc::slot_bar(slot);
    if (*(volatile int*)&s_abort[slot]) break;
    tile = next;
    next = s_next[slot][it & 1];
    ++it;
    p = pn;
  }
  tc::cp_async_wait<0>();  // no copy into shared memory outlives the loop
  // after a timed-out wait, give this slot's products in flight a bounded chance to finish
  if (t == 0 && s_abort[slot]) tc::mbar_wait(&mbar[slot], mma.phase ^ 1u, kWaitIters);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (tid < 32) tc::tmem_dealloc<256 * kSlots>(tmem_base);
  if (tid == 0) feed.leave();
}

}  // namespace

// The launcher of degree N (the kernels of that degree's translation unit).
template <int N>
int launch_local_tc_deg(const StepArgs& a, const Segs& g, int n_sms, void* stream, bool buffers, bool acoustic,
                        bool grav) {
  using K = void (*)(StepArgs, Segs);
  static const K plain = local_tc_kernel<N, Elastic, false, false>, buf = local_tc_kernel<N, Elastic, true, false>,
                 fluid = local_tc_kernel<N, Acoustic, false, false>, spec = local_tc_kernel<N, Elastic, true, true>;
  constexpr int bytes_el = LSmem<N, Elastic, false>::bytes, bytes_fl = LSmem<N, Acoustic, false>::bytes,
                bytes_sp = LSmem<N, Elastic, true>::bytes;
  const int rc = configure_on_device((const void*)plain, [] {
    cudaError_t ce = cudaFuncSetAttribute((const void*)plain, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes_el);
    if (ce == cudaSuccess)
      ce = cudaFuncSetAttribute((const void*)buf, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes_el);
    if (ce == cudaSuccess)
      ce = cudaFuncSetAttribute((const void*)fluid, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes_fl);
    if (ce == cudaSuccess)
      ce = cudaFuncSetAttribute((const void*)spec, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes_sp);
    return ce;
  });
  if (rc) return rc;
  const int64_t ntiles = g.n ? g.first[g.n] : 0;
  if (ntiles <= 0) return 0;
  if (acoustic && (buffers || grav)) return (int)cudaErrorInvalidValue;
  // one CTA per SM at most; fewer tiles than slots: a CTA each, so that no SM holds two
  const int64_t units = (ntiles + g.chunk - 1) / g.chunk;
  const unsigned grid = (unsigned)(units < n_sms ? units : n_sms);
  StepArgs b = a;
  b.tiles = a.tiles + 2 * (grav ? TILES_SPECIAL : acoustic ? TILES_FLUID : buffers ? TILES_BUFFER : TILES_ELASTIC);
  if (grav)
    spec<<<grid, LSmem<N, Elastic, true>::threads, bytes_sp, (cudaStream_t)stream>>>(b, g);
  else if (acoustic)
    fluid<<<grid, LSmem<N, Acoustic, false>::threads, bytes_fl, (cudaStream_t)stream>>>(b, g);
  else
    (buffers ? buf : plain)<<<grid, LSmem<N, Elastic, false>::threads, bytes_el, (cudaStream_t)stream>>>(b, g);
  return (int)cudaGetLastError();
}

// Host-side image of the operands of degree N from the modal face projections
// rfc[f][l][r] and the stiffness lists (kt[a][m][l], kvol[a][m][l] with l < B1
// of that degree's basis), split into tf32 hi / lo, canonical K-major.
template <int N>
void pack_local_tc_deg(const double* kt, const double* kvol, const double* rfc, float* out) {
  using I_ = LImg<N>;
  constexpr int B = I_::B, B1 = I_::B1, BF = I_::BF;
  for (int i = 0; i < I_::floats; ++i) out[i] = 0.f;
  auto put = [&](int off, int size, int R, int n, int k, double x) {
    const float xf = (float)x, hi = tc::tf32_trunc(xf);
    const int o = tc::canon(n, k, R);
    out[off + o] = hi;
    out[off + size + o] = xf - hi;
  };
  // row m, input l of the directions X, Y = eta - X/2, Z = zeta - X/2 - Y (sparse_ops.inc)
  auto place = [&](int m, int l, double x, double eta, double zeta, int nE, int nO, int oE, int sE, int NEc, int oO,
                   int sO, int NOc) {
    const double y = eta - 0.5 * x, z = zeta - 0.5 * x - y;
    const bool odd_in = parity(l) == 1, odd_out = parity(m) == 1;
    const int k = par_index(l), r = par_index(m);
    if (odd_in == odd_out) {
      if (odd_in) {
        put(oO, sO, NOc, r, k, y);
        put(oO, sO, NOc, nO + r, k, z);
      } else {
        put(oE, sE, NEc, r, k, y);
        put(oE, sE, NEc, nE + r, k, z);
      }
    } else if (odd_in) {
      put(oO, sO, NOc, 2 * nO + r, k, x);
    } else {
      put(oE, sE, NEc, 2 * nE + r, k, x);
    }
  };
  auto at = [](const double* p, size_t rows, size_t cols, size_t ax, size_t r, size_t c) {
    return p[(ax * rows + r) * cols + c];
  };
  for (int m = 0; m < B1; ++m)
    for (int l = 0; l < B; ++l)
      place(m, l, at(kt, B, B, 0, m, l), at(kt, B, B, 1, m, l), at(kt, B, B, 2, m, l), I_::ME, I_::MO, I_::oPE,
            I_::sPE, I_::nPE, I_::oPO, I_::sPO, I_::nPO);
  for (int m = 0; m < B; ++m)
    for (int l = 0; l < B1; ++l)
      place(m, l, at(kvol, B, B1, 0, m, l), at(kvol, B, B1, 1, m, l), at(kvol, B, B1, 2, m, l), I_::BE, I_::BO,
            I_::oVE, I_::sVE, I_::nVE, I_::oVO, I_::sVO, I_::nVO);
  auto face = [&](int f, int l, int r) { return rfc[((size_t)f * B + l) * BF + r]; };
  for (int l = 0; l < B; ++l) {
    const bool odd = parity(l) == 1;
    const int k = par_index(l);
    for (int r = 0; r < BF; ++r) {
      put(odd ? I_::oTO : I_::oTE, odd ? I_::sTO : I_::sTE, odd ? I_::nTO : I_::nTE, r, k, face(0, l, r));
      if (fparity(r) == (odd ? 1 : 0))
        for (int f = 2; f < 4; ++f)
          put(odd ? I_::oTO : I_::oTE, odd ? I_::sTO : I_::sTE, odd ? I_::nTO : I_::nTE,
              BF + (f - 2) * (odd ? I_::FO : I_::FE) + fpar_index(r), k, face(f, l, r));
    }
  }
}

}  // namespace adg
