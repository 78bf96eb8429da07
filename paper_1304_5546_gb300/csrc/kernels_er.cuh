// FP32 stage kernel of large meshes at N = 3..5: element-local products on
// the 5th-generation tensor cores with one GEMM row per element ("element
// rows").
//
// Same result as dg_stage_tc_kernel (kernels_tc.cuh) up to rounding: deflated
// operands, three TF32 products X_hi Op_hi + X_hi Op_lo + X_lo Op_hi with FP32
// accumulation, one fused LSRK(5,4) stage or the right-hand side.
//
// Why.  That kernel is bound by the instructions of its operand rows: a row
// per (element, output field) carries the geometric factors, so every deflated
// value is scaled, split and stored three to four times (K = 60 columns for
// each of 3 rows at N = 5; 154 warp instructions an element, 0.67 of measured
// HBM).  Here a row is an element and its thread does everything that belongs
// to the element, as in the element-thread kernel, while the products' FMAs --
// what limits that one from N = 3 on -- are on the tensor cores:
//
//   operands (TMEM columns)                 accumulators
//   z      deflated Ez                 ->   Dr z, Ds z
//   A, B   rx Hy - ry Hx, sx Hy - sy Hx,
//          deflated                    ->   C = Dr A + Ds B
//   f0..2  flux scalar of each face    ->   P_f = LIFT_f f_f
//
// With f = Fscale/2 ([Ht] - [Ez]), [Ht] = ny [Hx] - nx [Hy], the upwind (alpha
// = 1) and the media flux both lift (-Z ny f, Z nx f, f), and the normal is
// constant on a face, so one scalar per face node is computed, stored and
// multiplied by LIFT, and the accumulator's reader combines
//   dHx/dt = l0 - ry Dr z - sy Ds z - sum_f Z ny_f P_f
//   dHy/dt = l1 + rx Dr z + sx Ds z + sum_f Z nx_f P_f
//   dEz/dt = l2 + C + P_0 + P_1 + P_2
// (l: the linear part's derivatives).  The vertex nodes' deflated values are
// zero and have no columns: 18 + 36 + 18 columns an element at N = 5 instead
// of 3 * 60.
//
// Block: 128 elements, a full MMA tile.  Warp roles: two groups of 4 element
// warps that take blocks in turn (operands into tensor memory; then the
// accumulators back, chain rule, update in place in the stage buffers), 7 flux
// warps in one group, at N = 3 two groups of 5 (traces element-major, so that a
// warp's loads coalesce, from the stage where the neighbour is in the block;
// flux scalars into an array in shared memory), one MMA warp, one memory warp
// (1D TMA bulk loads into rings of q and geometry stages and of residual
// stages, bulk stores from both).  Every wait is bounded; on expiry the CTA sets
// the status word, drains its copies (bounded), frees its TMEM and returns.
#pragma once

#include <type_traits>

#include "kernels_tc.cuh"

namespace dgw {

// weights of vertices 2 and 3 in the linear interpolant, at the nodes that
// are not vertices (an FMA's constant operand)
template <int N>
struct ErWeights {
  static constexpr int NI = Order<N>::Np - 3;
  float l2[NI], l3[NI];
};

template <int N, bool MEDIA_>
struct ErLayout {
  static constexpr int Np = Order<N>::Np, Nfp = Order<N>::Nfp, Nafp = Order<N>::Nafp;
  static constexpr int E = kErElems;  // the rows of an MMA tile, a thread each
  static constexpr int GEO = MEDIA_ ? kGeoMedia : kGeo;
  static constexpr int NI = Np - 3;
  static constexpr int KZ = er_kz(N), KAB = er_kab(N), KF = kErKf;  // operand columns
  static constexpr int NP8 = er_np8(N), NZ = 2 * NP8, NF = er_nf(N);  // MMA N extents
  static constexpr int XC = KZ + KAB + 3 * KF;  // columns of X_hi, and of X_lo
  // LIFT as one block-diagonal product (P_f NP8 columns apart) or face by face
  static constexpr bool LIFT_ONE = er_lift_one(N, MEDIA_);
  static constexpr int NL = er_nl(N), PS = LIFT_ONE ? NP8 : NF;  // P_f to P_(f+1)
  static constexpr int OFF_C = NZ + (LIFT_ONE ? NL : 3 * NF);
  static constexpr int ACC = OFF_C + NF;  // Dr z | Ds z, P_0..2, C
  // accumulators (AB) and operands (XB) double-buffered where the 512 columns
  // allow; a second accumulator lets a block's MMAs run beside the update of
  // the block before
  static constexpr int AB = 2 * ACC + 2 * XC <= 512 ? 2 : 1;
  static constexpr int XB = AB * ACC + 4 * XC <= 512 ? 2 : 1;
  static constexpr int OFF_X = AB * ACC;
  // Flux warps, in one group or in two that take blocks in turn (us a step,
  // one group of 7 / two of 5 warps: N = 3, K = 999,698 511 / 445, N = 4, K =
  // 665,858 477 / 531, N = 5, K = 999,698 983 / 1312: from N = 4 on two
  // groups' gathers in flight hold up the element warps' shared-memory
  // accesses; one group of 6, 8, 10 warps at N = 5 982, 988, 1063)
  static constexpr int ELEM_WARPS = 8;
  static constexpr int FLUX_GROUPS = N == 3 ? 2 : 1, FLUX_WARPS = N == 3 ? 5 : 7;
  // groups of four nodes per copy of the update's code (N = 3 all, 445 against
  // 461; N = 5 one, 983 against 1098 with all)
  static constexpr int UPDATE_UNROLL = N == 3 ? 3 : 1;
  static constexpr int FLUX_WARP0 = ELEM_WARPS, MMA_WARP = FLUX_WARP0 + FLUX_GROUPS * FLUX_WARPS,
                       IO_WARP = MMA_WARP + 1;
  static constexpr int THREADS = 32 * (IO_WARP + 1);
  // flux threads of a group: PER elements at a time, face node fastest
  static constexpr int PER = 32 * FLUX_WARPS / Nafp, FT = PER * Nafp;
  static constexpr int FES = Nafp | 1;  // flux row stride, odd: conflict-free rows
  static constexpr int QB = E * Np * 4, GB = E * GEO * 4, FB = E * FES * 4;
  static constexpr int QSTAGE = round_up(3 * QB + GB, 128), RSTAGE = 3 * QB;
  static constexpr int ZT = NZ * KZ * 4, CT = NF * KAB * 4;
  static constexpr int LT = er_lift_floats(N, MEDIA_) * 4, FTILE = NF * KF * 4;
  static constexpr int OB = 2 * (ZT + LT + CT);  // operator tiles, each hi then lo
  static constexpr int HEADER = 512;
  static constexpr int OFF_OP = HEADER, OFF_F = OFF_OP + OB;
  static constexpr int SMAX = 232448;
  static constexpr int off_q(int fbuf) { return round_up(OFF_F + fbuf * FB, 128); }
  static constexpr int bytes(int qs, int rs, int fbuf) {
    return off_q(fbuf) + qs * QSTAGE + rs * RSTAGE;
  }
  // stages of q and of the residual, flux arrays
  static constexpr int FIT = bytes(4, 4, 2) <= SMAX   ? 442
                             : bytes(4, 3, 2) <= SMAX ? 432
                             : bytes(3, 3, 2) <= SMAX ? 332
                             : bytes(3, 2, 2) <= SMAX ? 322
                             : bytes(3, 2, 1) <= SMAX ? 321
                                                      : 222;
  static constexpr int QS = FIT / 100, RS = FIT / 10 % 10, FBUF = FIT % 10;
  // The element and flux groups see every other block.  A parity wait tells a
  // phase only from its neighbours, so each group has to see every phase of a
  // barrier it waits on: block j's loads complete on barrier j % QBAR (RBAR),
  // whose count is even, whatever the number of stages.
  static constexpr int QBAR = QS % 2 ? 2 * QS : QS, RBAR = RS % 2 ? 2 * RS : RS;
  static constexpr int OFF_Q = off_q(FBUF), OFF_R = OFF_Q + QS * QSTAGE;
  static constexpr int SMEM_BYTES = bytes(QS, RS, FBUF);
  static_assert(SMEM_BYTES <= SMAX && SMEM_BYTES > 118784, "one CTA per SM, which owns the TMEM");
  static_assert(AB * ACC + XB * 2 * XC <= 512, "tensor memory");
  // an element group waits on mma_done of its own blocks and of the blocks XB
  // before them: with one accumulator it sees every phase only if XB is odd
  static_assert(AB == 2 || XB == 1, "every phase of mma_done seen by both element groups");
  static_assert(Np <= 32 && E == 128, "5-bit node table; element warps");
  static_assert(NZ % 16 == 0 && NF % 16 == 0 && NL % 16 == 0 && NZ <= 256 && Nfp <= KF, "UMMA shape");
  static_assert(QB % 128 == 0 && GB % 16 == 0 && OB % 128 == 0, "TMA chunks");
  static_assert(OB == er_tile_floats(N, MEDIA_) * 4, "operator tiles");
};

// Eight operand columns, hi and lo parts, into tensor memory.
__device__ __forceinline__ void er_emit8(uint32_t xh, uint32_t xl, const float* v) {
  float h[8], l[8];
#pragma unroll
  for (int i = 0; i < 8; i += 2) {
    const f32x2 p = f32x2_pack(v[i], v[i + 1]);
    const f32x2 hh = f32x2_tf32_trunc(p);
    f32x2_unpack(hh, h[i], h[i + 1]);
    f32x2_unpack(f32x2_sub(p, hh), l[i], l[i + 1]);
  }
  tmem_st8(xh, h);
  tmem_st8(xl, l);
}

// Two consecutive values of a row of Np floats in shared memory, from an even
// node on (one: the first alone)
template <int Np>
__device__ __forceinline__ f32x2 er_ld2(const float* p, bool one) {
  if constexpr (Np % 2 == 0) {
    return *reinterpret_cast<const f32x2*>(p);
  } else {
    return f32x2_pack(p[0], one ? 0.f : p[1]);
  }
}
template <int Np>
__device__ __forceinline__ void er_st2(float* p, f32x2 v, bool one) {
  if constexpr (Np % 2 == 0) {
    *reinterpret_cast<f32x2*>(p) = v;
  } else {
    float a, b;
    f32x2_unpack(v, a, b);
    p[0] = a;
    if (!one) p[1] = b;
  }
}

template <int N, int MODE, bool MEDIA>
__global__ void __launch_bounds__(ErLayout<N, MEDIA>::THREADS, 1)
    dg_stage_er_kernel(const __grid_constant__ StageArgs<float> p,
                       const __grid_constant__ ErWeights<N> w) {
  using L = ErLayout<N, MEDIA>;
  constexpr int Np = L::Np, Nfp = L::Nfp, Nafp = L::Nafp, E = L::E, NI = L::NI, GEO = L::GEO;
  constexpr int UPD = L::UPDATE_UNROLL;
  constexpr int QS = L::QS, RS = L::RS, QBAR = L::QBAR, RBAR = L::RBAR, XB = L::XB, AB = L::AB, FES = L::FES;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* full_q = reinterpret_cast<uint64_t*>(smem);           // [QBAR] q and geometry landed
  uint64_t* full_r = reinterpret_cast<uint64_t*>(smem + 64);      // [RBAR] residual landed (or free)
  uint64_t* out_ready = reinterpret_cast<uint64_t*>(smem + 128);  // [QS] outputs written
  uint64_t* mma_done = reinterpret_cast<uint64_t*>(smem + 160);   // [AB] accumulators ready
  uint64_t* acc_free = reinterpret_cast<uint64_t*>(smem + 176);   // [AB] accumulators read
  uint64_t* xfull = reinterpret_cast<uint64_t*>(smem + 192);      // [XB] operands written
  uint64_t* fs_full = reinterpret_cast<uint64_t*>(smem + 208);    // [2] block j & 1: fluxes written
  uint64_t* fs_free = reinterpret_cast<uint64_t*>(smem + 224);    // [2] fluxes read
  uint64_t* op_bar = reinterpret_cast<uint64_t*>(smem + 240);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + 248);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + 252);
  float* Fs = reinterpret_cast<float*>(smem + L::OFF_F);  // [FBUF][E][FES]

  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int K = static_cast<int>(p.K);
  const int nblk = (K + E - 1) / E, G = gridDim.x, first = blockIdx.x;
  const int niter = first < nblk ? (nblk - 1 - first) / G + 1 : 0;
  const int64_t fs = p.fstride;
  auto q_stage = [&](int j) { return reinterpret_cast<float*>(smem + L::OFF_Q + (j % QS) * L::QSTAGE); };
  auto r_stage = [&](int j) { return reinterpret_cast<float*>(smem + L::OFF_R + (j % RS) * L::RSTAGE); };
  auto block_at = [&](int j, int& k0, int& n) {
    k0 = (first + j * G) * E;
    n = (K - k0) < E ? (K - k0) : E;
  };

  if (t == 0) {
    for (int s = 0; s < QBAR; ++s) mbar_init(&full_q[s], 1);
    for (int s = 0; s < RBAR; ++s) mbar_init(&full_r[s], 1);
    for (int s = 0; s < QS; ++s) mbar_init(&out_ready[s], E);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&mma_done[b], 1);
      mbar_init(&acc_free[b], E);
      mbar_init(&xfull[b], E);
      mbar_init(&fs_full[b], L::FT);
      mbar_init(&fs_free[b], E);
    }
    mbar_init(op_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(tmem_slot, 512);
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (warp == L::IO_WARP && lane == 0) {  // the operator tiles, which no kernel writes
    mbar_expect_tx(op_bar, L::OB);
    tma_load_1d(smem + L::OFF_OP, p.tc_op, L::OB, op_bar);
  }
  chain_wait();
  chain_trigger();

  auto fail = [&]() {
    *abort_flag = 1;
    atomicOr(p.status, kStatusTimeout);
  };

  if (warp == L::IO_WARP) {
    // ======================= memory warp: several lanes issue a block's copies;
    // lane 0 alone arms the mbarriers; every lane waits on its own bulk groups
    auto issue_q = [&](int j) {
      int k0, n;
      block_at(j, k0, n);
      const uint32_t qb = round16(static_cast<uint32_t>(n * Np * 4));
      const uint32_t gb = round16(static_cast<uint32_t>(n * GEO * 4));
      unsigned char* st = reinterpret_cast<unsigned char*>(q_stage(j));
      uint64_t* bar = &full_q[j % QBAR];
      if (lane == 0) mbar_expect_tx(bar, 3 * qb + gb);
      __syncwarp();
      if (lane < 3)
        tma_load_1d(st + lane * L::QB, p.qin + lane * fs + static_cast<int64_t>(k0) * Np, qb, bar);
      else if (lane == 3)
        tma_load_1d(st + 3 * L::QB, p.geo + static_cast<int64_t>(k0) * GEO, gb, bar);
    };
    auto issue_r = [&](int j) {
      if (MODE == kModeRhs) return;
      int k0, n;
      block_at(j, k0, n);
      uint64_t* bar = &full_r[j % RBAR];
      if (MODE == kModeFirstStage) {  // nothing to read: the stage is free
        if (lane == 0) mbar_arrive(bar);
        return;
      }
      const uint32_t qb = round16(static_cast<uint32_t>(n * Np * 4));
      unsigned char* st = reinterpret_cast<unsigned char*>(r_stage(j));
      if (lane == 0) mbar_expect_tx(bar, 3 * qb);
      __syncwarp();
      if (lane < 3)
        tma_load_1d(st + lane * L::QB, p.res + lane * fs + static_cast<int64_t>(k0) * Np, qb, bar);
    };
    int issued = 0;  // blocks whose q loads were issued
    for (int j = 0; j < niter && j < (QS > RS ? QS : RS); ++j) {
      if (j < QS) {
        issue_q(j);
        ++issued;
      }
      if (j < RS) issue_r(j);
    }
    bool ok = true;
    int j = 0;
    for (; j < niter; ++j) {
      ok = __all_sync(0xffffffffu,
                      mbar_wait_or_abort(&out_ready[j % QS], static_cast<uint32_t>((j / QS) & 1),
                                         abort_flag));
      if (!ok) break;
      int k0, nv;
      block_at(j, k0, nv);
      float* sq = q_stage(j);
      float* sr = r_stage(j);
      const int se = p.psrc_k - k0;
      if (static_cast<unsigned>(se) < static_cast<unsigned>(nv)) {  // the operator's point source
        float* y = sq + 2 * E * Np + se * Np;
        float* r = sr + 2 * E * Np + se * Np;
        if (nv != E) {
          const int64_t g = 2 * fs + static_cast<int64_t>(p.psrc_k) * Np;
          y = (MODE == kModeRhs ? p.rhs : p.qout) + g;
          r = p.res + g;
        }
        point_source_call<Np, MODE>(y, r, p.psrc_w, p.psrc_amp, p.b, lane, 32);
        fence_proxy_async();
      }
      __syncwarp();
      if (nv == E && lane < 6) {
        const int64_t g = static_cast<int64_t>(k0) * Np;
        if (MODE == kModeRhs) {
          if (lane < 3) tma_store_1d(p.rhs + lane * fs + g, sq + lane * E * Np, L::QB);
        } else if (lane < 3) {
          tma_store_1d(p.qout + lane * fs + g, sq + lane * E * Np, L::QB);
        } else {
          tma_store_1d(p.res + (lane - 3) * fs + g, sr + (lane - 3) * E * Np, L::QB);
        }
      }
      bulk_commit();
      if (j + QS < niter || j + RS < niter) {
        bulk_wait_read_all();
        __syncwarp();
        fence_proxy_async();
        if (j + QS < niter) {
          issue_q(j + QS);
          ++issued;
        }
        if (j + RS < niter) issue_r(j + RS);
      }
    }
    if (!ok && lane == 0) {
      fail();
      // let this CTA's loads in flight land (each wait bounded)
      for (int i = j; i < issued; ++i)
        mbar_wait_bounded(&full_q[i % QBAR], static_cast<uint32_t>((i / QBAR) & 1), kWaitLimitNs);
      for (int i = j; i < niter && i < j + RS; ++i)
        if (MODE == kModeStage)
          mbar_wait_bounded(&full_r[i % RBAR], static_cast<uint32_t>((i / RBAR) & 1), kWaitLimitNs);
    }
    bulk_wait_read_all();  // the end of the kernel completes the writes
  } else if (warp == L::MMA_WARP) {
    // ======================= MMA warp (lane 0)
    if (lane == 0) {
      bool ok = mbar_wait_or_abort(op_bar, 0, abort_flag);
      const uint32_t op = smem_u32(smem + L::OFF_OP);
      constexpr uint32_t IDZ = umma_idesc_tf32(128, L::NZ), IDF = umma_idesc_tf32(128, L::NF),
                         IDL = umma_idesc_tf32(128, L::NL);
      // X_hi Op_hi, X_hi Op_lo, X_lo Op_hi over K columns from column x of the
      // operands, into the accumulator columns from d
      auto product = [&](uint32_t d, uint32_t xh, uint32_t tile, int k, uint32_t idesc,
                         uint32_t tile_bytes) {
        const uint32_t sbo = static_cast<uint32_t>(k / 4) * 128;
#pragma unroll
        for (int pr = 0; pr < 3; ++pr) {
          const uint32_t x = xh + (pr == 2 ? L::XC : 0), b = tile + (pr == 1 ? tile_bytes : 0);
#pragma unroll
          for (int ks = 0; ks < k / 8; ++ks)
            umma_tf32_ta(d, x + 8 * ks, umma_desc(b + ks * 256, 128, sbo), idesc,
                         pr > 0 || ks > 0 ? 1u : 0u);
        }
      };
      int pending = -1;
      for (int j = 0; ok && j < niter; ++j) {
        const int xb = j % XB, ab = j % AB;
        ok = mbar_wait_or_abort(&xfull[xb], static_cast<uint32_t>((j / XB) & 1), abort_flag);
        if (ok && j >= AB)
          ok = mbar_wait_or_abort(&acc_free[ab], static_cast<uint32_t>(((j - AB) / AB) & 1),
                                  abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem + static_cast<uint32_t>(ab * L::ACC);
        const uint32_t x = tmem + static_cast<uint32_t>(L::OFF_X + xb * 2 * L::XC);
        const uint32_t xf = x + L::KZ + L::KAB, lift = op + 2 * L::ZT;
        product(d, x, op, L::KZ, IDZ, L::ZT);
        product(d + L::OFF_C, x + L::KZ, lift + 2 * L::LT, L::KAB, IDF, L::CT);
        if constexpr (L::LIFT_ONE) {
          product(d + L::NZ, xf, lift, 3 * L::KF, IDL, L::LT);
        } else {
#pragma unroll
          for (int f = 0; f < 3; ++f)
            product(d + L::NZ + f * L::PS, xf + f * L::KF, lift + 2 * f * L::FTILE, L::KF, IDF,
                    L::FTILE);
        }
        umma_commit(&mma_done[ab]);
        pending = j;
      }
      if (!ok) {
        fail();
        if (pending >= 0)
          mbar_wait_bounded(&mma_done[pending % AB], static_cast<uint32_t>((pending / AB) & 1),
                            kWaitLimitNs);
      }
    }
  } else if (warp >= L::FLUX_WARP0) {
    // ======================= flux warps, in FLUX_GROUPS groups that take blocks
    // in turn (one from N = 4 on: every block);
    // thread = face node jn of elements e0, e0 + PER, ... (U of them).  A
    // block's traces are asked for before its stage has landed, from face
    // codes that came straight from global memory a block of the group
    // earlier: half of the traces come from DRAM, for blocks that other CTAs
    // are about to load, and take 4000 cycles under load.  (One group, traces
    // asked for once the stage had landed: 7100 of 8500 cycles a block at N =
    // 5, the slowest role.)
    const int group = (warp - L::FLUX_WARP0) / L::FLUX_WARPS;
    const int ft = t - 32 * (L::FLUX_WARP0 + group * L::FLUX_WARPS);
    if (ft < L::FT) {
      constexpr int PER = L::PER, U = (E + PER - 1) / PER, FBUF = L::FBUF;
      const int e0 = ft / Nafp, jn = ft - e0 * Nafp, f = jn / Nfp, jj = jn - f * Nfp;
      const int nm = face_node_dev(N, f, jj);
      // the neighbour's node for each value of a face code's low bits, 5 bits each
      uint32_t nodes = 0;
      for (int c = 0; c < 6; ++c)
        nodes |= static_cast<uint32_t>(face_node_dev(N, c >> 1, (c & 1) ? N - jj : jj)) << (5 * c);
      const float* q0 = p.qin;
      const float* q1 = p.qin + fs;
      const float* q2 = p.qin + 2 * fs;
      int32_t code[U];  // -1: a wall, or no element
      auto fetch_codes = [&](int j) {
        const int k0 = (first + j * G) * E;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = e0 + u * PER;
          code[u] = -1;
          if (j < niter && (U * PER == E || e < E) && k0 + e < K)
            code[u] = __ldg(p.conn + static_cast<int64_t>(k0 + e) * 3 + f);
        }
      };
      fetch_codes(group);
      bool ok = true;
      for (int j = group; ok && j < niter; j += L::FLUX_GROUPS) {
        int k0, nv;
        block_at(j, k0, nv);
        // traces; for a neighbour in the block itself (two faces of three on a
        // mesh in row order) its place in the stage
        float tx[U], ty[U], tz[U];
        uint32_t open = 0, local = 0;  // bits: not a wall; in the block
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int32_t c = code[u];
          bool inner = c >= 0;
#ifdef DGW_DEVICE_CHECKS
          if (!nbr_code_ok(c, fs, Np)) {
            atomicOr(p.status, kStatusIndex);
            inner = false;
          }
#endif
          const int node = static_cast<int>((nodes >> (5 * (c & 7))) & 31u);
          const int le = (c >> 3) - k0;
          const bool in_block = inner && static_cast<unsigned>(le) < static_cast<unsigned>(nv);
          open |= inner ? 1u << u : 0u;
          local |= in_block ? 1u << u : 0u;
          tx[u] = __int_as_float(in_block ? le * Np + node : 0);
          ty[u] = tz[u] = 0.f;
          if (inner && !in_block) {
            const int g = (c >> 3) * Np + node;
            tx[u] = q0[g];
            ty[u] = q1[g];
            tz[u] = q2[g];
          }
        }
        fetch_codes(j + L::FLUX_GROUPS);
        ok = mbar_wait_or_abort(&full_q[j % QBAR], static_cast<uint32_t>((j / QBAR) & 1), abort_flag);
        if (!ok) break;
        const float* sq = q_stage(j);
        const float* sg = sq + 3 * E * Np;
        // neighbours in the block: no one updates the stage before its fluxes
        // are read
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (local >> u & 1u) {
            const float* n = sq + __float_as_int(tx[u]);
            tx[u] = n[0];
            ty[u] = n[E * Np];
            tz[u] = n[2 * E * Np];
          }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          // past the last element: some value of row 0, which no one reads
          const int e = U * PER == E || e0 + u * PER < E ? e0 + u * PER : 0;
          const float* q = sq + e * Np + nm;
          const float* gf = sg + e * GEO + 4 + (MEDIA ? 4 : 3) * f;
          const float hx = q[0], hy = q[E * Np], ez = q[2 * E * Np];
          const bool wall = !(open >> u & 1u);  // PEC wall: H+ = H-, Ez+ = -Ez-
          const float dHx = wall ? 0.f : hx - tx[u];
          const float dHy = wall ? 0.f : hy - ty[u];
          const float dEz = wall ? 2.f * ez : ez - tz[u];
          const float Ht = __fmaf_rn(gf[1], dHx, -__fmul_rn(gf[0], dHy));
          tx[u] = MEDIA ? __fmaf_rn(gf[2], Ht, -__fmul_rn(gf[3], dEz))
                        : __fmul_rn(gf[2], __fadd_rn(Ht, -dEz));
        }
        if (j >= FBUF)  // the element warps have read this array's last fluxes
          ok = mbar_wait_or_abort(&fs_free[(j - FBUF) & 1],
                                  static_cast<uint32_t>(((j - FBUF) >> 1) & 1), abort_flag);
        if (!ok) break;
        float* Fb = Fs + (j % FBUF) * (L::FB / 4) + jn;
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (U * PER == E || e0 + u * PER < E) Fb[(e0 + u * PER) * FES] = tx[u];
        mbar_arrive(&fs_full[j & 1]);
      }
      if (!ok) fail();
    }
  } else {
    // ======================= element warps: thread = element of the block
    const int group = warp >> 2, quarter = warp & 3;
    const int e = 32 * quarter + lane;
    const uint32_t lane_base = static_cast<uint32_t>(32 * quarter) << 16;
    bool ok = true;
    for (int j = group; j < niter; j += 2) {
      const int xb = j % XB, ab = j % AB;
      ok = mbar_wait_or_abort(&full_q[j % QBAR], static_cast<uint32_t>((j / QBAR) & 1), abort_flag);
      // the MMAs that last read this operand buffer are done
      if (ok && j >= XB)
        ok = mbar_wait_or_abort(&mma_done[(j - XB) % AB],
                                static_cast<uint32_t>(((j - XB) / AB) & 1), abort_flag);
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      tc_fence_after();
      int k0, nv;
      block_at(j, k0, nv);
      float* sq = q_stage(j);
      const float* ge = sq + 3 * E * Np + e * GEO;
      float* q0 = sq + e * Np;
      const uint32_t xh = tmem + lane_base + static_cast<uint32_t>(L::OFF_X + xb * 2 * L::XC);
      const float x1 = q0[0], x2 = q0[N], x3 = q0[Np - 1];
      const float y1 = q0[E * Np], y2 = q0[E * Np + N], y3 = q0[E * Np + Np - 1];
      const float z1 = q0[2 * E * Np], z2 = q0[2 * E * Np + N], z3 = q0[2 * E * Np + Np - 1];
      const float rx = ge[0], ry = ge[1], sx = ge[2], sy = ge[3];
      {  // ---- operands
        // the field at an interior node minus its linear interpolant
        auto deflated = [&](int field, int c, float v1, float d2, float d3) {
          const int n = c < N - 1 ? c + 1 : c + 2;
          return fmaf(d3, w.l3[c], fmaf(d2, w.l2[c], q0[field * E * Np + n] - v1));
        };
        const float dz2 = z1 - z2, dz3 = z1 - z3;
#pragma unroll
        for (int c0 = 0; c0 < L::KZ; c0 += 8) {
          float v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = c0 + i < NI ? deflated(2, c0 + i < NI ? c0 + i : 0, z1, dz2, dz3) : 0.f;
          __syncwarp();
          er_emit8(xh + c0, xh + L::XC + c0, v);
        }
        const float dx2 = x1 - x2, dx3 = x1 - x3, dy2 = y1 - y2, dy3 = y1 - y3;
#pragma unroll
        for (int c0 = 0; c0 < L::KAB; c0 += 8) {  // A then B of four nodes
          float v[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = c0 / 2 + i;
            if (c < NI) {
              const float hx = deflated(0, c, x1, dx2, dx3), hy = deflated(1, c, y1, dy2, dy3);
              v[i] = fmaf(rx, hy, -ry * hx);
              v[4 + i] = fmaf(sx, hy, -sy * hx);
            } else {
              v[i] = v[4 + i] = 0.f;
            }
          }
          __syncwarp();
          er_emit8(xh + L::KZ + c0, xh + L::XC + L::KZ + c0, v);
        }
      }
      ok = mbar_wait_or_abort(&fs_full[j & 1], static_cast<uint32_t>((j >> 1) & 1), abort_flag);
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      {
        const float* fr = Fs + (j % L::FBUF) * (L::FB / 4) + e * FES;
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          float v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = i < Nfp ? fr[f * Nfp + (i < Nfp ? i : 0)] : 0.f;
          __syncwarp();
          const uint32_t c = L::KZ + L::KAB + f * L::KF;
          er_emit8(xh + c, xh + L::XC + c, v);
        }
      }
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(&xfull[xb]);
      mbar_arrive(&fs_free[j & 1]);

      // ---- accumulators back, chain rule, update
      const float l0 = -0.5f * (ry * (z2 - z1) + sy * (z3 - z1));
      const float l1 = 0.5f * (rx * (z2 - z1) + sx * (z3 - z1));
      const float l2 = 0.5f * (rx * (y2 - y1) - ry * (x2 - x1) + sx * (y3 - y1) - sy * (x3 - x1));
      const float zm = MEDIA ? ge[16] : 1.f, sH = MEDIA ? ge[17] : 1.f, sE = MEDIA ? ge[18] : 1.f;
      constexpr int FG = MEDIA ? 4 : 3;
      float kx[3], ky[3];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        kx[f] = MEDIA ? zm * ge[4 + FG * f] : ge[4 + FG * f];
        ky[f] = MEDIA ? -zm * ge[5 + FG * f] : -ge[5 + FG * f];
      }
      ok = mbar_wait_or_abort(&mma_done[ab], static_cast<uint32_t>((j / AB) & 1), abort_flag);
      if (ok && MODE != kModeRhs)
        ok = mbar_wait_or_abort(&full_r[j % RBAR], static_cast<uint32_t>((j / RBAR) & 1), abort_flag);
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      tc_fence_after();
      float* r0 = r_stage(j) + e * Np;
      const uint32_t acc = tmem + lane_base + static_cast<uint32_t>(ab * L::ACC);
      const bool whole = nv == E, mine = e < nv;
      const int64_t g0 = static_cast<int64_t>(k0 + e) * Np;  // ragged last block: global memory
      // four nodes at a time: their accumulators, values and residuals are all
      // asked for before the first is used.  One copy of the code for all
      // whole groups of four: unrolled, the roles' instructions overran the
      // instruction cache.
      auto update = [&](int n0, auto count) {
        constexpr int CNT = decltype(count)::value;  // nodes of the group
        float zr[4], zs[4], pf[3][4], c[4];
        __syncwarp();
        tmem_ld4(acc + n0, zr);
        tmem_ld4(acc + L::NP8 + n0, zs);
#pragma unroll
        for (int f = 0; f < 3; ++f) tmem_ld4(acc + L::NZ + f * L::PS + n0, pf[f]);
        tmem_ld4(acc + L::OFF_C + n0, c);
        f32x2 qv[3][2], rv[3][2];
        if (MODE != kModeRhs) {
#pragma unroll
          for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int i = 0; i < CNT; i += 2) {
              qv[f][i / 2] = er_ld2<Np>(q0 + f * E * Np + n0 + i, CNT - i < 2);
              if (MODE == kModeStage)
                rv[f][i / 2] = er_ld2<Np>(r0 + f * E * Np + n0 + i, CNT - i < 2);
            }
        }
        tmem_ld_wait();
        if (n0 + CNT == Np) {  // the last columns are read
          tc_fence_before();
          mbar_arrive(&acc_free[ab]);
        }
#pragma unroll
        for (int i = 0; i < CNT; i += 2) {
          const f32x2 r2 = f32x2_pack(zr[i], zr[i + 1]), s2 = f32x2_pack(zs[i], zs[i + 1]);
          f32x2 rhs[3] = {f32x2_fma(f32x2_dup(-sy), s2, f32x2_fma(f32x2_dup(-ry), r2, f32x2_dup(l0))),
                          f32x2_fma(f32x2_dup(sx), s2, f32x2_fma(f32x2_dup(rx), r2, f32x2_dup(l1))),
                          f32x2_add(f32x2_pack(c[i], c[i + 1]), f32x2_dup(l2))};
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            const f32x2 p2 = f32x2_pack(pf[f][i], pf[f][i + 1]);
            rhs[0] = f32x2_fma(f32x2_dup(ky[f]), p2, rhs[0]);
            rhs[1] = f32x2_fma(f32x2_dup(kx[f]), p2, rhs[1]);
            rhs[2] = f32x2_add(p2, rhs[2]);
          }
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            const float sc = f < 2 ? sH : sE;
            f32x2 qn, rn;
            if (MODE == kModeRhs) {
              qn = MEDIA ? f32x2_mul(f32x2_dup(sc), rhs[f]) : rhs[f];
              rn = qn;
            } else {
              rn = f32x2_mul(f32x2_dup(MEDIA ? p.dt * sc : p.dt), rhs[f]);
              if (MODE == kModeStage) rn = f32x2_fma(f32x2_dup(p.a), rv[f][i / 2], rn);
              qn = f32x2_fma(f32x2_dup(p.b), rn, qv[f][i / 2]);
            }
            if (whole) {
              er_st2<Np>(q0 + f * E * Np + n0 + i, qn, CNT - i < 2);
              if (MODE != kModeRhs) er_st2<Np>(r0 + f * E * Np + n0 + i, rn, CNT - i < 2);
            } else if (mine) {
              float qa, qb, ra, rb;
              f32x2_unpack(qn, qa, qb);
              f32x2_unpack(rn, ra, rb);
              float* dq = (MODE == kModeRhs ? p.rhs : p.qout) + f * fs + g0 + n0 + i;
              float* dr = p.res + f * fs + g0 + n0 + i;
              dq[0] = qa;
              if (i + 1 < CNT) dq[1] = qb;
              if (MODE != kModeRhs) {
                dr[0] = ra;
                if (i + 1 < CNT) dr[1] = rb;
              }
            }
          }
        }
      };
#pragma unroll UPD
      for (int n0 = 0; n0 + 4 <= Np; n0 += 4) update(n0, std::integral_constant<int, 4>());
      if constexpr (Np % 4 != 0) update(Np / 4 * 4, std::integral_constant<int, Np % 4>());
      fence_proxy_async();
      mbar_arrive(&out_ready[j % QS]);
    }
    if (!ok) fail();
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

template <int N, int MODE, bool MEDIA>
cudaError_t launch_er_mode(const StageArgs<float>& args, const ErWeights<N>& w, int num_sms,
                           cudaStream_t stream) {
  using L = ErLayout<N, MEDIA>;
  static std::atomic<uint64_t> configured{0};
  cudaError_t err = configure_once_per_device(configured, [] {
    return cudaFuncSetAttribute(dg_stage_er_kernel<N, MODE, MEDIA>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM_BYTES);
  });
  if (err != cudaSuccess) return err;
  const int64_t nblk = (args.K + L::E - 1) / L::E;
  const int64_t grid = nblk < num_sms ? nblk : num_sms;  // one CTA per SM
  return launch_chained(dg_stage_er_kernel<N, MODE, MEDIA>, static_cast<unsigned>(grid),
                        L::THREADS, L::SMEM_BYTES, stream, args, w);
}

template <int N, bool MEDIA>
cudaError_t launch_er_modes(const StageArgs<float>& args, const ErWeights<N>& w, int mode,
                            int num_sms, cudaStream_t stream) {
  if (mode == kModeRhs) return launch_er_mode<N, kModeRhs, MEDIA>(args, w, num_sms, stream);
  if (mode == kModeFirstStage)
    return launch_er_mode<N, kModeFirstStage, MEDIA>(args, w, num_sms, stream);
  return launch_er_mode<N, kModeStage, MEDIA>(args, w, num_sms, stream);
}

// Definition of the launcher declared in launch.h; explicitly instantiated
// per order in kernels_er_N*.cu.
template <int N>
cudaError_t launch_stage_er(const StageArgs<float>& args, const float* weights, bool media,
                            int mode, int num_sms, cudaStream_t stream) {
  ErWeights<N> w;
  for (int c = 0; c < ErWeights<N>::NI; ++c) {
    const int n = c < N - 1 ? c + 1 : c + 2;
    w.l2[c] = weights[n];
    w.l3[c] = weights[Order<N>::Np + n];
  }
  return media ? launch_er_modes<N, true>(args, w, mode, num_sms, stream)
               : launch_er_modes<N, false>(args, w, mode, num_sms, stream);
}

}  // namespace dgw
