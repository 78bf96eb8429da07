// FP64 stage kernel: the same fused stage as dg_stage_kernel (kernels.cuh) --
// right-hand side of Eq. dg-strong-explicit (volume derivative by Dr/Ds and
// the chain rule of Eq. dg-diff-local-to-global, upwind flux of Eq.
// max2d-numflux, LIFT of Eq. dg-lift) and one LSRK(5,4) update -- for FP64
// fields.
//
// What bounds it.  A GB300 SM retires 1.6 to 2 FP64 operations a clock (a
// warp instruction holds the one FP64 pipe for 16 to 20 clocks, whatever its
// active lanes; 70 clocks latency) beside 128 integer ones, so the time of an
// FP64 stage is its count of FP64 instructions: 200 a node at N = 5 as plain
// arithmetic, of which 138 are the element-local products.  Here those are
// exact integer arithmetic instead, and the flux is one scalar:
//
// * Products in fixed point.  The operand vectors of an element (deflated
//   Ez; A = rx Hy - ry Hx and B = sx Hy - sy Hx, deflated; the face fluxes)
//   are scaled by a power of two taken from the vector's largest entry and
//   taken as 84-bit integers hi 2^56 + mid 2^28 + lo (28-bit signed limbs),
//   and so, on the host, are the rows of Dr, Ds and LIFT.  An entry keeps its
//   53 bits down to 2^-31 of its vector's (its row's) largest.  A term is six
//   32 x 32 -> 64 bit multiply-adds into the sums of hi hi, of hi mid + mid hi
//   and of hi lo + mid mid + lo hi, which are exact (operand limbs below 2^28,
//   table limbs at most 2^27, at most 66 terms); what is left out is 2^-82 of
//   the largest product.  One final rounding replaces the roundings of up to
//   60 FP64 multiply-adds, and a component that only small entries reach is
//   as precise as they are: rows of Dr at N = 3, 5, 7 times vectors with
//   entries over nine decades, largest relative error of a component, FMAs /
//   two limbs (56 bits) / three: 2.6e-14 / 1.3e-8 / 1.1e-16 (over twelve, where
//   entries lose bits, 1.7e-14 / 1.2e-5 / 2.9e-14).  With two limbs an element
//   beside one 1e8 times larger, on axis-aligned faces, had components off by
//   1e7 times 2^-53 of their own terms' sizes (now 32 at most).  They are
//   faster: GB300, us a step, two / three limbs: N = 1, K = 180,000 302 / 320; 2,
//   80,000 324 / 354; 3, 45,000 305 / 337; 4, 45,000 397 / 439; 5, 101,250 1270 /
//   1453; 6, 20,000 363 / 472; 7, 20,000 534 / 695; N = 4, K = 128 32.5 / 37.4.
// * An operand vector that fixed point cannot hold -- largest entry
//   infinite, NaN, or outside 2^-890 .. 2^870 -- keeps its FP64 values in the
//   same slots, and its element takes the products in FP64.
// * Flux.  With f = Fscale/2 ([Ht] - [Ez]), [Ht] = ny [Hx] - nx [Hy], the
//   upwind (alpha = 1) and the media flux both lift (-Z ny f, Z nx f, f), Z =
//   1 in a uniform medium, and the normal is constant on a face: LIFT is
//   applied to f alone, face by face, and the three faces' results combined
//   per row (Nafp products a node instead of 3 Nafp).  alpha != 1 has a
//   second scalar, Fscale/2 (alpha [Ht] - [Ez]), for the H rows.
//
// Measured: see the table at f64_max_elems (launch.h).
//
// Work decomposition.  A CTA walks blocks of E consecutive elements, one
// thread per (element, node); E is a run-time number (f64_block_elems).  A
// block's q, residual, geometry and face codes come in by 8- and 4-byte
// cp.async copies (no alignment demand on E) one block ahead, into a ring of
// two stage buffers; its neighbour traces are gathered into registers as the
// block before it starts its products.  Per block, between barriers:
//   0  differences of the vertex values per element and field
//   1  deflated operands of the own node, flux of the own face nodes, and
//      the largest entry of every operand vector (shared-memory atomics)
//   2  fixed-point operands into shared memory
//   3  products, chain rule, update, stores.
#pragma once

#include <atomic>

#include "kernels.cuh"

namespace dgw {

// Resident CTAs the register allocation aims at, and product columns per
// unrolled step.  More CTAs let one's products run beside another's FP64
// phases, until the registers spill (us a step on the meshes of
// f64_max_elems' table, CTAs aimed at: N = 1 2 / 3 / 4 / 5 377 / 332 / 320 /
// 337, N = 2 2 / 4 / 5 / 6 405 / 405 / 358 / 354, N = 3 2 / 3 / 4 / 5 432 / 379 /
// 337 / 348, N = 5 1713 / 1664 / 1510 / 1651, N = 7 720 / 760 / 717 / 726; three
// / four / six columns a step: N = 3 337 / 345 / 344, N = 4 439 / 439 / 465, N =
// 5 1510 / 1453 / 1565, N = 6 484 / 472 / 468, N = 7 717 / 695 / 695).
__host__ __device__ constexpr int f64_ctas(int N) { return N == 2 ? 6 : 4; }
__host__ __device__ constexpr int f64_unroll(int N) { return N <= 4 ? 3 : 4; }

template <int N, bool MEDIA>
struct F64Layout {
  static constexpr int Np = Order<N>::Np, Nfp = Order<N>::Nfp, Nafp = Order<N>::Nafp;
  static constexpr int GEO = MEDIA ? kGeoMedia : kGeo;
  static constexpr int NI = Np - 3;  // nodes that are not vertices
  static constexpr int TABLE = f64_table_ints(N);
  static constexpr int TPT = (Nafp + Np - 1) / Np;            // flux tasks per thread
  // shared memory of a block of E elements: table, then per stage buffer
  // q[3], res[3], geometry, codes; then operands, differences, linear terms,
  // maxima, the rest of the operands (two: with the second flux scalar's)
  __host__ __device__ static constexpr int stage_bytes(int E) {
    return (E * (6 * Np * 8 + GEO * 8 + 12) + 15) / 16 * 16;
  }
  __host__ __device__ static constexpr int smem_bytes(int E, bool two) {
    return 4 * TABLE + 2 * stage_bytes(E) +
           E * (NI * 36 + (two ? 2 : 1) * Nafp * 16 + 6 * 8 + 3 * 8 + 2 * 4 * 4);
  }
};

__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}

// |v| as an integer that orders like it; 0 for zero only
__device__ __forceinline__ int f64_size(double v) {
  return (__double2hiint(v) & 0x7fffffff) | (__double2loint(v) != 0 ? 1 : 0);
}
// biased exponents of a vector's largest entry that fixed point holds (0:
// the vector is zero)
__device__ __forceinline__ bool f64_fixed(int size) {
  const int e = size >> 20;
  return size == 0 || (e >= 128 && e <= 1900);
}

// A fixed-point number x 2^56 + y 2^28 + z.
struct F64Limbs {
  int x, y, z;
};

// v 2^(1106 - ex) cut to an integer below 2^84 in size, ex the biased exponent
// of its vector's largest entry (exact if v's is at least ex - 31)
__device__ __forceinline__ F64Limbs f64_limbs(double v, int ex) {
  const long long b = __double_as_longlong(v);
  const int e = static_cast<int>((b >> 52) & 0x7ff);
  const unsigned long long m =
      (static_cast<unsigned long long>(b) << 11) | (e ? 1ull << 63 : 0);
  const int sh = ex - (e ? e : 1);
  // the integer's upper 64 bits and the 20 below them
  const unsigned long long top = sh < 64 ? m >> sh : 0;
  const unsigned long long below =
      sh == 0 ? 0 : sh < 64 ? m << (64 - sh) : sh < 128 ? m >> (sh - 64) : 0;
  const int x = static_cast<int>(top >> 36);
  const int y = static_cast<int>((top >> 8) & 0xfffffff);
  const int z = static_cast<int>(((top & 0xff) << 20) | (below >> 44));
  return b < 0 ? F64Limbs{-x, -y, -z} : F64Limbs{x, y, z};
}

// A sum of fixed-point products, without their parts below 2^56: (hh 2^56 +
// hl 2^28 + ll) 2^56
struct F64Sum {
  long long hh = 0, hl = 0, ll = 0;
  __device__ __forceinline__ void term(const F64Limbs& a, const F64Limbs& b) {
    hh += static_cast<long long>(a.x) * b.x;
    hl += static_cast<long long>(a.x) * b.y;
    hl += static_cast<long long>(a.y) * b.x;
    ll += static_cast<long long>(a.x) * b.z;
    ll += static_cast<long long>(a.y) * b.y;
    ll += static_cast<long long>(a.z) * b.x;
  }
  __device__ __forceinline__ void add(const F64Sum& o) {
    hh += o.hh;
    hl += o.hl;
    ll += o.ll;
  }
};

// The FP64 value of a sum times its operands' powers of two, 2^(ex - 1106)
// and 2^scale; k = ex + scale
__device__ __forceinline__ double f64_value(const F64Sum& s, int k) {
  constexpr long long M28 = (1ll << 28) - 1;
  // the sum as hi 2^64 + lo in units of 2^-8, then its size
  const long long mid = s.hl + (s.ll >> 28);
  long long hi = s.hh + (mid >> 28);
  unsigned long long lo = static_cast<unsigned long long>((mid & M28) << 28 | (s.ll & M28)) << 8;
  const long long sign = hi & (1ll << 63);
  if (hi < 0) {
    lo = -lo;
    hi = ~hi + (lo == 0);
  }
  if (hi == 0) {
    if (lo == 0) return 0.0;
    hi = lo >> 8;
    lo = 0;
    k -= 56;
  }
  const int lz = __clzll(hi);
  const unsigned long long top = (static_cast<unsigned long long>(hi) << lz) | (lo >> 1 >> (63 - lz));
  const unsigned long long m = (top >> 11) + ((top >> 10) & 1);  // 53 bits, or 2^53
  const long long bits = (static_cast<long long>(k + 91 - lz) << 52) + static_cast<long long>(m);
  return __longlong_as_double(bits | sign);
}

template <int N, int MODE, bool MEDIA>
__global__ void __launch_bounds__(f64_max_elems(N) * Order<N>::Np, f64_ctas(N))
    dg_stage_f64_kernel(const StageArgs<double> p, const int E) {
  using L = F64Layout<N, MEDIA>;
  constexpr int Np = L::Np, Nfp = L::Nfp, Nafp = L::Nafp, GEO = L::GEO, NI = L::NI;
  constexpr int TPT = L::TPT, UNROLL = f64_unroll(N);
  extern __shared__ __align__(128) unsigned char smem[];
  const int NT = E * Np;  // threads of the CTA
  const int t = threadIdx.x;
  const int e = t / Np, i = t - e * Np;
  // interior column of the own node, -1 at a vertex node
  const int ci = (i == 0 || i == N || i == Np - 1) ? -1 : i < N ? i - 1 : i - 2;

  // the table (f64_table_ints)
  int4* tab4 = reinterpret_cast<int4*>(smem);
  int2* tab2 = reinterpret_cast<int2*>(tab4 + NI * Np);
  int2* tabl = tab2 + NI * Np;
  int* tablz = reinterpret_cast<int*>(tabl + Nafp * Np);
  unsigned char* stages = smem + 4 * L::TABLE;
  const int SB = L::stage_bytes(E);
  const bool two = !MEDIA && p.alpha != 1.0;  // a second flux scalar
  const int NF = two ? 2 * Nafp : Nafp;
  // per element and column {z x, y, A x, y}, {B x, y, z z, A z}; per face node {x, y, z}
  int4* vol = reinterpret_cast<int4*>(stages + 2 * SB);
  int4* flx = vol + 2 * NI * E;
  double* dif = reinterpret_cast<double*>(flx + NF * E);      // [E][3][2]
  double* lin = dif + 6 * E;                                  // [3][E]
  int* mx = reinterpret_cast<int*>(lin + 3 * E);              // [2][E][4]
  int* volb = mx + 8 * E;                                     // B z [E][NI]

  const int K = static_cast<int>(p.K);
  const int nblk = (K + E - 1) / E;
  const int G = gridDim.x, b0 = blockIdx.x;
  const int niter = b0 < nblk ? (nblk - 1 - b0) / G + 1 : 0;
  const int64_t fs = p.fstride;

  auto stage = [&](int it) { return reinterpret_cast<double*>(stages + (it & 1) * SB); };
  auto codes = [&](int it) {
    return reinterpret_cast<const int32_t*>(stage(it) + E * (6 * Np + GEO));
  };
  // geometry and codes of block it (nothing writes them), then its fields
  auto issue_geo = [&](int it) {
    const int k0 = (b0 + it * G) * E;
    const int n = (K - k0) < E ? (K - k0) : E;
    double* st = stage(it);
    for (int c = t; c < n * GEO; c += NT)
      cp_async8(st + 6 * NT + c, p.geo + static_cast<int64_t>(k0) * GEO + c);
    int32_t* sc = reinterpret_cast<int32_t*>(st + 6 * NT + E * GEO);
    for (int c = t; c < n * 3; c += NT) cp_async4(sc + c, p.conn + static_cast<int64_t>(k0) * 3 + c);
  };
  auto issue_q = [&](int it) {
    const int k0 = (b0 + it * G) * E;
    if (k0 + e < K) {
      double* st = stage(it) + t;
      const int64_t g = static_cast<int64_t>(k0) * Np + t;
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        cp_async8(st + f * NT, p.qin + f * fs + g);
        if (MODE == kModeStage) cp_async8(st + (3 + f) * NT, p.res + f * fs + g);
      }
    }
  };

  if (niter > 0) issue_geo(0);
  {
    const int4* src = static_cast<const int4*>(p.tc_op);
    for (int c = t; c < L::TABLE / 4; c += NT) cp_async16(tab4 + c, src + c);
  }
  // powers of two of this node's rows of Dr and Ds, and of LIFT
  const int2 scale = __ldg(static_cast<const int2*>(p.tc_op) + L::TABLE / 2 + i);
  const double lam2 = __ldg(p.lam + i), lam3 = __ldg(p.lam + Np + i);
  for (int c = t; c < 8 * E; c += NT) mx[c] = 0;

  // flux tasks of this thread (the same in every block)
  int task_e[TPT], task_j[TPT];
#pragma unroll
  for (int u = 0; u < TPT; ++u) {
    const int tau = t + u * NT;
    task_e[u] = tau < E * Nafp ? tau / Nafp : E;  // E: none
    task_j[u] = tau - (tau / Nafp) * Nafp;
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();

  double trc[TPT][3];
  auto gather = [&](int it) {
    const int32_t* sc = codes(it);
    const int k0 = (b0 + it * G) * E;
#pragma unroll
    for (int u = 0; u < TPT; ++u) {
      trc[u][0] = trc[u][1] = trc[u][2] = 0.0;
      if (task_e[u] < E && k0 + task_e[u] < K) {
        const int f = task_j[u] / Nfp, jj = task_j[u] - f * Nfp;
        const int32_t code = sc[task_e[u] * 3 + f];
#ifdef DGW_DEVICE_CHECKS
        if (!nbr_code_ok(code, fs, Np)) {
          atomicOr(p.status, kStatusIndex);
          continue;
        }
#endif
        if (code >= 0) {
          const int nb = face_node_dev(N, (code >> 1) & 3, (code & 1) ? N - jj : jj);
          const double* src = p.qin + static_cast<int64_t>(code >> 3) * Np + nb;
          trc[u][0] = src[0];
          trc[u][1] = src[fs];
          trc[u][2] = src[2 * fs];
        }
      }
    }
  };
  chain_wait();
  chain_trigger();
  if (niter > 0) {  // the first block's values and traces side by side
    issue_q(0);
    cp_async_commit();
    gather(0);
    cp_async_wait<0>();
  }
  __syncthreads();

  for (int it = 0; it < niter; ++it) {
    const int k0 = (b0 + it * G) * E;
    const bool valid = k0 + e < K;
    const double* sq = stage(it);
    const double* sg = sq + 6 * NT;
    const int32_t* sc = codes(it);
    int* m = mx + (it & 1) * 4 * E;  // largest z, (A, B), f, g of each element

    // ---- 0: vertex differences
    for (int c = t; c < 6 * E; c += NT) {
      const int ee = c / 6, r = c - 6 * ee, f = r >> 1;
      const double* q = sq + f * NT + ee * Np;
      dif[c] = q[(r & 1) ? Np - 1 : N] - q[0];
    }
    __syncthreads();

    // ---- 1: the next block's data; deflated operands, flux, linear part
    if (it + 1 < niter) {
      issue_geo(it + 1);
      issue_q(it + 1);
    }
    cp_async_commit();
    for (int c = t; c < 4 * E; c += NT) mx[((it + 1) & 1) * 4 * E + c] = 0;
    double z = 0, A = 0, B = 0;
    if (valid && ci >= 0) {
      const double* d = dif + 6 * e;
      const double* q = sq + e * Np;
      const double dhx = fma(-d[1], lam3, fma(-d[0], lam2, sq[t] - q[0]));
      const double dhy = fma(-d[3], lam3, fma(-d[2], lam2, sq[NT + t] - q[NT]));
      const double* ge = sg + e * GEO;
      z = fma(-d[5], lam3, fma(-d[4], lam2, sq[2 * NT + t] - q[2 * NT]));
      A = fma(-ge[1], dhx, ge[0] * dhy);
      B = fma(-ge[3], dhx, ge[2] * dhy);
      atomicMax(m + 4 * e, f64_size(z));
      atomicMax(m + 4 * e + 1, max(f64_size(A), f64_size(B)));
    }
    double fv[TPT], gv[TPT];
#pragma unroll
    for (int u = 0; u < TPT; ++u) {
      const int ee = task_e[u];
      fv[u] = gv[u] = 0.0;
      if (ee < E && k0 + ee < K) {
        const int f = task_j[u] / Nfp, jj = task_j[u] - f * Nfp;
        const double* q = sq + ee * Np + face_node_dev(N, f, jj);
        const double hx = q[0], hy = q[NT], ez = q[2 * NT];
        const bool wall = sc[ee * 3 + f] < 0;  // PEC wall: H+ = H-, Ez+ = -Ez-
        const double dHx = hx - (wall ? hx : trc[u][0]);
        const double dHy = hy - (wall ? hy : trc[u][1]);
        const double dEz = ez - (wall ? -ez : trc[u][2]);
        const double* gf = sg + ee * GEO + 4 + (MEDIA ? 4 : 3) * f;
        const double Ht = fma(-gf[0], dHy, gf[1] * dHx);
        if (MEDIA) {
          fv[u] = fma(-gf[3], dEz, gf[2] * Ht);
        } else {
          fv[u] = gf[2] * fma(-p.alpha, dEz, Ht);
          if (two) {
            gv[u] = gf[2] * fma(p.alpha, Ht, -dEz);
            atomicMax(m + 4 * ee + 3, f64_size(gv[u]));
          }
        }
        atomicMax(m + 4 * ee + 2, f64_size(fv[u]));
      }
    }
    if (t < E) {  // derivatives of the linear part along r and s, chain rule
      const double* d = dif + 6 * t;
      const double* ge = sg + t * GEO;
      lin[t] = -0.5 * (ge[1] * d[4] + ge[3] * d[5]);
      lin[E + t] = 0.5 * (ge[0] * d[4] + ge[2] * d[5]);
      lin[2 * E + t] = 0.5 * (ge[0] * d[2] - ge[1] * d[0] + ge[2] * d[3] - ge[3] * d[1]);
    }
    __syncthreads();

    // ---- 2: fixed-point operands
    auto slot = [&](double v, int size) {
      if (size == 0) return F64Limbs{0, 0, 0};
      return f64_fixed(size) ? f64_limbs(v, size >> 20)
                             : F64Limbs{__double2hiint(v), __double2loint(v), 0};
    };
    if (valid && ci >= 0) {
      const F64Limbs lz = slot(z, m[4 * e]), la = slot(A, m[4 * e + 1]), lb = slot(B, m[4 * e + 1]);
      int4* o = vol + 2 * (e * NI + ci);
      o[0] = make_int4(lz.x, lz.y, la.x, la.y);
      o[1] = make_int4(lb.x, lb.y, lz.z, la.z);
      volb[e * NI + ci] = lb.z;
    }
#pragma unroll
    for (int u = 0; u < TPT; ++u) {
      const int ee = task_e[u];
      if (ee < E && k0 + ee < K) {
        int4* o = flx + ee * NF + task_j[u];
        const F64Limbs lf = slot(fv[u], m[4 * ee + 2]);
        o[0] = make_int4(lf.x, lf.y, lf.z, 0);
        if (two) {
          const F64Limbs lg = slot(gv[u], m[4 * ee + 3]);
          o[Nafp] = make_int4(lg.x, lg.y, lg.z, 0);
        }
      }
    }
    cp_async_wait<0>();
    __syncthreads();
    if (it + 1 < niter) gather(it + 1);

    // ---- 3: products, chain rule, update
    if (valid) {
      const int4* vo = vol + 2 * e * NI;
      const int* vb = volb + e * NI;
      const int4* fo = flx + e * NF;
      auto lift = [&](int j) {
        const int2 h = tabl[j * Np + i];
        return F64Limbs{h.x, h.y, tablz[j * Np + i]};
      };
      auto flux = [&](int j) {
        const int4 h = fo[j];
        return F64Limbs{h.x, h.y, h.z};
      };
      const int sz = m[4 * e], sab = m[4 * e + 1], sf = m[4 * e + 2], sgg = m[4 * e + 3];
      const bool fixed = f64_fixed(sz) && f64_fixed(sab) && f64_fixed(sf) && f64_fixed(sgg);
      double zr, zs, c, lf[3], lsum;  // lf: LIFT of the H rows' scalar per face
      if (fixed) {
        F64Sum szr, szs, sc;
#pragma unroll UNROLL
        for (int k = 0; k < NI; ++k) {
          const int4 d = tab4[k * Np + i], u = vo[2 * k], w = vo[2 * k + 1];
          const int2 dz = tab2[k * Np + i];
          const F64Limbs dr = {d.x, d.y, dz.x}, ds = {d.z, d.w, dz.y};
          const F64Limbs vz = {u.x, u.y, w.z};
          szr.term(dr, vz);
          szs.term(ds, vz);
          sc.term(dr, F64Limbs{u.z, u.w, w.w});
          sc.term(ds, F64Limbs{w.x, w.y, vb[k]});
        }
        const int kz = (sz >> 20) + scale.x, kab = (sab >> 20) + scale.x;
        zr = f64_value(szr, kz);
        zs = f64_value(szs, kz);
        c = f64_value(sc, kab);
        const int kf = (sf >> 20) + scale.y;
        F64Sum all;
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          F64Sum face;
#pragma unroll UNROLL
          for (int jj = 0; jj < Nfp; ++jj) {
            const int j = f * Nfp + jj;
            face.term(lift(j), flux(j));
          }
          lf[f] = f64_value(face, kf);
          all.add(face);
        }
        lsum = f64_value(all, kf);
        if (two) {
          const int kg = (sgg >> 20) + scale.y;
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            F64Sum face;
#pragma unroll UNROLL
            for (int jj = 0; jj < Nfp; ++jj) {
              const int j = f * Nfp + jj;
              face.term(lift(j), flux(Nafp + j));
            }
            lf[f] = f64_value(face, kg);
          }
        }
      } else {
        // some operand has no fixed-point form: all of the element's in FP64
        auto at = [](int x, int y, int lo, int size) {
          if (!f64_fixed(size)) return __hiloint2double(x, y);
          const double low = static_cast<double>(y) * 268435456.0 + lo;
          return size == 0 ? 0.0
                           : scalbn(static_cast<double>(x) * 72057594037927936.0 + low,
                                    (size >> 20) - 1106);
        };
        zr = zs = c = lsum = 0.0;
#pragma unroll 1
        for (int k = 0; k < NI; ++k) {
          const int col = i * Np + (k < N - 1 ? k + 1 : k + 2);
          const double dr = __ldg(p.Dr + col), ds = __ldg(p.Ds + col);
          const int4 u = vo[2 * k], w = vo[2 * k + 1];
          const double vz = at(u.x, u.y, w.z, sz);
          zr += dr * vz;
          zs += ds * vz;
          c += dr * at(u.z, u.w, w.w, sab) + ds * at(w.x, w.y, vb[k], sab);
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          lf[f] = 0.0;
#pragma unroll 1
          for (int jj = 0; jj < Nfp; ++jj) {
            const int j = f * Nfp + jj;
            const double l = __ldg(p.LIFT + i * Nafp + j);
            const int4 a = fo[j], b = fo[two ? Nafp + j : j];
            const double v = at(a.x, a.y, a.z, sf);
            lsum += l * v;
            lf[f] += l * (two ? at(b.x, b.y, b.z, sgg) : v);
          }
        }
      }
      const double* ge = sg + e * GEO;
      double rhs[3] = {lin[e], lin[E + e], (lin[2 * E + e] + lsum) + c};
      if (MEDIA) {
        const double zm = ge[16];
        rhs[0] = fma(-zm, fma(ge[13], lf[2], fma(ge[9], lf[1], ge[5] * lf[0])), rhs[0]);
        rhs[1] = fma(zm, fma(ge[12], lf[2], fma(ge[8], lf[1], ge[4] * lf[0])), rhs[1]);
      } else {
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          rhs[0] = fma(-ge[5 + 3 * f], lf[f], rhs[0]);
          rhs[1] = fma(ge[4 + 3 * f], lf[f], rhs[1]);
        }
      }
      rhs[0] = fma(-ge[3], zs, fma(-ge[1], zr, rhs[0]));
      rhs[1] = fma(ge[2], zs, fma(ge[0], zr, rhs[1]));
      if (MEDIA) {
        rhs[0] *= ge[17];
        rhs[1] *= ge[17];
        rhs[2] *= ge[18];
      }
      const int64_t g = static_cast<int64_t>(k0) * Np + t;
      const bool src = k0 + e == p.psrc_k;
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        if (MODE == kModeRhs) {
          p.rhs[f * fs + g] = f == 2 && src ? fma(p.psrc_amp, p.psrc_w[i], rhs[f]) : rhs[f];
        } else {
          double r = p.dt * rhs[f];
          if (MODE == kModeStage) r = fma(p.a, sq[(3 + f) * NT + t], r);
          double q = fma(p.b, r, sq[f * NT + t]);
          if (f == 2 && src) {  // the operator's point source
            const double v = p.psrc_amp * p.psrc_w[i];
            r = __dadd_rn(r, v);
            q = fma(p.b, v, q);
          }
          p.res[f * fs + g] = r;
          p.qout[f * fs + g] = q;
        }
      }
    }
  }
}

template <int N, int MODE, bool MEDIA>
cudaError_t launch_f64_mode(const StageArgs<double>& args, int num_sms, cudaStream_t stream) {
  using L = F64Layout<N, MEDIA>;
  static std::atomic<uint64_t> configured{0};
  static std::atomic<int> blocks_per_sm{1};
  constexpr int EMAX = f64_max_elems(N);
  cudaError_t err = configure_once_per_device(configured, [] {
    cudaError_t e = cudaFuncSetAttribute(dg_stage_f64_kernel<N, MODE, MEDIA>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         L::smem_bytes(EMAX, !MEDIA));
    int nb = 0;
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, dg_stage_f64_kernel<N, MODE, MEDIA>,
                                                        EMAX * L::Np, L::smem_bytes(EMAX, false));
    if (e == cudaSuccess) blocks_per_sm.store(nb > 0 ? nb : 1);
    return e;
  });
  if (err != cudaSuccess) return err;
  const int E = f64_block_elems(N, args.K, num_sms);
  const int64_t nblk = (args.K + E - 1) / E;
  int64_t grid = static_cast<int64_t>(blocks_per_sm.load()) * num_sms;
  if (grid > nblk || E < EMAX) grid = nblk;
  return launch_chained(dg_stage_f64_kernel<N, MODE, MEDIA>, static_cast<unsigned>(grid),
                        E * L::Np, L::smem_bytes(E, !MEDIA && args.alpha != 1.0), stream, args, E);
}

template <int N, bool MEDIA>
cudaError_t launch_f64_modes(const StageArgs<double>& args, int mode, int num_sms,
                             cudaStream_t stream) {
  if (mode == kModeRhs) return launch_f64_mode<N, kModeRhs, MEDIA>(args, num_sms, stream);
  if (mode == kModeFirstStage)
    return launch_f64_mode<N, kModeFirstStage, MEDIA>(args, num_sms, stream);
  return launch_f64_mode<N, kModeStage, MEDIA>(args, num_sms, stream);
}

// Definition of the launcher declared in launch.h; explicitly instantiated
// per order in kernels_f64_N*.cu.
template <int N>
cudaError_t launch_stage_f64(const StageArgs<double>& args, bool media, int mode, int num_sms,
                             cudaStream_t stream) {
  return media ? launch_f64_modes<N, true>(args, mode, num_sms, stream)
               : launch_f64_modes<N, false>(args, mode, num_sms, stream);
}

}  // namespace dgw
