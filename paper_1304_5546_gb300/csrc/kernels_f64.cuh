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
//   rounded to 56-bit integers v = hi 2^28 + lo (28-bit signed limbs), and so,
//   on the host, are the rows of Dr, Ds and LIFT.  A term is four 32 x 32 ->
//   64 bit multiply-adds into the sums of hi hi, of hi lo + lo hi and of lo
//   lo, which are exact (|hi| <= 2^27, at most 66 terms).  Rounding an entry
//   to 2^-56 of its vector's (its row's) largest and one final rounding
//   replace the roundings of up to 60 FP64 multiply-adds.
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
// f64_max_elems' table, CTAs aimed at: N = 1 2 / 3 / 4 358 / 309 / 313, N = 2
// 4 / 6 383 / 326, N = 3 3 / 4 / 5 348 / 312 / 320, N = 5 2 / 3 / 4 / 5 1506 /
// 1395 / 1331 / 1364, N = 7 2 / 3 / 4 601 / 560 / 575; three columns a step
// instead of two: N = 5 1292, N = 6 371 against 378, N = 7 605 against 575).
__host__ __device__ constexpr int f64_ctas(int N) { return N == 1 || N == 7 ? 3 : N == 2 ? 6 : 4; }
__host__ __device__ constexpr int f64_unroll(int N) { return N == 7 ? 2 : 3; }

template <int N, bool MEDIA>
struct F64Layout {
  static constexpr int Np = Order<N>::Np, Nfp = Order<N>::Nfp, Nafp = Order<N>::Nafp;
  static constexpr int GEO = MEDIA ? kGeoMedia : kGeo;
  static constexpr int NI = Np - 3;  // nodes that are not vertices
  static constexpr int TABLE = f64_table_pairs(N);            // limb pairs
  static constexpr int TPT = (Nafp + Np - 1) / Np;            // flux tasks per thread
  // shared memory of a block of E elements: table, then per stage buffer
  // q[3], res[3], geometry, codes; then operands, differences, linear terms,
  // maxima
  __host__ __device__ static constexpr int stage_bytes(int E) {
    return E * (6 * Np * 8 + GEO * 8) + (E * 12 + 7) / 8 * 8;
  }
  static constexpr int OPS = 3 * NI + 2 * Nafp;  // operand slots (8 bytes) of an element
  __host__ __device__ static constexpr int smem_bytes(int E) {
    return 8 * TABLE + 2 * stage_bytes(E) + E * (OPS * 8 + 6 * 8 + 3 * 8 + 2 * 4 * 4);
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

// v / 2^(ex - 1077) rounded to an integer of at most 2^55, ex the biased
// exponent of its vector's largest entry, as limbs x 2^28 + y, |y| <= 2^27
__device__ __forceinline__ int2 f64_limbs(double v, int ex) {
  const long long b = __double_as_longlong(v);
  const int e = static_cast<int>((b >> 52) & 0x7ff);
  long long m = (b & 0xfffffffffffffll) | (e ? 1ll << 52 : 0);
  const int sh = ex - (e ? e : 1);
  m = (((m << 3) >> (sh < 63 ? sh : 63)) + 1) >> 1;
  if (b < 0) m = -m;
  const int lo = static_cast<int>(static_cast<unsigned>(m) << 4) >> 4;
  return make_int2(static_cast<int>((m - lo) >> 28), lo);
}

// A sum of fixed-point products, hh 2^56 + hl 2^28 + ll (|hh| < 2^61)
struct F64Sum {
  long long hh = 0, hl = 0, ll = 0;
  __device__ __forceinline__ void term(int2 a, int2 b) {
    hh += static_cast<long long>(a.x) * b.x;
    hl += static_cast<long long>(a.x) * b.y;
    hl += static_cast<long long>(a.y) * b.x;
    ll += static_cast<long long>(a.y) * b.y;
  }
  __device__ __forceinline__ void add(const F64Sum& o) {
    hh += o.hh;
    hl += o.hl;
    ll += o.ll;
  }
};

// The FP64 value of a sum times its operands' powers of two, 2^(ex - 1077)
// and 2^scale; k = ex + scale
__device__ __forceinline__ double f64_value(const F64Sum& s, int k) {
  const long long r = (s.hh << 2) + ((s.hl + (s.ll >> 28)) >> 26);
  if (r == 0) return 0.0;
  unsigned long long a = r < 0 ? -static_cast<unsigned long long>(r) : r;
  const int lz = __clzll(a);
  a = ((a << lz) + (1ull << 10)) >> 11;  // 53 bits, or 2^53 after a carry
  const long long bits = (static_cast<long long>(k + 62 - lz) << 52) + static_cast<long long>(a);
  return __longlong_as_double(bits | (r & (1ll << 63)));
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

  int2* tab = reinterpret_cast<int2*>(smem);  // Dr [NI][Np], Ds [NI][Np], LIFT [Nafp][Np]
  unsigned char* stages = smem + 8 * L::TABLE;
  const int SB = L::stage_bytes(E);
  int2* ops = reinterpret_cast<int2*>(stages + 2 * SB);  // per element: z, A, B [NI], f, g [Nafp]
  double* dif = reinterpret_cast<double*>(ops + E * L::OPS);  // [E][3][2]
  double* lin = dif + 6 * E;                                  // [3][E]
  int* mx = reinterpret_cast<int*>(lin + 3 * E);              // [2][E][4]

  const int K = static_cast<int>(p.K);
  const int nblk = (K + E - 1) / E;
  const int G = gridDim.x, b0 = blockIdx.x;
  const int niter = b0 < nblk ? (nblk - 1 - b0) / G + 1 : 0;
  const int64_t fs = p.fstride;
  const bool two = !MEDIA && p.alpha != 1.0;  // a second flux scalar

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
    for (int c = t; c < L::TABLE / 2; c += NT) cp_async16(tab + 2 * c, src + c);
  }
  // powers of two of this node's rows of Dr and Ds, and of LIFT
  const int2 scale = __ldg(static_cast<const int2*>(p.tc_op) + L::TABLE + i);
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
      if (size == 0) return make_int2(0, 0);
      return f64_fixed(size) ? f64_limbs(v, size >> 20)
                             : make_int2(__double2hiint(v), __double2loint(v));
    };
    if (valid && ci >= 0) {
      int2* o = ops + e * L::OPS + ci;
      o[0] = slot(z, m[4 * e]);
      o[NI] = slot(A, m[4 * e + 1]);
      o[2 * NI] = slot(B, m[4 * e + 1]);
    }
#pragma unroll
    for (int u = 0; u < TPT; ++u) {
      const int ee = task_e[u];
      if (ee < E && k0 + ee < K) {
        int2* o = ops + ee * L::OPS + 3 * NI + task_j[u];
        o[0] = slot(fv[u], m[4 * ee + 2]);
        if (two) o[Nafp] = slot(gv[u], m[4 * ee + 3]);
      }
    }
    cp_async_wait<0>();
    __syncthreads();
    if (it + 1 < niter) gather(it + 1);

    // ---- 3: products, chain rule, update
    if (valid) {
      const int2* o = ops + e * L::OPS;
      const int sz = m[4 * e], sab = m[4 * e + 1], sf = m[4 * e + 2], sgg = m[4 * e + 3];
      const bool fixed = f64_fixed(sz) && f64_fixed(sab) && f64_fixed(sf) && f64_fixed(sgg);
      double zr, zs, c, lf[3], lsum;  // lf: LIFT of the H rows' scalar per face
      if (fixed) {
        F64Sum szr, szs, sc;
#pragma unroll UNROLL
        for (int k = 0; k < NI; ++k) {
          const int2 dr = tab[k * Np + i], ds = tab[(NI + k) * Np + i];
          const int2 vz = o[k];
          szr.term(dr, vz);
          szs.term(ds, vz);
          sc.term(dr, o[NI + k]);
          sc.term(ds, o[2 * NI + k]);
        }
        const int2* lt = tab + 2 * NI * Np + i;
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
            face.term(lt[j * Np], o[3 * NI + j]);
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
              face.term(lt[j * Np], o[3 * NI + Nafp + j]);
            }
            lf[f] = f64_value(face, kg);
          }
        }
      } else {
        // some operand has no fixed-point form: all of the element's in FP64
        auto at = [&](int k, int size) {
          if (!f64_fixed(size)) return __hiloint2double(o[k].x, o[k].y);
          return size == 0 ? 0.0
                           : scalbn(static_cast<double>(o[k].x) * 268435456.0 + o[k].y,
                                    (size >> 20) - 1077);
        };
        zr = zs = c = lsum = 0.0;
#pragma unroll 1
        for (int k = 0; k < NI; ++k) {
          const int col = i * Np + (k < N - 1 ? k + 1 : k + 2);
          const double dr = __ldg(p.Dr + col), ds = __ldg(p.Ds + col);
          zr += dr * at(k, sz);
          zs += ds * at(k, sz);
          c += dr * at(NI + k, sab) + ds * at(2 * NI + k, sab);
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          lf[f] = 0.0;
#pragma unroll 1
          for (int jj = 0; jj < Nfp; ++jj) {
            const int j = f * Nfp + jj;
            const double l = __ldg(p.LIFT + i * Nafp + j), v = at(3 * NI + j, sf);
            lsum += l * v;
            lf[f] += l * (two ? at(3 * NI + Nafp + j, sgg) : v);
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
                                         L::smem_bytes(EMAX));
    int nb = 0;
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, dg_stage_f64_kernel<N, MODE, MEDIA>,
                                                        EMAX * L::Np, L::smem_bytes(EMAX));
    if (e == cudaSuccess) blocks_per_sm.store(nb > 0 ? nb : 1);
    return e;
  });
  if (err != cudaSuccess) return err;
  const int E = f64_block_elems(N, args.K, num_sms);
  const int64_t nblk = (args.K + E - 1) / E;
  int64_t grid = static_cast<int64_t>(blocks_per_sm.load()) * num_sms;
  if (grid > nblk || E < EMAX) grid = nblk;
  return launch_chained(dg_stage_f64_kernel<N, MODE, MEDIA>, static_cast<unsigned>(grid),
                        E * L::Np, L::smem_bytes(E), stream, args, E);
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
