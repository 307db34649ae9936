// a3-a5 of a step or Jacobian action (Sec. 3.1): inverse DFT in phi of the nine grid fields,
// U x omega and U.grad T (or their linearisation about a base state), forward DFT of the four
// products; and the base state's grid values on their own.
//
// The DFTs use the symmetries of the longitudes phi_j = 2 pi j / n.  With theta = a phi_j,
//   cos a phi_(n-j) = cos theta,             sin a phi_(n-j) = -sin theta,
//   cos a phi_(n/2-j) = (-1)^a cos theta,    sin a phi_(n/2-j) = -(-1)^a sin theta   (n even),
// so the four longitudes j, n - j, n/2 - j, n/2 + j share the sums over even and over odd a of
// the cosine and of the sine part: a quarter of the multiply-adds of the direct sums (a half
// for odd n, which has the first symmetry only).  The forward transform folds the products of
// the four longitudes the same way before it multiplies.
//
// Layout: a thread is one latitude and one quad of longitudes (J quads in FP32), lanes run over
// consecutive latitudes.  The coefficients of LT latitudes are staged in shared memory by
// coalesced loads (a warp per latitude gathered them with a stride of nlat, one sector per
// coefficient; the copies are asynchronous, so a block waits for one round trip of memory), read
// back without bank conflicts, and the twiddles are warp broadcasts.
//
// What bounds it: FP64 its multiply-adds (one warp instruction holds the FP64 pipe of a
// sub-partition for 64 cycles), FP32 the latency of its global loads.  Measured, one GB300, a warp
// per latitude with direct sums before -> this kernel (us per launch):
//   L = 127, M_s = 12 (n = 32): FP64 step 488 -> 170, FP32 step 45 -> 18, FP32 linearised 39 -> 24;
//   L = 255, M_s = 8 (n = 96): FP64 step 12001 -> 2630, FP32 step 584 -> 172, linearised 900 -> 277;
//   L = 31, M_s = 4 (n = 24): FP64 step 46 -> 21.
#pragma once

#include "kernels.cuh"

namespace rsc {

enum { kProdStep = 0, kProdLin = 1, kProdBase = 2 };

template <typename R>
struct alignas(16) ProdR4 {
  R x, y, z, w;
};

// Quads of the n longitudes: 0 .. n/4 for even n, pairs 0 .. (n-1)/2 for odd n.
__host__ __device__ __forceinline__ int prod_quads(int n) { return (n & 1) ? (n + 1) / 2 : n / 4 + 1; }

// Shape of a launch: latitudes per block LT, quads in flight S (threads LT S), shared memory.
struct ProdShape {
  int LT, S, Q, J;
  size_t smem;
};

// Quads per thread: two in FP32 when there are many (each staged coefficient then feeds four
// multiply-adds instead of two), one where that would leave too few threads.
template <typename R>
__host__ inline int prod_quads_per_thread(int Q) { return sizeof(R) == 4 && Q > 12 ? 2 : 1; }
template <typename R>
constexpr int prod_max_threads() { return sizeof(R) == 4 ? 288 : 256; }

template <typename R>
__host__ inline size_t prod_smem(int K1, int nphi, int LT, bool base) {
  const size_t Q = prod_quads(nphi), NK = (nphi & 1) ? 2 : 4;
  return 9 * (size_t)K1 * LT * 2 * sizeof(R) + Q * K1 * 2 * sizeof(R) +
         (base ? 0 : Q * NK * LT * 4 * sizeof(R));
}

// 32 latitudes per block (a full line per coefficient row) unless that leaves fewer than two
// blocks per SM or a block takes more than a third of an SM's shared memory: then 16 or 8.
template <typename R>
__host__ inline ProdShape prod_shape(int K1, int nphi, int nlat, int Nd, bool base) {
  ProdShape s;
  s.Q = prod_quads(nphi);
  s.LT = 32;
  while (s.LT > 8 && ((long)Nd * ((nlat + s.LT - 1) / s.LT) < 2 * 152 ||
                      prod_smem<R>(K1, nphi, s.LT, base) > 74 * 1024))
    s.LT /= 2;
  s.J = prod_quads_per_thread<R>(s.Q);
  const int tasks = (s.Q + s.J - 1) / s.J;
  const int cap = prod_max_threads<R>() / s.LT;
  const int rounds = (tasks + cap - 1) / cap;
  s.S = max((tasks + rounds - 1) / rounds, 128 / s.LT);   // a warp group at least, for the loads
  s.smem = prod_smem<R>(K1, nphi, s.LT, base);
  return s;
}

// Fields v: 0 u_r, 1 u_th, 2 u_ph, 3-5 omega, 6-8 grad T.
template <typename R>
__device__ __forceinline__ ProdR4<R> prod_point(const R (&v)[9], R Ek) {
  return {Ek * (v[1] * v[5] - v[2] * v[4]), Ek * (v[2] * v[3] - v[0] * v[5]),
          Ek * (v[0] * v[4] - v[1] * v[3]), v[0] * v[6] + v[1] * v[7] + v[2] * v[8]};
}

// Linearised about U.
template <typename R>
__device__ __forceinline__ ProdR4<R> prod_point_lin(const R (&u)[9], const R (&U)[9], R Ek) {
  return {Ek * ((U[1] * u[5] - U[2] * u[4]) + (u[1] * U[5] - u[2] * U[4])),
          Ek * ((U[2] * u[3] - U[0] * u[5]) + (u[2] * U[3] - u[0] * U[5])),
          Ek * ((U[0] * u[4] - U[1] * u[3]) + (u[0] * U[4] - u[1] * U[3])),
          U[0] * u[6] + U[1] * u[7] + U[2] * u[8] + u[0] * U[6] + u[1] * U[7] + u[2] * U[8]};
}

template <typename R>
__device__ __forceinline__ ProdR4<R> prod_add(ProdR4<R> a, ProdR4<R> b) {
  return {a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w};
}
template <typename R>
__device__ __forceinline__ ProdR4<R> prod_sub(ProdR4<R> a, ProdR4<R> b) {
  return {a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w};
}

// MODE kProdStep: F = Ek U x omega, N = U.grad T from FC.  kProdLin: their linearisation, u from
// FC and U from UG.  kProdBase: UG[f][i][j][th] from FC (once per base state).  EVEN: nphi even.
// grid = (Nd, ceil(nlat / LT)), block = LT S.
template <typename R, int MODE, bool EVEN, int J>
__global__ void __launch_bounds__(prod_max_threads<R>(), 2)
k_products(DevGeom g, DevLegendre<R> T, R Ek, const typename C2<R>::T* __restrict__ FC,
           typename C2<R>::T* __restrict__ FA, R* __restrict__ UG, int LT, int S, int Q) {
  grid_begin();
  using V = typename C2<R>::T;
  constexpr int NK = EVEN ? 4 : 2, NPT = EVEN ? 4 : 2;
  extern __shared__ __align__(16) unsigned char pr_sh[];
  const int K1 = g.K + 1, n = g.nphi, nlat = g.nlat, Nd = g.Nd;
  ProdR4<R>* fold = reinterpret_cast<ProdR4<R>*>(pr_sh);                  // [Q][NK][LT]
  V* coef = reinterpret_cast<V*>(fold + (MODE == kProdBase ? 0 : Q * NK * LT));   // [a][f][LT]
  V* tw = coef + 9 * K1 * LT;                                             // [q][a] (cos, sin)
  const int i = blockIdx.x;
  const int th0 = blockIdx.y * LT;
  const int lat = threadIdx.x % LT, slot = threadIdx.x / LT;
  {
    // coefficients by asynchronous copies, all of a thread's in flight together
    int f = 0, a = slot;   // coefficient row slot, slot + S, ... = (f, a)
    const bool in = th0 + lat < nlat;
    const V* src = FC + (long)i * K1 * nlat + (in ? th0 + lat : 0);
    for (int c = slot; c < 9 * K1; c += S, a += S) {
      while (a >= K1) {
        a -= K1;
        ++f;
      }
      const unsigned dst = (unsigned)__cvta_generic_to_shared(coef + (a * 9 + f) * LT + lat);
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst),
                   "l"(src + ((long)f * Nd * K1 + a) * nlat), "n"(sizeof(V)), "r"(in ? (int)sizeof(V) : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // twiddles, doubled for a > 0 (the conjugate half of the real field); the forward transform halves
  for (int idx = threadIdx.x; idx < Q * K1; idx += blockDim.x) {
    const int q = idx / K1, a = idx - q * K1;
    const R w = a ? (R)2 : (R)1;
    tw[idx] = mk<R>(w * T.twc[a * n + q], w * T.tws[a * n + q]);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const int th = th0 + lat;
  const bool live = th < nlat;
  const V* cl = coef + lat;
  const int half = n / 2;
  // base state at longitude jj of this latitude
  const R* ub = UG + (long)i * n * nlat + th;
  auto load_base = [&](int jj, R (&U)[9]) {
#pragma unroll
    for (int f = 0; f < 9; ++f) U[f] = live ? ub[((long)f * Nd * n + jj) * nlat] : (R)0;
  };
  for (int q0 = slot * J; q0 < Q; q0 += S * J) {
    // sums over even a (e) and odd a (o; EVEN only) of the cosine (C) and sine (D) parts
    R Ce[J][9], De[J][9], Co[EVEN ? J : 1][9], Do[EVEN ? J : 1][9];
    const V* tq[J];
    R U[9], Un[9];
    if (MODE == kProdLin) load_base(q0, Un);   // the next longitude's base state, loaded ahead
#pragma unroll
    for (int u = 0; u < J; ++u) {
      tq[u] = tw + min(q0 + u, Q - 1) * K1;
#pragma unroll
      for (int f = 0; f < 9; ++f) {
        Ce[u][f] = De[u][f] = 0;
        if (EVEN) Co[u][f] = Do[u][f] = 0;
      }
    }
    for (int a = 0; a < K1; a += EVEN ? 2 : 1) {
      V t0[J], t1[J];
      const bool two = EVEN && a + 1 < K1;
#pragma unroll
      for (int u = 0; u < J; ++u) {
        t0[u] = tq[u][a];
        if (EVEN) t1[u] = tq[u][two ? a + 1 : a];
      }
#pragma unroll
      for (int f = 0; f < 9; ++f) {
        const V c = cl[(a * 9 + f) * LT];
#pragma unroll
        for (int u = 0; u < J; ++u) {
          Ce[u][f] += c.x * t0[u].x;
          De[u][f] += c.y * t0[u].y;
        }
      }
      if (two) {
#pragma unroll
        for (int f = 0; f < 9; ++f) {
          const V c = cl[((a + 1) * 9 + f) * LT];
#pragma unroll
          for (int u = 0; u < J; ++u) {
            Co[u][f] += c.x * t1[u].x;
            Do[u][f] += c.y * t1[u].y;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < J; ++u) {
      const int j = q0 + u;
      if (j >= Q) break;
      // the longitudes of this quad; duplicates at j = 0 and j = n / 4 count once
      const int jj[4] = {j, j ? n - j : 0, half - j, half + j};
      ProdR4<R> F[NPT];
#pragma unroll
      for (int k = 0; k < NPT; ++k) {
        R v[9];
#pragma unroll
        for (int f = 0; f < 9; ++f) {
          R c, s;
          if (!EVEN) {
            c = Ce[u][f];
            s = De[u][f];
          } else if (k < 2) {
            c = Ce[u][f] + Co[u][f];
            s = De[u][f] + Do[u][f];
          } else {
            c = Ce[u][f] - Co[u][f];
            s = Do[u][f] - De[u][f];
          }
          v[f] = (k & 1) ? c + s : c - s;
        }
        if (MODE == kProdBase) {
          if (live) {
#pragma unroll
            for (int f = 0; f < 9; ++f) UG[(((long)f * Nd + i) * n + jj[k]) * nlat + th] = v[f];
          }
        } else if (MODE == kProdLin) {
#pragma unroll
          for (int f = 0; f < 9; ++f) U[f] = Un[f];
          if (k + 1 < NPT) load_base(jj[k + 1], Un);
          else if (u + 1 < J && j + 1 < Q) load_base(j + 1, Un);
          F[k] = prod_point_lin<R>(v, U, Ek);
        } else {
          F[k] = prod_point<R>(v, Ek);
        }
      }
      if (MODE != kProdBase) {
        const ProdR4<R> zero = {0, 0, 0, 0};
        ProdR4<R> p = j ? prod_add(F[0], F[1]) : F[0];
        ProdR4<R> m = j ? prod_sub(F[0], F[1]) : zero;
        ProdR4<R>* o = fold + (long)j * NK * LT + lat;
        if (!EVEN) {
          o[0] = p;
          o[LT] = m;
        } else {
          ProdR4<R> p2 = j ? prod_add(F[2], F[3]) : F[2];
          ProdR4<R> m2 = j ? prod_sub(F[2], F[3]) : zero;
          const bool quarter = 4 * j == n;   // j = n/2 - j
          o[0] = quarter ? p : prod_add(p, p2);
          o[LT] = quarter ? zero : prod_sub(p, p2);
          o[2 * LT] = quarter ? zero : prod_sub(m, m2);
          o[3 * LT] = quarter ? m : prod_add(m, m2);
        }
      }
    }
  }
  if (MODE == kProdBase) return;
  __syncthreads();
  // forward DFT: a thread sums wavenumber a of the four products over the quads
  const R inv = (R)1 / (R)n;
  for (int a = slot; a < K1; a += S) {
    const R w = a ? (R)0.5 * inv : inv;
    const ProdR4<R>* fc = fold + (EVEN ? (a & 1) : 0) * LT + lat;
    const ProdR4<R>* fs = fold + (EVEN ? 2 + (a & 1) : 1) * LT + lat;
    R re[4] = {0, 0, 0, 0}, im[4] = {0, 0, 0, 0};
    for (int q = 0; q < Q; ++q) {
      const V t = tw[q * K1 + a];
      const ProdR4<R> c = fc[(long)q * NK * LT], s = fs[(long)q * NK * LT];
      re[0] += c.x * t.x; im[0] -= s.x * t.y;
      re[1] += c.y * t.x; im[1] -= s.y * t.y;
      re[2] += c.z * t.x; im[2] -= s.z * t.y;
      re[3] += c.w * t.x; im[3] -= s.w * t.y;
    }
    if (live) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        FA[(((long)q * Nd + i) * K1 + a) * nlat + th] = mk<R>(re[q] * w, im[q] * w);
    }
  }
}

}  // namespace rsc
