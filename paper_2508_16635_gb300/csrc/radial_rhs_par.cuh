// The radial stages with FP64 sums (the FP64 path; the mass products of mixed steps): the radial
// evaluation (a1) and the right-hand side (a7), by the reflection x -> -x of the Gauss-Lobatto radii.
//
// T_k(-x) = (-1)^k T_k(x), so rows j and j' = N - 1 - j of a Chebyshev table differ in signs only:
// with S_e, S_o the sums over even and odd k of one row, the other is S_e - S_o (even derivatives)
// or S_o - S_e (odd ones).  The projection onto the collocation radii R[j][i] obeys
// R[j'][i'] = +-R[j][i]: with P, M = (R[j][i] +- R[j][i']) / 2 and the inputs folded to a_i +- a_i',
// rows j and j' are sum P a+ +- sum M a-.  Either way two rows for the multiply-adds of one.
//
// What bounds it: the FP64 pipe (a warp instruction holds its sub-partition for 64 cycles however
// few lanes take part), so lanes run over (row pair, pair of the block) packed together, PPB
// pairs per block chosen to fill warps, and the sums of one pair are shared out over several
// warps (real / imaginary part, mass / projection): a warp per pair left 1.2 warps per sub-partition
// at L = 127.  Measured (us per launch, one GB300, a thread per row summing every k -> this):
//   L = 127, N_r = 64: radial FP64 120 -> 79; right-hand side FP64 step 125 -> 67, action 169 -> 90,
//   mixed step 97 (44 at its best block shape) -> 35;
//   L = 255, N_r = 96: radial 1511 -> 791; FP64 step 1426 -> 713, mixed step 647 -> 333;
//   L = 52, N_r = 60, second-order mixed step: 75 -> 26.
#pragma once

#include "kernels.cuh"

namespace rsc {

struct ParTables {
  // [i][j], i < ceil(Nd / 2), j < ceil(Nr / 2): P, M of R0 and of R1 r_i (FP64 and FP32)
  const double *P0, *M0, *P1, *M1;
  const float *P0f, *M0f, *P1f, *M1f;
  const double* irc;   // 1 / r_j
  const double* ird;   // 1 / r_i of the de-aliased radii
  double Ra_rout;      // Ra / r_out
};

template <typename R> struct ParTab;
template <> struct ParTab<double> {
  static __device__ __forceinline__ const double* P0(const ParTables& t) { return t.P0; }
  static __device__ __forceinline__ const double* M0(const ParTables& t) { return t.M0; }
  static __device__ __forceinline__ const double* P1(const ParTables& t) { return t.P1; }
  static __device__ __forceinline__ const double* M1(const ParTables& t) { return t.M1; }
};
template <> struct ParTab<float> {
  static __device__ __forceinline__ const float* P0(const ParTables& t) { return t.P0f; }
  static __device__ __forceinline__ const float* M0(const ParTables& t) { return t.M0f; }
  static __device__ __forceinline__ const float* P1(const ParTables& t) { return t.P1f; }
  static __device__ __forceinline__ const float* M1(const ParTables& t) { return t.M1f; }
};

// Pairs per block: the fewest that fill their warps to 15/16, or the best of 1..8.
__host__ inline int par_pairs(int rows) {
  int best = 1;
  double eff = 0.0;
  for (int p = 1; p <= 8; ++p) {
    const int n = p * rows, w = (n + 31) / 32 * 32;
    if (w > 160) break;
    if ((double)n / w > eff + 1e-9) {
      eff = (double)n / w;
      best = p;
    }
    if (eff >= 15.0 / 16.0) break;
  }
  return best;
}
__host__ inline int par_task_threads(int rows) { return (par_pairs(rows) * rows + 31) / 32 * 32; }

// Dynamic shared memory of k_radial_par, k_rhs_par.
__host__ inline size_t radial_par_smem(int Nr, int Nd) {
  return (size_t)par_pairs((Nd + 1) / 2) * (6 * (size_t)Nr + 14 * (size_t)Nd) * sizeof(double);
}
__host__ inline size_t rhs_par_smem(int Nr, int Nd, bool second, size_t real) {
  return (size_t)par_pairs((Nr + 1) / 2) *
         (((second ? 12 : 6) + 8 + (second ? 8 : 0)) * (size_t)Nr * sizeof(double) +
          8 * (size_t)Nr * real + 16 * (size_t)((Nd + 1) / 2) * real + 4 * sizeof(double));
}

// Rows j (S_e + S_o) and j' of a table with even (sg = 1) or odd (sg = -1) derivative order.
__device__ __forceinline__ void par_rows(double* z, int n, int j, double se, double so, double sg) {
  z[j] = se + so;
  z[n - 1 - j] = sg * (se - so);   // the middle row of an odd n is written twice: so (se) is zero
}

// SR[(p Nd + i) 8 + q] as k_radial.  grid = ceil(P / PPB), block = 2 TW: the threads of the first
// half sum real parts, of the second imaginary ones; thread l of a half = (pair l / NdH, row l % NdH).
__global__ void __launch_bounds__(320) k_radial_par(DevGeom g, ParTables pt, const double2* __restrict__ x,
                                                    double2* __restrict__ SR, int PPB) {
  grid_begin();
  extern __shared__ double pa_sh[];
  const int Nr = g.Nr, Nd = g.Nd, P = g.P, NH = (Nd + 1) / 2;
  double* xs = pa_sh;                       // [part][pl][f][k]
  double* zs = xs + 6 * PPB * Nr;           // [part][pl][7][Nd]: e0 e1 f0 f1 f2 T0 T1
  const int pb = blockIdx.x * PPB, np = min(PPB, P - pb);
  for (int idx = threadIdx.x; idx < np * 3 * Nr; idx += blockDim.x) {
    const int pl = idx / (3 * Nr), fk = idx - pl * 3 * Nr, f = fk / Nr, k = fk - f * Nr;
    const double2 v = x[((long)f * P + pb + pl) * Nr + k];
    xs[idx] = v.x;
    xs[3 * PPB * Nr + idx] = v.y;
  }
  __syncthreads();
  const int TW = blockDim.x >> 1, part = threadIdx.x >= TW ? 1 : 0;
  const int l = threadIdx.x - part * TW;
  const int pl = l / NH, ii = l - pl * NH;
  if (pl < np) {
    const double* e = xs + (part * PPB + pl) * 3 * Nr;
    const double *f = e + Nr, *T = f + Nr;
    double se[7] = {0, 0, 0, 0, 0, 0, 0}, so[7] = {0, 0, 0, 0, 0, 0, 0};
    auto step = [&](double (&s)[7], int k) {
      const double a0 = g.EdT0[k * Nd + ii], a1 = g.EdT1[k * Nd + ii], a2 = g.EdT2[k * Nd + ii];
      const double ek = e[k], fk = f[k], Tk = T[k];
      s[0] = fma(a0, ek, s[0]); s[1] = fma(a1, ek, s[1]);
      s[2] = fma(a0, fk, s[2]); s[3] = fma(a1, fk, s[3]); s[4] = fma(a2, fk, s[4]);
      s[5] = fma(a0, Tk, s[5]); s[6] = fma(a1, Tk, s[6]);
    };
    for (int k = 0; k + 1 < Nr; k += 2) {
      step(se, k);
      step(so, k + 1);
    }
    if (Nr & 1) step(se, Nr - 1);
    double* z = zs + (part * PPB + pl) * 7 * Nd;
#pragma unroll
    for (int q = 0; q < 7; ++q) par_rows(z + q * Nd, Nd, ii, se[q], so[q], (q == 1 || q == 3 || q == 6) ? -1.0 : 1.0);
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < np * Nd; idx += blockDim.x) {
    const int q = idx / Nd, i = idx - q * Nd;
    const double *zr = zs + q * 7 * Nd + i, *zi = zr + PPB * 7 * Nd;
    auto c = [&](int s) { return make_double2(zr[s * Nd], zi[s * Nd]); };
    const int lp = g.pair_l[pb + q];
    const double lam = lp * (lp + 1.0), ir = pt.ird[i], lr2 = lam * (ir * ir);
    auto sc = [](double a, double2 v) { return make_double2(a * v.x, a * v.y); };
    const double2 f0 = sc(lr2, c(2)), f2 = c(4);
    double2* o = SR + ((long)(pb + q) * Nd + i) * 8;
    o[0] = f0;                                                   // u_r
    o[1] = sc(ir, c(3));                                         // S_u
    o[2] = sc(ir, c(0));                                         // T_u
    o[3] = sc(lr2, c(0));                                        // omega_r
    o[4] = sc(ir, c(1));                                         // S_w
    o[5] = make_double2(-(f2.x - f0.x) * ir, -(f2.y - f0.y) * ir);   // T_w
    o[6] = c(6);                                                 // d_r T
    o[7] = sc(ir, c(5));                                         // S_T
  }
}

// The right-hand side with the Coriolis terms implicit, as k_rhs (modes 0, 1, 2, 3 of RhsParams):
// projections in precision R, everything else FP64.  U2: the base state (drift term of mode 1), the
// state of the linear explicit terms (mode 3 when it is not x), else null.
// grid = ceil(P / PPB), block = NT TW, task t = thread / TW: 0, 1 the mass products of x (real,
// imaginary parts), 2, 3 the projections, 4, 5 the mass products of U2 (NT = 6).
template <typename R>
__global__ void __launch_bounds__(960) k_rhs_par(DevGeom g, RhsParams rp, ParTables pt,
                                                 const typename C2<R>::T* __restrict__ AR,
                                                 const double2* __restrict__ x, const double2* __restrict__ U2,
                                                 const double* __restrict__ u_orig, double2* __restrict__ rhs,
                                                 int PPB, int TW) {
  grid_begin();
  using V = typename C2<R>::T;
  extern __shared__ double pa_sh[];
  const int Nr = g.Nr, Nd = g.Nd, P = g.P, NH = (Nr + 1) / 2, DH = (Nd + 1) / 2;
  const int nv = U2 ? 2 : 1;                 // vectors with mass products
  double* xs = pa_sh;                        // [vector][part][pl][f][k]
  double* zm = xs + nv * 6 * PPB * Nr;       // [vector][part][pl][e0 f0 f2 T0][j]
  R* zp = reinterpret_cast<R*>(zm + nv * 8 * PPB * Nr);   // [part][pl][Q T N dS][j]
  R* fold = zp + 8 * PPB * Nr;               // [part][pl][+/-][Q T N S][i]
  const int pb = blockIdx.x * PPB, np = min(PPB, P - pb);
  for (int idx = threadIdx.x; idx < nv * np * 3 * Nr; idx += blockDim.x) {
    const int v = idx / (np * 3 * Nr), r = idx - v * np * 3 * Nr;
    const int pl = r / (3 * Nr), fk = r - pl * 3 * Nr, f = fk / Nr, k = fk - f * Nr;
    const double2 z = (v ? U2 : x)[((long)f * P + pb + pl) * Nr + k];
    double* o = xs + v * 6 * PPB * Nr + r;
    o[0] = z.x;
    o[3 * PPB * Nr] = z.y;
  }
  const R* rdv = Tab<R>::rd(g);
  for (int idx = threadIdx.x; idx < np * DH * 4; idx += blockDim.x) {
    const int pl = idx / (DH * 4), r = idx - pl * DH * 4, i = r >> 2, c = r & 3;   // c: Q S T N
    const int im = Nd - 1 - i;
    const V* src = AR + (long)(pb + pl) * Nd * 4 + c;
    V a = src[i * 4], b = src[im * 4];
    if (c == 1) {   // r S, whose derivative is projected
      a = mk<R>(a.x * rdv[i], a.y * rdv[i]);
      b = mk<R>(b.x * rdv[im], b.y * rdv[im]);
    }
    if (im == i) b = mk<R>(0, 0);
    const int s = c == 0 ? 0 : c == 1 ? 3 : c - 1;
    R* o = fold + (pl * 8 + s) * DH + i;
    o[0] = a.x + b.x;
    o[4 * DH] = a.x - b.x;
    o += PPB * 8 * DH;
    o[0] = a.y + b.y;
    o[4 * DH] = a.y - b.y;
  }
  __syncthreads();
  const int task = threadIdx.x / TW, l = threadIdx.x - task * TW;
  const int pl = l / NH, jj = l - pl * NH, part = task & 1;
  if (pl < np && task != 2 && task != 3) {
    const int v = task >= 4 ? 1 : 0;
    const double* e = xs + ((v * 2 + part) * PPB + pl) * 3 * Nr;
    const double *f = e + Nr, *T = f + Nr;
    double se[4] = {0, 0, 0, 0}, so[4] = {0, 0, 0, 0};
    auto step = [&](double (&s)[4], int k) {
      const double c0 = g.EcT0[k * Nr + jj], c2 = g.EcT2[k * Nr + jj], fk = f[k];
      s[0] = fma(c0, e[k], s[0]);
      s[1] = fma(c0, fk, s[1]);
      s[2] = fma(c2, fk, s[2]);
      s[3] = fma(c0, T[k], s[3]);
    };
    for (int k = 0; k + 1 < Nr; k += 2) {
      step(se, k);
      step(so, k + 1);
    }
    if (Nr & 1) step(se, Nr - 1);
    double* z = zm + ((v * 2 + part) * PPB + pl) * 4 * Nr;
#pragma unroll
    for (int q = 0; q < 4; ++q) par_rows(z + q * Nr, Nr, jj, se[q], so[q], 1.0);
  } else if (pl < np) {
    const R* ap = fold + (part * PPB + pl) * 8 * DH;
    const R *P0 = ParTab<R>::P0(pt), *M0 = ParTab<R>::M0(pt), *P1 = ParTab<R>::P1(pt), *M1 = ParTab<R>::M1(pt);
    R sp[4] = {0, 0, 0, 0}, sm[4] = {0, 0, 0, 0};
    for (int i = 0; i < DH; ++i) {
      const R p0 = P0[i * NH + jj], m0 = M0[i * NH + jj], p1 = P1[i * NH + jj], m1 = M1[i * NH + jj];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        sp[q] += (q == 3 ? p1 : p0) * ap[q * DH + i];
        sm[q] += (q == 3 ? m1 : m0) * ap[(4 + q) * DH + i];
      }
    }
    R* z = zp + (part * PPB + pl) * 4 * Nr;
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // dS has an odd derivative: the signs of row j' swap
      z[q * Nr + jj] = sp[q] + sm[q];
      z[q * Nr + Nr - 1 - jj] = q == 3 ? sm[q] - sp[q] : sp[q] - sm[q];
    }
  }
  // mode 3: d_r f at the walls from x, sum_k (+-1)^(k+1) k^2 f_k dx/dr (one warp per pair)
  double* wall = reinterpret_cast<double*>(fold + 16 * PPB * DH);   // [pl][r_out, r_in][part]
  if (rp.mode == 3) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int q = warp; q < np; q += nw) {
#pragma unroll
      for (int pt2 = 0; pt2 < 2; ++pt2) {
        const double* f = xs + ((pt2 * PPB + q) * 3 + 1) * Nr;
        double a = 0.0, b = 0.0;
        for (int k = lane; k < Nr; k += 32) {
          a = fma(g.EcT1[k * Nr], f[k], a);
          b = fma(g.EcT1[k * Nr + Nr - 1], f[k], b);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          a += __shfl_xor_sync(0xffffffffu, a, o);
          b += __shfl_xor_sync(0xffffffffu, b, o);
        }
        if (lane == 0) {
          wall[q * 4 + pt2] = a;
          wall[q * 4 + 2 + pt2] = b;
        }
      }
    }
  }
  __syncthreads();
  const double cdrift = rp.J >= 0 ? u_orig[rp.J] : 0.0;
  for (int idx = threadIdx.x; idx < np * Nr; idx += blockDim.x) {
    const int q = idx / Nr, j = idx - q * Nr, p = pb + q;
    const int lp = g.pair_l[p], m = g.pair_m[p];
    const double lam = lp * (lp + 1.0), ir = pt.irc[j], ir2 = ir * ir;
    auto zc = [&](int v, int s) {
      const double* z = zm + (v * 2 * PPB + q) * 4 * Nr + s * Nr + j;
      return make_double2(z[0], z[4 * PPB * Nr]);
    };
    auto pc = [&](int s) {
      const R* z = zp + q * 4 * Nr + s * Nr + j;
      return make_double2((double)z[0], (double)z[4 * PPB * Nr]);
    };
    const double ce = lam * rp.Ek * ir2, lr2 = lam * ir2;
    auto mass = [&](int v, double2 (&o)[3]) {
      const double2 e0 = zc(v, 0), f0 = zc(v, 1), f2 = zc(v, 2);
      o[0] = make_double2(ce * e0.x, ce * e0.y);
      o[1] = make_double2(-ce * (f2.x - lr2 * f0.x), -ce * (f2.y - lr2 * f0.y));
      o[2] = zc(v, 3);
    };
    const double2 Qc = pc(0), Tc = pc(1), Nc = pc(2), dS = pc(3);
    const double2 MT = zc(rp.mode == 3 && U2 ? 1 : 0, 3);   // temperature whose buoyancy enters
    const double cb = lam * ir * pt.Ra_rout, lr = lam * ir;
    double2 o[3] = {make_double2(lr * Tc.x, lr * Tc.y),
                    make_double2(lr2 * (Qc.x - dS.x) + cb * MT.x, lr2 * (Qc.y - dS.y) + cb * MT.y),
                    make_double2(-Nc.x, -Nc.y)};
    if (rp.mode != 2) {
      const double fr = rp.inv_dt, fi = rp.C * m;   // (1/dt + i C m) M x
      double2 M[3];
      mass(0, M);
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        o[f].x += fr * M[f].x - fi * M[f].y;
        o[f].y += fr * M[f].y + fi * M[f].x;
      }
      if (rp.J >= 0) {
        double2 Mu[3];
        mass(1, Mu);
        const double cmv = cdrift * m;              // c i m M U
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          o[f].x -= cmv * Mu[f].y;
          o[f].y += cmv * Mu[f].x;
        }
      }
      // boundary rows (Sec. 3.1) and identity rows of e_00, f_00
      const bool w0 = j == 0 || j == Nr - 1, w1 = j == 1 || j == Nr - 2;
      if (w0) o[0] = o[2] = make_double2(0, 0);
      if (w0 || w1) o[1] = make_double2(0, 0);
      if ((rp.mode == 0 || rp.mode == 3) && lp == 0 && j == Nr - 1) o[2] = make_double2(1.0, 0.0);   // T(r_in) = 1
      if (lp == 0) o[0] = o[1] = make_double2(0, 0);
      if (rp.mode == 3) {   // boundary rows (bc + B x) / 2 of the half step
        auto half = [](double2 a, double2 b) { return make_double2(0.5 * (a.x + b.x), 0.5 * (a.y + b.y)); };
        if (w0) {
          o[0] = half(o[0], zc(0, 0));
          o[1] = half(o[1], zc(0, 1));
          o[2] = half(o[2], zc(0, 3));
        }
        if (w1) {
          const double* wl = wall + q * 4 + (j == 1 ? 0 : 2);
          o[1] = half(o[1], make_double2(wl[0], wl[1]));
        }
        if (lp == 0) {      // identity rows of e_00, f_00: y = x / 2 keeps them at zero
          const double* xr = xs + q * 3 * Nr + j;
          o[0] = make_double2(0.5 * xr[0], 0.5 * xr[3 * PPB * Nr]);
          o[1] = make_double2(0.5 * xr[Nr], 0.5 * xr[3 * PPB * Nr + Nr]);
        }
      }
      if (m == 0) o[0].y = o[1].y = o[2].y = 0;
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) rhs[((long)f * P + p) * Nr + j] = o[f];
  }
}

}  // namespace rsc
