// The passes of chain_cr.cuh in FP64, for the FP64 chain solve on odd-even reduced chains: the same
// blocks, couplings and order, factors and tables FP64 (double2 per complex entry).
//
// What bounds it: the FP64 pipe, one warp instruction in 64 cycles per SM quarter whatever its active
// lanes.  Hence four lanes per row instead of eight (two steps of reduction, in each of which a lane
// passes on what it does not keep: 2 FP64 additions per 64 multiply-adds at N_r = 64), both rows
// of a pair j, N_r - 1 - j from one pair of table sums, and factors, never divisions, in the rows.
// Measured (one GB300): mean of the three passes 41 us at L = 127, M_s = 12, N_r = 64 (the FP64 pipe 82 %
// active), 377 us at L = 255, M_s = 8, N_r = 96; a sweep over every second block 63 us (115 over
// all, L = 127).  Unreduced -> reduced chains: two FP64 steps at L = 127 3851 -> 3638 us, one at L = 255
// 20186 -> 19738, ten monitored ones at L = 31 2548 -> 2280, a refined solve at L = 45, M_s = 5, N_r = 37
// 270 -> 196 us.
// Grid of each kernel: 2 CTAs (e and f block) per pair (m, l) of the given parity of l - m, 256 threads.
#pragma once

#include "chain_cr.cuh"
#include "factor_gpu.cuh"

namespace rsc {

__device__ __forceinline__ double cr_flip(double x, bool neg) {   // no FP64 instruction
  return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}

__device__ __forceinline__ void cr_prefetch(const double2* M, int Nr) {
  cr_prefetch(reinterpret_cast<const float4*>(M), Nr);
}

// y = M v for one Nr x Nr block M (row-major), v in shared memory, y in shared or global memory and not
// v.  A lane's columns are s + 4 q.
__device__ __forceinline__ void cr_gemv(const double2* __restrict__ M, const double2* v, int Nr,
                                        bool real_op, double2* y) {
  constexpr int QC = 4;
  const int s = threadIdx.x & 3, rows = blockDim.x >> 2;
  for (int r0 = 0; r0 < Nr; r0 += rows) {
    const int r = r0 + (threadIdx.x >> 2);
    if (r0 + ((threadIdx.x & ~31) >> 2) >= Nr) break;   // no row for this warp
    const double2* Mr = M + (long)r * Nr;
    double re = 0.0, im = 0.0, re1 = 0.0, im1 = 0.0;
#pragma unroll 1
    for (int k0 = s; k0 - s < Nr; k0 += 4 * QC) {
      double2 a[QC];
#pragma unroll
      for (int q = 0; q < QC; ++q) {
        const int k = k0 + 4 * q;
        a[q] = r < Nr && k < Nr ? Mr[k] : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int q = 0; q < QC; ++q) {
        if (k0 - s + 4 * q >= Nr) break;   // the same for the whole warp
        const int k = k0 + 4 * q;
        const double2 x = k < Nr ? v[k] : make_double2(0.0, 0.0);
        re = fma(a[q].x, x.x, re);
        im = fma(a[q].x, x.y, im);
        if (!real_op) {
          re1 = fma(a[q].y, x.y, re1);
          im1 = fma(a[q].y, x.x, im1);
        }
      }
    }
    if (!real_op) {
      re -= re1;
      im += im1;
    }
    const bool odd = s & 1;
    double t = odd ? im : re;
    t += __shfl_xor_sync(0xffffffffu, odd ? re : im, 1);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    if (r < Nr && s < 2) reinterpret_cast<double*>(y)[2 * r + s] = t;
  }
}

// (E0 v0)_j and (E1 v1)_j for every row j (E01[j][k] = {E0, E1}); as cr_e01 of chain_cr.cuh.
__device__ __forceinline__ void cr_e01(const double2* __restrict__ E01, const double2* v0,
                                       const double2* v1, int Nr, double2* e0, double2* e1) {
  constexpr int QC = 4;
  const int s = threadIdx.x & 3, rows = blockDim.x >> 2, NH = (Nr + 1) >> 1;
  for (int r0 = 0; r0 < NH; r0 += rows) {
    const int j = r0 + (threadIdx.x >> 2);
    if (r0 + ((threadIdx.x & ~31) >> 2) >= NH) break;
    const double2* Ej = E01 + (long)j * Nr;
    double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
#pragma unroll 1
    for (int k0 = s; k0 - s < Nr; k0 += 4 * QC) {
      double2 e[QC];
#pragma unroll
      for (int q = 0; q < QC; ++q) {
        const int k = k0 + 4 * q;
        e[q] = j < NH && k < Nr ? Ej[k] : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int q = 0; q < QC; ++q) {
        if (k0 - s + 4 * q >= Nr) break;
        const int k = k0 + 4 * q;
        const bool in = k < Nr;
        const double2 x = in ? v0[k] : make_double2(0.0, 0.0), y = in ? v1[k] : make_double2(0.0, 0.0);
        a = fma(e[q].x, x.x, a);
        b = fma(e[q].x, x.y, b);
        c = fma(e[q].y, y.x, c);
        d = fma(e[q].y, y.y, d);
      }
    }
    // lanes 0, 1 keep E0 v0 (even and odd columns), lanes 2, 3 E1 v1; then the even lane joins row j
    // (even + odd), the odd one row Nr - 1 - j (even - odd of E0, odd - even of E1)
    const bool hi = s & 2, odd = s & 1;
    double p = hi ? c : a, q = hi ? d : b;
    p += __shfl_xor_sync(0xffffffffu, hi ? a : c, 2);
    q += __shfl_xor_sync(0xffffffffu, hi ? b : d, 2);
    const double po = __shfl_xor_sync(0xffffffffu, p, 1), qo = __shfl_xor_sync(0xffffffffu, q, 1);
    p = cr_flip(p, odd && !hi) + cr_flip(po, odd && hi);
    q = cr_flip(q, odd && !hi) + cr_flip(qo, odd && hi);
    const int row = odd ? Nr - 1 - j : j;
    if (j < NH && !(odd && row == j)) (hi ? e1 : e0)[row] = make_double2(p, q);
  }
}

// (re, im) += k v
__device__ __forceinline__ void cr_axpy(double2& z, double k, double2 v) {
  z.x = fma(k, v.x, z.x);
  z.y = fma(k, v.y, z.y);
}

// Odd blocks, first pass: u = D^-1 b, then w0 = E0 u and w1 = E1 u (w: [2][2 P Nr]).
// Dynamic shared memory: 2 Nr double2.
__global__ void __launch_bounds__(256, 5) k_cr_odd(DevGeom g, const int* __restrict__ odd_pairs,
                                                   const long* __restrict__ odd_off,
                                                   const double2* __restrict__ Dinv,
                                                   const double2* __restrict__ E01,
                                                   const double2* __restrict__ rhs,
                                                   double2* __restrict__ w) {
  extern __shared__ double2 cr64_sh[];
  const int Nr = g.Nr;
  const CrBlock b = cr_block(g, odd_pairs);
  const double2* Di = Dinv + (odd_off[b.c] + (b.i >> 1)) * (long)Nr * Nr;
  cr_prefetch(Di, Nr);
  grid_begin();
  double2* sb = cr64_sh;
  double2* su = cr64_sh + Nr;
  for (int k = threadIdx.x; k < Nr; k += blockDim.x) sb[k] = rhs[b.row0 + k];
  __syncthreads();
  cr_gemv(Di, sb, Nr, b.m == 0, su);
  __syncthreads();
  cr_e01(E01, su, su, Nr, w + b.row0, w + 2L * g.P * Nr + b.row0);
}

// Even blocks: b' = b - A u_{i-1} - C u_{i+1} from the neighbours' w, then g' = G' b' into out.
// Dynamic shared memory: Nr double2.
__global__ void __launch_bounds__(256, 5) k_cr_even(DevGeom g, const int* __restrict__ even_pairs,
                                                    const long* __restrict__ red_off,
                                                    const double2* __restrict__ Gr,
                                                    const double2* __restrict__ rowf,
                                                    const CrPair* __restrict__ pairf,
                                                    const double2* __restrict__ rhs,
                                                    const double2* __restrict__ w,
                                                    double2* __restrict__ out) {
  extern __shared__ double2 cr64_sh[];
  const int Nr = g.Nr;
  const CrBlock b = cr_block(g, even_pairs);
  const double2* Gt = Gr + (red_off[b.c] + (b.i >> 1)) * (long)Nr * Nr;
  cr_prefetch(Gt, Nr);
  grid_begin();
  double2* sb = cr64_sh;
  const long half = 2L * g.P * Nr;
  const bool left = b.i >= 1, right = b.i + 1 <= b.nb - 1;
  const long rowL = ((long)(1 - b.fld) * g.P + b.p - 1) * Nr;
  const long rowR = ((long)(1 - b.fld) * g.P + b.p + 1) * Nr;
  const CrPair pf = pairf[b.p];
  for (int j = threadIdx.x; j < Nr; j += blockDim.x) {
    double2 z = rhs[b.row0 + j];
    if (cr_coupled_row(b.fld, j, Nr) && b.l > 0) {
      const double2 rf = rowf[j];
      if (left) {   // - A u_{i-1} = -(s ir a l) E0 u + (s a) E1 u
        cr_axpy(z, -(rf.x * pf.x), w[rowL + j]);
        cr_axpy(z, rf.y * pf.y, w[half + rowL + j]);
      }
      if (right) {  // - C u_{i+1} = (s ir c (l+1)) E0 u + (s c) E1 u
        cr_axpy(z, rf.x * pf.z, w[rowR + j]);
        cr_axpy(z, rf.y * pf.w, w[half + rowR + j]);
      }
    }
    sb[j] = z;
  }
  __syncthreads();
  cr_gemv(Gt, sb, Nr, b.m == 0, out + b.row0);
}

// Odd blocks, last pass: x_i = D^-1 (b - A x_{i-1} - C x_{i+1}), A x_{i-1} + C x_{i+1} = s ir E0 y0 - s E1 y1
// as in k_cr_back_df.  Dynamic shared memory: 4 Nr double2.
__global__ void __launch_bounds__(256, 5) k_cr_back(DevGeom g, const int* __restrict__ odd_pairs,
                                                    const long* __restrict__ odd_off,
                                                    const double2* __restrict__ Dinv,
                                                    const double2* __restrict__ E01,
                                                    const double2* __restrict__ rowf,
                                                    const CrPair* __restrict__ pairf,
                                                    const double2* __restrict__ rhs,
                                                    double2* __restrict__ out) {
  extern __shared__ double2 cr64_sh[];
  const int Nr = g.Nr;
  const CrBlock b = cr_block(g, odd_pairs);
  const double2* Di = Dinv + (odd_off[b.c] + (b.i >> 1)) * (long)Nr * Nr;
  cr_prefetch(Di, Nr);
  grid_begin();
  double2* y0 = cr64_sh;
  double2* y1 = cr64_sh + Nr;
  double2* e0 = cr64_sh + 2 * Nr;
  double2* e1 = cr64_sh + 3 * Nr;
  const bool right = b.i + 1 <= b.nb - 1;
  const long rowL = ((long)(1 - b.fld) * g.P + b.p - 1) * Nr;
  const long rowR = ((long)(1 - b.fld) * g.P + b.p + 1) * Nr;
  const CrPair pf = pairf[b.p];
  for (int k = threadIdx.x; k < Nr; k += blockDim.x) {
    const double2 xl = out[rowL + k];
    double2 a = make_double2(pf.x * xl.x, pf.x * xl.y), c = make_double2(pf.y * xl.x, pf.y * xl.y);
    if (right) {
      const double2 xr = out[rowR + k];
      cr_axpy(a, -pf.z, xr);
      cr_axpy(c, pf.w, xr);
    }
    y0[k] = a;
    y1[k] = c;
  }
  __syncthreads();
  cr_e01(E01, y0, y1, Nr, e0, e1);
  __syncthreads();
  for (int j = threadIdx.x; j < Nr; j += blockDim.x) {
    double2 z = rhs[b.row0 + j];
    if (cr_coupled_row(b.fld, j, Nr)) {   // - s ir E0 y0 + s E1 y1
      const double2 rf = rowf[j];
      cr_axpy(z, -rf.x, e0[j]);
      cr_axpy(z, rf.y, e1[j]);
    }
    y0[j] = z;
  }
  __syncthreads();
  cr_gemv(Di, y0, Nr, b.m == 0, out + b.row0);
}

}  // namespace rsc
