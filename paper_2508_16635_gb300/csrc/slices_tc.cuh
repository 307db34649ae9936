// FP64 matrix products on the BF16 tensor cores, exactly: the Legendre synthesis and analysis of
// the FP64 path (Sec. 3.1 transforms).
//
// Splitting (Ozaki, Ogita, Oishi, Rumpf, "Error-free transformations of matrix multiplication",
// Numer. Algorithms 59, 2012, with a fixed grid of digits): a row of the table and a column of the
// data are scaled by powers of two to |x| < 1 and cut into kSl = 7 digits base 256,
//     x = 2^e sum_i d_i 2^(-7-8i),   d_i an integer in [-128, 128],
// 55 bits after the binary point.  Every digit is exact in BF16, a product of two digits is an
// integer of at most 14 bits, and a sum over K <= 128 terms and up to 7 digit pairs stays below 2^24,
// so the FP32 accumulators hold the sums of each diagonal i + j = d exactly whatever their order.
// The diagonals d <= 6 are kept (28 of 49 digit products); the rest weighs less than 2^-55 of
// (row maximum)(column maximum) per term.  The seven sums are joined in 64-bit integers and rounded once
// to FP64.  Measured on the tables of L = 127 against 64-digit sums: 0.4 to 0.9 of the error of
// an FP64 loop over the degrees.
//
// Why: GB300 does 1.26 TFLOP/s of FP64 and 2 PFLOP/s of BF16; 28 digit products cost 1/60 of the
// FP64 sums.  What is left on the FP64 pipe is the combination i m X + Y of the vector fields.
// All digit slices of the data lie side by side along N, so one MMA multiplies slice i of the table
// with slices 0 .. 6 - i of the data and adds them onto the diagonals i .. 6 (7 MMAs per 16 terms).
//
// A CTA: epilogue warps (TMEM lane = row, warpgroup = radius) also cut the data into digits; one
// thread of a warp of its own copies table digits through a ring of stages, one of another issues
// the MMAs (in one thread, and with the descriptors built for every MMA, its instruction latency
// took 1900 cycles per step against 450 at the tensor rate); the accumulators of the phases (table
// type, parity) alternate between tensor-memory buffers, so the MMAs of a phase run under the
// epilogue of the one before.
// A column with an infinity or NaN gives NaN.  All waits are bounded; a wait that gives up sets
// *status and everything in flight is waited for before the tensor memory is freed.
// Measured (us per launch, one GB300, sums on the FP64 pipe before -> this): synthesis 500 -> 75 at
// L = 127, M_s = 12, N_r = 64 and 6175 -> 700 at L = 255, M_s = 8, N_r = 96; analysis 447 -> 60 and
// 5015 -> 404.  At L = 127 a CTA of the synthesis (m = 0) spends 6.5 of 52 thousand cycles on the
// digits of P, 5 on those of the vector types, the MMAs run underneath (950 per step: a 128-row
// MMA takes 135 cycles however few its columns), and 38 on reading, joining and combining the sums.
#pragma once

#include <stdint.h>

#include "kernels.cuh"
#include "legendre_tc.cuh"

namespace rsc {

constexpr int kSl = 7;                        // digits
constexpr int kSlStage = kSl * 128 * 32;      // bytes of a 16-term step of a full table tile
constexpr int kSlNaN = 0x40000000;            // exponent mark of a column that holds Inf or NaN

// x = v 2^(eb - 55) rounded to the nearest integer v; needs |x| < 2^eb (|v| <= 2^55).
__device__ __forceinline__ long long sl_fixed(double x, int eb) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7FF;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const int sh = e - 1020 - eb;               // at most 2
  unsigned long long v = 0;
  if (e != 0) {
    if (sh >= 0)
      v = m << min(sh, 2);
    else if (sh >= -54)
      v = (m + (1ull << (-sh - 1))) >> (-sh);
  }
  return (b >> 63) ? -(long long)v : (long long)v;
}

// The smallest exponent eb with |x| < 2^eb for every x whose largest exponent field is ef.
__device__ __forceinline__ int sl_exponent(int ef) { return ef == 0x7FF ? kSlNaN : ef ? ef - 1022 : 0; }

__device__ __forceinline__ int sl_field(double x) {
  return (int)((unsigned)__double2hiint(x) >> 20) & 0x7FF;
}

// Digit i (0 = highest) of v as a BF16 in the upper half of the result: v plus 128 in every digit
// place has non-negative bytes, 2^23 + byte - (2^23 + 128) is exact.
__device__ __forceinline__ uint32_t sl_digit(unsigned long long biased, int i) {
  const uint32_t t = i == 0 ? (uint32_t)(biased >> 48) : (uint32_t)(biased >> (48 - 8 * i)) & 0xFFu;
  return __float_as_uint(__uint_as_float(0x4B000000u | (t & 0x1FFu)) - 8388736.0f);
}

// The seven slices of eight consecutive terms of one row / column: 16 bytes each.
__device__ __forceinline__ void sl_store8(unsigned char* dst, int slice_stride, const long long (&v)[8]) {
  unsigned long long b[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) b[u] = (unsigned long long)(v[u] + 0x0080808080808080ll);
#pragma unroll
  for (int i = 0; i < kSl; ++i) {
    uint32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      w[u] = __byte_perm(sl_digit(b[2 * u], i), sl_digit(b[2 * u + 1], i), 0x7632);
    *reinterpret_cast<uint4*>(dst + (long)i * slice_stride) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// acc 2^e as a double, rounded to nearest (ties away); magnitudes below the normal range give 0.
// (A call: expanded at its 50 places in the synthesis epilogue, the code missed the instruction
// cache, 14000 cycles per vector phase.)
__device__ __noinline__ double sl_join(long long acc, int e) {
  if (acc == 0) return 0.0;
  const unsigned long long sg = (unsigned long long)acc & 0x8000000000000000ull;
  unsigned long long u = acc < 0 ? (unsigned long long)(-acc) : (unsigned long long)acc;
  const int lz = __clzll((long long)u);
  u = (u << lz) + 0x400ull;
  int ex = 63 - lz + e + 1023;
  if (u < 0x400ull) {                         // rounded up to the next power of two
    u = 0x8000000000000000ull;
    ex += 1;
  }
  if (ex < 1) return 0.0;
  if (ex > 2046) return __longlong_as_double((long long)(sg | 0x7FF0000000000000ull));
  return __longlong_as_double((long long)(sg | (((unsigned long long)(ex - 1) << 52) + (u >> 11))));
}

// Join of the seven diagonal sums (exact integers): units of 2^-40 of the first.
__device__ __forceinline__ long long sl_sum(const float (&d)[kSl]) {
  long long a = (long long)__float2int_rn(d[0]) * (1ll << 40);
#pragma unroll
  for (int i = 1; i < kSl - 1; ++i) a += (long long)__float2int_rn(d[i]) * (1ll << (40 - 8 * i));
  return a + ((__float2int_rn(d[kSl - 1]) + 128) >> 8);
}
// Exponent of sl_sum's unit for row and column exponents ea, eb.
__device__ __forceinline__ int sl_unit(int ea, int eb) { return ea + eb - 54; }

// kind::f16 instruction descriptor: D = F32, A = B = BF16, both K-major, M = 128.
__device__ __forceinline__ uint32_t sl_idesc(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
}

__device__ __forceinline__ void sl_mma(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void sl_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

__device__ __forceinline__ void sl_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

template <int X>
__device__ __forceinline__ void sl_ld(uint32_t taddr, float (&v)[X]);
template <>
__device__ __forceinline__ void sl_ld<2>(uint32_t taddr, float (&v)[2]) { tc_ld<2>(taddr, v); }
template <>
__device__ __forceinline__ void sl_ld<4>(uint32_t taddr, float (&v)[4]) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = __uint_as_float(r[q]);
}

// The joined sums of X columns from column c of an accumulator of NC columns per diagonal.
template <int X, int NC>
__device__ __forceinline__ void sl_read(uint32_t taddr, int c, long long (&o)[X]) {
  float d[kSl][X];
#pragma unroll
  for (int i = 0; i < kSl; ++i) sl_ld<X>(taddr + i * NC + c, d[i]);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int q = 0; q < X; ++q) {
    float e[kSl];
#pragma unroll
    for (int i = 0; i < kSl; ++i) e[i] = d[i][q];
    o[q] = sl_sum(e);
  }
}

// Table digits.  Tile of (m index, parity s, type w, row tile t): per 16-term step, seven slices of
// G groups of 8 rows, each group two 128-byte core matrices (8 rows x 8 terms, K-major, no swizzle).
struct SlTables {
  const unsigned char* tiles;
  const long* off;    // byte offset of tile ((a 2 + s) 3 + w) nt + t
  const int* ea;      // row exponents (see the kernels)
  int nt;             // row tiles of 128
  int ksmax;          // largest number of 16-term steps
  int* status;
};

// Row exponents: ea[row] with |table| < 2^ea over the row.  Synthesis (ANAL = false): rows are
// the north latitudes, ea[(a 3 + w) n2 + t] over every degree of m (both parities); table layout
// [q][t].  Analysis: rows are the degrees, ea[(a 3 + w)(L + 1) + q] over the latitudes; layout [t][q].
// grid = (nm, 3), block = 256.
template <bool ANAL>
__global__ void k_slice_exponents(DevGeom g, const double* __restrict__ T0, const double* __restrict__ T1,
                                  const double* __restrict__ T2, int* __restrict__ ea) {
  const int a = blockIdx.x, w = blockIdx.y;
  const double* T = (w == 0 ? T0 : w == 1 ? T1 : T2) + g.leg_off[a];
  const int nl = g.L - g.m_of[a] + 1, n2 = g.nlat2;
  const int rows = ANAL ? nl : n2, cols = ANAL ? n2 : nl;
  for (int r = threadIdx.x; r < rows; r += blockDim.x) {
    int ef = 0;
    for (int k = 0; k < cols; ++k) ef = max(ef, sl_field(T[(long)k * rows + r]));
    ea[(a * 3 + w) * (ANAL ? g.L + 1 : n2) + r] = sl_exponent(ef);
  }
}

// The tiles.  grid = (nm 2 3, nt), block = 256; terms past the last are zero digits.
template <bool ANAL>
__global__ void k_slice_tables(DevGeom g, const double* __restrict__ T0, const double* __restrict__ T1,
                               const double* __restrict__ T2, SlTables tt, unsigned char* __restrict__ tiles) {
  const int w = blockIdx.x % 3, s = (blockIdx.x / 3) & 1, a = blockIdx.x / 6, t = blockIdx.y;
  const double* T = (w == 0 ? T0 : w == 1 ? T1 : T2) + g.leg_off[a];
  const int nl = g.L - g.m_of[a] + 1, n2 = g.nlat2;
  const int deg = (nl - s + 1) / 2;
  const int nrow = ANAL ? deg : n2, nk = ANAL ? n2 : deg;
  const int rows = min(128, nrow - 128 * t), G = (rows + 7) / 8, ks = (nk + 15) / 16;
  if (rows <= 0) return;
  unsigned char* dst = tiles + tt.off[((a * 2 + s) * 3 + w) * tt.nt + t];
  const int* ea = tt.ea + (a * 3 + w) * (ANAL ? g.L + 1 : n2);
  for (int idx = threadIdx.x; idx < G * 8 * ks * 2; idx += blockDim.x) {
    const int r = idx % (G * 8), ko = idx / (G * 8);     // row, octet of terms
    const int row = t * 128 + r;
    long long v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = ko * 8 + u;
      double x = 0.0;
      int e = 0;
      if (r < rows && k < nk) {
        x = ANAL ? T[(long)k * nl + s + 2 * row] : T[(long)(s + 2 * k) * n2 + row];
        e = ea[ANAL ? s + 2 * row : row];
      }
      v[u] = sl_fixed(x, e);
    }
    sl_store8(dst + (long)(ko >> 1) * (kSl * G * 256) + (r >> 3) * 256 + (ko & 1) * 128 + (r & 7) * 16,
              G * 256, v);
  }
}

// Bounded wait that also ends when another thread of the CTA has given up (*fail).
__device__ __forceinline__ bool sl_wait(uint32_t bar, uint32_t parity, volatile int* fail) {
  for (int it = 0; it < (1 << 14); ++it) {
    uint32_t done = 0;
    for (int q = 0; q < (1 << 10) && !done; ++q)
      asm volatile(
          "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(done)
          : "r"(bar), "r"(parity)
          : "memory");
    if (done) return true;
    if (*fail) return false;
  }
  *fail = 1;
  return false;
}

// Barriers of a CTA (shared memory): ring stages, accumulator buffers.
struct SlBars {
  uint32_t full, empty, tfull, tempty, drain;   // addresses; 8 bytes per barrier
  volatile int* fail;
};

// One thread copies the table steps: phase p has ks(p) steps of seven slices of G(p) row groups
// from src(p).  Ends when its copies have arrived (also after a failure).
template <class GR, class KS, class SRC>
__device__ __forceinline__ void sl_copy(const SlBars& sb, int nphase, int nst, uint32_t ring, GR G, KS ks,
                                        SRC src) {
  int st = 0, n = 0;
  uint32_t par = 1;                // a fresh barrier counts as the end of parity 1
  bool ok = true;
  for (int p = 0; p < nphase && ok; ++p) {
    const int steps = ks(p);
    if (steps == 0) continue;
    const uint32_t bytes = (uint32_t)(kSl * G(p) * 256);
    const unsigned char* from = src(p);
    for (int k = 0; k < steps; ++k, from += bytes) {
      ok = sl_wait(sb.empty + 8 * st, par, sb.fail);
      if (!ok) break;
      const uint32_t bar = sb.full + 8 * st;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              ring + (uint32_t)st * kSlStage),
          "l"(from), "r"(bytes), "r"(bar)
          : "memory");
      ++n;
      if (++st == nst) {
        st = 0;
        par ^= 1u;
      }
    }
  }
  // the last copy of every stage used has arrived (bounded, whatever the others do)
  for (int q = 0; q < min(n, nst); ++q) {
    if (--st < 0) {
      st = nst - 1;
      par ^= 1u;
    }
    tc_wait(sb.full + 8 * st, par ^ 1u);
  }
}

// One thread issues the MMAs: data digits of phase p at shared address b(p) (steps of kSl NC 32
// bytes), accumulator in buffer p % NB (stride BC columns); before(p) runs before its first MMA.
template <int NC, int NB, int BC, class GR, class KS, class BA, class BEFORE>
__device__ __forceinline__ bool sl_issue(const SlBars& sb, int nphase, int nst, uint32_t ring, uint32_t tmem,
                                         GR G, KS ks, BA b, BEFORE before) {
  int st = 0;
  uint32_t par = 0;
  bool ok = true;
  for (int p = 0; p < nphase && ok; ++p) {
    const int buf = p % NB, steps = ks(p);
    if (p >= NB) ok = sl_wait(sb.tempty + 8 * buf, (uint32_t)((p / NB - 1) & 1), sb.fail);
    if (ok) ok = before(p);
    if (!ok) break;
    const uint32_t d = tmem + buf * BC;
    const uint64_t slice = (uint64_t)(G(p) * 16);   // descriptor units of 16 bytes
    uint64_t db = tc_desc(b(p), 128, 256);
    for (int k = 0; k < steps; ++k) {
      ok = sl_wait(sb.full + 8 * st, par, sb.fail);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint64_t da = tc_desc(ring + (uint32_t)st * kSlStage, 128, 256);
#pragma unroll
      for (int i = 0; i < kSl; ++i) {
        sl_mma(d + i * NC, da, db, sl_idesc((kSl - i) * NC), (i > 0 || k > 0) ? 1u : 0u);
        da += slice;
      }
      sl_commit(sb.empty + 8 * st);
      db += (uint64_t)(kSl * NC * 2);
      if (++st == nst) {
        st = 0;
        par ^= 1u;
      }
    }
    if (ok) sl_commit(sb.tfull + 8 * buf);
  }
  if (!ok) {   // every MMA issued so far
    sl_commit(sb.drain);
    tc_wait(sb.drain, 0u);
  }
  return ok;
}

// ---- synthesis --------------------------------------------------------------------------------
// CTA = (3 radii, m, 128 latitudes); 12 epilogue warps (warpgroup = radius), MMA and copy warps.
// Phases P(s=0), P(1), dP(0), dP(1), P/sin(0), P/sin(1); columns (radius, component, re/im): 18 of
// kSsNC for P (u_r, omega_r, d_r T), 30 for the vector types (S_u, T_u, S_w, T_w, S_T).
// The data digits of both parities are resident.
constexpr int kSsRad = 3, kSsNC = 32, kSsEpi = 32 * 4 * kSsRad, kSsThreads = kSsEpi + 64;
constexpr int kSsBuf = 256;   // tensor-memory columns per accumulator buffer (224 used)

// Digits of P and of the vector types resident together (up to 64 terms) beside two stages.
__host__ __device__ constexpr bool ss_both(int ksmax) { return ksmax <= 4; }
__host__ __device__ constexpr size_t ss_smem(int ksmax, int nst) {
  return (size_t)nst * kSlStage + (ss_both(ksmax) ? 4 : 2) * (size_t)ksmax * kSl * kSsNC * 32 + 512;
}

__device__ __forceinline__ int ss_comp(bool vec, int c) {
  return vec ? (c < 2 ? c + 1 : (c < 4 ? c + 2 : 7)) : 3 * c;   // 1, 2, 4, 5, 7 / 0, 3, 6
}

// grid = (ceil(Nd / 3), nm, nt): the long sums (small m) of every radius first.
__global__ void __launch_bounds__(kSsThreads, 1) k_synth_sl(DevGeom g, SlTables tt, int nst,
                                                         const double2* __restrict__ SR,
                                                         double2* __restrict__ FC) {
  grid_begin();
  extern __shared__ __align__(1024) unsigned char sl_raw[];
  const int a = blockIdx.y, i0 = blockIdx.x * kSsRad, mt = blockIdx.z;
  const int m = g.m_of[a], p0 = g.pstart[a], nl = g.L - m + 1, Nd = g.Nd;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rows = min(128, g.nlat2 - mt * 128), G = (rows + 7) / 8;
  int deg[2], ks[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    deg[s] = (nl - s + 1) / 2;
    ks[s] = (deg[s] + 15) / 16;
  }
  unsigned char* ring = sl_raw;
  unsigned char* B = ring + (size_t)nst * kSlStage;               // [s][step][slice][NC][16]
  const uint32_t bpar = (uint32_t)(tt.ksmax * kSl * kSsNC * 32);   // bytes per parity
  // the vector types' digits have a region of their own where both fit, else they replace those of P
  const bool both = ss_both(tt.ksmax);
  const uint32_t bvec = both ? 2 * bpar : 0;
  uint64_t* bar = reinterpret_cast<uint64_t*>(B + (both ? 4 : 2) * bpar);
  uint64_t *full = bar, *empty = bar + 4, *tfull = bar + 8, *tempty = bar + 10, *drain = bar + 12;
  uint64_t* conv = bar + 13;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 14);
  volatile int* fail = reinterpret_cast<int*>(tslot + 1);
  int* eb = reinterpret_cast<int*>(tslot + 2);                     // [3 radii][8][2]
  const SlBars sb{tc_smem(full), tc_smem(empty), tc_smem(tfull), tc_smem(tempty), tc_smem(drain), fail};
  if (tid < kSsRad * 16) eb[tid] = 0;
  if (warp == 12) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(tslot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    if (lane == 0) {
      *fail = 0;
      for (int q = 0; q < 14; ++q)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem(&bar[q])),
                     "r"(q == 10 || q == 11 || q == 13 ? 12 : 1)
                     : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  // column exponents over the degrees of both parities (they are added as integers later)
  if (tid < kSsEpi) {
    // thread = one component of one radius, every 16th degree: its loads are independent
    const int c = tid % (kSsRad * 8), i = i0 + (c >> 3);
    int ex = 0, ey = 0;
    if (i < Nd) {
      const double2* src = SR + ((long)p0 * Nd + i) * 8 + (c & 7);
#pragma unroll 8
      for (int q = tid / (kSsRad * 8); q < nl; q += kSsEpi / (kSsRad * 8)) {
        const double2 v = src[(long)q * Nd * 8];
        ex = max(ex, sl_field(v.x));
        ey = max(ey, sl_field(v.y));
      }
    }
    atomicMax(&eb[2 * c], ex);
    atomicMax(&eb[2 * c + 1], ey);
  }
  __syncthreads();
  if (tid < kSsRad * 16) eb[tid] = sl_exponent(eb[tid]);
  __syncthreads();
  // digits of the P (3) or vector (5) components of both parities; item = (column, octet of terms)
  auto convert = [&](bool vec) {
    const int per = 2 * kSsRad * (vec ? 5 : 3);
    const int items0 = per * ks[0] * 2, items = items0 + per * ks[1] * 2;
    unsigned char* dst = B + (vec ? bvec : 0);
    for (int it = tid; it < items; it += kSsEpi) {
      const int s = it >= items0 ? 1 : 0;
      const int idx = it - (s ? items0 : 0);
      const int n = idx % per, ko = idx / per;
      const int cc = n >> 1, nc = vec ? 5 : 3, rr = cc / nc, comp = ss_comp(vec, cc - rr * nc);
      const int i = i0 + rr, e = eb[(rr * 8 + comp) * 2 + (n & 1)];
      const int dg = (nl - s + 1) / 2;
      const double* src = reinterpret_cast<const double*>(SR + ((long)(p0 + s) * Nd + i) * 8 + comp) + (n & 1);
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = ko * 8 + u;
        x[u] = (k < dg && i < Nd && e != kSlNaN) ? src[(long)k * Nd * 32] : 0.0;
      }
      long long v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = sl_fixed(x[u], e);
      sl_store8(dst + s * bpar + (ko >> 1) * (kSl * kSsNC * 32) + (ko & 1) * 128 + (n >> 3) * 256 + (n & 7) * 16,
                kSsNC * 32, v);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  };
  if (tid < kSsEpi) convert(false);
  __syncthreads();   // digits of P written
  if (warp == 12) {
    if (lane == 0) {
      const uint32_t b0 = tc_smem(B);
      if (!sl_issue<kSsNC, 2, kSsBuf>(
              sb, 6, nst, tc_smem(ring), tmem, [&](int) { return G; },
              [&](int p) { return p & 1 ? ks[1] : ks[0]; },
              [&](int p) { return b0 + (uint32_t)(p & 1) * bpar + (p >= 2 ? bvec : 0u); },
              [&](int p) { return p != 2 || sl_wait(tc_smem(conv), 0u, fail); }))   // vector digits
        atomicExch(tt.status, 7);
    }
    __syncwarp();
  } else if (warp == 13) {
    if (lane == 0)
      sl_copy(sb, 6, nst, tc_smem(ring), [&](int) { return G; }, [&](int p) { return p & 1 ? ks[1] : ks[0]; },
              [&](int p) { return tt.tiles + tt.off[((a * 2 + (p & 1)) * 3 + (p >> 1)) * tt.nt + mt]; });
    __syncwarp();
  } else {
    const int quad = warp & 3, rr = warp >> 2;
    const int row = quad * 32 + lane, t = mt * 128 + row;
    const int i = i0 + rr;
    const bool live = row < rows && i < Nd;
    const bool work = quad * 32 < rows && i < Nd;      // any live lane in this warp
    const int* ebr = eb + rr * 16;
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16);
    const int nlat = g.nlat, K1 = g.K + 1;
    bool ok = true;
    auto wait_full = [&](int p) {
      if (ok) ok = sl_wait(sb.tfull + 8 * (p & 1), (uint32_t)((p >> 1) & 1), fail);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto release = [&](int p) {
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) sl_arrive(sb.tempty + 8 * (p & 1));
    };
    auto row_exp = [&](int w) { return live ? tt.ea[(a * 3 + w) * g.nlat2 + t] : 0; };
    const double nan = __longlong_as_double(0x7FF8000000000000ll);
    auto val = [&](long long v, int ea, int e) { return e == kSlNaN ? nan : sl_join(v, sl_unit(ea, e)); };
    auto put = [&](int fld, int hemi, double x, double y) {
      const int th = hemi ? nlat - 1 - t : t;
      if (live) FC[(((long)fld * Nd + i) * K1 + a) * nlat + th] = make_double2(x, y);
    };
    // P: u_r, omega_r, d_r T (even about the equator for s = 0)
    long long E[10];
    const int ea0 = row_exp(0), ea1 = row_exp(1), ea2 = row_exp(2);
    // columns of the even class
    auto read_even = [&](int n, int buf) {
#pragma unroll
      for (int c = 0; c < 10; c += 2) {
        if (c < n) {
          long long v[2];
          sl_read<2, kSsNC>(tl + buf * kSsBuf, rr * n + c, v);
          E[c] = v[0]; E[c + 1] = v[1];
        }
      }
    };
    if (both) {
      convert(true);
      __syncwarp();
      if (lane == 0) sl_arrive(tc_smem(conv));
    }
    wait_full(0);
    if (work) read_even(6, 0);
    release(0);
    wait_full(1);
    if (!both) {   // the MMAs of P have read their digits
      convert(true);
      __syncwarp();
      if (lane == 0) sl_arrive(tc_smem(conv));
    }
    if (work) {
#pragma unroll
    for (int c = 0; c < 6; c += 2) {
      long long v[2];
      sl_read<2, kSsNC>(tl + kSsBuf, rr * 6 + c, v);
      const long long ox = ks[1] ? v[0] : 0, oy = ks[1] ? v[1] : 0;
      const int ex = ebr[3 * c], ey = ebr[3 * c + 1];
      put(3 * (c >> 1), 0, val(E[c] + ox, ea0, ex), val(E[c + 1] + oy, ea0, ey));
      put(3 * (c >> 1), 1, val(E[c] - ox, ea0, ex), val(E[c + 1] - oy, ea0, ey));
    }
    }
    release(1);
    // dP: north E + O, south O - E
    double DN[10], DS[10];
    wait_full(2);
    if (work) read_even(10, 0);
    release(2);
    wait_full(3);
    if (work) {
#pragma unroll
    for (int c = 0; c < 10; c += 2) {
      long long v[2];
      sl_read<2, kSsNC>(tl + kSsBuf, rr * 10 + c, v);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const long long o = ks[1] ? v[u] : 0;
        const int e = ebr[2 * ss_comp(true, c >> 1) + u];
        DN[c + u] = val(E[c + u] + o, ea1, e);
        DS[c + u] = val(o - E[c + u], ea1, e);
      }
    }
    put(7, 0, DN[8], DN[9]);                                        // (1/r) d_th T
    put(7, 1, DS[8], DS[9]);
    }
    release(3);
    // P/sin: north E + O, south E - O; then the combinations i m X + Y
    wait_full(4);
    if (work) read_even(10, 0);
    release(4);
    wait_full(5);
    const double mm = (double)m;
    if (work) {
#pragma unroll
    for (int u = 0; u < 3; ++u) {       // (S_u, T_u), (S_w, T_w), S_T
      double SN[4], SS[4];
      const int nv = u < 2 ? 4 : 2;
#pragma unroll
      for (int c = 0; c < 4; c += 2) {
        if (c < nv) {
          long long v[2];
          sl_read<2, kSsNC>(tl + kSsBuf, rr * 10 + 4 * u + c, v);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const long long o = ks[1] ? v[q] : 0;
            const int e = ebr[2 * ss_comp(true, 2 * u + (c >> 1)) + q];
            SN[c + q] = val(E[4 * u + c + q] + o, ea2, e);
            SS[c + q] = val(E[4 * u + c + q] - o, ea2, e);
          }
        }
      }
      if (u < 2) {
        // v_th = dS + i m T/s, v_ph = i m S/s - dT
        const double *dn = DN + 4 * u, *ds = DS + 4 * u;
        put(1 + 3 * u, 0, dn[0] - mm * SN[3], dn[1] + mm * SN[2]);
        put(2 + 3 * u, 0, -mm * SN[1] - dn[2], mm * SN[0] - dn[3]);
        put(1 + 3 * u, 1, ds[0] - mm * SS[3], ds[1] + mm * SS[2]);
        put(2 + 3 * u, 1, -mm * SS[1] - ds[2], mm * SS[0] - ds[3]);
      } else {
        put(8, 0, -mm * SN[1], mm * SN[0]);                         // (1/(r s)) d_ph T
        put(8, 1, -mm * SS[1], mm * SS[0]);
      }
    }
    }
    if (!ok && lane == 0) atomicExch(tt.status, 7);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 12) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// ---- analysis ---------------------------------------------------------------------------------
// CTA = (4 radii, m); 16 epilogue warps (warpgroup = radius), MMA and copy warps.  Rows are the
// degrees of a parity class, terms the north latitudes; data columns (radius, field, re/im) of the
// equatorially symmetric and antisymmetric parts n +- s, formed as integers: blocks
// [sym | ant][(r, U.grad T) | (theta, phi)], resident.  Phases (s, w): P with (r, U.grad T) and P/sin
// with (theta, phi) of sym for s = 0 (ant for s = 1), dP/dtheta with (theta, phi) of the other.
constexpr int kSaRad = 4, kSaNC = 16, kSaEpi = 32 * 4 * kSaRad, kSaThreads = kSaEpi + 64;
constexpr int kSaBuf = 128, kSaNB = 4;

__host__ __device__ constexpr size_t sa_smem(int ks, int nst) {
  return (size_t)nst * kSlStage + 4 * (size_t)ks * kSl * kSaNC * 32 + 512;
}

// grid = (ceil(Nd / 4), nm).
__global__ void __launch_bounds__(kSaThreads, 1) k_analysis_sl(DevGeom g, SlTables tt, int nst,
                                                            const double2* __restrict__ FA,
                                                            double2* __restrict__ AR) {
  grid_begin();
  extern __shared__ __align__(1024) unsigned char sl_raw[];
  const int a = blockIdx.y, i0 = blockIdx.x * kSaRad;
  const int m = g.m_of[a], p0 = g.pstart[a], nl = g.L - m + 1, Nd = g.Nd;
  const int n2 = g.nlat2, nlat = g.nlat, K1 = g.K + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ks = (n2 + 15) / 16;
  unsigned char* ring = sl_raw;
  unsigned char* B = ring + (size_t)nst * kSlStage;               // [blk][half][step][slice][NC][16]
  const uint32_t bblk = (uint32_t)(ks * kSl * kSaNC * 32);
  uint64_t* bar = reinterpret_cast<uint64_t*>(B + 4 * bblk);
  uint64_t *full = bar, *empty = bar + 4, *tfull = bar + 8, *tempty = bar + 12, *drain = bar + 16;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 17);
  volatile int* fail = reinterpret_cast<int*>(tslot + 1);
  int* eb = reinterpret_cast<int*>(tslot + 2);                    // [4 radii][4 fields][2]
  const SlBars sb{tc_smem(full), tc_smem(empty), tc_smem(tfull), tc_smem(tempty), tc_smem(drain), fail};
  if (warp == 16) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(tslot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    if (lane == 0) {
      *fail = 0;
      for (int q = 0; q < 17; ++q)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem(&bar[q])),
                     "r"(q >= 12 && q < 16 ? 16 : 1)
                     : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  // fields in the order r, U.grad T, theta, phi: FA fields 0, 3, 1, 2
  auto src_of = [&](int f, int rr) {
    const int q = f == 0 ? 0 : f == 1 ? 3 : f - 1;
    return FA + (((long)q * Nd + i0 + rr) * K1 + a) * nlat;
  };
  if (tid < kSaEpi) {   // a warp per (radius, field)
    int ex = 0, ey = 0;
    if (i0 + (warp >> 2) < Nd) {
      const double2* src = src_of(warp & 3, warp >> 2);
#pragma unroll 6
      for (int th = lane; th < nlat; th += 32) {
        const double2 v = src[th];
        ex = max(ex, sl_field(v.x));
        ey = max(ey, sl_field(v.y));
      }
    }
    ex = __reduce_max_sync(0xffffffffu, ex);
    ey = __reduce_max_sync(0xffffffffu, ey);
    if (lane == 0) {
      eb[2 * warp] = ex;
      eb[2 * warp + 1] = ey;
    }
  }
  __syncthreads();
  if (tid < kSaRad * 8) {
    const int e = sl_exponent(eb[tid]);
    eb[tid] = e == kSlNaN ? e : e + 1;      // |n +- s| < 2^(e + 1)
  }
  __syncthreads();
  if (tid < kSaEpi) {
    // a warp per (radius, field), lanes over latitudes (coalesced loads)
    const int c = warp, rr = c >> 2, f = c & 3, ex = eb[2 * c], ey = eb[2 * c + 1];
    const double2* src = src_of(f, rr);
    const int n = rr * 4 + (f & 1) * 2;
    unsigned char* d0 = B + (f >> 1) * bblk + (n >> 3) * 256 + (n & 7) * 16;
    for (int t = lane; t < ks * 16; t += 32) {
      double2 vn = make_double2(0, 0), vz = make_double2(0, 0);
      if (i0 + rr < Nd && t < n2) {
        vn = src[t];
        vz = src[nlat - 1 - t];
      }
      unsigned char* d = d0 + (t >> 4) * (kSl * kSaNC * 32) + ((t >> 3) & 1) * 128 + (t & 7) * 2;
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        const int e = part ? ey : ex;
        const long long p = e == kSlNaN ? 0 : sl_fixed(part ? vn.y : vn.x, e);
        const long long q = e == kSlNaN ? 0 : sl_fixed(part ? vz.y : vz.x, e);
        const unsigned long long bs = (unsigned long long)(p + q + 0x0080808080808080ll);
        const unsigned long long ba = (unsigned long long)(p - q + 0x0080808080808080ll);
#pragma unroll
        for (int i = 0; i < kSl; ++i) {
          unsigned char* o = d + part * 16 + i * (kSaNC * 32);
          *reinterpret_cast<unsigned short*>(o) = (unsigned short)(sl_digit(bs, i) >> 16);
          *reinterpret_cast<unsigned short*>(o + 2 * bblk) = (unsigned short)(sl_digit(ba, i) >> 16);
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  const int deg0 = (nl + 1) / 2, deg1 = nl / 2;
  const int nph = deg1 > 0 ? 6 : 3;
  auto groups = [&](int p) { return ((p < 3 ? deg0 : deg1) + 7) / 8; };
  bool ok = true;
  if (warp == 16) {
    if (lane == 0) {
      const uint32_t b0 = tc_smem(B);
      if (!sl_issue<kSaNC, kSaNB, kSaBuf>(
              sb, nph, nst, tc_smem(ring), tmem, groups, [&](int) { return ks; },
              [&](int p) {
                const int s = p / 3, w = p % 3;
                const int blk = w == 1 ? 1 - s : s;
                return b0 + (uint32_t)(blk * 2 + (w == 0 ? 0 : 1)) * bblk;
              },
              [&](int) { return true; }))
        atomicExch(tt.status, 7);
    }
    __syncwarp();
  } else if (warp == 17) {
    if (lane == 0)
      sl_copy(sb, nph, nst, tc_smem(ring), groups, [&](int) { return ks; },
              [&](int p) { return tt.tiles + tt.off[((a * 2 + p / 3) * 3 + p % 3) * tt.nt]; });
    __syncwarp();
  } else {
    const int quad = warp & 3, rr = warp >> 2;
    const int row = quad * 32 + lane, i = i0 + rr;
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16);
    const double nan = __longlong_as_double(0x7FF8000000000000ll);
    const double mm = (double)m;
    const int* ebr = eb + rr * 8;
    for (int s = 0; s < nph / 3; ++s) {
      const int q = s + 2 * row;
      const bool live = q < nl && i < Nd;
      double X[4], Y[4];
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        const int p = s * 3 + w;
        if (ok) ok = sl_wait(sb.tfull + 8 * (p % kSaNB), (uint32_t)((p / kSaNB) & 1), fail);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const bool work = s + 2 * quad * 32 < nl && i < Nd;   // any live lane in this warp
        long long v[4] = {0, 0, 0, 0};
        if (work) sl_read<4, kSaNC>(tl + (p % kSaNB) * kSaBuf, rr * 4, v);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) sl_arrive(sb.tempty + 8 * (p % kSaNB));
        if (!work) continue;
        const int ea = live ? tt.ea[(a * 3 + w) * (g.L + 1) + q] : 0;
        double o[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int e = ebr[(w == 0 ? 0 : 4) + c];
          o[c] = e == kSlNaN ? nan : sl_join(v[c], sl_unit(ea, e));
        }
        double2* dst = AR + ((long)(p0 + q) * Nd + i) * 4;
        if (w == 0) {
          if (live) {
            dst[0] = make_double2(o[0], o[1]);
            dst[3] = make_double2(o[2], o[3]);
          }
        } else if (w == 1) {
#pragma unroll
          for (int c = 0; c < 4; ++c) Y[c] = o[c];
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) X[c] = o[c];
          if (live) {
            const int l = m + q;
            const double il = l > 0 ? 1.0 / ((double)l * (double)(l + 1)) : 0.0;
            // S = dP F_th - i m P/s F_ph,  T = -i m P/s F_th - dP F_ph
            dst[1] = make_double2((Y[0] + mm * X[3]) * il, (Y[1] - mm * X[2]) * il);
            dst[2] = make_double2((mm * X[1] - Y[2]) * il, (-mm * X[0] - Y[3]) * il);
          }
        }
      }
    }
    if (!ok && lane == 0) atomicExch(tt.status, 7);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 16) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

}  // namespace rsc
