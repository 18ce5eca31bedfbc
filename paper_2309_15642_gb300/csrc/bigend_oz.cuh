// Gram and update products of the larger end of a bond in complex128 on the
// tensor cores: error-free splitting into fixed-point digits (the scheme of
// Ozaki, Ogita, Oishi and Rump), tcgen05.mma of kind::f16 with FP32 accumulators.
//
// GB300 runs FP64 at 1.2 TFLOP/s (an FP64 instruction of a warp holds its SMSP's
// unit for 64 cycles) and f16 products at 2 PFLOP/s, so the two streaming
// products, which are plain contractions, are formed from integers:
//
//   x = 2^(E-6) sum_i d_i 2^(-8 i),  i = 0..6,  |d_i| <= 128 integers (|d_0| <= 65),
//
// with one exponent E per operand row (|x| < 2^E over the contraction), that is
// x rounded to a multiple of 2^-54 of its row's power of two.  The digits are
// exact in f16, their products and the FP32 sums of up to 7 x 128 of them are
// below 2^24, so every accumulator is an exact integer whatever the order:
//
//   sum_k x_k y_k = 2^(Ex+Ey-12) sum_{l=0..7} 2^(-8 l) v_l,  v_l = sum_{i+j=l} sum_k d_i(x_k) d_j(y_k).
//
// The eight v_l of an output are combined in a 64-bit integer of unit 2^(Ex+Ey-53), to
// nearest, and rounded once to FP64.  Error of a sum of K products, in units of
// 2^(Ex+Ey): K 2^-54 from the 54 bits of x and y, 5 K 2^-62 from the levels l > 7 that
// are left out, 2^-54 from the combination.  Over Gaussian rows it is 0.41, 0.53 and 0.64
// x 2^-53 rms for K = 16, 64 and 128; a chain of FP64 multiply-adds makes 0.58, 1.25 and
// 2.47 (seven levels and a low part cut off rather than rounded made 1.9, 3.6 and 5.1, with a
// mean of -0.9, in 28 digit products instead of 34; one class of 127 + 433 + 1121 qubits, D = 32:
// Gram 1.95 -> 2.07, bonds 11.3 -> 11.4, update 1.39 -> 1.58 ms).  Against the terms
// themselves it is an FP64 sum's only as far as they are within a few bits of the row
// maxima: the passes scale their operands for that (the Gram's columns are summed over rows
// against their own norms, the update balances k).
//
// The digits of a double cost about 30 integer instructions and no FP64 one.
// Slices are stored as K-major operands without swizzle, slice after slice, so
// that one instruction multiplies slice i of A with several slices j of B at once
// (N = slices x columns) and lands on the adjacent accumulators of the levels
// i + j.
//
//   oz_gram_kernel    one CTA per row tile (and spin, beyond D = 32): kicks the
//       rows (writing them, unweighted, to `at` for the update), weights them, and
//       writes the upper triangles of the tile's Gram blocks in FP64 (they are Hermitian to
//       the bit: both triangles come from the same integers).
//   oz_update_kernel  one CTA per 128 rows, spin and 32 new bond indices:
//       Gamma_a'[s] = mask (Ã_s Y_s) from `at`, the bond index balanced first.
//
// Included by su_kernels.cu after its row/element helpers.
#pragma once
#include "oz_mma.cuh"
#include "tcgen05.cuh"

namespace gpeps {

constexpr int kOzThreads = 512;
constexpr int kOzOperand = kOzSlices * 128 * 64 * 2;  // bytes of 7 slices of 8192 digits
constexpr int kOzDumpLd = 129;                        // row stride (doubles) of the Gram readout
constexpr size_t kOzGramSmem = (size_t)128 * kOzDumpLd * 8;
constexpr size_t kOzUpdateSmem = (size_t)kOzOperand + kOzOperand / 2;

// The digits of 8 consecutive K values of one operand row: one 16-byte store per slice.
__device__ __forceinline__ void oz_store(unsigned char* p, uint32_t slice_bytes, const unsigned long long* v) {
#pragma unroll
  for (int i = 0; i < kOzSlices; ++i) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = oz_pair(v[2 * q], v[2 * q + 1], i);
    *reinterpret_cast<uint4*>(p + (size_t)i * slice_bytes) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, int n, uint32_t accumulate) {
  // FP32 accumulator, f16 operands, both K-major, M = 128
  const uint32_t idesc = (1u << 4) | ((uint32_t)(n >> 3) << 17) | (8u << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// 32 lanes x 8 consecutive FP32 columns (the caller waits: tcgen05.wait::ld)
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Slice i is the first to add to level l (its seven slices j reach level 7 from i = 1 on).
__device__ __forceinline__ bool oz_first(int i, int l) { return i == (l == kOzLevels - 1 ? 1 : 0); }

// Commit the issued products and wait (bounded) for them; the outcome is uniform over the CTA.
__device__ __forceinline__ bool oz_wait(uint64_t* bar, uint32_t& phase) {
  const bool ok = tc_wait(bar, phase, kTcWaitCycles);
  tc::fence_after_sync();
  return ok;
}

// cos and sin of half the pending kick of end a, once per bond (an FP64 sincos per
// thread of every tile would cost more than the tile's products).
__global__ void oz_kick_kernel(const BondDesc* __restrict__ bonds, int n, const double* __restrict__ pending,
                               double2* __restrict__ cs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double h = 0.5 * pending[bonds[i].a.site];
  cs[i] = make_double2(cos(h), sin(h));
}

// Slot of one row tile in `at`: Ã [s][row][re/im][k] (doubles).
__device__ __forceinline__ int64_t oz_at(int part, int s, int row, int ri, int tr, int D) {
  return (int64_t)part * 4 * tr * D + ((int64_t)(s * tr + row) * 2 + ri) * D;
}

// kMode 0: D <= 32, one CTA per 64-row tile, operand rows (s, re/im, k), k padded to 32;
// kMode 1: D <= 64, one per tile and spin, rows (re/im, k), k padded to 64;
// kMode 2: D <= 128, one per 32-row tile and spin, rows (re/im, k), k padded to 128: two
//          products, Re = re re^T + im im^T and T = re im^T (Im = T - T^T).
// In each, 16 warps take 8 rows x 32 bond indices of one spin: 8192 digits per slice.
template <int kMode>
__global__ void __launch_bounds__(kOzThreads, 1)
    oz_gram_kernel(const TileDesc* __restrict__ tiles, const BondDesc* __restrict__ bonds,
                   const double2* __restrict__ gamma, const double* __restrict__ lam, const double2* __restrict__ cs,
                   double2* __restrict__ partials, double* __restrict__ at, int* flags, int D) {
  constexpr int Kt = kMode == 2 ? 32 : 64, kRows = kMode == 2 ? 256 : 128;
  constexpr uint32_t kSlice = kRows * Kt * 2, kSbo = Kt * 16;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int cmax[kMode == 2 ? 128 : 64];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ uint32_t tslot;
  const TileDesc t = tiles[blockIdx.x];
  const SideDesc sa = bonds[t.bond].a;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < (int)(sizeof(cmax) / 4)) cmax[threadIdx.x] = 0;
  const uint32_t tmem = tc_setup(&tslot, bars, 512);
  // rows of this warp: 8 rows from rg * 8, bond index k, spin s
  const int rg = kMode == 2 ? (warp & 3) : (warp & 7);
  const int kb = kMode == 0 ? 0 : kMode == 1 ? (warp >> 3) : (warp >> 2);
  const int s = kMode == 0 ? (warp >> 3) : (int)blockIdx.y;
  const int k = kb * 32 + lane;
  const int tr = kMode == 2 ? 32 : 64;
  double2 x[8];
  {
    const double2 c = cs[t.bond];
    double2 g0[8], g1[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = rg * 8 + i;
      g0[i] = g1[i] = make_double2(0.0, 0.0);
      if (r < t.nrows && k < D) {
        const int64_t e = elem(sa, 0, row_pos(sa, t.row0 + r), k);
        g0[i] = gamma[e];
        g1[i] = gamma[e + sa.str_s];
      }
    }
    int cm = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = rg * 8 + i;
      double2 a = make_double2(0.0, 0.0);
      double w = 0.0;
      if (r < t.nrows) {
        // component s of exp(-i theta X / 2) (as kick2)
        const double2 p = s ? g1[i] : g0[i], q = s ? g0[i] : g1[i];
        a = make_double2(c.x * p.x + c.y * q.y, c.x * p.y - c.y * q.x);
        w = row_weight(sa, lam, row_pos(sa, t.row0 + r));
        if (k < D) {
          at[oz_at(t.part, s, r, 0, tr, D) + k] = a.x;
          at[oz_at(t.part, s, r, 1, tr, D) + k] = a.y;
        }
      }
      x[i] = make_double2(a.x * w, a.y * w);
      cm = max(cm, max(oz_row_exp(x[i].x), oz_row_exp(x[i].y)));
    }
    if (cm) atomicMax(cmax + (kMode == 0 ? s * 32 : 0) + k, cm);
  }
  __syncthreads();
  {
    const int em = cmax[(kMode == 0 ? s * 32 : 0) + k];
#pragma unroll
    for (int ri = 0; ri < 2; ++ri) {
      const int c = kMode == 0 ? (s * 2 + ri) * 32 + k : ri * (kRows / 2) + k;
      unsigned long long v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = oz_fixed(ri ? x[i].y : x[i].x, em);
      oz_store(smem_raw + (uint32_t)(c >> 3) * kSbo + rg * 128 + (c & 7) * 16, kSlice, v);
    }
  }
  tc::fence_async_smem();
  __syncthreads();
  const uint32_t base = tc::smem_u32(smem_raw);
  // levels [l0, l0 + 4) of product `prod` into the accumulators at column (l - l0) * 128
  auto issue = [&](int prod, int l0) {
    if (threadIdx.x != 0) return;
    tc::fence_after_sync();
    for (int ks = 0; ks < Kt / 16; ++ks) {
      auto desc = [&](int slice, int row) {
        return tc::smem_desc(base + slice * kSlice + (uint32_t)(row >> 3) * kSbo + ks * 256, 128, kSbo);
      };
      for (int i = 0; i < min(l0 + 4, kOzSlices); ++i) {
        const int j1 = min(l0 + 4 - i, kOzSlices);
        for (int j = max(l0 - i, 0); j < j1;) {
          const uint32_t d = tmem + (uint32_t)(i + j - l0) * 128u;
          const bool first = !ks && oz_first(i, i + j);  // these accumulators hold nothing yet
          // two slices j at once where both accumulators are in the same state
          const int w = kMode != 2 && j + 1 < j1 && first == (!ks && oz_first(i, i + j + 1)) ? 2 : 1;
          mma_f16(d, desc(i, 0), desc(j, kMode == 2 && prod ? 128 : 0), 128 * w, first ? 0u : 1u);
          if (kMode == 2 && !prod) mma_f16(d, desc(i, 128), desc(j, 128), 128, 1u);
          j += w;
        }
      }
    }
    tc::mma_commit(bars);
  };
  uint32_t phase = 0;
  bool ok = true;
  const int m = 32 * (warp & 3) + lane, n0 = 32 * (warp >> 2);
  const uint32_t tq = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)n0;
  double* dump = reinterpret_cast<double*>(smem_raw);
  const int half = D * (D + 1) / 2;
  double2* out = partials + (int64_t)t.part * 2 * half + (kMode == 0 ? 0 : s * half);
  for (int prod = 0; prod < (kMode == 2 ? 2 : 1) && ok; ++prod) {
    long long acc[32];
    issue(prod, 0);
    ok = oz_wait(bars, phase);
    if (!ok) break;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      uint32_t v[4][8];
#pragma unroll
      for (int l = 0; l < 4; ++l) tmem_ld8(tq + l * 128 + b * 8, v[l]);
      tmem_ld_wait();
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        long long h = 0;
#pragma unroll
        for (int l = 0; l < 4; ++l) h += oz_weigh(__uint_as_float(v[l][q]), l);
        acc[8 * b + q] = h;
      }
    }
    tc::fence_before_sync();
    __syncthreads();
    issue(prod, 4);
    ok = oz_wait(bars, phase);
    if (!ok) break;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      uint32_t v[4][8];
#pragma unroll
      for (int l = 0; l < 4; ++l) tmem_ld8(tq + l * 128 + b * 8, v[l]);
      tmem_ld_wait();
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        long long low = 0;
#pragma unroll
        for (int l = 0; l < 4; ++l) low += oz_weigh(__uint_as_float(v[l][q]), l);
        acc[8 * b + q] = oz_sum(acc[8 * b + q], low);
      }
    }
    tc::fence_before_sync();
    // both passes are complete: the digits are free unless a second product follows
    if (kMode == 2 && prod == 0) {
      const int ea = cmax[m];
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        const int l = n0 + q;
        if (m <= l && l < D) out[upper_pos(m, l, D)].x = oz_value(acc[q], ea, cmax[l]);
      }
    } else {
      auto ce = [&](int c) { return cmax[kMode == 0 ? (c >> 6) * 32 + (c & 31) : kMode == 1 ? (c & 63) : c]; };
      const int ea = ce(m);
#pragma unroll
      for (int q = 0; q < 32; ++q) dump[m * kOzDumpLd + n0 + q] = oz_value(acc[q], ea, ce(n0 + q));
    }
    __syncthreads();
  }
  if (ok) {
    if (kMode == 2) {
      for (int o = threadIdx.x; o < half; o += kOzThreads) {
        int a, b;
        upper_index(o, D, a, b);
        out[o].y = dump[a * kOzDumpLd + b] - dump[b * kOzDumpLd + a];
      }
    } else {
      constexpr int kp = kMode == 0 ? 32 : 64;
      for (int o = threadIdx.x; o < (kMode == 0 ? 2 : 1) * half; o += kOzThreads) {
        const int sp = kMode == 0 && o >= half ? 1 : 0;  // (D <= 32: both spins)
        int ra, rb;
        upper_index(o - sp * half, D, ra, rb);
        ra += sp * 64;
        rb += sp * 64;
        out[o] = make_double2(dump[ra * kOzDumpLd + rb] + dump[(ra + kp) * kOzDumpLd + rb + kp],
                              dump[ra * kOzDumpLd + rb + kp] - dump[(ra + kp) * kOzDumpLd + rb]);
      }
    }
  } else if (threadIdx.x == 0) {
    atomicOr(flags, 4);
  }
  tc_teardown(tmem, 512);
}

// Balance of the bond index in the update, per bond and spin (blockIdx.x, blockIdx.y).
//
// Y[k][k'] = lambda_k W[k][k'] / s_k', W formed in FP64 to eps of its row, and near the
// canonical form Ã[r][k] grows like 1 / lambda_k in rows of small lambda on the other legs.
// A digit holds 54 bits below its operand row's largest element, so k is balanced before the
// split: Ã[.][k] 2^b_k, Y[k][.] 2^-b_k, b_k the exponent of max_k' |Y[k][k']| s_k' (exact,
// integers added to exponents).  The error of an output is then 2^-54 of
// max_k |Ã[r][k]| 2^b_k / s_k', which the rounding of W alone already makes.  Without it
// the tensor loses digits like 1 / lambda_min: 9e-11 of a row's scale at 1e-6, 8e-7 at 1e-10.
// Update of one class of 127 + 433 + 1121 qubits, D = 32: 1.26 -> 1.38 ms.
//
// Once per bond and spin: in each of the update's CTAs it would be three dependent passes of
// loads.  bal: b_k [D], the largest exponents of Y's balanced columns [D], and whether Y = I.
__device__ __forceinline__ int64_t oz_bal(int bond, int s, int D) { return ((int64_t)bond * 2 + s) * (2 * D + 1); }
__global__ void __launch_bounds__(kThreads)
    oz_balance_kernel(const BondDesc* __restrict__ bonds, const double* __restrict__ lam,
                      const double2* __restrict__ Yall, int* __restrict__ balance, int D) {
  __shared__ int snew[kMaxDc128], bal[kMaxDc128], ymax[kMaxDc128];
  const int s = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kThreads / 32;
  const double2* Y = Yall + ((int64_t)blockIdx.x * 2 + s) * D * D;
  int* out = balance + oz_bal(blockIdx.x, s, D);
  for (int k = threadIdx.x; k < D; k += kThreads) {
    snew[k] = oz_exp(lam[bonds[blockIdx.x].lam_e + k]) - 2046;  // the bond's new lambda
    ymax[k] = kOzNone;
  }
  __syncthreads();
  bool one = true;
  for (int k = warp; k < D; k += nw) {
    int e = kOzNone;
    for (int kp = lane; kp < D; kp += 32) {
      const double2 y = Y[k * D + kp];
      const int ey = max(oz_exp(y.x), oz_exp(y.y));
      one = one && __double2hiint(y.x) == (k == kp ? 0x3ff00000 : 0) &&
            (__double2loint(y.x) | __double2hiint(y.y) | __double2loint(y.y)) == 0;
      if (ey) e = max(e, ey + snew[kp]);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) bal[k] = e;
  }
  one = __syncthreads_and(one);
  for (int kp = lane; kp < D; kp += 32) {
    int e = kOzNone;
    for (int k = warp; k < D; k += nw) {
      const double2 y = Y[k * D + kp];
      const int ey = max(oz_row_exp(y.x), oz_row_exp(y.y));
      if (ey) e = max(e, ey >= kOzNan ? 2 * kOzNan : ey - bal[k]);
    }
    atomicMax(ymax + kp, e);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < D; k += kThreads) {
    out[k] = bal[k];
    out[D + k] = ymax[k];
  }
  if (threadIdx.x == 0) out[2 * D] = one;
}

// Rows [row0, row0 + 128) of end a, spin blockIdx.y, new bond indices [32 blockIdx.z, +32):
// Gamma_a'[s][r][k'] = mask_r sum_k Ã_s[r][k] Y_s[k][k'] as a real product over K = (re/im, k),
// 32 k at a time: M = 128 rows, N = (re/im, k') = 64.  Launched over the row tiles; the tiles
// that do not start a 128-row block return at once.
//
// Y = I (a bond that bond_fail leaves as it was) copies the kicked rows unrounded.
//
// kMore: beyond D = 64, where the accumulators (exact to 128 K values) are read and added up
// after every second chunk; up to there once, after the last.
template <bool kMore>
__global__ void __launch_bounds__(kOzThreads, 1)
    oz_update_kernel(const TileDesc* __restrict__ tiles, const BondDesc* __restrict__ bonds, double2* gamma,
                     const double* __restrict__ lam, const double2* __restrict__ Yall, const double* __restrict__ at,
                     const int* __restrict__ balance, int* flags, int D) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kPad = kMore ? kMaxDc128 : 64;
  __shared__ int ymax[32], rmax[128], bal[kPad];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ uint32_t tslot;
  __shared__ float mask[128];
  __shared__ double cut[2];
  const TileDesc t = tiles[blockIdx.x];
  if (t.row0 & 127) return;
  const SideDesc sa = bonds[t.bond].a;
  const int s = blockIdx.y, kp0 = 32 * blockIdx.z, D2 = D * D;
  const double2* Y = Yall + ((int64_t)t.bond * 2 + s) * D2;
  const int nrows = sa.rows - t.row0 < 128 ? sa.rows - t.row0 : 128;
  const int tr = tile_rows(D, 16);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int* plan = balance + oz_bal(t.bond, s, D);
  if (threadIdx.x < 32) ymax[threadIdx.x] = kp0 + threadIdx.x < D ? plan[D + kp0 + threadIdx.x] : kOzNone;
  if (threadIdx.x < kPad) bal[threadIdx.x] = threadIdx.x < D ? plan[threadIdx.x] : kOzNone;
  const uint32_t tmem = tc_setup(&tslot, bars, 512);
  tc_row_mask<false>(sa, lam, t.row0, nrows, D, mask, cut);
  if (plan[2 * D]) {
    __syncthreads();
    for (int i = threadIdx.x; i < nrows * 32; i += kOzThreads) {
      const int r = i >> 5, kp = kp0 + lane;
      if (kp >= D) continue;
      const int64_t src = oz_at(t.part + r / tr, s, r % tr, 0, tr, D) + kp;
      const double2 v = make_double2(at[src], at[src + D]);
      gamma[elem(sa, s, row_pos(sa, t.row0 + r), kp)] = mask[r] == 0.f ? cscale(v, 0.0) : v;
    }
    tc_teardown(tmem, 512);
    return;
  }
  // left operand: 8 rows x 4 groups of 8 k per warp and part (re, im); from the last chunk of
  // 32 k down for the rows' exponents, so that the first is in registers when its digits follow
  const int nchunk = (D + 31) / 32;
  const int ra = warp * 8 + (lane & 7), kg = lane >> 3;
  const double* arow = at + oz_at(t.part + ra / tr, s, ra % tr, 0, tr, D) + kg * 8;
  double a[2][8];
  auto load = [&](int ch) {
    const int left = ra < nrows ? D - 32 * ch - kg * 8 : 0;
#pragma unroll
    for (int ri = 0; ri < 2; ++ri) {
      const double* src = arow + ri * D + 32 * ch;
#pragma unroll
      for (int e = 0; e < 8; ++e) a[ri][e] = 0.0;
      if ((D & 7) == 0 && left > 0) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const double2 d = *reinterpret_cast<const double2*>(src + 2 * e);
          a[ri][2 * e] = d.x;
          a[ri][2 * e + 1] = d.y;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (e < left) a[ri][e] = src[e];
      }
    }
  };
  int em = kOzNone;
  for (int ch = nchunk - 1; ch >= 0; --ch) {
    load(ch);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int ea = max(oz_row_exp(a[0][e]), oz_row_exp(a[1][e]));
      if (ea) em = max(em, ea >= kOzNan ? 2 * kOzNan : ea + bal[32 * ch + kg * 8 + e]);
    }
  }
  em = max(em, __shfl_xor_sync(0xffffffffu, em, 8));
  em = max(em, __shfl_xor_sync(0xffffffffu, em, 16));
  if (kg == 0) rmax[ra] = em;
  __syncthreads();
  unsigned char* sb = smem_raw + kOzOperand;
  constexpr uint32_t kSa = 128 * 64 * 2, kSb = 64 * 64 * 2, kSbo = 64 * 16;
  const uint32_t abase = tc::smem_u32(smem_raw), bbase = tc::smem_u32(sb);
  const int m = 32 * (warp & 3) + lane, q0 = 8 * (warp >> 2);
  const uint32_t tq = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)q0;
  long long ar[8], ai[8];
  if (kMore)
#pragma unroll
    for (int q = 0; q < 8; ++q) ar[q] = ai[q] = 0;
  uint32_t phase = 0;
  bool ok = true;
  for (int ch = 0; ch < nchunk && ok; ++ch) {
    const int k0 = 32 * ch;
    if (ch) load(ch);
#pragma unroll
    for (int ri = 0; ri < 2; ++ri) {
      unsigned long long v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = oz_fixed(a[ri][e], em - bal[k0 + kg * 8 + e]);
      oz_store(smem_raw + warp * kSbo + (ri * 4 + kg) * 128 + (lane & 7) * 16, kSa, v);
    }
    // right operand: row n = (ro, k'), K = (ri, k): ro = ri -> yr; (0, 1) -> -yi; (1, 0) -> yi
    {
      const int ro = warp >> 3, ri = (warp >> 2) & 1, kp = (warp & 3) * 8 + (lane & 7), ey = ymax[kp];
      unsigned long long v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int k = k0 + kg * 8 + e;
        double2 y = make_double2(0.0, 0.0);
        if (k < D && kp0 + kp < D) y = Y[k * D + kp0 + kp];
        v[e] = oz_fixed(ro == ri ? y.x : y.y, ey + bal[k], ro < ri);
      }
      oz_store(sb + (uint32_t)(ro * 4 + (warp & 3)) * kSbo + (ri * 4 + kg) * 128 + (lane & 7) * 16, kSb, v);
    }
    tc::fence_async_smem();
    __syncthreads();
    const bool fresh = kMore ? (ch & 1) == 0 : ch == 0;
    if (threadIdx.x == 0) {
      tc::fence_after_sync();
      for (int ks = 0; ks < 4; ++ks)
        for (int i = 0; i < kOzSlices; ++i) {
          const int j1 = min(kOzLevels - i, kOzSlices);
          for (int j = 0; j < j1;) {
            // up to four slices j at once, level 7 by itself where its accumulators hold nothing yet
            const bool start = fresh && !ks, first = start && oz_first(i, i + j);
            int w = min(j1 - j, 4);
            if (start && i == 1 && i + j + w == kOzLevels && w > 1) --w;
            mma_f16(tmem + (uint32_t)(i + j) * 64u, tc::smem_desc(abase + i * kSa + ks * 256, 128, kSbo),
                    tc::smem_desc(bbase + j * kSb + ks * 256, 128, kSbo), 64 * w, first ? 0u : 1u);
            j += w;
          }
        }
      tc::mma_commit(bars);
    }
    ok = oz_wait(bars, phase);
    if (ok && ((kMore && !fresh) || ch + 1 == nchunk)) {
      long long hr[8], hi[8], lr[8], li[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) hr[q] = hi[q] = lr[q] = li[q] = 0;
#pragma unroll
      for (int l = 0; l < kOzLevels; ++l) {
        uint32_t vr[8], vi[8];
        tmem_ld8(tq + l * 64, vr);
        tmem_ld8(tq + l * 64 + 32, vi);
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          (l < 4 ? hr : lr)[q] += oz_weigh(__uint_as_float(vr[q]), l);
          (l < 4 ? hi : li)[q] += oz_weigh(__uint_as_float(vi[q]), l);
        }
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        ar[q] = (kMore ? ar[q] : 0) + oz_sum(hr[q], lr[q]);
        ai[q] = (kMore ? ai[q] : 0) + oz_sum(hi[q], li[q]);
      }
      tc::fence_before_sync();
    }
    __syncthreads();
  }
  if (ok && m < nrows) {
    const int er = rmax[m];
    const bool cut_row = mask[m] == 0.f;
    const RowPos p = row_pos(sa, t.row0 + m);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int kp = kp0 + q0 + q;
      if (kp < D) {
        const int ey = ymax[q0 + q];
        double2 v = make_double2(oz_value(ar[q], er, ey), oz_value(ai[q], er, ey));
        if (cut_row) v = cscale(v, 0.0);
        gamma[elem(sa, s, p, kp)] = v;
      }
    }
  }
  if (!ok && threadIdx.x == 0) atomicOr(flags, 4);
  tc_teardown(tmem, 512);
}

}  // namespace gpeps
