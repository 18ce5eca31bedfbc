// Integer digits of FP64 values, and the products of the small square matrices of a
// bond from them on the tensor cores (mma.sync).
//
// The digit form is that of bigend_oz.cuh: x = 2^(E-6) sum_i d_i 2^(-8 i), seven digits
// exact in f16, one exponent per row of an operand, the sums of 2 x 7 x 64 digit
// products below 2^24 and so exact in FP32; error bound there.  Columns of the solve's
// operands are unit vectors or scaled to norms in [1, 2), so that the row maxima are the
// scale that an FP64 sum rounds against too.
#pragma once
#include <cuda_fp16.h>

#include <cstdint>

namespace gpeps {

constexpr int kOzSlices = 7, kOzLevels = 8;

// One more block of accumulators: high = levels 0..3 in units of level 3, low = levels 4..7 in
// units of level 7, as an integer of unit 2^(Ea+Eb-53), rounded to nearest (a shift alone would
// bias every output downwards by half a unit).
__device__ __forceinline__ long long oz_sum(long long high, long long low) {
  return high * (1ll << 17) + ((low + (1ll << 14)) >> 15);
}
__device__ __forceinline__ long long oz_weigh(float v, int l) {
  return (long long)__float2int_rn(v) * (1ll << (8 * (3 - (l & 3))));
}

__device__ __forceinline__ int oz_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Row exponents: kOzNan marks a row that holds a value that is not finite, kOzNone (or
// any exponent more than 55 below the others') one that holds nothing.
constexpr int kOzNan = 1 << 16, kOzNone = -(1 << 16);
__device__ __forceinline__ int oz_row_exp(double x) {
  const int e = oz_exp(x);
  return e == 0x7ff ? kOzNan : e;
}

// Biased fixed point: round(x 2^(54 - E)) + 0x80 in each of the 7 digit bytes, E =
// em - 1022 for the row's largest biased exponent em: byte 6 - i minus 128 is d_i.
__device__ __forceinline__ unsigned long long oz_fixed(double x, int em, bool negate = false) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7ff, d = em - ex;
  unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 1;
  m = (m + ((1ull << (d & 63)) >> 1)) >> (d & 63);
  if (d > 55 || ex == 0) m = 0;
  const bool neg = ((long long)b < 0) != negate;
  return (neg ? 0ull - m : m) + 0x0080808080808080ull;
}

// t 2^(ea + eb - 2044 - 53) rounded to FP64 (ea, eb: biased exponents of the two rows);
// NaN when a row held a value that is not finite.
__device__ __forceinline__ double oz_value(long long t, int ea, int eb) {
  if (ea >= kOzNan || eb >= kOzNan) return __longlong_as_double(0x7ff8000000000000ll);
  const unsigned long long u = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;
  if (u == 0) return 0.0;
  const int n = __clzll((long long)u);
  const unsigned long long m = u << n;  // top bit at 63: value m 2^(-n) 2^(...)
  const int e = 1023 + 63 - n + ea + eb - 2044 - 53;
  if (e <= 0) return 0.0;
  if (e >= 0x7ff) return __longlong_as_double(t < 0 ? 0xfff0000000000000ll : 0x7ff0000000000000ll);
  const unsigned long long r = ((unsigned long long)(e - 1) << 52) + (m >> 11) + ((m >> 10) & 1ull);
  return __longlong_as_double((long long)(r | (t < 0 ? 0x8000000000000000ull : 0ull)));
}

// Digit i of two values at consecutive k as a pair of f16 (the first in the low half).
__device__ __forceinline__ uint32_t oz_pair(unsigned long long v0, unsigned long long v1, int i) {
  const int byte = 6 - i;
  const uint32_t a = (uint32_t)(v0 >> (byte >= 4 ? 32 : 0)), b = (uint32_t)(v1 >> (byte >= 4 ? 32 : 0));
  const uint32_t s = byte & 3;
  // two bytes -> f16 1024 + byte -> byte - 128
  const uint32_t t = (__byte_perm(a, b, s | (s << 4) | ((4 + s) << 8) | ((4 + s) << 12)) & 0x00ff00ffu) | 0x64006400u;
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&t), __half2half2(__ushort_as_half(0x6480)));
  return *reinterpret_cast<const uint32_t*>(&h);
}

// One operand: element (i, k) at p[i si + k sk], zero for k > i with tri; e[i]: the largest
// biased exponent of row i.
struct OzOperand {
  const double2* p;
  int si, sk;
  bool tri;
  int* e;
  __device__ __forceinline__ const double2* elem(int i, int k) const { return p + i * si + k * sk; }
  __device__ __forceinline__ int exponent(int i, int n) const { return i < n ? e[i] : 0; }
};

// e of the n rows of K elements, by the whole CTA; e is zero and visible before.
__device__ __forceinline__ void oz_exponents(const OzOperand& o, int n, int K) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nu = o.sk == 1 ? n : K, nv = o.sk == 1 ? K : n;
  for (int u = warp; u < nu; u += nw)
    for (int w = lane; w < nv; w += 32) {
      const int i = o.sk == 1 ? u : w, k = o.sk == 1 ? w : u;
      if (o.tri && k > i) continue;
      const double2 x = *o.elem(i, k);
      atomicMax(o.e + i, max(oz_row_exp(x.x), oz_row_exp(x.y)));
    }
}

// One 16 x 8 tile of sum_{k < K} A(i, k) B(j, k) (i < ni, j < nj), A conjugated with conj, by one warp: a lane gets
// rows i0 + lane/4 (out[0], out[1]) and 8 more (out[2], out[3]), columns j0 + 2 (lane % 4)
// and the next.
//
// A real 16 x 8 x 16 product takes 34 mma.sync.m16n8k16 and about 450 instructions for the
// digits of both tiles, taken from the FP64 values each time (kept in shared memory they
// would need 28 bytes an element); as FP64 multiply-adds it is 64 instructions of 64
// cycles each on the SMSP's FP64 unit.  Bound by issue slots.  Registers: 32 accumulators, 16 of
// A's fixed-point values, 14 of B's digits.  E and Q of a 256-wide core: D = 128, one colour
// class 355 -> 335 ms.
__device__ __noinline__ void oz_tile(const OzOperand A, const OzOperand B, bool conj, int i0, int j0, int ni, int nj,
                                     int K, double2* out) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t2 = 2 * (lane & 3);
  const int rc = j0 + g;
  const int kend = A.tri ? min(K, i0 + 16) : K;
  const int ea0 = A.exponent(i0 + g, ni), ea1 = A.exponent(i0 + g + 8, ni), ebf = B.exponent(rc, nj);
#pragma unroll 1
  for (int part = 0; part < 2; ++part) {
    long long tot[4] = {0, 0, 0, 0};
#pragma unroll 1
    for (int kc = 0; kc < kend; kc += 64) {
      float acc[kOzLevels][4];
#pragma unroll
      for (int l = 0; l < kOzLevels; ++l)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[l][q] = 0.f;
#pragma unroll 1
      for (int s = 0; s < 2 * ((min(kend - kc, 64) + 15) >> 4); ++s) {
        // re = Ar Br -+ Ai Bi, im = Ar Bi +- Ai Br
        const int h = s & 1, kb = kc + 16 * (s >> 1) + t2;
        const bool neg = h && (part ? conj : !conj);
        unsigned long long fa[8], fb[4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int z = 0; z < 2; ++z) {
            const int i = i0 + g + 8 * (r & 1), k = kb + 8 * (r >> 1) + z;
            double x = 0.0;
            if (i < ni && k < kend && !(A.tri && k > i)) x = reinterpret_cast<const double*>(A.elem(i, k))[h];
            fa[2 * r + z] = oz_fixed(x, r & 1 ? ea1 : ea0, neg);
          }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int k = kb + 8 * (r >> 1) + (r & 1);
          double x = 0.0;
          if (rc < nj && k < kend) x = reinterpret_cast<const double*>(B.elem(rc, k))[h ^ part];
          fb[r] = oz_fixed(x, ebf);
        }
        uint32_t bd[kOzSlices][2];
#pragma unroll
        for (int j = 0; j < kOzSlices; ++j) {
          bd[j][0] = oz_pair(fb[0], fb[1], j);
          bd[j][1] = oz_pair(fb[2], fb[3], j);
        }
#pragma unroll
        for (int i = 0; i < kOzSlices; ++i) {
          uint32_t ad[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) ad[r] = oz_pair(fa[2 * r], fa[2 * r + 1], i);
#pragma unroll
          for (int j = 0; j < (i ? kOzLevels - i : kOzSlices); ++j)
            asm volatile(
                "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                : "+f"(acc[i + j][0]), "+f"(acc[i + j][1]), "+f"(acc[i + j][2]), "+f"(acc[i + j][3])
                : "r"(ad[0]), "r"(ad[1]), "r"(ad[2]), "r"(ad[3]), "r"(bd[j][0]), "r"(bd[j][1]));
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        long long h = 0, low = 0;
#pragma unroll
        for (int l = 0; l < kOzLevels; ++l) (l < 4 ? h : low) += oz_weigh(acc[l][q], l);
        tot[q] += oz_sum(h, low);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = j0 + t2 + (q & 1);
      const double v = oz_value(tot[q], q & 2 ? ea1 : ea0, B.exponent(j, nj));
      if (part) out[q].y = v;
      else out[q].x = v;
    }
  }
}

// C(i, j) = sum_k A(i, k) B(j, k), n x n at C[i ci + j cj], A conjugated with conj, tiles
// below the diagonal left out with upper.  ex: 2n ints.  By the whole CTA; the operands are
// visible before, C after the caller's barrier.
__device__ __noinline__ void oz_product(const double2* a, int ai, int ak, bool conj, const double2* b, int bj, int bk,
                                           int* ex, double2* C, int ci, int cj, int n, bool upper) {
  const OzOperand A{a, ai, ak, false, ex}, B{b, bj, bk, false, ex + n};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = threadIdx.x; i < 2 * n; i += blockDim.x) ex[i] = 0;
  __syncthreads();
  oz_exponents(A, n, n);
  oz_exponents(B, n, n);
  __syncthreads();
  const int nt = (n + 7) >> 3;
  for (int t = warp; t < ((n + 15) >> 4) * nt; t += nw) {
    const int i0 = 16 * (t / nt), j0 = 8 * (t - (t / nt) * nt);
    if (upper && j0 + 7 < i0) continue;
    double2 out[4];
    oz_tile(A, B, conj, i0, j0, n, n, n, out);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + (lane >> 2) + (q & 2) * 4, j = j0 + 2 * (lane & 3) + (q & 1);
      if (i < n && j < n) C[i * ci + j * cj] = out[q];
    }
  }
}

// V += V M in place, M upper triangular (row stride ldm; below its diagonal anything).  A
// warp takes 8 rows of V and goes over their columns from the right: columns j0.. of the
// result read columns up to j0 + 15 only.
__device__ __noinline__ void oz_correct(double2* V, int n, const double2* M, int ldm, int* ex) {
  const OzOperand A{M, 1, ldm, true, ex}, B{V, n, 1, false, ex + n};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = threadIdx.x; i < 2 * n; i += blockDim.x) ex[i] = 0;
  __syncthreads();
  oz_exponents(A, n, n);
  oz_exponents(B, n, n);
  __syncthreads();
  for (int r0 = 8 * warp; r0 < n; r0 += 8 * nw)
    for (int j0 = ((n - 1) >> 4) << 4; j0 >= 0; j0 -= 16) {
      double2 out[4];
      oz_tile(A, B, false, j0, r0, n, n, n, out);
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = j0 + (lane >> 2) + (q & 2) * 4, r = r0 + 2 * (lane & 3) + (q & 1);
        if (j < n && r < n) {
          double2* v = V + r * n + j;
          *v = make_double2(v->x + out[q].x, v->y + out[q].y);
        }
      }
      __syncwarp();
    }
}

}  // namespace gpeps
