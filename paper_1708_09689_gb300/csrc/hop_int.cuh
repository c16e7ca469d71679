// The hopping sum of the complex128 TI sweeps on the integer pipes.
//
// Each real part of T = Gamma^1 S + sum_j (-i Gamma^{j+1}) d_j (sweep.cuh) is a sum of twelve
// neighbour values with signs.  The fp64 pipe of this part has two lanes per SM, its integer
// pipes 64: aligning the twelve values to one exponent and adding them as 64-bit integers takes
// about 140 integer instructions for a part and one fp64 instruction (the conversion back), where
// the projected fp64 sum takes 8 fp64 instructions of 32 times the cost.
//
// Accuracy.  E: the largest exponent field among the twelve inputs of this part (of these alone:
// a part whose inputs are small keeps its own scale).  An input m 2^(e - 1081), m its 53-bit
// significand shifted to the bits 58 .. 6, enters as m >> (E - e), cut off below 2^-58 of the
// power of two above the largest input; inputs within six binary places of the largest enter
// exactly.  The sum of twelve stays below 2^63 and is exact.  The error, at most 12 2^(E - 1081)
// and typically 2^(E - 1080), is below one rounding of a partial sum of that size in fp64
// (2^(E - 1076)), of which the fp64 sum makes up to eleven; the conversion rounds once.  This is a bound
// against the magnitude of the inputs, not against the result: where the large inputs of a part cancel
// exactly, inputs below 2^-58 of them are lost, which an fp64 sum keeps if it happens to add the
// cancelling ones first.  Parts with an exponent field outside [128, 1900] (zeros, subnormals, infinities, NaN) are left to the
// fp64 sum.
#pragma once

#include <cuda_runtime.h>

namespace pvsc {

struct FixTerm {
  unsigned lo, hi;  // 53-bit significand at bits 58 .. 6
  int e;            // exponent field
  unsigned s;       // all ones if negative
};

__device__ __forceinline__ FixTerm fix_term(double v) {
  const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
  FixTerm t;
  t.e = (int)((h & 0x7fffffffu) >> 20);
  t.s = (unsigned)((int)h >> 31);
  const unsigned mh = (h & 0xfffffu) | 0x100000u;
  t.hi = __funnelshift_l(l, mh, 6);
  t.lo = l << 6;
  return t;
}

// One real part of the sum: terms are added as one's complements and the count of the negative
// ones, kept negative in neg, completes them.
struct FixSum {
  unsigned long long a;
  int neg, E;
};

template <bool MINUS>
__device__ __forceinline__ unsigned long long fix_aligned(const FixTerm& t, int E) {
  const unsigned long long m = ((unsigned long long)t.hi << 32) | t.lo;
  unsigned long long v;
  // shifts by 64 and more give 0 (the PTX shift clamps)
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"((unsigned)(E - t.e)));
  const unsigned s = MINUS ? ~t.s : t.s;
  return v ^ (((unsigned long long)s << 32) | s);
}

// Both neighbours of an axis at once: three-operand additions.
template <bool MA, bool MB>
__device__ __forceinline__ void fix_add2(FixSum& f, const FixTerm& ta, const FixTerm& tb) {
  f.a = f.a + fix_aligned<MA>(ta, f.E) + fix_aligned<MB>(tb, f.E);
  f.neg = f.neg + (int)(MA ? ~ta.s : ta.s) + (int)(MB ? ~tb.s : tb.s);
}

__device__ __forceinline__ unsigned fix_mag(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// Index (2 component + part) that part c of a neighbour's component k enters besides its own: the
// axes are 0 z, 1 x, 2 y.
__host__ __device__ constexpr int hop_partner(int axis, int k, int c) {
  return axis == 0 ? 2 * (k ^ 1) + c : (axis == 1 ? 2 * (3 - k) + c : 2 * (3 - k) + 1 - c);
}
// Its sign there for the neighbour at n - e_j (the one at n + e_j enters with the other sign):
// z: T_0 += d_1, T_1 -= d_0, T_2 += d_3, T_3 -= d_2; x: T_0 += d_3, T_1 += d_2, T_2 -= d_1, T_3 -= d_0;
// y: T_{3-k} += -i d_k = (d_k.im, -d_k.re); d = x(n - e_j) - x(n + e_j).
__host__ __device__ constexpr bool hop_partner_minus(int axis, int k, int c) {
  return axis == 0 ? (k & 1) == 0 : (axis == 1 ? k < 2 : c == 0);
}

// H: T in units of 2^(E - 1081) per part (as doubles); off: (E - 1081) << 20, to be added to the high
// word of a factor.  False (nothing written): some part is outside the exponent range.
// get(axis, a, b): the neighbour blocks at n - e_j and n + e_j, asked for twice (the exponents come
// first); RELOAD: they are cheap to read again (shared memory) and are not kept between the passes.
template <bool RELOAD, class Get>
__device__ __forceinline__ bool hop_int(Get&& get, Blk<double, 1>& H, int (&off)[8]) {
  unsigned m[8] = {};  // largest magnitude (high words) that enters each part
#pragma unroll
  for (int axis = 0; axis < 3; ++axis) {
    Blk<double, 1> a, b;
    get(axis, a, b);
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const unsigned g = c ? max(fix_mag(a.v[k][0].im), fix_mag(b.v[k][0].im))
                             : max(fix_mag(a.v[k][0].re), fix_mag(b.v[k][0].re));
        m[2 * k + c] = max(m[2 * k + c], g);
        m[hop_partner(axis, k, c)] = max(m[hop_partner(axis, k, c)], g);
      }
  }
  FixSum f[8];
  bool ok = true;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    f[i].E = (int)(m[i] >> 20);
    f[i].a = 0;
    f[i].neg = 0;
    ok = ok && (unsigned)(f[i].E - 128) <= 1900u - 128u;
  }
  if (!ok) return false;
  if constexpr (RELOAD) asm volatile("" ::: "memory");
#pragma unroll
  for (int axis = 0; axis < 3; ++axis) {
    Blk<double, 1> a, b;
    get(axis, a, b);
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const FixTerm ta = fix_term(c ? a.v[k][0].im : a.v[k][0].re), tb = fix_term(c ? b.v[k][0].im : b.v[k][0].re);
        FixSum &own = f[2 * k + c], &par = f[hop_partner(axis, k, c)];
        if (k & 1) fix_add2<true, true>(own, ta, tb);  // Gamma^1 = diag(1, -1, 1, -1)
        else fix_add2<false, false>(own, ta, tb);
        if (hop_partner_minus(axis, k, c)) fix_add2<true, false>(par, ta, tb);
        else fix_add2<false, true>(par, ta, tb);
      }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const double v = (double)((long long)f[i].a - f[i].neg);
    if (i & 1) H.v[i / 2][0].im = v; else H.v[i / 2][0].re = v;
    off[i] = (f[i].E - 1081) << 20;
  }
  return true;
}

// A factor whose exponent field lies well inside the range, so that the offsets of hop_int keep it normal.
__device__ __forceinline__ bool hop_int_factor(double kt) {
  return (unsigned)(((__double2hiint(kt) & 0x7fffffff) >> 20) - 960) <= 1200u - 960u;
}

}  // namespace pvsc
