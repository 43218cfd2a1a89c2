// Preparation of one FP64 position (a1, Sec. 2.3): wrapped into [0, L), split into the integer cell and the FP32
// offset of the grid. Shared by the preparation kernels and by the adjoint's gather, which rounds
// positions as the forward path did.
#pragma once

#include "internal.cuh"

namespace pk {

// floor(u) and the fraction u - floor(u) rounded to FP32 (to nearest, ties to even) for 0 <= u < 2^20,
// read from u's bits with integer operations: FP64 arithmetic is scarce on this GPU, and the fraction
// of a double is exact in its significand, so this equals float(u - floor(u)) bit for bit. (A call: as an inlined
// branch its FP64 conversion would be issued, predicated off, for every particle.)
static __device__ __noinline__ void split_units_any(double u, int* c, float* f) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(u));
  const int e = int((b >> 52) & 0x7ff) - 1023;
  if (e < 0) {  // u in [0, 1), or -0: floor 0 (+ 0.0f makes -0 the +0 that u - floor(u) gives)
    *c = 0;
    *f = __double2float_rn(u) + 0.0f;
    return;
  }
  const int sh = 52 - e;  // fraction bits of the significand (32 < sh <= 52 for u < 2^20)
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  *c = int(m >> sh);
  const unsigned long long fr = m & ((1ull << sh) - 1);  // u - floor(u) = fr 2^-sh exactly
  if (fr == 0) {
    *f = 0.0f;
    return;
  }
  const int top = 63 - __clzll(static_cast<long long>(fr));  // fr in [2^top, 2^(top+1)), top < sh
  unsigned long long m24;  // 24-bit significand, rounded; 2^24 when the rounding carries
  if (top >= 24) {
    const int d = top - 23;
    m24 = fr >> d;
    const unsigned long long rem = fr & ((1ull << d) - 1), half = 1ull << (d - 1);
    if (rem > half || (rem == half && (m24 & 1ull))) ++m24;
  } else {
    m24 = fr << (23 - top);
  }
  const int ex = top - sh + 127;  // biased exponent of 2^(top - sh), >= 75
  *f = __int_as_float(int((unsigned(ex - 1) << 23) + unsigned(m24)));
}

// The same from 32-bit instructions, for all u but the rare ones (u below 2^-60, fractions below 2^-32). The significand
// left-aligned in 64 bits, M = Mh:Ml, is u 2^(63 - e); shifted left by e + 1 its integer part is gone and
// the fraction is FR 2^-64. Normalised, the top 32 bits with a sticky last bit hold 32 > 25 significant
// bits, so the integer-to-float conversion rounds them as the whole fraction would round (to nearest, ties
// to even), and the power of two is exact. (k_prepare_hist was bound by the 64-bit shifts and
// comparisons of split_units_any: 421 instructions per warp of particles; 256^3 particles 243 us, now 202.)
__device__ __forceinline__ void split_units(double u, int* c, float* f) {
  const unsigned hi = unsigned(__double2hiint(u)), lo = unsigned(__double2loint(u));
  const int e = int(hi >> 20) - 1023;  // u >= 0 (the sign bit of -0 makes e large: the rare path)
  const unsigned mh = __funnelshift_l(lo, (hi & 0x000fffffu) | 0x00100000u, 11), ml = lo << 11;
  unsigned fh = mh, fl = ml;
  int sc = e - 31;  // f = (top 32 bits) 2^sc
  int ci = 0;
  if (e >= 0) {
    ci = int(mh >> (31 - (e & 31)));
    fh = __funnelshift_l(ml, mh, e + 1);
    fl = ml << ((e + 1) & 31);
    const int nz = __clz(int(fh));
    fh = __funnelshift_l(fl, fh, nz);
    fl = fl << (nz & 31);
    sc = -32 - nz;
  }
  if (unsigned(e + 60) < 80u && fh != 0u) {  // -60 <= e < 20
    *c = ci;
    *f = __uint2float_rn(fh | (fl != 0u ? 1u : 0u)) * __int_as_float((127 + sc) << 23);
  } else {
    split_units_any(u, c, f);
  }
}

// One FP64 position as a packed cell and FP32 offsets; *nonfinite: a coordinate is NaN or infinite, and the record
// is cell 0, offset 0.
__device__ __forceinline__ pk_cellpos prepare_one(const double* p, int ng, double box, double scale, bool* nonfinite) {
  pk_cellpos r;
  int c[3];
  float fo[3];
  bool bad = false;
  const unsigned long long box_bits = static_cast<unsigned long long>(__double_as_longlong(box));
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double x = p[a];
    const unsigned long long xb = static_cast<unsigned long long>(__double_as_longlong(x));
    if (xb >= box_bits) {  // negative (sign bit), >= L (another periodic image), or not finite
      if (((xb >> 52) & 0x7ff) == 0x7ff) {
        bad = true;
        x = 0.0;
      } else {
        x = fmod(x, box);
        if (x < 0.0) x += box;
      }
    }
    int ci;
    float ff;
    split_units(x * scale, &ci, &ff);
    if (ci >= ng) { ci -= ng; }
    if (ff >= 1.0f) {  // f rounded up to 1 in FP32: the particle sits on the next node
      ff = 0.0f;
      ci = ci + 1 == ng ? 0 : ci + 1;
    }
    c[a] = ci;
    fo[a] = ff;
  }
  *nonfinite = bad;
  if (bad) {
    c[0] = c[1] = c[2] = 0;
    fo[0] = fo[1] = fo[2] = 0.0f;
  }
  r.cell = pack_cell(c[0], c[1], c[2]);
  r.fx = fo[0];
  r.fy = fo[1];
  r.fz = fo[2];
  return r;
}

}  // namespace pk
