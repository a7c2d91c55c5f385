// Device helpers shared by the query kernels.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "uhnsw.h"

namespace uhnsw_dev {

constexpr uint32_t kExpanded = 0x80000000u;  // beam entry already expanded
constexpr uint32_t kIdMask = 0x7fffffffu;
constexpr int32_t kEmpty = -1;
constexpr unsigned kFull = 0xffffffffu;

// (da, ia) before (db, ib) in the (distance, id) order used everywhere.
__device__ __forceinline__ bool pair_lt(float da, int32_t ia, float db, int32_t ib) {
  return da < db || (da == db && ia < ib);
}

// Row storage types: 16 bytes hold 4 FP32 or 8 FP16/BF16 values.
template <typename T> struct Elems16;
template <> struct Elems16<float> { static constexpr int n = 4; };
template <> struct Elems16<__half> { static constexpr int n = 8; };
template <> struct Elems16<__nv_bfloat16> { static constexpr int n = 8; };

template <typename T>
__device__ __forceinline__ void unpack16(const uint4& v, float* out);

template <>
__device__ __forceinline__ void unpack16<float>(const uint4& v, float* out) {
  out[0] = __uint_as_float(v.x);
  out[1] = __uint_as_float(v.y);
  out[2] = __uint_as_float(v.z);
  out[3] = __uint_as_float(v.w);
}

template <>
__device__ __forceinline__ void unpack16<__half>(const uint4& v, float* out) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __half2 h = *reinterpret_cast<const __half2*>(&w[i]);
    float2 f = __half22float2(h);
    out[2 * i] = f.x;
    out[2 * i + 1] = f.y;
  }
}

template <>
__device__ __forceinline__ void unpack16<__nv_bfloat16>(const uint4& v, float* out) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&w[i]);
    float2 f = __bfloat1622float2(h);
    out[2 * i] = f.x;
    out[2 * i + 1] = f.y;
  }
}

// Hardware base-2 logarithm and exponential (the SFU instructions).
__device__ __forceinline__ float hw_lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float hw_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float hw_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// |a|^p for the verification modes: general p as 2^(p log2 |a|) (two SFU
// operations; |0|^p = 2^-inf = 0), p = 0.5 and p = 1.5 through one square
// root (Section 2.1's fast cases), p = 1 and p = 2 without the SFU.
enum PMode { kPGeneral = 0, kPHalf = 1, kPThreeHalves = 2, kPOne = 3, kPTwo = 4 };

__device__ __forceinline__ int pmode_of(float p) {
  if (p == 1.0f) return kPOne;
  if (p == 2.0f) return kPTwo;
  if (p == 0.5f) return kPHalf;
  if (p == 1.5f) return kPThreeHalves;
  return kPGeneral;
}

template <int PM>
__device__ __forceinline__ float pow_term(float a, float p) {
  if (PM == kPOne) return a;
  if (PM == kPTwo) return a * a;
  if (PM == kPHalf) return hw_sqrt(a);
  if (PM == kPThreeHalves) return a * hw_sqrt(a);
  return hw_ex2(p * hw_lg2(a));
}

// Records the first error code of a launch into the sticky device word
// (err[0]; err[1..3] hold the site, value and limit of a failed index check).
__device__ __forceinline__ void set_error(int32_t* err, int32_t code) {
  if (err) atomicCAS(err, 0, code);
}

// Index check of the diagnostic build (compiled with -DUHNSW_CHECK): an index
// outside [0, limit) is recorded (code UHNSW_ECAPACITY, site, value, limit)
// and replaced by 0 so that the access stays inside the buffer.  In the
// normal build it is the identity.
__device__ __forceinline__ int64_t chk_idx(int64_t i, int64_t limit, int site, int32_t* err) {
#ifdef UHNSW_CHECK
  if (i < 0 || i >= limit) {
    if (err && atomicCAS(err, 0, UHNSW_ECAPACITY) == 0) {
      err[1] = site;
      err[2] = (int32_t)i;
      err[3] = (int32_t)limit;
    }
    return 0;
  }
#else
  (void)limit;
  (void)site;
  (void)err;
#endif
  return i;
}

__device__ __forceinline__ uint32_t hash_slot(int32_t id, int bits) {
  return ((uint32_t)id * 0x9E3779B1u) >> (32 - bits);
}

// Insert `id` into the open-addressing table (linear probing); true if it was
// absent.  The caller keeps the load at or below one half, so a free slot is
// always found within the table size.
__device__ __forceinline__ bool hash_insert(int32_t* tab, int bits, int32_t id, int32_t* err) {
  const uint32_t mask = (1u << bits) - 1u;
  uint32_t s = hash_slot(id, bits);
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    int32_t old = atomicCAS(&tab[s], kEmpty, id);
    if (old == kEmpty) return true;
    if (old == id) return false;
    s = (s + 1u) & mask;
  }
  set_error(err, UHNSW_ECAPACITY);
  return false;
}

// Number of entries of the ascending (d, id) list [0, n) that precede (x, xi).
__device__ __forceinline__ int lower_bound_pair(const float* d, const uint32_t* id, int n, float x,
                                                int32_t xi) {
  int lo = 0, hi = n;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (pair_lt(d[mid], (int32_t)(id[mid] & kIdMask), x, xi)) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Two FP32 lanes in one 64-bit register: Blackwell's paired FP32 instructions
// (sub / add / fma .f32x2, IEEE round-to-nearest per element).
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ float f2_hsum(uint64_t v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a + b;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// s^(1/p) for a sum s >= 0 and p in (0, 2], to within 2^-44 of the exact value
// before the one rounding to FP32 (p = 1/2, 1 and 2 are correctly rounded).
// Measured on a host restatement with the reciprocals off by up to one unit, 48
// million s and p in [0.001, 2] whose roots cover the normal FP32 range: at most
// 2^-44.6, and one FP32 value beside the correctly rounded one, as with FP64's pow.
//
// This chip retires 2 FP64 operations a clock and SM, so a pow per returned
// distance was 0.07 of 0.29 ms of a verification of 5,003 queries at K = 50.
// Here log2 is the atanh series of (m - 1) / (m + 1) for the mantissa m in
// [sqrt(1/2), sqrt(2)), 2^f is e^(f ln 2)'s Taylor series for |f| <= 1/2, and
// the tails of both, 2^-20 of the sum or less, are summed in FP32.
__device__ __forceinline__ float root_p(float s, float p) {
  if (p == 1.0f) return s;
  if (p == 2.0f) return __fsqrt_rn(s);
  if (p == 0.5f) return __double2float_rn((double)s * (double)s);
  if (!(s > 0.0f) || s == __int_as_float(0x7f800000)) return s;  // 0, +inf, NaN
  // s = m 2^e (a subnormal FP32 value is a normal FP64 one)
  const double sd = (double)s;
  const int hi = __double2hiint(sd);
  const int e = (hi - 0x3fe6a09e) >> 20;  // the high word of sqrt(1/2)
  const double m = __hiloint2double(hi - (e << 20), __double2loint(sd));
  const double num = m - 1.0, den = m + 1.0;
  float rden;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rden) : "f"((float)den));
  const double rd = (double)rden;
  double u = num * rd;
  // 2^-46, then as far as FP64 goes (as a loop: unrolled, the step moves registers in
  // the search kernels, and 1,000 queries of 1M x 96 FP16 at ef 512 take 1 % longer)
#pragma unroll 1
  for (int i = 0; i < 2; ++i) u = fma(fma(-u, den, num), rd, u);
  const double w = u * u;
  const float wf = (float)w;
  float lt = fmaf(wf, 1.0f / 19, 1.0f / 17);
  lt = fmaf(wf, lt, 1.0f / 15);
  lt = fmaf(wf, lt, 1.0f / 13);
  lt = fmaf(wf, lt, 1.0f / 11);
  double l = fma(w, (double)lt, 1.0 / 9);
  l = fma(w, l, 1.0 / 7);
  l = fma(w, l, 1.0 / 5);
  l = fma(w, l, 1.0 / 3);
  l = fma(w, l, 1.0);
  constexpr double kLn2 = 0.693147180559945309417232;
  l = fma(u * (2.0 / kLn2), l, (double)e);
  // (the hardware reciprocal flushes p below 2^-126 and gives +inf; any s but 1
  // leaves FP32's range long before 2^100.  Bounding p itself took 4 % more time in
  // the search of 1,000 queries of 1M x 96 FP16 at ef 512, by its registers.)
  float rp;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rp) : "f"(p));
  rp = fminf(rp, 0x1p100f);
  const double pd = (double)p;
  double inv = (double)rp;
  inv = fma(inv, fma(-pd, inv, 1.0), inv);
  inv = fma(inv, fma(-pd, inv, 1.0), inv);
  // an exponent beyond FP32's range rounds to 0 or +inf all the same
  const double z = fmin(fmax(l * inv, -1000.0), 1000.0);
  const int n = __double2int_rn(z);
  const double t = (z - (double)n) * kLn2;
  const float tf = (float)t;
  float et = fmaf(tf, 1.0f / 479001600, 1.0f / 39916800);
  et = fmaf(tf, et, 1.0f / 3628800);
  et = fmaf(tf, et, 1.0f / 362880);
  et = fmaf(tf, et, 1.0f / 40320);
  double x = fma(t, (double)et, 1.0 / 5040);
  x = fma(t, x, 1.0 / 720);
  x = fma(t, x, 1.0 / 120);
  x = fma(t, x, 1.0 / 24);
  x = fma(t, x, 1.0 / 6);
  x = fma(t, x, 0.5);
  x = fma(t, x, 1.0);
  x = fma(t, x, 1.0);
  return __double2float_rn(__hiloint2double(__double2hiint(x) + (n << 20), __double2loint(x)));
}

}  // namespace uhnsw_dev
