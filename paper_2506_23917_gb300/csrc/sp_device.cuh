// sp_device.cuh -- device code of libsp: Philox streams, the per-cell
// collision step and the free-flight / wall / reservoir step of the hybrid
// stochastic-particle Shakhov / DSMC method (arXiv:2506.23917, Sec. III.B).
//
// Templated on the particle precision T (double: FP64 mode, float: FP32
// mode) and the spatial dimension DIM.  Per-cell quantities (moments, tau,
// dt_c, the DSMC/Shakhov split, exp(-dt/tau), rescale factors, time
// averages) are always FP64; per-particle arithmetic runs in T.
#pragma once
#include <cstddef>
#include <cstdint>
#include <type_traits>

#include "sp_internal.h"

namespace sp {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr double kPi = 3.141592653589793238462643383279502884;

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): 10 rounds of two 32x32->64
// multiplications with Weyl-bumped keys.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                          uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return make_uint4(c0, c1, c2, c3);
}

// FP64 uniform in (0,1): 52 bits from two words, (2k+1) 2^-53.  Formed as
// (1 + k 2^-52) - (1 - 2^-53), exact in one subtraction: on GB300 an FP64
// operation or 64-bit conversion holds the SM's FP64 pipe for ~17 cycles.
__device__ __forceinline__ double u01d(uint32_t a, uint32_t b) {
  const unsigned long long k = ((unsigned long long)(a >> 6) << 26) | (unsigned long long)(b >> 6);
  return __longlong_as_double((long long)(0x3FF0000000000000ull | k)) -
         __longlong_as_double(0x3FEFFFFFFFFFFFFFll);
}
// The same uniform in FP32, to 2^-22 relative.
__device__ __forceinline__ float u01d_approx(uint32_t a, uint32_t b) {
  return fmaf((float)(a >> 6), 1.490116119384765625e-8f, (float)(2u * (b >> 6) + 1u) * 1.1102230246251565e-16f);
}
// An FP64 value in FP32 (truncated, relative error below 2^-23) by integer
// operations only; zero below FP32's normal range, infinity above it.
__device__ __forceinline__ float approx_f32(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t e = (hi >> 20) & 0x7FFu;
  uint32_t m = (((hi & 0x7FFFFFFFu) - (896u << 20)) << 3) | (lo >> 29);
  if (e < 897u) m = 0u;
  if (e > 1150u) m = 0x7F800000u;
  return __uint_as_float(m | (hi & 0x80000000u));
}
// FP32 uniform in (0,1): 23 bits from one word, (2k+1) 2^-24.
__device__ __forceinline__ float u01f(uint32_t a) {
  return (float)(2u * (a >> 9) + 1u) * 5.9604644775390625e-8f;
}

// An FP32 value widened exactly, by integer operations (the conversion
// instruction goes through the FP64 pipe); subnormals take the instruction.
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x), m = u & 0x7FFFFFFFu;
  if ((m < 0x00800000u && m != 0u) || m >= 0x7F800000u) return (double)x;
  const uint32_t hi = m ? (u & 0x80000000u) | ((m >> 3) + 0x38000000u) : u;
  return __hiloint2double((int)hi, (int)(u << 29));
}

// A uniform stream addressed by (step, a, b, purpose<<24 | sub); the q-th
// uniform lives in block q/2 (FP64) or q/4 (FP32) of the counter word 3.
template <class T>
struct Uni;

template <>
struct Uni<double> {
  uint32_t c0, c1, c2, c3, k0, k1;
  int blk;
  uint4 w;
  __device__ Uni(uint32_t step, uint32_t a, uint32_t b, uint32_t c3base, uint32_t key0, uint32_t key1)
      : c0(step), c1(a), c2(b), c3(c3base), k0(key0), k1(key1), blk(-1) {}
  __device__ __forceinline__ double get(int q) {
    const int bq = q >> 1;
    if (bq != blk) {
      w = philox10(c0, c1, c2, c3 + (uint32_t)bq, k0, k1);
      blk = bq;
    }
    return (q & 1) ? u01d(w.z, w.w) : u01d(w.x, w.y);
  }
};

template <>
struct Uni<float> {
  uint32_t c0, c1, c2, c3, k0, k1;
  int blk;
  uint4 w;
  __device__ Uni(uint32_t step, uint32_t a, uint32_t b, uint32_t c3base, uint32_t key0, uint32_t key1)
      : c0(step), c1(a), c2(b), c3(c3base), k0(key0), k1(key1), blk(-1) {}
  __device__ __forceinline__ float get(int q) {
    const int bq = q >> 2;
    if (bq != blk) {
      w = philox10(c0, c1, c2, c3 + (uint32_t)bq, k0, k1);
      blk = bq;
    }
    const int r = q & 3;
    return u01f(r == 0 ? w.x : r == 1 ? w.y : r == 2 ? w.z : w.w);
  }
};

// Asynchronous global -> shared copy of one 4- or 8-byte element (no
// register staging), and the wait for all of this thread's copies.
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(gsrc), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// Precision helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ double tsqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float tsqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double tlog(double x) { return log(x); }
__device__ __forceinline__ float tlog(float x) { return logf(x); }
__device__ __forceinline__ double tpow(double x, double e) { return pow(x, e); }
__device__ __forceinline__ float tpow(float x, float e) { return powf(x, e); }
__device__ __forceinline__ double tfloor(double x) { return floor(x); }
__device__ __forceinline__ float tfloor(float x) { return floorf(x); }
__device__ __forceinline__ double tfabs(double x) { return fabs(x); }
__device__ __forceinline__ float tfabs(float x) { return fabsf(x); }
// Division and power of the per-cell scalars and of the pairs' sigma c:
// FP64 mode keeps the IEEE operations (the oracle's rounding); FP32 mode,
// where these only set rates, split weights and acceptance probabilities,
// uses the hardware approximations (division within 2 ulp for divisors
// below 2^126, power through exp2/log2), which shorten the dependent chains
// on the lanes.
__device__ __forceinline__ double cdiv(double x, double y) { return x / y; }
__device__ __forceinline__ float cdiv(float x, float y) { return __fdividef(x, y); }
__device__ __forceinline__ double cpow(double x, double e) { return pow(x, e); }
__device__ __forceinline__ float cpow(float x, float e) { return __powf(x, e); }
// Square root and natural logarithm on the per-particle sampling paths
// (pair speeds, Box-Muller radii): FP32 mode uses the hardware
// approximations (sqrt.approx, lg2.approx scaled by ln 2).
__device__ __forceinline__ double csqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float csqrt(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double clog(double x) { return log(x); }
__device__ __forceinline__ float clog(float x) { return __logf(x); }
__device__ __forceinline__ double tmax0(double x) { return x; }  // exact log: -log(R) >= 0 already
__device__ __forceinline__ float tmax0(float x) { return fmaxf(x, 0.0f); }

// cos / sin of 2 pi u
__device__ __forceinline__ void sincos2pi(double u, double* s, double* c) {
  sincospi(2.0 * u, s, c);
}
__device__ __forceinline__ void sincos2pi(float u, float* s, float* c) { sincospif(2.0f * u, s, c); }
__device__ __forceinline__ double cos2pi(double u) { return cospi(2.0 * u); }
__device__ __forceinline__ float cos2pi(float u) { return cospif(2.0f * u); }

// The five uniforms of NTC candidate kk: pair (u1, u2), acceptance u3,
// scattering cos(chi) from u4 and azimuth from u5.  FP64 mode: three Philox
// blocks (shared layout with the oracle), the third formed for accepted
// candidates only.  FP32 mode: one block; u4 and u5
// take 16 bits each of the fourth word ((2k+1) 2^-17), ample for angles.
template <class T>
struct NtcDraw;
template <>
struct NtcDraw<double> {
  uint4 w0, w1;  // u1 u2, u3 u4
  double u1, u2;
  __device__ __forceinline__ double u3() const { return u01d(w1.x, w1.y); }
  __device__ __forceinline__ float u3_approx() const { return u01d_approx(w1.x, w1.y); }
  __device__ __forceinline__ double u4() const { return u01d(w1.z, w1.w); }
};
template <>
struct NtcDraw<float> {
  float u1, u2, u3, u4, u5;
};
__device__ __forceinline__ NtcDraw<double> ntc_draw(double, uint32_t step, uint32_t kl, uint32_t kk,
                                                    uint32_t key0, uint32_t key1) {
  NtcDraw<double> d;
  d.w0 = philox10(step, kl, kk, kPurpNtc << 24, key0, key1);
  d.w1 = philox10(step, kl, kk, (kPurpNtc << 24) + 1u, key0, key1);
  d.u1 = u01d(d.w0.x, d.w0.y);
  d.u2 = u01d(d.w0.z, d.w0.w);
  return d;
}
__device__ __forceinline__ double ntc_u5(uint32_t step, uint32_t kl, uint32_t kk, uint32_t key0, uint32_t key1) {
  const uint4 w = philox10(step, kl, kk, (kPurpNtc << 24) + 2u, key0, key1);
  return u01d(w.x, w.y);
}
__device__ __forceinline__ NtcDraw<float> ntc_draw(float, uint32_t step, uint32_t kl, uint32_t kk,
                                                   uint32_t key0, uint32_t key1) {
  const uint4 w = philox10(step, kl, kk, kPurpNtc << 24, key0, key1);
  NtcDraw<float> d;
  d.u1 = u01f(w.x);
  d.u2 = u01f(w.y);
  d.u3 = u01f(w.z);
  d.u4 = (float)(2u * (w.w >> 16) + 1u) * 7.62939453125e-6f;
  d.u5 = (float)(2u * (w.w & 0xFFFFu) + 1u) * 7.62939453125e-6f;
  return d;
}

// FP64 mode's test of an NTC candidate: sigma c = coef c_r^ex costs a square
// root and a power, over 100 operations of the FP64 pipe, and is needed only
// for decisions -- whether it raises (sigma c)_max, and whether
// u3 < sigma c / (sigma c)_max.  An FP32 estimate (relative error below 1e-5,
// the sum of the rounding of its inputs, powf and ex ln c_r) settles both
// unless it comes within 1e-4 of the line; only then is the FP64 value
// formed, so that every decision is the FP64 one.  (With the flight's and the
// Shakhov step's filters: Sod tube of 11 k particles 0.43 -> 0.31 ms per step.)
struct NtcTest {
  double sc;   // sigma c where it was formed, else -1 (then below S)
  float est;   // estimate of sigma c / S, S = (sigma c)_max before the round
  bool exact;  // sc was formed
};
__device__ __forceinline__ double ntc_sigc(double g0, double g1, double g2, double coef, double ex) {
  return coef * cpow(csqrt(g0 * g0 + g1 * g1 + g2 * g2), ex);
}
__device__ __forceinline__ NtcTest ntc_test(double g0, double g1, double g2, double S, double coef, double ex,
                                            float coef32, float ex32) {
  NtcTest o;
  const float x = approx_f32(g0), y = approx_f32(g1), z = approx_f32(g2), S32 = approx_f32(S);
  const float c2 = x * x + y * y + z * z;
  const float sc32 = coef32 * powf(sqrtf(c2), ex32);
  o.est = sc32 / S32;
  const bool sure = c2 > 1e-30f && c2 < 1e30f && S32 > 1e-30f && S32 < 1e30f && sc32 > 1e-30f && o.est < 0.9999f;
  o.exact = !sure;
  o.sc = -1.0;
  if (!sure) o.sc = ntc_sigc(g0, g1, g2, coef, ex);
  return o;
}
// u3 < sigma c / smL, with smL >= S the running maximum up to the candidate.
__device__ __forceinline__ bool ntc_pass(const NtcTest& o, const NtcDraw<double>& dr, double g0, double g1, double g2,
                                         double S, double smL, double coef, double ex) {
  if (!o.exact && smL == S) {
    const float u = dr.u3_approx();
    if (u < o.est * 0.9999f) return true;
    if (u > o.est * 1.0001f) return false;
  }
  const double sc = o.exact ? o.sc : ntc_sigc(g0, g1, g2, coef, ex);
  return dr.u3() < sc / smL;
}

template <class T>
__device__ __forceinline__ T tinf();
template <>
__device__ __forceinline__ double tinf<double>() { return __longlong_as_double(0x7FF0000000000000ll); }
template <>
__device__ __forceinline__ float tinf<float>() { return __int_as_float(0x7F800000); }

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(kFull, v, m);
  return v;
}

// ---------------------------------------------------------------------------
// Geometry: cell index, free flight with walls and body (Step 2).
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ const Geo<T>& geo(const InstParams& P);
template <>
__device__ __forceinline__ const Geo<double>& geo<double>(const InstParams& P) { return P.g64; }
template <>
__device__ __forceinline__ const Geo<float>& geo<float>(const InstParams& P) { return P.g32; }

template <class T, int DIM>
__device__ __forceinline__ uint32_t cell_of(const InstParams& P, const T* x) {
  const Geo<T>& G = geo<T>(P);
  uint32_t idx[3] = {0, 0, 0};
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    const T f = tfloor((x[d] - G.lo[d]) * G.inv_d[d]);
    int i = (int)f;
    if (f < (T)0) i = 0;
    if (i > P.n[d] - 1) i = P.n[d] - 1;
    idx[d] = (uint32_t)i;
  }
  return idx[0] + (uint32_t)P.n[0] * (idx[1] + (uint32_t)P.n[1] * idx[2]);
}

// Whether the crossing point x of face f lies in the face's open window.
template <class T, int DIM>
__device__ __forceinline__ bool face_open(const Geo<T>& G, int f, const T* x) {
  const int ax = f >> 1;
  int i = 0;
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    if (d == ax) continue;
    const T w0 = G.win_lo[f][i], w1 = G.win_hi[f][i];
    if (w0 < w1 && (x[d] < w0 || x[d] > w1)) return false;
    ++i;
  }
  return true;
}

// Bird's sub-cells (option): the sub-cell of a particle at x in the
// instance-local cell kl -- on each axis the cell coordinate
// u = (x - lo) n / L (cell_of's expression) minus the cell's index, split
// into P.subcells equal parts (clamped).
template <class T, int DIM>
__device__ __forceinline__ int subcell_of(const InstParams& P, int64_t kl, const T* x) {
  const Geo<T>& G = geo<T>(P);
  const int ns = P.subcells;
  int64_t kk = kl;
  int sub = 0, mul = 1;
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    const int64_t id = kk % P.n[d];
    kk /= P.n[d];
    const T u = (x[d] - G.lo[d]) * G.inv_d[d];
    const T f = tfloor((u - (T)id) * (T)ns);
    int t = (int)f;
    if (f < (T)0) t = 0;
    if (t > ns - 1) t = ns - 1;
    sub += mul * t;
    mul *= ns;
  }
  return sub;
}

// The pair of an NTC candidate (Sec. II.A: "selected randomly within the
// cell") from its uniforms u1, u2: i uniform over the N slots, j uniform
// over the other N - 1; with sub-cells (so = the cell's sub-cell offsets,
// nsub > 1) j uniform over the other particles of i's sub-cell when it
// holds one.  Slots relative to the cell.
template <class T, class O>
__device__ __forceinline__ void select_pair(int N, T u1, T u2, const O* so, int nsub, int* pi, int* pj) {
  int i = (int)(u1 * (T)N);
  if (i > N - 1) i = N - 1;
  int a0 = 0, b0 = N;
  if (nsub > 1) {
    int t = 0;
    while ((int)so[t + 1] <= i) ++t;
    if ((int)so[t + 1] - (int)so[t] >= 2) {
      a0 = so[t];
      b0 = so[t + 1];
    }
  }
  int j = a0 + (int)(u2 * (T)(b0 - a0 - 1));
  if (j > b0 - 2) j = b0 - 2;
  if (j >= i) j += 1;
  *pi = i;
  *pj = j;
}

// Diffuse re-emission at a wall with R T_w = RTw: normal speed
// c_n = sqrt(-2 R T_w ln R1), tangential Box-Muller pair (R3, R4).
template <class T>
__device__ __forceinline__ void diffuse_sample(T RTw, Uni<T>& r, T* cn, T* t1, T* t2) {
  const T R1 = r.get(0), R3 = r.get(1), R4 = r.get(2);
  *cn = tsqrt((T)-2.0 * RTw * tlog(R1));
  const T r4 = tsqrt(-tlog(R4));
  const T s = tsqrt((T)2.0 * RTw);
  T sn, cs;
  sincos2pi(R3, &sn, &cs);
  *t1 = s * cs * r4;
  *t2 = s * sn * r4;
}

// Whether the straight flight over trem stays inside the box by the rounding
// margin and misses the body (the first test of move_particle, without its
// square root and division: for a particle approaching the body,
// t < trem <=> -b - trem a < sqrt(disc)); if so x is moved to the end point.
// In 2-D FP32 the comparison decides as it stands; elsewhere only a
// particle that misses by a margin far above rounding is cleared, so that
// move_particle's quotient decides every close case.
template <class T, int DIM>
__device__ __forceinline__ bool flight_fast(const InstParams& P, T* x, const T* v, T trem) {
  const Geo<T>& G = geo<T>(P);
  T xe[DIM];
  bool ok = true;
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    xe[d] = x[d] + v[d] * trem;
    ok = ok && xe[d] > G.lo[d] + G.eps[d] && xe[d] < G.hi[d] - G.eps[d];
  }
  if (P.body != 0) {
    T bb = 0, aa = 0, cc = 0;
#pragma unroll
    for (int d = 0; d < (DIM < 3 ? DIM : 3); ++d) {
      if (d == 2 && P.body == 1) break;
      const T dx = x[d] - G.body_c[d];
      bb += v[d] * dx;
      aa += v[d] * v[d];
      cc += dx * dx;
    }
    cc -= G.body_r * G.body_r;
    const T disc = bb * bb - aa * cc;
    T q = -bb - trem * aa;
    bool hit;
    if constexpr (sizeof(T) == 4 && DIM == 2) {
      hit = bb < (T)0 && aa > (T)0 && disc >= (T)0 && (q < (T)0 || q * q < disc);
    } else {
      q += bb * (sizeof(T) == 4 ? (T)1e-5 : (T)1e-12);  // (b < 0: towards a hit)
      hit = bb < (T)0 && aa > (T)0 && disc >= -(bb * bb) * (sizeof(T) == 4 ? (T)1e-5 : (T)1e-12) &&
            (q < (T)0 || q * q < disc);
    }
    ok = ok && !hit;
  }
  if (ok) {
#pragma unroll
    for (int d = 0; d < DIM; ++d) x[d] = xe[d];
  }
  return ok;
}

// FP64 state: the same question asked in FP32 first, on truncated positions
// and velocities (relative error below 2^-22; P.g32.eps is 1e-5 of the span,
// the magnitude of the box's coordinates).  A particle that starts and ends
// inside the box by that margin, and whose path keeps further from the
// body's centre than r by 4e-6 of the lengths involved plus the rounding of
// the coordinates, flies straight in FP64 too (there the margins are 1e10
// roundings wide): 2 DIM operations of the FP64 pipe instead of about 45.
template <int DIM>
__device__ __forceinline__ bool flight_clear(const InstParams& P, const double* x, const double* v, double trem) {
  const Geo<float>& G = P.g32;
  const float dt = approx_f32(trem);
  float xf[DIM], vf[DIM];
  bool ok = true;
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    xf[d] = approx_f32(x[d]);
    vf[d] = approx_f32(v[d]);
    const float xe = fmaf(vf[d], dt, xf[d]);
    ok = ok && xe > G.lo[d] + G.eps[d] && xe < G.hi[d] - G.eps[d] && fabsf(xf[d]) + fabsf(vf[d]) * dt < 2e5f * G.eps[d];
  }
  if (P.body != 0) {
    float dx[DIM], bb = 0, aa = 0, dd = 0, m = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      if (d == 2 && P.body == 1) break;
      dx[d] = xf[d] - G.body_c[d];
      bb = fmaf(vf[d], dx[d], bb);
      aa = fmaf(vf[d], vf[d], aa);
      dd = fmaf(dx[d], dx[d], dd);
      m += 0.05f * G.eps[d] + 4e-7f * fabsf(G.body_c[d]) + 4e-6f * (fabsf(dx[d]) + fabsf(vf[d]) * dt);
    }
    // the path's closest point (a clamped time; its own error counts only
    // in second order)
    const float ts = fminf(fmaxf(__fdividef(-bb, aa), 0.0f), dt);
    float pp = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      if (d == 2 && P.body == 1) break;
      const float p = fmaf(vf[d], ts, dx[d]);
      pp = fmaf(p, p, pp);
    }
    const float rm = G.body_r + m;
    ok = ok && aa > 1e-30f && aa < 1e30f && dd < 1e30f && pp > rm * rm * 1.00001f;
  }
  return ok;
}
// cell_of for an FP64 state: the FP32 coordinate decides where it lies in the
// grid and not within 1e-6 of the box's magnitude of a cell face.
template <int DIM>
__device__ __forceinline__ uint32_t cell_of_clear(const InstParams& P, const double* x) {
  const Geo<float>& G = P.g32;
  uint32_t idx[3] = {0, 0, 0};
  bool ok = true;
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    const float u = (approx_f32(x[d]) - G.lo[d]) * G.inv_d[d], f = floorf(u);
    const float mg = 0.1f * G.eps[d] * G.inv_d[d];
    ok = ok && u - f > mg && u - f < 1.0f - mg && f >= 0.0f && f < (float)P.n[d];
    idx[d] = (uint32_t)(int)f;
  }
  if (!ok) return cell_of<double, DIM>(P, x);
  return idx[0] + (uint32_t)P.n[0] * (idx[1] + (uint32_t)P.n[1] * idx[2]);
}

// Wall tallies of one body hit while sampling (FP64 atomics): the momentum
// and energy the wall receives, binned by the polar angle of the inward
// normal nv at the hit point.
template <class T>
__device__ __forceinline__ void tally_hit(const InstParams& P, double* surf_all, uint32_t step, const T* nv,
                                          T vin0, T vin1, T vin2, const T* v) {
  if (!(surf_all != nullptr && P.n_surf > 0 && (int64_t)step >= (int64_t)P.n_steady)) return;
  // momentum and energy the wall receives from this hit (FP64 tallies)
  double frac;
  if (P.body == 1) {
    frac = ((double)atan2(nv[1], nv[0]) + kPi) / (2.0 * kPi);
  } else {
    const double cx = (double)nv[0] < -1.0 ? -1.0 : ((double)nv[0] > 1.0 ? 1.0 : (double)nv[0]);
    frac = acos(cx) / kPi;
  }
  int bin = (int)floor(frac * (double)P.n_surf);
  if (bin < 0) bin = 0;
  if (bin > P.n_surf - 1) bin = P.n_surf - 1;
  double* t = surf_all + kSurfFields * (P.surf_off + bin);
  const double ein = (double)vin0 * vin0 + (double)vin1 * vin1 + (double)vin2 * vin2;
  const double eout = (double)v[0] * v[0] + (double)v[1] * v[1] + (double)v[2] * v[2];
  const double dp0 = P.FnM * ((double)vin0 - (double)v[0]);
  const double dp1 = P.FnM * ((double)vin1 - (double)v[1]);
  const double dp2 = P.FnM * ((double)vin2 - (double)v[2]);
  // direction of increasing polar angle at the hit point
  double et0 = 0, et1 = 0, et2 = 0;
  if (P.body == 1) {
    et0 = -(double)nv[1];
    et1 = (double)nv[0];
  } else {
    const double sn = sqrt((double)nv[1] * nv[1] + (double)nv[2] * nv[2]);
    if (sn > 0) {
      et0 = -sn;
      et1 = (double)nv[0] * nv[1] / sn;
      et2 = (double)nv[0] * nv[2] / sn;
    }
  }
  atomicAdd(t + 0, 1.0);
  atomicAdd(t + 1, dp0);
  atomicAdd(t + 2, dp1);
  atomicAdd(t + 3, dp2);
  atomicAdd(t + 4, 0.5 * P.FnM * (ein - eout));
  atomicAdd(t + 5, -(dp0 * nv[0] + dp1 * nv[1] + dp2 * nv[2]));
  atomicAdd(t + 6, dp0 * et0 + dp1 * et1 + dp2 * et2);
}

// Moves one particle for time trem.  Returns true when it left the domain.
// Draw stream of bounce b: (step, sa, sb, purpose<<24 | subbase + 2b).
template <class T, int DIM>
__device__ __forceinline__ bool move_particle(const InstParams& P, double* surf_all, T* x, T* v, T trem,
                              uint32_t step, uint32_t purpose, uint32_t sa, uint32_t sb,
                              uint32_t subbase, unsigned long long* err) {
  const Geo<T>& G = geo<T>(P);
  for (int bounce = 0;; ++bounce) {
    if (bounce >= kMaxBounce) {
      atomicAdd(&err[kErrBounce], 1ull);
      return false;
    }
    T tf = tinf<T>();
    int fa = -1, fs = 0;
    // straight end point inside the box by a margin far above rounding: no
    // face can be reached, the exit times need not be formed
    bool inside = true;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const T xe = x[d] + v[d] * trem;
      inside = inside && xe > G.lo[d] + G.eps[d] && xe < G.hi[d] - G.eps[d];
    }
    if (!inside) {
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        if (v[d] > (T)0) {
          const T t = (G.hi[d] - x[d]) / v[d];
          if (t < tf) { tf = t; fa = d; fs = 1; }
        } else if (v[d] < (T)0) {
          const T t = (G.lo[d] - x[d]) / v[d];
          if (t < tf) { tf = t; fa = d; fs = 0; }
        }
      }
    }
    T tb = tinf<T>();
    if (P.body != 0) {
      const int D = P.body == 1 ? 2 : 3;
      T bb = 0, aa = 0, cc = 0;
      for (int d = 0; d < D; ++d) {
        const T dx = x[d] - G.body_c[d];
        bb += v[d] * dx;
        aa += v[d] * v[d];
        cc += dx * dx;
      }
      cc -= G.body_r * G.body_r;
      if (bb < (T)0 && aa > (T)0) {
        const T disc = bb * bb - aa * cc;
        if (disc >= (T)0) {
          const T t = (-bb - tsqrt(disc)) / aa;
          tb = t < (T)0 ? (T)0 : t;
        }
      }
    }
    const T th = tf < tb ? tf : tb;
    if (!(th < trem)) {
#pragma unroll
      for (int d = 0; d < DIM; ++d) x[d] += v[d] * trem;
      return false;
    }
    const uint32_t c3 = (purpose << 24) | (subbase + 2u * (uint32_t)bounce);
    // the wall reached first: the body (diffuse at T_w) or a face; diffuse
    // re-emission of either runs through one copy of the sampling code,
    // in the frame (inward normal nv, tangents e1, e2) of the surface hit
    T nv[3] = {0, 0, 0}, e1[3] = {0, 0, 0}, e2[3] = {0, 0, 0};
    T RTw;
    const bool body_hit = tb <= tf;
    if (body_hit) {
#pragma unroll
      for (int d = 0; d < DIM; ++d) x[d] += v[d] * tb;
      trem -= tb;
      const int D = P.body == 1 ? 2 : 3;
      for (int d = 0; d < D; ++d) nv[d] = (x[d] - G.body_c[d]) / G.body_r;
      if (P.body == 1) {
        e1[0] = -nv[1]; e1[1] = nv[0]; e1[2] = 0;
        e2[0] = 0; e2[1] = 0; e2[2] = 1;
      } else {
        T ax[3] = {0, 0, 0};
        if (tfabs(nv[0]) < (T)0.9) ax[0] = 1; else ax[1] = 1;
        const T cx = nv[1] * ax[2] - nv[2] * ax[1];
        const T cy = nv[2] * ax[0] - nv[0] * ax[2];
        const T cz = nv[0] * ax[1] - nv[1] * ax[0];
        const T cn = tsqrt(cx * cx + cy * cy + cz * cz);
        e1[0] = cx / cn; e1[1] = cy / cn; e1[2] = cz / cn;
        e2[0] = nv[1] * e1[2] - nv[2] * e1[1];
        e2[1] = nv[2] * e1[0] - nv[0] * e1[2];
        e2[2] = nv[0] * e1[1] - nv[1] * e1[0];
      }
      RTw = G.body_RT;
    } else {
      // (static indices only: x and v stay in registers)
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        if (d != fa) x[d] += v[d] * tf;
        else x[d] = fs ? G.hi[d] : G.lo[d];
      }
      trem -= tf;
      const int f = 2 * fa + fs;
      int bc = P.face_bc[f];
      if (bc >= 2 && ((P.face_win >> f) & 1) && !face_open<T, DIM>(G, f, x)) bc = 1;  // orifice lips
      if (bc == 0) {
#pragma unroll
        for (int d = 0; d < DIM; ++d)
          if (d == fa) v[d] = -v[d];
        continue;
      }
      if (bc != 1) return true;
      // diffuse face: normal into the domain, tangents along the next axes
      const int f1 = fa == 2 ? 0 : fa + 1, f2 = fa == 0 ? 2 : fa - 1;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        nv[d] = d == fa ? (fs ? (T)-1 : (T)1) : (T)0;
        e1[d] = d == f1 ? (T)1 : (T)0;
        e2[d] = d == f2 ? (T)1 : (T)0;
      }
      RTw = G.face_RT[f];
    }
    Uni<T> r(step, sa, sb, c3, P.key0, P.key1);
    T cn, t1, t2;
    diffuse_sample<T>(RTw, r, &cn, &t1, &t2);
    const T vin0 = v[0], vin1 = v[1], vin2 = v[2];
#pragma unroll
    for (int d = 0; d < 3; ++d) v[d] = cn * nv[d] + t1 * e1[d] + t2 * e2[d];
    if (body_hit) tally_hit<T>(P, surf_all, step, nv, vin0, vin1, vin2, v);
  }
}

// ---------------------------------------------------------------------------
// Body-fitted O-grid (mesh = 1, 2-D): point location by face crossing.
// ---------------------------------------------------------------------------
// Walk of one particle of local cell kl for time trem.  In its cell it
// leaves through the face whose line its straight path meets first among
// the faces it moves towards (outward normal . v > 0; exit times below zero
// count as zero, so a point that rounding left just outside a face leaves
// at once); interior faces hand it to the neighbour (inner i-1, outer i+1,
// sectors j-1, j+1), the body polygon (inner face of ring 0) re-emits it
// diffusely at T_w, the outer polygon (outer face of the last ring) removes
// it (inflow, outflow), reflects it (specular) or re-emits it (diffuse at
// face_T[1]).  locate: the point location walk, where a boundary face ends
// the walk as "outside".  Draws of wall event b: (step, sa, sb, purpose<<24
// | subbase + 2b), as for the Cartesian walls.  Returns true when the
// particle left the domain (or, locating, the point lies outside).
template <class T>
__device__ __forceinline__ bool mesh_walk(const InstParams& P, const T* mface, double* surf_all, int64_t& kl,
                                          T* x, T* v, T trem, uint32_t step, uint32_t purpose, uint32_t sa,
                                          uint32_t sb, uint32_t subbase, unsigned long long* err, bool locate) {
  const Geo<T>& G = geo<T>(P);
  const int nr = P.n[0], nt = P.n[1];
  int bounce = 0;
  for (int cross = 0;; ++cross) {
    if (cross >= kMaxCross) {
      if (locate) return true;
      atomicAdd(&err[kErrBounce], 1ull);
      return false;
    }
    const T* f = mface + 12 * (P.cell_off + kl);
    if constexpr (sizeof(T) == 4) {
      // FP32 state: the flight that ends inside the cell (t_e >= trem on
      // every face it approaches, i.e. s_e >= trem (n_e . v)) is settled
      // without the four divisions; the FP64 state keeps the quotient
      // test of the oracle (the two can differ only at a tie)
      bool stay = true;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const T nvv = f[3 * e] * v[0] + f[3 * e + 1] * v[1];
        const T se = f[3 * e + 2] - (f[3 * e] * x[0] + f[3 * e + 1] * x[1]);
        stay = stay && !(nvv > (T)0 && se < trem * nvv);
      }
      if (stay) {
        x[0] += v[0] * trem;
        x[1] += v[1] * trem;
        return false;
      }
    }
    T tmin = tinf<T>();
    int fm = -1;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const T nvv = f[3 * e] * v[0] + f[3 * e + 1] * v[1];
      if (nvv > (T)0) {
        T t = (f[3 * e + 2] - (f[3 * e] * x[0] + f[3 * e + 1] * x[1])) / nvv;
        if (t < (T)0) t = 0;
        if (t < tmin) {
          tmin = t;
          fm = e;
        }
      }
    }
    if (!(tmin < trem)) {
      x[0] += v[0] * trem;
      x[1] += v[1] * trem;
      return false;
    }
    x[0] += v[0] * tmin;
    x[1] += v[1] * tmin;
    trem -= tmin;
    const int i = (int)(kl % nr), j = (int)(kl / nr);
    if (fm == 2) { kl = i + (int64_t)nr * ((j + nt - 1) % nt); continue; }
    if (fm == 3) { kl = i + (int64_t)nr * ((j + 1) % nt); continue; }
    if (fm == 0 && i > 0) { kl -= 1; continue; }
    if (fm == 1 && i < nr - 1) { kl += 1; continue; }
    if (locate) return true;
    if (bounce >= kMaxBounce) {
      atomicAdd(&err[kErrBounce], 1ull);
      return false;
    }
    const uint32_t c3 = (purpose << 24) | (subbase + 2u * (uint32_t)bounce);
    ++bounce;
    // a boundary face: normal into the domain
    T nv[3] = {-f[3 * fm], -f[3 * fm + 1], (T)0};
    T RTw;
    if (fm == 1) {
      const int bc = P.face_bc[1];
      if (bc >= 2) return true;  // outflow, inflow
      if (bc == 0) {             // specular
        const T vn = f[3] * v[0] + f[4] * v[1];
        v[0] -= (T)2.0 * vn * f[3];
        v[1] -= (T)2.0 * vn * f[4];
        continue;
      }
      RTw = G.face_RT[1];
    } else {
      RTw = G.body_RT;
    }
    const T e1[3] = {-nv[1], nv[0], (T)0}, e2[3] = {(T)0, (T)0, (T)1};
    Uni<T> r(step, sa, sb, c3, P.key0, P.key1);
    T cn, t1, t2;
    diffuse_sample<T>(RTw, r, &cn, &t1, &t2);
    const T vin0 = v[0], vin1 = v[1], vin2 = v[2];
#pragma unroll
    for (int d = 0; d < 3; ++d) v[d] = cn * nv[d] + t1 * e1[d] + t2 * e2[d];
    if (fm == 0) tally_hit<T>(P, surf_all, step, nv, vin0, vin1, vin2, v);
  }
}

// The local cell of point x (O-grid): a first guess from its polar
// coordinates, then the walk from that cell's centroid to x; -1 outside
// the mesh (inside the body polygon or beyond the outer polygon).
template <class T>
__device__ __forceinline__ int64_t mesh_locate(const InstParams& P, const T* mface, const T* mnode,
                                               const double* mrad, const T* x) {
  const int nr = P.n[0], nt = P.n[1];
  const double kTwoPi = 2.0 * 3.14159265358979323846;
  const double dx = (double)x[0] - P.body_c[0], dy = (double)x[1] - P.body_c[1];
  const double r = sqrt(dx * dx + dy * dy);
  double th = atan2(dy, dx);
  if (th < 0) th += kTwoPi;
  int j = (int)floor(th * (double)nt / kTwoPi);
  if (j < 0) j = 0;
  if (j > nt - 1) j = nt - 1;
  const double* rad = mrad + P.mrad_off;
  int i = 0;
  while (i < nr - 1 && rad[i + 1] <= r) ++i;
  int64_t kl = i + (int64_t)nr * j;
  const T* nd = mnode + 2 * P.mnode_off;
  const int j1 = (j + 1) % nt;
  const T* A = nd + 2 * ((int64_t)i * nt + j);
  const T* B = nd + 2 * ((int64_t)(i + 1) * nt + j);
  const T* C = nd + 2 * ((int64_t)(i + 1) * nt + j1);
  const T* D = nd + 2 * ((int64_t)i * nt + j1);
  T p[2] = {(T)0.25 * (A[0] + B[0] + C[0] + D[0]), (T)0.25 * (A[1] + B[1] + C[1] + D[1])};
  T w[3] = {x[0] - p[0], x[1] - p[1], (T)0};
  if (mesh_walk<T>(P, mface, nullptr, kl, p, w, (T)1, 0u, 0u, 0u, 0u, 0u, nullptr, true)) return -1;
  return kl;
}

// ---------------------------------------------------------------------------
// Warp-cooperative pieces of the per-cell step.
// ---------------------------------------------------------------------------
// Warp-aggregated histogram increment (key == kSentinel is skipped).
__device__ __forceinline__ void warp_count(uint32_t key, uint32_t* count) {
  const unsigned peers = __match_any_sync(kFull, key);
  const int lane = threadIdx.x & 31;
  if (key != kSentinel && lane == __ffs(peers) - 1) atomicAdd(&count[key], (uint32_t)__popc(peers));
}

struct CellMoments {
  double U[3], T, q[3], n, tau, dtc;
};

__device__ __forceinline__ double dsmc_ratio(const InstParams& P, int N, const CellMoments& m) {
  if (P.mode == 1) return 1.0;
  if (P.mode == 2) return 0.0;
  if (N < 2 || !(m.T > 0) || m.dtc <= m.tau) return 1.0;
  return m.tau / m.dtc;
}

// Precision modes of the collision kernel: T = particle state and
// per-particle arithmetic, A = per-cell sums and per-cell arithmetic.
// T == A: FP64 mode (double) or the opt-in all-FP32 mode (float).
// T = float, A = double: FP32 state with FP64 per-cell sums and arithmetic.
template <class T, class A>
__host__ __device__ constexpr bool mixed_prec() {
  return sizeof(T) < sizeof(A);
}

// Per-cell constants of a batch that the particle-parallel phases read
// (one warp's batch of at most 32 cells).
template <class T, class A>
struct __align__(16) CellTab {
  int off[33];   // slot range of cell i: [off[i], off[i+1])
  int inst[32];
  uint8_t ne[32];  // the cells that hold particles, in order
  int nres[32];
  int nar[32];
  int nacc[32];
  int coff[33];  // candidate offsets of the flattened NTC loop
  int pad[2];
  uint16_t hpart[32];  // helper lane -> (cell << 8 | part) of the split sums
  T U[3][32];
  T q[3][32];    // (from the rescale on: its factor f, high and low part, in q[0], q[1])
  T RT[32], s2RT[32], Amax[32], Pres[32], omp[32];
  // Conservation rescale c' = U + (c - U_p) f, applied slot by slot.
  // T == A: Up = U_p and f.  Mixed precision: the same map written as
  // c' = c f + K with f = f[] + fl[] and K = Up[] + Kl[] as FP32 pairs
  // (high part + rounding remainder of the FP64 values).  The mean-shift
  // of the second moment pass uses Up / Kl the same way (U = Up + Kl).
  T Up[3][32];
  T Kl[3][32];
  T smax[32];    // (sigma_T c_r)_max while candidates run
};

// Staging per particle: velocities (3 T), source index, and two bytes that
// hold the NTC clash tags (a table of cap / 2 words that the slots are folded
// into), then the list of resampled slots.  In FP32 modes the source indices
// live in the x-velocity array until the gather overwrites them slot by slot.
// 14 bytes per particle (FP32) let 16 warps of 812 particles share an SM;
// with 4-byte tags and a cell byte per slot (17) it was 12 of 864.
template <class T>
__host__ __device__ constexpr bool idx_in_velocity() {
  return sizeof(T) == 4;
}
template <class T>
__host__ __device__ constexpr size_t stage_bytes_per_particle() {
  return 3 * sizeof(T) + (idx_in_velocity<T>() ? 0 : 4) + 2;
}
// sub-cells on: their offsets within each cell of the batch
constexpr size_t kSubBytes = 32 * (kMaxSub + 1) * sizeof(uint16_t);
template <class T, class A>
__host__ __device__ constexpr size_t warp_stage_bytes(int cap, bool subcells) {
  return (sizeof(CellTab<T, A>) + (subcells ? kSubBytes : 0) + ((size_t)cap * stage_bytes_per_particle<T>() + 3) / 4 * 4 +
          15) / 16 * 16;
}

// ---------------------------------------------------------------------------
// Error-free transformations in FP32 (Knuth's two-sum; Dekker's product,
// here with a fused multiply-add): a + b = s + e and a * b = p + e exactly.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float two_sum(float a, float b, float* e) {
  const float s = a + b;
  const float bv = s - a;
  const float av = s - bv;
  *e = (a - av) + (b - bv);
  return s;
}
__device__ __forceinline__ float two_prod(float a, float b, float* e) {
  const float p = a * b;
  *e = fmaf(a, b, -p);
  return p;
}

// Accumulators of a lane's run of terms.  Each term comes as x plus an
// exact low part lo (zero for plain terms; the remainder of an exact
// product).
//   PlainSum<T>: x added in T (lo is zero in the modes that use it).
//   ExactSum: FP32 terms carried without rounding loss: every addition is
//   split by two_sum, and the remainders (with the low parts) collect in e,
//   whose own rounding is of order eps^2 of the total; s + e, formed in
//   FP64, is the run's sum to FP64 accuracy.  On GB300 an FP64 add (and the
//   FP32 -> FP64 conversion of its operand) goes through the FP64 pipe at
//   about 1/56 of the FP32 rate, so these seven FP32 operations per term
//   are several times cheaper than widening each term and adding in FP64.
// add1(x) takes a term without a low part (one FP32 add fewer);
// combine(o) adds another accumulator's run; shfl_xor(o) is the lane
// o-apart copy (for butterflies across a warp).
template <class T>
struct PlainSum {
  using term = T;
  using result = T;
  static constexpr bool kExact = false;
  T s;
  __device__ __forceinline__ void init() { s = 0; }
  __device__ __forceinline__ void add(T x, T) { s += x; }
  __device__ __forceinline__ void add1(T x) { s += x; }
  __device__ __forceinline__ void combine(const PlainSum& o) { s += o.s; }
  __device__ __forceinline__ PlainSum shfl_xor(int o) const {
    PlainSum r;
    r.s = __shfl_xor_sync(kFull, s, o);
    return r;
  }
  __device__ __forceinline__ PlainSum shfl_from(int src) const {
    PlainSum r;
    r.s = __shfl_sync(kFull, s, src);
    return r;
  }
  __device__ __forceinline__ T get() const { return s; }
};
struct ExactSum {
  using term = float;
  using result = double;
  static constexpr bool kExact = true;
  float s, e;
  __device__ __forceinline__ void init() { s = 0.0f; e = 0.0f; }
  __device__ __forceinline__ void add(float x, float lo) {
    float r;
    s = two_sum(s, x, &r);
    e += r + lo;
  }
  __device__ __forceinline__ void add1(float x) {  // a term without a low part
    float r;
    s = two_sum(s, x, &r);
    e += r;
  }
  __device__ __forceinline__ void combine(const ExactSum& o) {
    float r;
    s = two_sum(s, o.s, &r);
    e += o.e + r;
  }
  __device__ __forceinline__ ExactSum shfl_xor(int o) const {
    ExactSum r;
    r.s = __shfl_xor_sync(kFull, s, o);
    r.e = __shfl_xor_sync(kFull, e, o);
    return r;
  }
  __device__ __forceinline__ ExactSum shfl_from(int src) const {
    ExactSum r;
    r.s = __shfl_sync(kFull, s, src);
    r.e = __shfl_sync(kFull, e, src);
    return r;
  }
  __device__ __forceinline__ double get() const { return widen(s) + widen(e); }
};
template <class T, class A>
using CellAcc = typename std::conditional<mixed_prec<T, A>(), ExactSum, PlainSum<T>>::type;
// An FP32 accumulator as the pair (s, e) whose FP64 sum is its value.
__device__ __forceinline__ float2 acc_pair(const ExactSum& x) { return make_float2(x.s, x.e); }
__device__ __forceinline__ float2 acc_pair(const PlainSum<float>& x) { return make_float2(x.s, 0.0f); }
__device__ __forceinline__ float2 acc_pair(const PlainSum<double>&) { return make_float2(0.0f, 0.0f); }

// Parameters of instance i.  With a single instance (ONE) they come from
// the copy in the kernel's parameter space, so that the geometry and gas
// constants reach the arithmetic as constant-bank operands rather than as
// per-particle loads.
template <bool ONE>
__device__ __forceinline__ const InstParams& inst_params(const StepArgs& a, uint32_t i) {
  if constexpr (ONE) return a.P0;
  else return a.P[i];
}

// Per-cell sums with an order fixed by the cell alone (so results do not
// depend on how cells are grouped into batches).  A cell of at most
// kLaneSumMax particles is summed by its own lane (lane i <-> cell i) in
// slot order (FP64 terms: by about N / 8 lanes, as many cells at a time as
// fill the warp); with an FP32 state a cell above kSplitLanes particles is cut
// into P = cell_lanes(N) contiguous parts of ceil(N / P) slots, part 0 on
// its own lane and parts 1..P-1 on helper lanes of the batch (lanes G,
// G+1, ... in cell order), and its lane adds the parts in part order -- so
// that a dense batch's loops run over ~N / P slots instead of N.  A larger
// cell is summed by the warp, one contiguous share of its slots per lane,
// then a butterfly over the lanes (the order again fixed by the cell's
// particle count).  f(s, c, v, lo) gives the K terms of slot s of cell c
// (and their exact low parts); lane i receives the sums of its own cell i
// in out[] (cells with own false are skipped).
constexpr int kLaneSumMaxExact = kLaneSumMax;
// Cells above kHugeCell particles (sp_internal.h) are collided by one
// block of kHugeThreads threads each (k_collide_huge).
constexpr int kHugeThreads = 256;
constexpr int kHugeWarps = kHugeThreads / 32;
// NTC candidates up to which a cell runs its collision loop on its own lane:
// in 3-D (sphere: +18 %; thresholds 8-32 gave -7 % to +9 %); not in 2-D,
// where the flattened loop is as fast or faster (cylinder: -1 % to -3 %;
// again -3 % / -4 % for 64 / 256 with FP64-accurate cells)
template <int DIM>
constexpr int kLaneNtcMax = DIM == 3 ? 256 : 0;
// Cells above lane_sum_max<Acc> particles are summed by the whole warp.
// (With the error-free accumulator, thresholds of 32 / 64 / 128 were 60 /
// 26 / 6 % slower on the cylinder than 256: the warp's error-free butterfly
// costs more than the lanes a dense cell leaves idle.)
template <class Acc>
constexpr int lane_sum_max = Acc::kExact ? kLaneSumMaxExact : kLaneSumMax;
// Parts split per cell for state type T (0: one lane per cell): 2-D FP32
// state only (in 1-D and 3-D the fewer cells per batch cost more than the
// shorter loops gain: the sphere 1.55e10 -> 1.24e10, the 1-D batch -4 %).
template <class T, int DIM>
constexpr int kSplitOf = (sizeof(T) == 4 && DIM == 2) ? kSplitLanes : 0;

// The part of the per-cell sums a lane of the batch serves: owner lanes
// (lane < G) part 0 of their own cell, helper lanes a later part of
// another cell.  c = -1: none.  own_parts / h0: for an owner lane, its
// cell's part count and the helper lane of part 1.  kSplit = 0: no parts
// (an empty record; every cell is summed by its own lane).
template <int kSplit>
struct LanePart {
  static constexpr int split = kSplit;
  int c, b, e;
  int own_parts, h0;
  uint16_t* scratch;  // [32] shared, for the FP64 sums
  int home;           // an owner lane's cell above kLaneSumMax: home_lane
};
template <>
struct LanePart<0> {
  static constexpr int split = 0;
  uint16_t* scratch;
  int home;
};

// The lanes' parts of a batch of G cells (cells with Ni > kLaneSumMax: one
// part, summed by the warp path); helper lanes read their (cell, part) from
// the table.  Called by the whole warp.
template <int split, class TabT>
__device__ __forceinline__ LanePart<split> lane_parts(TabT* ct, int G, bool own, int offi, int Ni) {
  LanePart<split> lp;
  lp.scratch = ct->hpart;
  lp.home = 0;
  if constexpr (split == 0) {
    return lp;
  } else {
    const int lane = threadIdx.x & 31;
    lp.c = -1;
    lp.b = lp.e = 0;
    lp.own_parts = 1;
    lp.h0 = 0;
    int L = own ? cell_lanes(Ni, split) : 1;
    int hs = L - 1;  // inclusive scan of the helpers over the cells
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, hs, o);
      if (lane >= o) hs += y;
    }
    int nhelp = __shfl_sync(kFull, hs, 31);
    hs -= L - 1;  // exclusive
    if (G + nhelp > 32) {  // (the batch plan never makes such a batch)
      L = 1;
      hs = 0;
      nhelp = 0;
    }
    if (own) {
      const int h = (Ni + L - 1) / L;
      lp.c = lane;
      lp.b = offi;
      lp.e = offi + (h < Ni ? h : Ni);
      lp.own_parts = L;
      lp.h0 = G + hs;
      for (int p = 1; p < L; ++p) ct->hpart[hs + p - 1] = (uint16_t)((lane << 8) | p);
    }
    __syncwarp();
    if (lane >= G && lane - G < nhelp) {
      const int hp = ct->hpart[lane - G];
      const int c = hp >> 8, p = hp & 255;
      const int o0 = ct->off[c], n = ct->off[c + 1] - o0;
      const int Lc = cell_lanes(n, split);
      const int h = (n + Lc - 1) / Lc;
      lp.c = c;
      lp.b = o0 + p * h;
      lp.e = o0 + ((p + 1) * h < n ? (p + 1) * h : n);
    }
    return lp;
  }
}

// The lane whose FP32 pair stands for the butterfly's sum of cell k (of
// kLaneSumMax + 1 to kHomeCap particles; lane 0 above): the cell's place among
// the cells of a partition of its chunk of 32 cells into runs of at most
// kHomeCap particles and 32 lanes.  That is the batch partition of the
// schedule that most FP32 flows are tuned to, whose sums are thus kept bit for
// bit; taken from the actual batches, the lane -- and with it the last bits
// of Shakhov cells -- would depend on the schedule.
constexpr int kHomeCap = 864;
__device__ __forceinline__ int home_lane(const uint32_t* start, int64_t NC, int64_t k, int split) {
  const int lane = threadIdx.x & 31;
  const int64_t c0 = k & ~(int64_t)31;
  const int at = (int)(k - c0), nc = (int)(NC - c0 < 32 ? NC - c0 : 32);
  uint32_t cum = lane < nc ? start[c0 + lane + 1] - start[c0 + lane] : 0u;
  int lcum = lane < nc ? cell_lanes((int)(cum < 0x7FFFFFFFu ? cum : 0x7FFFFFFFu), split) : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, cum, o);
    const int z = __shfl_up_sync(kFull, lcum, o);
    if (lane >= o) {
      cum += y;
      lcum += z;
    }
  }
  for (int kk = 0; kk <= at;) {
    const uint32_t before = kk > 0 ? __shfl_sync(kFull, cum, kk - 1) : 0u;
    const int lbefore = kk > 0 ? __shfl_sync(kFull, lcum, kk - 1) : 0;
    const int G = __popc(__ballot_sync(kFull, lane >= kk && lane < nc && cum - before <= (uint32_t)kHomeCap &&
                                                  lcum - lbefore <= 32));
    if (at < kk + G) return at - kk;
    kk += G > 0 ? G : 1;
  }
  return 0;
}

// Lanes that share the FP64 sum of a cell of n particles (a power of two,
// about eight particles each).
__device__ __forceinline__ int fp64_lanes(int n) {
  const int q = (n + 7) >> 3;  // ceil(n / 8), rounded up to a power of two
  return q <= 1 ? 1 : 1 << (32 - __clz(q - 1));
}

// kLo: the terms come with exact low parts (else lo is ignored).
template <class Acc, int K, bool kLo = false, class LP, class F>
__device__ __forceinline__ void cell_sums_acc(const LP& lp, bool own, int offi, int Ni, Acc (&out)[K], F f) {
  using Tm = typename Acc::term;
  const int lane = threadIdx.x & 31;
  const bool small = own && Ni <= lane_sum_max<Acc>;
#pragma unroll
  for (int k = 0; k < K; ++k) out[k].init();
  if constexpr (sizeof(Tm) == 8) {
    // FP64 terms (FP64 mode; the FP32 mode's FP64 record sums): an FP64
    // instruction holds the pipe as long for one lane as for 32, so a cell's
    // slots are dealt to P = fp64_lanes(N) neighbouring lanes (every P-th
    // slot each, then a tree over the P lanes), as many cells at a time as
    // fill the warp
    const int P = small && Ni > 0 ? fp64_lanes(Ni) : 0;
    int incl = P;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    for (unsigned todo = __ballot_sync(kFull, P > 0); todo;) {
      const int first = __ffs(todo) - 1;
      const int before = __shfl_sync(kFull, incl - P, first);
      const bool fit = P > 0 && lane >= first && incl - before <= 32;
      const unsigned round = __ballot_sync(kFull, fit);
      const int start = incl - P - before;  // the cell's first lane
      const unsigned heads = __reduce_or_sync(kFull, fit ? 1u << start : 0u);
      const int tot = __shfl_sync(kFull, incl, 31 - __clz((int)round)) - before;
      if (fit) lp.scratch[start] = (uint16_t)lane;
      __syncwarp();
      const int hs = 31 - __clz((int)(heads & (0xFFFFFFFFu >> (31 - lane)))), p = lane - hs;
      const int c = lp.scratch[hs];
      const int o0 = __shfl_sync(kFull, offi, c), n = __shfl_sync(kFull, Ni, c), Pc = __shfl_sync(kFull, P, c);
      Acc acc[K];
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k].init();
      if (lane < tot)
        for (int s = o0 + p; s < o0 + n; s += Pc) {
          Tm v[K], lo[K];
          f(s, c, v, lo);
#pragma unroll
          for (int k = 0; k < K; ++k) {
            if constexpr (kLo) acc[k].add(v[k], lo[k]);
            else acc[k].add1(v[k]);
          }
        }
      const int pmax = (int)__reduce_max_sync(kFull, (unsigned)P & (fit ? ~0u : 0u));
      for (int o = pmax >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const Acc y = acc[k].shfl_from(lane + o < 32 ? lane + o : lane);
          if (o < Pc && p < o) acc[k].combine(y);
        }
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const Acc y = acc[k].shfl_from(fit ? start : lane);
        if (fit) out[k] = y;
      }
      todo &= ~round;
      __syncwarp();
    }
  } else if constexpr (LP::split == 0) {
    // no split parts: one lane per cell, in slot order
    if (small) {
      for (int s = offi; s < offi + Ni; ++s) {
        Tm v[K], lo[K];
        f(s, lane, v, lo);
#pragma unroll
        for (int k = 0; k < K; ++k) {
          if constexpr (kLo) out[k].add(v[k], lo[k]);
          else out[k].add1(v[k]);
        }
      }
    }
  } else {
    // this lane's part: its own small cell, or a helper's part of a small
    // cell that takes part in this call
    const int cp = lp.c >= 0 ? lp.c : lane;
    const bool on = __shfl_sync(kFull, small, cp) && lp.c >= 0;
    if (on) {
      for (int s = lp.b; s < lp.e; ++s) {
        Tm v[K], lo[K];
        f(s, lp.c, v, lo);
#pragma unroll
        for (int k = 0; k < K; ++k) {
          if constexpr (kLo) out[k].add(v[k], lo[k]);
          else out[k].add1(v[k]);
        }
      }
    }
    // the owner adds parts 1.. in part order
    if (__any_sync(kFull, small && lp.own_parts > 1)) {
#pragma unroll
      for (int p = 1; p < kMaxParts; ++p) {
        const bool take = small && p < lp.own_parts;
        const int src = take ? lp.h0 + p - 1 : lane;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const Acc o = out[k].shfl_from(src);
          if (take) out[k].combine(o);
        }
      }
    }
  }
  for (unsigned b = __ballot_sync(kFull, own && !small); b; b &= b - 1) {
    const int c = __ffs(b) - 1;
    const int o0 = __shfl_sync(kFull, offi, c), n = __shfl_sync(kFull, Ni, c);
    const int per = (n + 31) / 32;
    const int s0 = o0 + lane * per;
    const int s1 = s0 + per < o0 + n ? s0 + per : o0 + n;
    Acc acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k].init();
    for (int s = s0; s < s1; ++s) {
      Tm v[K], lo[K];
      f(s, c, v, lo);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if constexpr (kLo) acc[k].add(v[k], lo[k]);
        else acc[k].add1(v[k]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k].combine(acc[k].shfl_xor(o));
    // one lane's sum, fixed by the state (home_lane), whichever lane c the
    // cell has in this batch: the lanes' error terms of the exact sums differ
    // in their last bits
    const int src = Acc::kExact ? __shfl_sync(kFull, lp.home, c) : 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const Acc y = acc[k].shfl_from(src);
      if (lane == c) out[k] = y;
    }
  }
  __syncwarp();
}

template <class Acc, int K, bool kLo = false, class LP, class F>
__device__ __forceinline__ void cell_sums(const LP& lp, bool own, int offi, int Ni,
                                          typename Acc::result (&out)[K], F f) {
  Acc acc[K];
  cell_sums_acc<Acc, K, kLo>(lp, own, offi, Ni, acc, f);
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = acc[k].get();
}

// c f + K for an FP32 c, with f = fh + fl and K = Kh + Kl given as FP32
// pairs (the splits of FP64 values): the product c fh is split exactly, the
// small parts are added in FP32, and s + *lo (s returned) is the FP64 value
// to about 2^-48 relative.
__device__ __forceinline__ float affine_ff(float c, float fh, float fl, float Kh, float Kl, float* lo) {
  float pe, se;
  const float p = two_prod(c, fh, &pe);
  const float s = two_sum(p, Kh, &se);
  *lo = se + (pe + fmaf(c, fl, Kl));
  return s;
}

// Record mode: conservation of the rescale in FP64, per cell:
// cons[0..2] = sum c'_d - N U_d, cons[3] = sum |c' - U|^2 - 3 R (N-1) T,
// cons[4] = 3 R (N-1) T, cons[5] = N sqrt(|U|^2 + 3 R T) (momentum scale),
// with U, T the Step 3 moments and r = (sum c'_x, sum c'_y, sum c'_z,
// sum |c'|^2) of the rescaled velocities before the FP32 store, summed in
// FP64 (sum |c' - U|^2 = sum |c'|^2 - 2 U . sum c' + N |U|^2).
template <class A>
__device__ __forceinline__ void record_conservation(const StepArgs& a, int64_t kc, int Ni, const InstParams& P,
                                                    const A* U, A T, const double* r) {
  const int64_t NC = a.NC;
  const double N = (double)Ni;
  double uu = 0, us = 0;
  for (int d = 0; d < 3; ++d) {
    a.cons[d * NC + kc] = r[d] - N * (double)U[d];
    uu += (double)U[d] * (double)U[d];
    us += (double)U[d] * r[d];
  }
  const double E = 3.0 * P.R * (N - 1.0) * (double)T;
  a.cons[3 * NC + kc] = (r[3] - 2.0 * us + N * uu) - E;
  a.cons[4 * NC + kc] = E;
  a.cons[5 * NC + kc] =
      N * sqrt((double)U[0] * U[0] + (double)U[1] * U[1] + (double)U[2] * U[2] + 3.0 * P.R * (double)T);
}

// Step 3 scalars and the Step 4 split of one cell, in A (Sec. III.B): from
// the cell's sums (m = sum c, mS2 = sum |C|^2, mS3 = sum |C|^2 C about the
// mean) to U, n, the unbiased T and q_s, tau = mu / p with the VHS
// viscosity, dt_c (Eq. "local time step"), the DSMC ratio and the sub-step
// durations (Eqs. "tDSMC", "tShakhov"), the NTC candidate count (Eq.
// "Ncol_DSMC", fractional part by stochastic rounding or the carried
// remainder), the resampling probability 1 - exp(-dt_SBGK / tau) (FP64) and
// the Shakhov sampling constants (A_max at |C| = 5 sqrt(RT), C parallel to
// q_s).  FP64 mode: the oracle's expressions, operation for operation, on
// the sums.
template <class A>
struct CellMath {
  A U[3], T, q[3], n, tau, dtc, ratio;
  A RT, s2RT, Amax, omp;  // Shakhov sampling constants (shk)
  double Pres;            // resampling probability (shk)
  int64_t ncol;
  unsigned long long dtbits;  // dt_c as ordered bits (~0: not a candidate)
  bool shk;
  __device__ __forceinline__ void clear() {
    U[0] = U[1] = U[2] = 0;
    T = 0;
    q[0] = q[1] = q[2] = 0;
    n = 0;
    tau = dtc = tinf<A>();
    ratio = 1;
    RT = s2RT = Amax = omp = 0;
    Pres = 0;
    ncol = 0;
    dtbits = ~0ull;
    shk = false;
  }
};

// The same quantities in FP64 for the FP32-state mode, with fewer FP64
// instructions (the FP64 pipe of GB300 runs at 1/56 of the FP32 rate, and an
// instruction costs the same whether one lane or 32 execute it): the
// reciprocals 1/N, 1/(N-1), 1/(N-2), 1/V once; one square root sqrt(R T)
// for the sound speed, sqrt(2RT) and (RT)^(3/2); and the viscosity power
// through tau = tau_k T^(omega-1) / n = tau_k exp((omega-1) ln T) / n with
// tau_k = mu_ref T_ref^-omega / (m R) from the host (one logarithm and one
// exponential instead of pow).  tau enters a result only through the split:
// where an FP32 bound of Delta t_c / tau is below 0.99 (its error is below
// 1e-5, so Delta t_c <= tau holds exactly) the cell is pure DSMC and tau is
// not formed; q_s and the Shakhov constants only in cells with a Shakhov
// part.  FP64 throughout; the rounding differs from the oracle's order by a
// few ulps (this mode is checked statistically).  ivol_k = 1 / V.  kQ
// false: q_s and A_max are left to shakhov_q_amax.
template <class T, bool kQ = true>
__device__ __forceinline__ void cell_math_lean(const StepArgs& a, const InstParams& Pi, int64_t kc, uint32_t kl,
                                               int Ni, double m0, double m1, double m2, double mS2, double mS3x,
                                               double mS3y, double mS3z, double ivol_k, T smaxT, double dt_cur,
                                               uint32_t step, CellMath<double>& o) {
  o.ratio = Pi.mode == 2 ? 0.0 : 1.0;  // cells without a split: the forced mode, else DSMC
  if (Ni <= 0) return;
  // 1/N, 1/(N-1), 1/(N-2) from the table of reciprocals (cells of the
  // warp launches) and 1/V from the per-cell array: no FP64 division
  const bool tab = Ni <= kHugeCell;
  const double fN = (double)Ni, iN = tab ? a.rcp[Ni] : 1.0 / fN, iV = ivol_k;
  const double Lk = a.Lc ? a.Lc[kc] : Pi.Lmin;  // the cell size of Delta t_c
  o.U[0] = m0 * iN;
  o.U[1] = m1 * iN;
  o.U[2] = m2 * iN;
  const double nt = fN * Pi.Fn * iV;
  o.n = nt;
  if (Ni < 2) return;
  const double iN1 = tab ? a.rcp[Ni - 1] : 1.0 / (fN - 1.0);
  const double Tt = mS2 * iN1 * Pi.inv3R;
  o.T = Tt;
  const double umag = sqrt(o.U[0] * o.U[0] + o.U[1] * o.U[1] + o.U[2] * o.U[2]);
  double taut = tinf<double>(), dtct = tinf<double>(), itau = 0, sRT = 0;
  bool dsmc_only = true;  // Delta t_c <= tau (or no split: T = 0, DSMC forced)
  if (Tt > 0.0) {
    sRT = sqrt(Pi.R * Tt);
    dtct = Lk / (umag + Pi.sqrt_gamma * sRT);
    if (Pi.mode != 1) {
      // Delta t_c / tau = Delta t_c n T^(1-omega) / tau_k; the FP32 power has
      // a relative error below 1e-5 for T in [1e-30, 1e30]
      bool sure = false;
      if (Pi.mode == 0 && Tt > 1e-30 && Tt < 1e30) {
        const double k = dtct * nt * Pi.inv_tau_k;
        sure = k * (double)__powf((float)Tt, Pi.omf) < 0.99;
      }
      if (!sure) {
        // 1/tau = n T^(1-omega) / tau_k
        itau = nt * exp((1.0 - Pi.omega) * log(Tt)) * Pi.inv_tau_k;
        taut = 1.0 / itau;
        dsmc_only = Pi.mode == 0 && dtct <= taut;
      }
    }
  } else if (umag > 0.0) {
    dtct = Lk / umag;
  }
  if (dtct < tinf<double>()) o.dtbits = (unsigned long long)__double_as_longlong(dtct);
  o.tau = taut;
  o.dtc = dtct;
  // r = tau / dt_c = tau (|U| + c_s) / L_min
  const double r = dsmc_only ? 1.0 : taut * (umag + Pi.sqrt_gamma * sRT) * (a.Lc ? a.iLc[kc] : Pi.inv_Lmin);
  if (Pi.mode == 1) o.ratio = 1;
  else if (Pi.mode == 2) o.ratio = 0;
  else o.ratio = r;
  if (!(Tt > 0.0)) return;
  const double dtG = dt_cur;
  double dsmc, sbgk;
  if (Pi.mode == 2) { dsmc = 0; sbgk = dtG; }
  else if (dsmc_only) { dsmc = dtG; sbgk = 0; }
  else { dsmc = r * dtG; sbgk = (1.0 - r) * dtG; }
  if (dsmc > 0.0) {
    const double ncr = 0.5 * fN * (fN - 1.0) * Pi.Fn * (double)smaxT * dsmc * iV;
    if (Pi.ntc_carry) {
      const double x = ncr + a.rem[kc];
      o.ncol = (int64_t)floor(x);
      a.rem[kc] = x - (double)o.ncol;
    } else {
      Uni<T> rr(step, kl, kSentinel, kPurpNtc << 24, Pi.key0, Pi.key1);
      o.ncol = (int64_t)floor(ncr + (double)rr.get(0));
    }
    if (o.ncol > kNcolCap) {
      o.ncol = kNcolCap;
      atomicAdd(&a.err[kErrNcol], 1ull);
    }
  }
  if (sbgk > 0.0 && Ni >= 3) {
    o.shk = true;
    const double RTt = Pi.R * Tt;
    o.RT = RTt;
    o.s2RT = 1.4142135623730950488 * sRT;
    o.omp = 1.0 - Pi.Pr;
    o.Pres = 1.0 - exp(-sbgk * itau);
    if constexpr (kQ) {
      const double fq = 0.5 * fN * iN1 * (tab ? a.rcp[Ni - 2] : 1.0 / (fN - 2.0));
      o.q[0] = fq * mS3x;
      o.q[1] = fq * mS3y;
      o.q[2] = fq * mS3z;
      const double qn = sqrt(o.q[0] * o.q[0] + o.q[1] * o.q[1] + o.q[2] * o.q[2]);
      o.Amax = 1.0 + 20.0 * (1.0 - Pi.Pr) * qn / (RTt * sRT);
    }
  }
}

// q_s = N/(2 (N-1)(N-2)) sum |C|^2 C and A_max = 1 + 20 (1 - Pr) |q_s| /
// (RT)^(3/2) of a Shakhov cell (Step 3, Sec. II.B), from o.RT and o.s2RT
// of cell_math_lean (mixed precision: the sums are taken after Step 4,
// in the Shakhov cells only).
__device__ __forceinline__ void shakhov_q_amax(const StepArgs& a, const InstParams& Pi, int Ni, double S3x,
                                               double S3y, double S3z, CellMath<double>& o) {
  const double fN = (double)Ni;
  const bool tab = Ni <= kHugeCell;
  const double fq = 0.5 * fN * (tab ? a.rcp[Ni - 1] * a.rcp[Ni - 2] : 1.0 / ((fN - 1.0) * (fN - 2.0)));
  o.q[0] = fq * S3x;
  o.q[1] = fq * S3y;
  o.q[2] = fq * S3z;
  const double qn = sqrt(o.q[0] * o.q[0] + o.q[1] * o.q[1] + o.q[2] * o.q[2]);
  const double sRT = o.s2RT * 0.70710678118654752440;
  o.Amax = 1.0 + 20.0 * (1.0 - Pi.Pr) * qn / (o.RT * sRT);
}

// vol_k: the cell volume V (FP64 and all-FP32 modes) or 1/V (mixed).
// kQ false (mixed precision): sum |C|^2 C is not given; q_s and A_max come
// later from shakhov_q_amax.
template <class T, class A, bool kQ = true>
__device__ __forceinline__ void cell_math(const StepArgs& a, const InstParams& Pi, int64_t kc, uint32_t kl, int Ni,
                                          A m0, A m1, A m2, A mS2, A mS3x, A mS3y, A mS3z, double vol_k,
                                          T smaxT, double dt_cur, uint32_t step, CellMath<A>& o) {
  if constexpr (mixed_prec<T, A>()) {
    cell_math_lean<T, kQ>(a, Pi, kc, kl, Ni, m0, m1, m2, mS2, mS3x, mS3y, mS3z, vol_k, smaxT, dt_cur, step, o);
    return;
  }
  const A V = (A)vol_k;
  const double Lk = a.Lc ? a.Lc[kc] : Pi.Lmin;  // the cell size of Delta t_c
  A Tt = 0, qt[3] = {0, 0, 0}, nt = 0;
  A taut = tinf<A>(), dtct = tinf<A>();
  if (Ni > 0) {
    o.U[0] = cdiv(m0, (A)Ni);
    o.U[1] = cdiv(m1, (A)Ni);
    o.U[2] = cdiv(m2, (A)Ni);
    nt = cdiv((A)Ni * (A)Pi.Fn, V);
  }
  if (Ni >= 2) {
    Tt = cdiv(mS2, (A)3.0 * (A)Pi.R * (A)(Ni - 1));
    if (Ni >= 3) {
      const A den = (A)(Ni - 1) * (A)(Ni - 2);
      qt[0] = cdiv((A)0.5 * (A)Ni * mS3x, den);
      qt[1] = cdiv((A)0.5 * (A)Ni * mS3y, den);
      qt[2] = cdiv((A)0.5 * (A)Ni * mS3z, den);
    }
    const A umag = tsqrt(o.U[0] * o.U[0] + o.U[1] * o.U[1] + o.U[2] * o.U[2]);
    if (Tt > (A)0) {
      const A p = nt * (A)Pi.m * (A)Pi.R * Tt;
      const A mu = (A)Pi.mu_ref * cpow(cdiv(Tt, (A)Pi.T_ref), (A)Pi.omega);
      taut = cdiv(mu, p);
      dtct = cdiv((A)Lk, umag + tsqrt((A)Pi.gamma * (A)Pi.R * Tt));
    } else if (umag > (A)0) {
      dtct = cdiv((A)Lk, umag);
    }
    if (dtct < tinf<A>()) o.dtbits = (unsigned long long)__double_as_longlong((double)dtct);
  }
  o.T = Tt;
  o.q[0] = qt[0];
  o.q[1] = qt[1];
  o.q[2] = qt[2];
  o.n = nt;
  o.tau = taut;
  o.dtc = dtct;
  // DSMC ratio of the split (Eqs. tDSMC, tShakhov)
  if (Pi.mode == 1) o.ratio = 1;
  else if (Pi.mode == 2) o.ratio = 0;
  else if (Ni < 2 || !(Tt > (A)0) || dtct <= taut) o.ratio = 1;
  else o.ratio = cdiv(taut, dtct);
  const A dtG = (A)dt_cur;
  if (Ni >= 2 && Tt > (A)0) {
    A dsmc, sbgk;
    if (Pi.mode == 1) { dsmc = dtG; sbgk = 0; }
    else if (Pi.mode == 2) { dsmc = 0; sbgk = dtG; }
    else if (dtct <= taut) { dsmc = dtG; sbgk = 0; }
    else {
      const A r = cdiv(taut, dtct);
      dsmc = r * dtG;
      sbgk = ((A)1.0 - r) * dtG;
    }
    if (dsmc > (A)0) {
      const A ncr = cdiv((A)0.5 * (A)Ni * (A)(Ni - 1) * (A)Pi.Fn * (A)smaxT * dsmc, V);
      if (Pi.ntc_carry) {  // Bird's carried remainder (FP64 state per cell)
        const double x = (double)ncr + a.rem[kc];
        o.ncol = (int64_t)floor(x);
        a.rem[kc] = x - (double)o.ncol;
      } else {
        Uni<T> rr(step, kl, kSentinel, kPurpNtc << 24, Pi.key0, Pi.key1);
        o.ncol = (int64_t)tfloor(ncr + (A)rr.get(0));
      }
      if (o.ncol > kNcolCap) {
        o.ncol = kNcolCap;
        atomicAdd(&a.err[kErrNcol], 1ull);
      }
    }
    if (sbgk > (A)0 && Ni >= 3) {
      o.shk = true;
      const A RTt = (A)Pi.R * Tt;
      const A qn = tsqrt(qt[0] * qt[0] + qt[1] * qt[1] + qt[2] * qt[2]);
      o.RT = RTt;
      o.s2RT = tsqrt((A)2.0 * RTt);
      o.Amax = (A)1.0 + cdiv((A)20.0 * ((A)1.0 - (A)Pi.Pr) * qn, RTt * tsqrt(RTt));
      o.omp = (A)1.0 - (A)Pi.Pr;
      o.Pres = 1.0 - exp(-(double)sbgk / (double)taut);
    }
  }
}

// One acceptance-rejection attempt t of the Shakhov resampling of a slot
// (Sec. II.B, Eqs. "Maxwell" and "A_cal"): a Box-Muller Maxwellian C at RT
// from the slot's stream r, accepted when R5 A_max < A(C) with
// A = 1 + (1 - Pr) (q_s . C) / (5 (RT)^2) (|C|^2 / RT - 5).  FP64 mode: five
// uniforms 1 + 5t .. 5 + 5t of the stream (the oracle's layout).  FP32
// modes: one Philox block per attempt (block 1 + t; block 0 holds the
// Bernoulli draw), the two angles sharing a word, 16 bits each, and A formed
// with the per-particle constants kA = (1 - Pr) / (5 (RT)^2), iRT = 1 / RT.
// FP64 mode: an attempt costs some 250 operations of the FP64 pipe (two
// logarithms, two square roots, three sines or cosines), and most attempts
// are rejected.  In units of sqrt(RT), A = 1 + (kq . c)(|c|^2 - 5) with
// kq = (1 - Pr) q_s / (5 (RT)^(3/2)): an FP32 evaluation rejects the attempts
// that are beyond a margin of 1e-5 |kq|_1 (1 + r2 + r4)(|c|^2 + 5); the others
// are evaluated in FP64, so that every decision and every accepted velocity is
// the FP64 one.  (A component's error goes with its radius r2 or r4, not with
// the component: a phase error of a few 2^-23 turns it.  Largest error found
// over 24 M attempts, half of them with extreme radii: 5.5e-7 of that bound's
// terms, plus a rounding or two of CUDA's sine, cosine and logarithm.)
struct ShakhovFilter {
  float kx, ky, kz, amax;  // amax < 0: no filter (values outside FP32's range)
};
__device__ __forceinline__ ShakhovFilter shakhov_filter(double RT, double Amax, double omp, double q0, double q1,
                                                        double q2) {
  ShakhovFilter f;
  const float rt = approx_f32(RT), k = 0.2f * approx_f32(omp) / (rt * sqrtf(rt));
  f.kx = k * approx_f32(q0);
  f.ky = k * approx_f32(q1);
  f.kz = k * approx_f32(q2);
  f.amax = approx_f32(Amax);
  const float big = fabsf(f.kx) + fabsf(f.ky) + fabsf(f.kz) + f.amax;
  if (!(rt > 1e-20f && rt < 1e20f && big < 1e15f)) f.amax = -1.0f;
  return f;
}
__device__ __forceinline__ ShakhovFilter shakhov_filter(float, float, float, float, float, float) { return {}; }
// -ln(u) of the uniform with words (a, b), relative error of a few 1e-7 also
// near u = 1
__device__ __forceinline__ float neg_log_approx(uint32_t a, uint32_t b) {
  if (a >> 31) {  // 1 - u = (2 k' + 1) 2^-53, k' the complement
    const float d = u01d_approx(~a, ~b);
    return -log1pf(-d);
  }
  return -logf(u01d_approx(a, b));
}
__device__ __forceinline__ bool shakhov_surely_rejected(const uint32_t* wa, const uint32_t* wb,
                                                        const ShakhovFilter& f) {
  if (!(f.amax > 0.0f)) return false;
  const float r2 = sqrtf(2.0f * neg_log_approx(wa[1], wb[1])), r4 = sqrtf(2.0f * neg_log_approx(wa[3], wb[3]));
  float sn, cs;
  sincospif(2.0f * u01d_approx(wa[2], wb[2]), &sn, &cs);
  const float c0 = r2 * cospif(2.0f * u01d_approx(wa[0], wb[0])), c1 = r4 * cs, c2 = r4 * sn;
  const float cc = c0 * c0 + c1 * c1 + c2 * c2;
  const float A = 1.0f + (f.kx * c0 + f.ky * c1 + f.kz * c2) * (cc - 5.0f);
  const float err = 1e-5f * (fabsf(f.kx) + fabsf(f.ky) + fabsf(f.kz)) *
                        (1.0f + r2 + r4) * (cc + 5.0f);
  const float lim = u01d_approx(wa[4], wb[4]) * f.amax;
  return lim * 0.99999f > A + err + 1e-5f;
}

// The words of attempt t's five uniforms: uniform q = 1 + 5 t + j in half
// q & 1 of block q / 2.
template <class U>
__device__ __forceinline__ void shakhov_words(const U& r, int t, uint32_t* wa, uint32_t* wb) {
  const int q0 = 1 + 5 * t;
#pragma unroll 1
  for (int b = q0 >> 1; b <= (q0 + 4) >> 1; ++b) {
    const uint4 w = philox10(r.c0, r.c1, r.c2, r.c3 + (uint32_t)b, r.k0, r.k1);
#pragma unroll
    for (int j = 0; j < 5; ++j)
      if ((q0 + j) >> 1 == b) {
        wa[j] = (q0 + j) & 1 ? w.z : w.x;
        wb[j] = (q0 + j) & 1 ? w.w : w.y;
      }
  }
}
// The first attempt from t on that the filter does not reject (FP64 mode; the
// last one, armax - 1, is kept whatever it is): the lanes of a warp then take
// their FP64 attempts together.
template <class T>
__device__ __forceinline__ int shakhov_skip(const Uni<T>& r, int t, int armax, const ShakhovFilter& fl) {
  if constexpr (sizeof(T) == 8) {
    for (; t < armax - 1; ++t) {
      uint32_t wa[5], wb[5];
      shakhov_words(r, t, wa, wb);
      if (!shakhov_surely_rejected(wa, wb, fl)) break;
    }
  }
  return t;
}

template <class T>
__device__ __forceinline__ bool shakhov_attempt(const Uni<T>& r, int t, T s2RT, T Amax, T omp, T RT, T kA, T iRT,
                                                T q0, T q1, T q2, T* C0, T* C1, T* C2) {
  T R1, R2, R3, R4, R5;
  if constexpr (sizeof(T) == 4) {
    const uint4 w = philox10(r.c0, r.c1, r.c2, r.c3 + 1u + (uint32_t)t, r.k0, r.k1);
    R2 = u01f(w.x);
    R4 = u01f(w.y);
    R1 = (float)(2u * (w.z >> 16) + 1u) * 7.62939453125e-6f;
    R3 = (float)(2u * (w.z & 0xFFFFu) + 1u) * 7.62939453125e-6f;
    R5 = u01f(w.w);
  } else {
    uint32_t wa[5], wb[5];
    shakhov_words(r, t, wa, wb);
    R1 = u01d(wa[0], wb[0]); R2 = u01d(wa[1], wb[1]); R3 = u01d(wa[2], wb[2]);
    R4 = u01d(wa[3], wb[3]); R5 = u01d(wa[4], wb[4]);
  }
  // (max: near R = 1 the approximate logarithm may round above 0)
  const T r2 = csqrt(tmax0(-clog(R2))), r4 = csqrt(tmax0(-clog(R4)));
  T sn3, cs3;
  sincos2pi(R3, &sn3, &cs3);
  *C0 = s2RT * cos2pi(R1) * r2;
  *C1 = s2RT * cs3 * r4;
  *C2 = s2RT * sn3 * r4;
  const T qC = q0 * *C0 + q1 * *C1 + q2 * *C2;
  const T CC = *C0 * *C0 + *C1 * *C1 + *C2 * *C2;
  T A;
  if constexpr (sizeof(T) == 4) A = (T)1.0 + kA * qC * (CC * iRT - (T)5.0);
  else A = (T)1.0 + omp * qC / ((T)5.0 * RT * RT) * (CC / RT - (T)5.0);
  return R5 * Amax < A;
}

// Mixed precision: the outcome of cell_math_lean for a cell whose decisions
// FP32 estimates settle -- a pure DSMC split (Delta t_c well below tau), a
// Delta t_c well above the smallest found so far, and a candidate count whose
// fractional draw is not close to an integer.  The estimates' relative
// errors (sums of a dozen roundings, __powf's 1e-5) stay below 3e-5.  A
// batch whose cells are all settled skips the FP64 arithmetic (60 to 130
// operations of the FP64 pipe in one dependent chain).  s: the cell's sums of
// c; S2: of |C|^2 (high parts of the exact pairs).
__device__ __forceinline__ bool cell_settled(const InstParams& Pi, uint32_t kl, int Ni, const float* s, float S2,
                                             double iV, const double* iLc, int64_t kc, float smaxT, double dt_cur,
                                             unsigned long long dt_min, uint32_t step, CellMath<double>& o) {
  if (Pi.mode == 2 || Pi.ntc_carry || Ni < 2) return false;
  const float fN = (float)Ni, iN = 1.0f / fN;
  const float ux = s[0] * iN, uy = s[1] * iN, uz = s[2] * iN;
  const float T = S2 * Pi.inv3R_f / (fN - 1.0f);
  const float iL = approx_f32(iLc ? iLc[kc] : Pi.inv_Lmin);
  const float idtc = (sqrtf(ux * ux + uy * uy + uz * uz) + sqrtf(Pi.gR_f * T)) * iL;  // 1 / Delta t_c
  // (1 / Delta t_c above 0.999 of the largest so far: the FP64 value counts)
  const float lim = 1.0f / approx_f32(__longlong_as_double((long long)dt_min));
  const float nv = fN * approx_f32(iV);
  bool ok = T > 1e-30f && T < 1e30f && idtc > 1e-30f && idtc < 1e30f && idtc < 0.999f * lim;
  if (Pi.mode == 0) {
    const float k = nv * Pi.Fn_itau_f * __powf(T, Pi.omf);  // 1 / tau
    ok = ok && k > 1e-30f && k < 0.98f * idtc;
  }
  if (!ok) return false;
  const float ncr = Pi.hFn_f * (fN - 1.0f) * nv * smaxT * approx_f32(dt_cur);
  Uni<float> rr(step, kl, kSentinel, kPurpNtc << 24, Pi.key0, Pi.key1);
  const float x = ncr + rr.get(0), f = floorf(x), m = 1e-4f * x + 1e-6f;
  if (!(ncr > 1e-30f && x < 4096.0f && x - f > m && x - f < 1.0f - m)) return false;
  o.ncol = (int64_t)(int)f;
  return true;
}

// ---------------------------------------------------------------------------
// One batch of G consecutive cells [k0, k0+G) whose particles fit the warp's
// staging area: gather through perm -> Step 3 moments -> Step 4 split, DSMC,
// Shakhov, rescale -> Step 5 sums -> velocities stored in cell order for the
// free flight (k_flight).  Particle work is spread over the lanes across the
// whole batch; per-cell FP64 arithmetic runs lane-per-cell (lane i <-> cell i).
// Bound by latency, of the dependent chains and the shared-memory round trips
// at 16 resident warps per SM (FP32 state), and in FP64 mode by the FP64
// pipe.  The phases stay in one kernel because they share the gather: sums
// and cell arithmetic as kernels of their own cost the 600 x 300 cylinder
// 98 us per step and saved 98.
// ---------------------------------------------------------------------------
template <class T, class A, int DIM, bool ONE>
__device__ void process_batch(const StepArgs& a, int64_t k0, int G, CellTab<T, A>* ct, uint32_t* sidx,
                              int* tags, int ntag, uint16_t (*soff)[kMaxSub + 1], T* svx, T* svy, T* svz) {
  using Acc = CellAcc<T, A>;
  constexpr bool kMixed = mixed_prec<T, A>();
  const int lane = threadIdx.x & 31;
  const int64_t NC = a.NC;
  const uint32_t step = *a.step;
  const uint32_t p0 = a.start[k0];
  const int M = (int)(a.start[k0 + G] - p0);
  // ---- lane-per-cell bookkeeping
  const bool own = lane < G;
  const int64_t kc = k0 + (own ? lane : 0);
  int Ni = 0, offi = 0;
  uint32_t inst = 0;
  // loaded early: used by the cell math (mixed precision: 1/V)
  double vol_k = 1.0, smax_k = 0.0, dt_k = 0.0;
  unsigned long long dt_min_k = 0;  // the instance's minimum so far
  if (own) {
    vol_k = kMixed ? a.ivol[kc] : a.vol[kc];
    smax_k = a.smax[kc];
    const uint32_t s0 = a.start[kc];
    Ni = (int)(a.start[kc + 1] - s0);
    offi = (int)(s0 - p0);
    inst = a.cell_inst[kc];
    dt_k = a.dt_cur[inst];
    if constexpr (kMixed) dt_min_k = *(volatile const unsigned long long*)&a.dt_min[inst];
    ct->off[lane] = offi;
    ct->inst[lane] = (int)inst;
    ct->nres[lane] = 0;
    ct->nar[lane] = 0;
  }
  if (lane == 0) ct->off[G] = M;
  __syncwarp();
  // the lanes' parts of the per-cell sums (split cells: FP32 state only)
  auto lp = lane_parts<kSplitOf<T, DIM>>(ct, G, own, offi, Ni);
  if constexpr (Acc::kExact) {
    for (unsigned b = __ballot_sync(kFull, own && Ni > kLaneSumMax && Ni <= kHomeCap); b; b &= b - 1) {
      const int c = __ffs(b) - 1, h = home_lane(a.start, NC, k0 + c, kSplitOf<T, DIM>);
      if (lane == c) lp.home = h;
    }
  }
  // ---- 1. source indices (in source order within each cell when the run is
  // reproducible: k_order_small, k_order_large) and cell of each slot
#pragma unroll 4
  for (int s = lane; s < M; s += 32) cp_async<4>(&sidx[s], &a.perm[p0 + s]);
  // the cell of slot sb + lane, for the 32 slots from sb (by the whole warp):
  // the cells that start up to it, from the lanes' own offsets
  const unsigned ne = __ballot_sync(kFull, own && Ni > 0);
  if (own && Ni > 0) ct->ne[__popc(ne & ((1u << lane) - 1u))] = (uint8_t)lane;
  const unsigned upto = 0xFFFFFFFFu >> (31 - lane);
  const auto slot_cell = [&](int sb) -> int {
    const bool has = own && Ni > 0;
    const unsigned heads = __reduce_or_sync(kFull, has && offi > sb && offi < sb + 32 ? 1u << (offi - sb) : 0u);
    const int before = __popc(__ballot_sync(kFull, has && offi <= sb));
    return ct->ne[before - 1 + __popc(heads & upto)];
  };
  // instance-local index of the batch's cell c (Philox counter)
  const auto kl_of = [&](int c) -> uint32_t {
    if constexpr (ONE) return (uint32_t)(k0 + c);
    else return (uint32_t)(k0 + c - a.P[ct->inst[c]].cell_off);
  };
  cp_async_wait_all();
  __syncwarp();
  // ---- 1b. Bird's sub-cells (option): each cell's slots in a stable order
  // by sub-cell (the sub-cell of a slot from its particle's position), so
  // that every sub-cell is a run of slots; offsets in soff
  const int nsub_i = own ? inst_params<ONE>(a, inst).nsub : 1;
  const unsigned subs = __ballot_sync(kFull, nsub_i > 1);
  if (subs) {
    uint16_t* slot_sub = (uint16_t*)tags;
    for (int sb = 0; sb < M; sb += 32) {
      const int s = sb + lane, c = slot_cell(sb);
      int sub = 0;
      if (s < M && ((subs >> c) & 1u)) {
        const InstParams& P = inst_params<ONE>(a, ct->inst[c]);
        T x[3] = {0, 0, 0};
        const uint32_t o = sidx[s];
#pragma unroll
        for (int d = 0; d < DIM; ++d) x[d] = ((const T*)a.Apos[d])[o];
        sub = subcell_of<T, DIM>(P, kl_of(c), x);
      }
      if (s < M) slot_sub[s] = (uint16_t)sub;
    }
    __syncwarp();
    if (nsub_i > 1) {  // lane i: a counting sort of cell i's slots (stable)
      uint16_t* so = soff[lane];
      for (int t = 0; t <= nsub_i; ++t) so[t] = 0;
      for (int s = offi; s < offi + Ni; ++s) so[slot_sub[s] + 1] += 1;
      for (int t = 0; t < nsub_i; ++t) so[t + 1] += so[t];
      uint32_t* tmp = (uint32_t*)svy;  // free until the gather
      for (int s = offi; s < offi + Ni; ++s) tmp[offi + so[slot_sub[s]]++] = sidx[s];
      for (int t = nsub_i; t > 0; --t) so[t] = so[t - 1];
      so[0] = 0;
      for (int s = offi; s < offi + Ni; ++s) sidx[s] = tmp[s];
    }
    __syncwarp();
    // the free flight reads the source indices from perm: store the sub-cell
    // order there
    if (nsub_i > 1)
      for (int s = offi; s < offi + Ni; ++s) a.perm[p0 + s] = sidx[s];
    __syncwarp();
  }
  // ---- 2. gather velocities (with the indices in the x-velocity array,
  // each lane reads slot s's index before it writes slot s's velocity);
  // every lane issues all of its copies before waiting once
  {
    const T* Av0 = (const T*)a.Avel[0];
    const T* Av1 = (const T*)a.Avel[1];
    const T* Av2 = (const T*)a.Avel[2];
#pragma unroll 4
    for (int s = lane; s < M; s += 32) {
      const uint32_t o = sidx[s];
      cp_async<sizeof(T)>(&svx[s], &Av0[o]);
      cp_async<sizeof(T)>(&svy[s], &Av1[o]);
      cp_async<sizeof(T)>(&svz[s], &Av2[o]);
    }
    for (int s = lane; s < ntag; s += 32) tags[s] = 0x7FFFFFFF;
    cp_async_wait_all();
  }
  __syncwarp();
  // ---- 3. moment sums per cell, kept by lane i (lane i <-> cell i).
  // All-FP32 mode, cells of at most kLaneSumMax particles: one pass, shifted
  // by the velocity D = c - c_1 of the cell's first particle (close to the
  // mean, so FP32 loses little to cancellation): sums of D, of D D^T and of
  // |D|^2 D, from which the central sums follow exactly (below).  All other
  // cases: two passes, the second about the cell mean U (FP64 mode: C = c - U
  // in FP64; FP32 state with FP64 cells: C = (c - U_h) -
  // U_l in FP32, with U = U_h + U_l the FP64 mean split into an FP32 pair, and
  // both passes summed without loss into FP64).
  bool one_pass = false;
  A m0 = 0, m1 = 0, m2 = 0, mS2 = 0, mS3x = 0, mS3y = 0, mS3z = 0;
  float sum_h[4] = {0, 0, 0, 0};  // mixed precision: the sums' high parts
  if constexpr (sizeof(A) == 4) {
    one_pass = own && Ni > 0 && Ni <= kLaneSumMax;
    if (one_pass) {
      const T c0x = svx[offi], c0y = svy[offi], c0z = svz[offi];
      T sx = 0, sy = 0, sz = 0, mxx = 0, myy = 0, mzz = 0, mxy = 0, mxz = 0, myz = 0, tx = 0, ty = 0, tz = 0;
#pragma unroll 2
      for (int q = offi; q < offi + Ni; ++q) {
        const T dx = svx[q] - c0x, dy = svy[q] - c0y, dz = svz[q] - c0z;
        sx += dx;
        sy += dy;
        sz += dz;
        mxx += dx * dx;
        myy += dy * dy;
        mzz += dz * dz;
        mxy += dx * dy;
        mxz += dx * dz;
        myz += dy * dz;
        const T d2 = dx * dx + dy * dy + dz * dz;
        tx += d2 * dx;
        ty += d2 * dy;
        tz += d2 * dz;
      }
      const T fN = (T)Ni, iN = cdiv((T)1, fN);
      const T ex = sx * iN, ey = sy * iN, ez = sz * iN;  // U - c_1
      m0 = fN * c0x + sx;
      m1 = fN * c0y + sy;
      m2 = fN * c0z + sz;
      if (Ni >= 2) {
        // C = D - e: sum |C|^2 = tr M - N |e|^2 and
        // sum |C|^2 C = T3 - e tr M - 2 M e + 2 e (e.S) + |e|^2 S - N |e|^2 e
        const T trM = mxx + myy + mzz, e2 = ex * ex + ey * ey + ez * ez, eS = ex * sx + ey * sy + ez * sz;
        mS2 = trM - fN * e2;
        const T Mex = mxx * ex + mxy * ey + mxz * ez;
        const T Mey = mxy * ex + myy * ey + myz * ez;
        const T Mez = mxz * ex + myz * ey + mzz * ez;
        mS3x = tx - ex * trM - (T)2 * Mex + (T)2 * ex * eS + e2 * sx - fN * e2 * ex;
        mS3y = ty - ey * trM - (T)2 * Mey + (T)2 * ey * eS + e2 * sy - fN * e2 * ey;
        mS3z = tz - ez * trM - (T)2 * Mez + (T)2 * ez * eS + e2 * sz - fN * e2 * ez;
      }
    }
  }
  const bool two_pass = own && !one_pass;
  if (__any_sync(kFull, two_pass)) {
    A r1[3];
    Acc a1[3];
    cell_sums_acc<Acc, 3>(lp, two_pass, offi, Ni, a1, [&](int s, int c, T* v, T* lo) {
      v[0] = svx[s];
      v[1] = svy[s];
      v[2] = svz[s];
      lo[0] = lo[1] = lo[2] = 0;
    });
#pragma unroll
    for (int d = 0; d < 3; ++d) r1[d] = a1[d].get();
    if (two_pass && Ni > 0) {  // the shift of the central sums: the cell mean
      if constexpr (kMixed) {
        // U = (s + e) / N as an FP32 pair U_h + U_l without FP64 work: the
        // residual s - U_h N is exact (an FMA), so U_h + U_l is the mean to
        // ~eps^2 relative
        const float fN = (float)Ni, rN = 1.0f / fN;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float uh = a1[d].s * rN;
          const float r = fmaf(-uh, fN, a1[d].s) + a1[d].e;
          ct->Up[d][lane] = uh;
          ct->Kl[d][lane] = r * rN;
        }
      } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) ct->Up[d][lane] = (T)cdiv(r1[d], (A)Ni);
      }
    }
    __syncwarp();
    // the second pass: sum |C|^2 and sum |C|^2 C (mixed precision: sum |C|^2
    // only; sum |C|^2 C, needed by the Shakhov cells alone, after Step 4)
    constexpr int K2 = kMixed ? 1 : 4;
    Acc a2[K2];
    cell_sums_acc<Acc, K2>(lp, two_pass, offi, Ni, a2, [&](int s, int c, T* v, T* lo) {
      T C0 = svx[s] - ct->Up[0][c], C1 = svy[s] - ct->Up[1][c], C2 = svz[s] - ct->Up[2][c];
      if constexpr (kMixed) {
        C0 -= ct->Kl[0][c];
        C1 -= ct->Kl[1][c];
        C2 -= ct->Kl[2][c];
      }
      const T c2 = C0 * C0 + C1 * C1 + C2 * C2;
      v[0] = c2;
      lo[0] = 0;
      if constexpr (K2 == 4) {
        v[1] = c2 * C0;
        v[2] = c2 * C1;
        v[3] = c2 * C2;
        lo[1] = lo[2] = lo[3] = 0;
      }
    });
    if (two_pass) {
      m0 = r1[0];
      m1 = r1[1];
      m2 = r1[2];
      if (Ni >= 2) {
        mS2 = a2[0].get();
        if constexpr (K2 == 4) {
          mS3x = a2[1].get();
          mS3y = a2[2].get();
          mS3z = a2[3].get();
        }
      }
      if constexpr (kMixed) {
#pragma unroll
        for (int d = 0; d < 3; ++d) sum_h[d] = a1[d].s;
        sum_h[3] = a2[0].s;
      }
    }
    __syncwarp();
  }
  // ---- 4. per-cell arithmetic in A, lane i <-> cell i (cell_math)
  const InstParams& Pi = inst_params<ONE>(a, inst);
  CellMath<A> cm;
  cm.clear();
  T smaxT = 0;
  bool sample = false;
  if (own) {
    sample = (int64_t)step >= (int64_t)Pi.n_steady;
    smaxT = (T)smax_k;
    bool settled = false;
    if constexpr (kMixed)
      settled = cell_settled(Pi, kl_of(lane), Ni, sum_h, sum_h[3], vol_k, a.iLc, kc, smaxT, dt_k, dt_min_k,
                             step, cm);
    if (!settled)
      cell_math<T, A, !kMixed>(a, Pi, kc, kl_of(lane), Ni, m0, m1, m2, mS2, mS3x, mS3y, mS3z, vol_k,
                               smaxT, dt_k, step, cm);
    ct->Pres[lane] = 0;
    if (cm.shk) {
      ct->RT[lane] = (T)cm.RT;
      ct->s2RT[lane] = (T)cm.s2RT;
      ct->omp[lane] = (T)cm.omp;
      if constexpr (!kMixed) ct->Amax[lane] = (T)cm.Amax;
    }
    if constexpr (kMixed) {  // the FP32 mean of the shift (U_h), no conversion
      ct->U[0][lane] = ct->Up[0][lane];
      ct->U[1][lane] = ct->Up[1][lane];
      ct->U[2][lane] = ct->Up[2][lane];
    } else {
      ct->U[0][lane] = (T)cm.U[0];
      ct->U[1][lane] = (T)cm.U[1];
      ct->U[2][lane] = (T)cm.U[2];
    }
    if (!kMixed && cm.shk) {  // the Shakhov sampling reads q_s in these cells only
      ct->q[0][lane] = (T)cm.q[0];
      ct->q[1][lane] = (T)cm.q[1];
      ct->q[2][lane] = (T)cm.q[2];
    }
  }
  if constexpr (kMixed) {
    // sum |C|^2 C about the Step 3 mean (the pair U_h + U_l), in the cells
    // with a Shakhov part only, before the DSMC sub-step moves any velocity
    const bool qsh = own && cm.shk;
    if (__any_sync(kFull, qsh)) {
      A r3[3];
      cell_sums<Acc, 3>(lp, qsh, offi, Ni, r3, [&](int s, int c, T* v, T* lo) {
        const T C0 = (svx[s] - ct->Up[0][c]) - ct->Kl[0][c];
        const T C1 = (svy[s] - ct->Up[1][c]) - ct->Kl[1][c];
        const T C2 = (svz[s] - ct->Up[2][c]) - ct->Kl[2][c];
        const T c2 = C0 * C0 + C1 * C1 + C2 * C2;
        v[0] = c2 * C0;
        v[1] = c2 * C1;
        v[2] = c2 * C2;
        lo[0] = lo[1] = lo[2] = 0;
      });
      if (qsh) {
        shakhov_q_amax(a, Pi, Ni, r3[0], r3[1], r3[2], cm);
        ct->q[0][lane] = (T)cm.q[0];
        ct->q[1][lane] = (T)cm.q[1];
        ct->q[2][lane] = (T)cm.q[2];
        ct->Amax[lane] = (T)cm.Amax;
      }
    }
  }
  const int64_t ncol = cm.ncol;
  const bool shk = cm.shk;
  const unsigned long long dtbits = cm.dtbits;
  A* UA = cm.U;
  const A TA = cm.T;
  // the instance's minimum Delta t_c: with one instance the warp's minimum
  // goes in one atomic (32 atomics per batch on one address otherwise)
  if constexpr (ONE) {
    unsigned long long mn = dtbits;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(kFull, mn, o);
      mn = y < mn ? y : mn;
    }
    if (lane == 0 && mn != ~0ull) atomicMin(&a.dt_min[0], mn);
  } else {
    if (dtbits != ~0ull) atomicMin(&a.dt_min[inst], dtbits);
  }
  // resampling probability 1 - exp(-dt_SBGK/tau) in FP64, only when a cell
  // of the batch has a Shakhov part
  if (__any_sync(kFull, shk) && shk) ct->Pres[lane] = (T)cm.Pres;
  const double ratio = (double)cm.ratio;
  __syncwarp();
  // ---- 5. DSMC sub-step.  In 3-D a cell with at most kLaneNtcMax
  // candidates runs its NTC loop on its own lane (lane i <-> cell i),
  // candidate after candidate: the one-by-one loop itself, with no clash
  // tags or scans.  The candidates of the other cells are flattened cell by
  // cell and taken 32 at a time, one per lane (below).
  const bool lane_ntc = kLaneNtcMax<DIM> > 0 && own && ncol > 0 && ncol <= kLaneNtcMax<DIM>;
  {
    int c_incl = lane_ntc ? 0 : (int)ncol;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, c_incl, o);
      if (lane >= o) c_incl += y;
    }
    if (own) {
      ct->coff[lane + 1] = c_incl;
      ct->smax[lane] = smaxT;
      ct->nacc[lane] = 0;
    }
    if (lane == 0) ct->coff[0] = 0;
  }
  __syncwarp();
  if constexpr (kLaneNtcMax<DIM> > 0) {
    const int nround = (int)__reduce_max_sync(kFull, lane_ntc ? (unsigned)ncol : 0u);
    if (nround > 0) {
      T smx = smaxT;
      int nacc_l = 0;
      const T coef = geo<T>(Pi).sigc_coef, ex = geo<T>(Pi).sigc_exp;
      for (int k = 0; k < nround; ++k) {
        if (lane_ntc && k < (int)ncol) {
          const int N = Ni;
          const NtcDraw<T> dr = ntc_draw((T)0, step, kl_of(lane), (uint32_t)k, Pi.key0, Pi.key1);
          int ci, cj;
          select_pair(N, dr.u1, dr.u2, soff[lane], nsub_i, &ci, &cj);
          ci += offi;
          cj += offi;
          const T ax = svx[ci], ay = svy[ci], az = svz[ci];
          const T bx = svx[cj], by = svy[cj], bz = svz[cj];
          const T g0 = ax - bx, g1 = ay - by, g2 = az - bz;
          T cr, u4, u5;
          bool pass;
          if constexpr (sizeof(T) == 4) {
            cr = csqrt(g0 * g0 + g1 * g1 + g2 * g2);
            const T sc = coef * cpow(cr, ex);
            if (sc > smx) smx = sc;  // the inclusive running maximum
            pass = dr.u3 * smx < sc;
            u4 = dr.u4;
            u5 = dr.u5;
          } else {
            const NtcTest tt = ntc_test(g0, g1, g2, smx, coef, ex, Pi.g32.sigc_coef, Pi.g32.sigc_exp);
            const T S = smx;
            if (tt.sc > smx) smx = tt.sc;
            pass = ntc_pass(tt, dr, g0, g1, g2, S, smx, coef, ex);
            if (pass) {
              cr = csqrt(g0 * g0 + g1 * g1 + g2 * g2);
              u4 = dr.u4();
              u5 = ntc_u5(step, kl_of(lane), (uint32_t)k, Pi.key0, Pi.key1);
            }
          }
          if (pass) {
            ++nacc_l;
            const T cchi = (T)2.0 * u4 - (T)1.0;
            const T schi = csqrt((T)1.0 - cchi * cchi);
            T sn, cs;
            sincos2pi(u5, &sn, &cs);
            const T w0 = cchi, w1 = schi * cs, w2 = schi * sn;
            const T q0 = ax + bx, q1 = ay + by, q2 = az + bz;
            svx[ci] = (T)0.5 * (q0 - cr * w0);
            svy[ci] = (T)0.5 * (q1 - cr * w1);
            svz[ci] = (T)0.5 * (q2 - cr * w2);
            svx[cj] = (T)0.5 * (q0 + cr * w0);
            svy[cj] = (T)0.5 * (q1 + cr * w1);
            svz[cj] = (T)0.5 * (q2 + cr * w2);
          }
        }
      }
      if (lane_ntc) {
        ct->smax[lane] = smx;
        ct->nacc[lane] = nacc_l;
      }
      __syncwarp();
    }
  }
  const int ctot = ct->coff[G];
  for (int base = 0; base < ctot; base += 32) {
    const int g = base + lane;
    const bool valid = g < ctot;
    int c = 255, ci = 0, cj = 0;
    NtcDraw<T> dr = {};
    if (valid) {
      int lo = 0, hi = G - 1;  // largest cell index with coff <= g
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (ct->coff[mid] <= g) lo = mid; else hi = mid - 1;
      }
      c = lo;
      const int N = ct->off[c + 1] - ct->off[c];
      const InstParams& P = inst_params<ONE>(a, ct->inst[c]);
      dr = ntc_draw((T)0, step, kl_of(c), (uint32_t)(g - ct->coff[c]), P.key0, P.key1);
      select_pair(N, dr.u1, dr.u2, soff[c], P.nsub, &ci, &cj);
      ci += ct->off[c];
      cj += ct->off[c];
    }
    const int cnext = __shfl_down_sync(kFull, c, 1), cprev = __shfl_up_sync(kFull, c, 1);
    const bool seg_last = valid && (lane == 31 || cnext != c);
    // the slots' entries in the folded tag table (ntag entries, slots below
    // 2 ntag + 2): two slots that share one only wait for each other
    const auto fold = [&](int s) {
      s = s < ntag ? s : s - ntag;
      return s < ntag ? s : s - ntag;
    };
    const int ti = fold(ci), tj = fold(cj);
    // the first lane of this lane's cell
    const int seg0 = 31 - __clz((int)(__ballot_sync(kFull, lane == 0 || c != cprev) & upto));
    const T coef = valid ? geo<T>(inst_params<ONE>(a, ct->inst[c])).sigc_coef : (T)0;
    const T ex = valid ? geo<T>(inst_params<ONE>(a, ct->inst[c])).sigc_exp : (T)0;
    const T smc = valid ? ct->smax[c] : (T)0;  // the cell's (sigma c)_max before this round
    unsigned pending = __ballot_sync(kFull, valid);
    // The one-by-one loop over a cell's candidates, run several at a time.
    // A candidate is evaluated (relative speed and sigma c from its pair's
    // current velocities) once no earlier pending candidate of its cell
    // shares a particle with it: its velocities are then final.  Its
    // acceptance test needs (sigma c)_max as the inclusive prefix maximum
    // over all earlier candidates of the cell.  It is decided when every
    // earlier candidate of the cell has been evaluated (the exact test), or
    // when it fails already against the prefix maximum of the evaluated
    // ones (the full maximum can only be larger, so it fails too: rejected,
    // nothing changes).  Accepted candidates of one pass share no particle,
    // and every pass decides at least the first pending candidate, so the
    // outcome is that of the one-by-one loop.
    bool known = false;
    T ax = 0, ay = 0, az = 0, bx = 0, by = 0, bz = 0, cr = 0, sc = (T)-1;
    NtcTest tt = {-1.0, 0.0f, false};
    while (pending) {
      const bool mine = (pending >> lane) & 1u;
      if (mine) {
        atomicMin(&tags[ti], lane);
        atomicMin(&tags[tj], lane);
      }
      __syncwarp();
      const bool ev = mine && tags[ti] == lane && tags[tj] == lane;
      __syncwarp();
      if (mine) {
        tags[ti] = 0x7FFFFFFF;
        tags[tj] = 0x7FFFFFFF;
      }
      if (ev && !known) {
        ax = svx[ci]; ay = svy[ci]; az = svz[ci];
        bx = svx[cj]; by = svy[cj]; bz = svz[cj];
        const T g0 = ax - bx, g1 = ay - by, g2 = az - bz;
        if constexpr (sizeof(T) == 4) {
          cr = csqrt(g0 * g0 + g1 * g1 + g2 * g2);
          sc = coef * cpow(cr, ex);
        } else {
          const Geo<float>& G32 = inst_params<ONE>(a, ct->inst[c]).g32;
          tt = ntc_test(g0, g1, g2, smc, coef, ex, G32.sigc_coef, G32.sigc_exp);
          sc = tt.sc;
        }
        known = true;
      }
      // inclusive prefix over the cell's lanes: maximum of the evaluated
      // sigma c, and whether all of them are evaluated
      const bool all = !(~__ballot_sync(kFull, known) & upto & (0xFFFFFFFFu << seg0));
      T pm = known ? sc : (T)-1;
      // (FP64 mode: sigma c is formed only where it may exceed the maximum)
      if (sizeof(T) == 4 || __any_sync(kFull, tt.exact)) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const T y = __shfl_up_sync(kFull, pm, o);
          if (lane - o >= seg0 && y > pm) pm = y;
        }
      }
      const T smL = pm > smc ? pm : smc;
      // P_c = sigma c / (sigma c)_max against u3; FP32 mode compares the
      // product (also monotone in (sigma c)_max, as the early rejection needs)
      bool pass;
      if constexpr (sizeof(T) == 4) pass = ev && dr.u3 * smL < sc;
      else pass = ev && ntc_pass(tt, dr, ax - bx, ay - by, az - bz, smc, smL, coef, ex);
      const bool decided = ev && (all || !pass);
      if (decided && pass) {
        atomicAdd(&ct->nacc[c], 1);
        T u4, u5;
        if constexpr (sizeof(T) == 4) {
          u4 = dr.u4;
          u5 = dr.u5;
        } else {
          const InstParams& P = inst_params<ONE>(a, ct->inst[c]);
          const T g0 = ax - bx, g1 = ay - by, g2 = az - bz;
          cr = csqrt(g0 * g0 + g1 * g1 + g2 * g2);
          u4 = dr.u4();
          u5 = ntc_u5(step, kl_of(c), (uint32_t)(g - ct->coff[c]), P.key0, P.key1);
        }
        const T cchi = (T)2.0 * u4 - (T)1.0;
        const T schi = csqrt((T)1.0 - cchi * cchi);
        T sn, cs;
        sincos2pi(u5, &sn, &cs);
        const T w0 = cchi, w1 = schi * cs, w2 = schi * sn;
        const T q0 = ax + bx, q1 = ay + by, q2 = az + bz;
        svx[ci] = (T)0.5 * (q0 - cr * w0);
        svy[ci] = (T)0.5 * (q1 - cr * w1);
        svz[ci] = (T)0.5 * (q2 - cr * w2);
        svx[cj] = (T)0.5 * (q0 + cr * w0);
        svy[cj] = (T)0.5 * (q1 + cr * w1);
        svz[cj] = (T)0.5 * (q2 + cr * w2);
      }
      pending &= ~__ballot_sync(kFull, decided);
      __syncwarp();
    }
    // the round's candidates raise the cell's (sigma c)_max
    T pm = sc;
    if (sizeof(T) == 4 || __any_sync(kFull, tt.exact)) {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(kFull, pm, o);
        if (lane - o >= seg0 && y > pm) pm = y;
      }
    }
    if (seg_last && pm > smc) ct->smax[c] = pm;
    __syncwarp();
  }
  int nacc_i = 0;
  if (own && ncol > 0) {
    nacc_i = ct->nacc[lane];
    a.smax[kc] = (double)ct->smax[lane];
  }
  // ---- 6. Shakhov sub-step.  First the Bernoulli draw of every slot, with
  // the resampled slots compacted into a list (the tags' bytes, free after the DSMC
  // loop); then the acceptance-rejection loops as a lane pool: a lane that
  // finishes a particle takes the next one from the list, so the warp's
  // iterations follow the total number of attempts instead of the slowest
  // lane of every 32 slots.  Every draw is keyed by (cell, slot, attempt),
  // so the order of the work changes no result.
  if (__any_sync(kFull, shk)) {
    int nlist = 0;
    uint16_t* list = (uint16_t*)tags;  // cell << 10 | slot (at most 1024 slots)
    for (int sb = 0; sb < M; sb += 32) {
      const int s = sb + lane, c = slot_cell(sb);
      bool res = false;
      if (s < M) {
        const T Pres = ct->Pres[c];
        if (Pres > (T)0) {
          const InstParams& P = inst_params<ONE>(a, ct->inst[c]);
          Uni<T> r(step, kl_of(c), (uint32_t)(s - ct->off[c]), kPurpShk << 24, P.key0, P.key1);
          res = r.get(0) < Pres;
        }
      }
      const unsigned bal = __ballot_sync(kFull, res);
      if (res) {
        list[nlist + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(c << 10 | s);
        atomicAdd(&ct->nres[c], 1);
        if (a.resamp) a.resamp[p0 + s] = 1;
      }
      nlist += __popc(bal);
    }
    __syncwarp();
    if (nlist > 0) {
      int s = lane < nlist ? list[lane] : -1;
      int next = 32, t = 0, c = 0, armax = 1;
      T RT = 0, s2RT = 0, Amax = 0, omp = 0, q0 = 0, q1 = 0, q2 = 0, kA = 0, iRT = 0;
      ShakhovFilter fl = {};
      Uni<T> r(0u, 0u, 0u, 0u, 0u, 0u);
      auto take = [&](int slot) {
        s = slot;
        t = 0;
        if (s < 0) return;
        c = s >> 10;
        s &= 1023;
        const InstParams& P = inst_params<ONE>(a, ct->inst[c]);
        r = Uni<T>(step, kl_of(c), (uint32_t)(s - ct->off[c]), kPurpShk << 24, P.key0, P.key1);
        armax = P.ar_max;
        RT = ct->RT[c];
        s2RT = ct->s2RT[c];
        Amax = ct->Amax[c];
        omp = ct->omp[c];
        if constexpr (sizeof(T) == 4) {  // FP32: the attempts' divisions as products
          kA = omp / ((T)5.0 * RT * RT);
          iRT = (T)1.0 / RT;
        }
        q0 = ct->q[0][c];
        q1 = ct->q[1][c];
        q2 = ct->q[2][c];
        if constexpr (sizeof(T) == 8) fl = shakhov_filter(RT, Amax, omp, q0, q1, q2);
      };
      take(s);
      while (__any_sync(kFull, s >= 0)) {
        bool done = false;
        if (s >= 0) {
          T C0, C1, C2;
          t = shakhov_skip(r, t, armax, fl);
          const bool acc = shakhov_attempt<T>(r, t, s2RT, Amax, omp, RT, kA, iRT, q0, q1, q2, &C0, &C1, &C2);
          if (acc || t == armax - 1) {
            if (!acc) atomicAdd(&a.err[kErrAr], 1ull);
            atomicAdd(&ct->nar[c], t + 1);
            svx[s] = ct->U[0][c] + C0;
            svy[s] = ct->U[1][c] + C1;
            svz[s] = ct->U[2][c] + C2;
            done = true;
          } else {
            ++t;
          }
        }
        const unsigned fin = __ballot_sync(kFull, done);
        if (done) {
          const int idx = next + __popc(fin & ((1u << lane) - 1u));
          take(idx < nlist ? list[idx] : -1);
        }
        next += __popc(fin);
      }
    }
  }
  __syncwarp();
  // ---- 7. conservation rescale c' = U + (c_p - U_p) sqrt(T/T_p) of every
  // particle of a cell with a resampled particle; U, T are the Step 3
  // moments (the targets), U_p, T_p those after the Shakhov sub-step.
  const int nres_i = own ? ct->nres[lane] : 0;
  const unsigned rcells = __ballot_sync(kFull, nres_i > 0);
  const bool rown = own && nres_i > 0;
  // Step 5 squares of the post-collision velocities of a rescaled cell (FP64
  // cells: from the rescale; else phase 8's pass)
  A bsq[3] = {0, 0, 0};
  if (rcells) {
    if constexpr (!kMixed) {
      // the U_p pass, then T_p about U_p (as the oracle; inside a sum the
      // order is cell_sums_acc's)
      A r1[3];
      cell_sums<Acc, 3>(lp, rown, offi, Ni, r1, [&](int s, int c, T* v, T* lo) {
        v[0] = svx[s];
        v[1] = svy[s];
        v[2] = svz[s];
        lo[0] = lo[1] = lo[2] = 0;
      });
      if (rown) {
        ct->Up[0][lane] = (T)(r1[0] / (A)Ni);
        ct->Up[1][lane] = (T)(r1[1] / (A)Ni);
        ct->Up[2][lane] = (T)(r1[2] / (A)Ni);
      }
      __syncwarp();
      A r2[1];
      cell_sums<Acc, 1>(lp, rown, offi, Ni, r2, [&](int s, int c, T* v, T* lo) {
        const T C0 = svx[s] - ct->Up[0][c], C1 = svy[s] - ct->Up[1][c], C2 = svz[s] - ct->Up[2][c];
        v[0] = C0 * C0 + C1 * C1 + C2 * C2;
        lo[0] = 0;
      });
      if (rown) {
        const double Tp = (double)r2[0] / (3.0 * Pi.R * (double)(Ni - 1));
        ct->q[0][lane] = Tp > 0 ? (T)sqrt((double)TA / Tp) : (T)-1;
        if constexpr (sizeof(A) == 8) {  // (T_p = 0: not rescaled, every velocity is U_p)
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const A u = Tp > 0 ? UA[d] : (A)ct->Up[d][lane];
            bsq[d] = (A)Ni * u * u;
          }
          if (Tp > 0) bsq[0] += (A)3.0 * (A)Pi.R * (A)(Ni - 1) * TA;
        }
      }
      __syncwarp();
      for (int sb = 0; sb < M; sb += 32) {
        const int s = sb + lane, c = slot_cell(sb);
        if (s >= M || !((rcells >> c) & 1u)) continue;
        const T f = ct->q[0][c];
        if (!(f > (T)0)) continue;
        svx[s] = ct->U[0][c] + (svx[s] - ct->Up[0][c]) * f;
        svy[s] = ct->U[1][c] + (svy[s] - ct->Up[1][c]) * f;
        svz[s] = ct->U[2][c] + (svz[s] - ct->Up[2][c]) * f;
      }
      __syncwarp();
    } else {
      // FP32 state, FP64 cells: one pass of exact sums of the deviations
      // d = c - U_h from the Step 3 mean U_h (as stored in FP32) and of
      // their squares; two_sum gives each deviation exactly as d_h + d_l
      // and two_prod its square, so that in FP64 U_p = U_h + sum d / N and
      // sum (c_i - U_p,i)^2 = sum d_i^2 - N (sum d_i / N)^2 are accurate to
      // a few 1e-13 (the deviations are thermal-sized: no cancellation).
      // The map is then applied as c' = c f + K, K = U - U_p f, with f and
      // K as FP32 pairs.
      A r[6];
      cell_sums<Acc, 6, true>(lp, rown, offi, Ni, r, [&](int s, int c, T* v, T* lo) {
        const T x[3] = {svx[s], svy[s], svz[s]};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          float dl;
          const float dh = two_sum(x[d], -ct->U[d][c], &dl);
          v[d] = dh;
          lo[d] = dl;
          float pe;
          v[3 + d] = two_prod(dh, dh, &pe);
          lo[3 + d] = fmaf(2.0f * dh, dl, pe);
        }
      });
      if (rown) {
        A Upd[3], Sii[3], Sp = 0;
        const A iN = (A)1 / (A)Ni;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const A e = r[d] * iN;
          Upd[d] = (A)ct->U[d][lane] + e;
          Sii[d] = r[3 + d] - r[d] * e;
          Sp += Sii[d];
        }
        if (Sp > 0) {
          // f = sqrt(T / T_p), T_p = sum |c - U_p|^2 / (3 R (N - 1))
          const A f = sqrt(TA * (A)3.0 * (A)Pi.R * (A)(Ni - 1) / Sp);
          ct->q[0][lane] = (T)f;
          ct->q[1][lane] = (T)(f - (A)(T)f);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const A K = UA[d] - Upd[d] * f;
            ct->Up[d][lane] = (T)K;
            ct->Kl[d][lane] = (T)(K - (A)(T)K);
            // sum (c'_d)^2 = f^2 sum (c_d - U_p,d)^2 + N U_d^2, since
            // sum (c'_d - U_d) = f sum (c_d - U_p,d) = 0
            bsq[d] = f * f * Sii[d] + (A)Ni * UA[d] * UA[d];
          }
        } else {
          ct->q[0][lane] = (T)-1;
#pragma unroll
          for (int d = 0; d < 3; ++d) bsq[d] = Sii[d] + (A)Ni * Upd[d] * Upd[d];
        }
      }
      __syncwarp();
      if (a.cons) {
        // record mode: the FP64 values of the rescaled velocities (before
        // they are rounded to FP32) summed in FP64, against the targets
        const bool chk = rown && ct->q[0][lane] > (T)0;
        double r3[4];
        cell_sums<PlainSum<double>, 4>(lp, chk, offi, Ni, r3, [&](int s, int c, double* v, double* lo) {
          const T x[3] = {svx[s], svy[s], svz[s]};
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            float l;
            const float h = affine_ff(x[d], ct->q[0][c], ct->q[1][c], ct->Up[d][c], ct->Kl[d][c], &l);
            v[d] = (double)h + (double)l;
            lo[d] = 0;
          }
          v[3] = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
          lo[3] = 0;
        });
        if (chk) record_conservation(a, kc, Ni, Pi, UA, TA, r3);
      }
      for (int sb = 0; sb < M; sb += 32) {
        const int s = sb + lane, c = slot_cell(sb);
        if (s >= M || !((rcells >> c) & 1u)) continue;
        const T f = ct->q[0][c];
        if (!(f > (T)0)) continue;
        float l;
        float h = affine_ff(svx[s], f, ct->q[1][c], ct->Up[0][c], ct->Kl[0][c], &l);
        svx[s] = h + l;
        h = affine_ff(svy[s], f, ct->q[1][c], ct->Up[1][c], ct->Kl[1][c], &l);
        svy[s] = h + l;
        h = affine_ff(svz[s], f, ct->q[1][c], ct->Up[2][c], ct->Kl[2][c], &l);
        svz[s] = h + l;
      }
      __syncwarp();
    }
    if constexpr (sizeof(T) == 8) {
      if (a.cons) {
        // record mode, FP64 mode: the rescaled velocities summed in FP64
        const bool chk = rown && ct->q[0][lane] > (T)0;
        double r3[4];
        cell_sums<PlainSum<double>, 4>(lp, chk, offi, Ni, r3, [&](int s, int c, double* v, double* lo) {
          v[0] = svx[s];
          v[1] = svy[s];
          v[2] = svz[s];
          v[3] = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
          lo[0] = lo[1] = lo[2] = lo[3] = 0;
        });
        if (chk) record_conservation(a, kc, Ni, Pi, UA, TA, r3);
      }
    }
  }
  // ---- 8. time-averaged sums (Step 5).  Both collision sub-steps conserve
  // each cell's momentum (the DSMC pair rule and the rescale to U), so the
  // momentum sums are those of Step 3 up to rounding.  With FP64 cells (FP64
  // and mixed mode) only the total sum |c|^2 is kept, in the first square's
  // slot (the averaged T needs no more): a cell without a rescale had DSMC
  // collisions alone, which conserve its energy, so its total is
  // sum |C|^2 + |sum c|^2 / N of Step 3; a rescaled cell's comes from the
  // rescale (mixed: its exact sums; FP64: its targets, sum |c'|^2 =
  // 3 R (N-1) T + N |U|^2).  The all-FP32 mode sums the per-component squares
  // of the post-collision velocities.
  constexpr bool kEnergy = sizeof(A) == 8;
  const bool need_sq = !kEnergy && own && sample && Ni > 0;
  const A a0 = m0, a1 = m1, a2 = m2;
  A b0 = bsq[0], b1 = bsq[1], b2 = bsq[2];
  if constexpr (kEnergy) {
    if (own && sample && Ni > 0) {
      if (nres_i > 0) {
        b0 = b0 + b1 + b2;
      } else {
        const A iN = Ni <= kHugeCell ? a.rcp[Ni] : (A)1 / (A)Ni;
        b0 = mS2 + (m0 * m0 + m1 * m1 + m2 * m2) * iN;
      }
      b1 = b2 = 0;
    }
  }
  constexpr unsigned kSampSlots = kEnergy ? 0x9Fu : 0xFFu;  // FP64 cells: slots 5, 6 unused
  double sv[8];  // the accumulators, requested before the sums
  if (own && sample) {
#pragma unroll
    for (int k = 0; k < 8; ++k) sv[k] = (kSampSlots >> k & 1u) ? a.samp[k * NC + kc] : 0.0;
  }
  if (__any_sync(kFull, need_sq)) {
    A r[3];
    cell_sums<Acc, 3>(lp, need_sq, offi, Ni, r, [&](int s, int c, T* v, T* lo) {
      const T x0 = svx[s], x1 = svy[s], x2 = svz[s];
      v[0] = x0 * x0;
      v[1] = x1 * x1;
      v[2] = x2 * x2;
      lo[0] = lo[1] = lo[2] = 0;
    });
    if (need_sq) {
      b0 = r[0];
      b1 = r[1];
      b2 = r[2];
    }
  }
  if (own) {
    if (sample) {
      double* S = a.samp;
      S[0 * NC + kc] = sv[0] + (double)Ni;
      if (Ni > 0) {
        S[1 * NC + kc] = sv[1] + (double)a0;
        S[2 * NC + kc] = sv[2] + (double)a1;
        S[3 * NC + kc] = sv[3] + (double)a2;
        S[4 * NC + kc] = sv[4] + (double)b0;
        if constexpr (!kEnergy) {
          S[5 * NC + kc] = sv[5] + (double)b1;
          S[6 * NC + kc] = sv[6] + (double)b2;
        }
      }
      S[7 * NC + kc] = sv[7] + ratio;
    }
    if (a.rec) {
      a.rec[0 * NC + kc] = (int32_t)ncol;
      a.rec[1 * NC + kc] = nacc_i;
      a.rec[2 * NC + kc] = nres_i;
      a.rec[3 * NC + kc] = ct->nar[lane];
    }
  }
  // ---- 9. the post-collision velocities in the current cell order, for the
  // free flight (k_flight)
  T* Bv0 = (T*)a.Bvel[0] + p0;
  T* Bv1 = (T*)a.Bvel[1] + p0;
  T* Bv2 = (T*)a.Bvel[2] + p0;
#pragma unroll 4
  for (int s = lane; s < M; s += 32) {
    Bv0[s] = svx[s];
    Bv1[s] = svy[s];
    Bv2[s] = svz[s];
  }
  __syncwarp();
}

template <class T, class A, int DIM, bool ONE>
__global__ void __launch_bounds__(32 * kMaxWarpsPerBlock, sizeof(T) == 4 ? 2 : 1) k_collide(StepArgs a, int big) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cap = big ? a.big_cap : a.cap_small;
  if (big && warp != 0) return;
  const bool subs = a.subcells != 0;
  unsigned char* base = smem + (size_t)(big ? 0 : warp) * warp_stage_bytes<T, A>(cap, subs);
  CellTab<T, A>* ct = (CellTab<T, A>*)base;
  uint16_t(*soff)[kMaxSub + 1] = (uint16_t(*)[kMaxSub + 1])(base + sizeof(CellTab<T, A>));
  T* svx = (T*)(base + sizeof(CellTab<T, A>) + (subs ? kSubBytes : 0));
  T* svy = svx + cap;
  T* svz = svy + cap;
  unsigned char* tail = (unsigned char*)(svz + cap);
  uint32_t* sidx = (uint32_t*)svx;
  if (!idx_in_velocity<T>()) {
    sidx = (uint32_t*)tail;
    tail += 4 * (size_t)cap;
  }
  int* tags = (int*)tail;
  // One call site of process_batch for both launches, so that every cell
  // runs through the same inlined code (identical rounding whichever launch
  // or batch takes it).  Main launch: batches from the plan's class lists by
  // work stealing, most expensive class first.  Big-cell
  // launch: a block per cell of the big list.
  // the end of each class in ticket order (main launch)
  uint32_t cend[kBatchClasses];
  uint32_t nb = 0;
#pragma unroll
  for (int k = 0; k < kBatchClasses; ++k) {
    nb += big ? 0u : a.nbatch[k];
    cend[k] = nb;
  }
  if (big) nb = *a.big_count;
  uint32_t it = big ? blockIdx.x : 0u;
  for (;;) {
    int64_t k0;
    int G;
    if (!big) {
      uint32_t t = 0;
      if (lane == 0) t = atomicAdd(a.ticket, 1u);
      t = __shfl_sync(kFull, t, 0);
      if (t >= nb) break;
      int cls = 0;
      uint32_t c0 = 0;
#pragma unroll
      for (int k = 0; k + 1 < kBatchClasses; ++k)
        if (t >= cend[k]) {
          cls = k + 1;
          c0 = cend[k];
        }
      const uint2 b = a.batches[(int64_t)cls * a.NC + (int64_t)(t - c0)];
      k0 = (int64_t)b.x;
      G = (int)b.y;
    } else {
      if (it >= nb) break;
      k0 = (int64_t)a.big_list[it];
      it += gridDim.x;
      G = 1;
      if ((int)(a.start[k0 + 1] - a.start[k0]) > kHugeCell) continue;  // k_collide_huge's cell
    }
    const long long t0 = clock64();
    process_batch<T, A, DIM, ONE>(a, k0, G, ct, sidx, tags, cap / 2, soff, svx, svy, svz);
    if (!big) {
      // the batch's cost steers the next step's plan (no effect on results):
      // its cycles per particle in units of cyc[2] (1/16 of the last step's
      // mean), saturating at 255, as the cost byte of each of its cells
      const unsigned long long cyc = (unsigned long long)(clock64() - t0);
      const unsigned long long Mb = a.start[k0 + G] - a.start[k0];
      if (lane == 0) {
        atomicAdd(&a.cyc[0], cyc);
        atomicAdd(&a.cyc[1], Mb);
      }
      const unsigned long long unit = a.cyc[2];
      unsigned long long w = 16;
      if (unit != ~0ull && unit > 0 && Mb > 0) {
        w = cyc / (unit * Mb);
        if (w < 1) w = 1;
        if (w > 255) w = 255;
      }
      if (lane < G) a.cost[k0 + lane] = (uint8_t)w;
    }
  }
}

// ---------------------------------------------------------------------------
// Cells above kHugeCell particles: one block of kHugeThreads threads per
// cell (the big-cell list is shared with the one-warp launch, which takes
// the cells up to kHugeCell).  The threshold is fixed, not the schedule's
// staging capacity, so that which code runs a cell depends on the cell
// alone (results do not depend on the schedule).  The block stages the
// cell in shared memory when it fits the launch's staging area and
// otherwise in the cell's own output slots in global memory (velocities in
// the B velocity arrays, source indices in the key array, clash tags in the
// first B position array; k_flight overwrites all three afterwards), so
// no cell size is refused.  The steps are those of process_batch for one
// cell: gather, two-pass moments, cell_math, the NTC loop
// with exactly the one-by-one outcome (candidates of a round evaluated as
// soon as their pair is final, decided against the prefix maximum of
// sigma c), Shakhov resampling, the conservation rescale, Step 5 sums and
// the velocities in cell order for k_flight.
// ---------------------------------------------------------------------------
template <class T, class A>
struct __align__(16) HugeTab {
  using acc_t = A;
  A red[kHugeWarps][8];  // per-warp partial sums
  A sum[8];              // the block's sums
  T wpm[kHugeWarps];     // prefix scans across warps (NTC passes)
  int wall[kHugeWarps];
  T U[3], q[3], RT, s2RT, Amax, Pres, omp, f, fl, Kh[3], Kl[3], smax;
  A UA[3], TA;
  int ncol, nacc, nres, nar;
  double ratio;
  int shk;
  int soff[kMaxSub + 1];  // sub-cell offsets (sub-cells on)
};

// Bytes of staging per particle in shared memory: velocities, source
// index, clash tag.
template <class T>
__host__ __device__ constexpr size_t huge_bytes_per_particle() {
  return 3 * sizeof(T) + 4 + 4;
}
// Particles staged in shared memory by the huge-cell launch.
template <class T>
__host__ __device__ constexpr int huge_smem_cap() {
  return sizeof(T) == 4 ? 4096 : 2048;
}
template <class T, class A>
__host__ __device__ constexpr size_t huge_smem_bytes() {
  return (sizeof(HugeTab<T, A>) + 15) / 16 * 16 + (size_t)huge_smem_cap<T>() * huge_bytes_per_particle<T>();
}

// Block-wide sums over n slots with an order fixed by n and the block size:
// thread t sums its contiguous share (the accumulator Acc), a butterfly
// combines each warp, and thread 0 adds the warp totals in warp order.
// Every thread returns the sums in out[].
template <class Acc, int K, bool kLo = false, class TabT, class F>
__device__ __forceinline__ void block_sums(TabT* tb, int n, typename Acc::result (&out)[K], F f) {
  using Tm = typename Acc::term;
  using R = typename Acc::result;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = (n + kHugeThreads - 1) / kHugeThreads;
  const int s0 = tid * per;
  const int s1 = s0 + per < n ? s0 + per : n;
  Acc acc[K];
#pragma unroll
  for (int k = 0; k < K; ++k) acc[k].init();
  for (int s = s0; s < s1; ++s) {
    Tm v[K], lo[K];
    f(s, v, lo);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if constexpr (kLo) acc[k].add(v[k], lo[k]);
      else acc[k].add1(v[k]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k].combine(acc[k].shfl_xor(o));
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) tb->red[w][k] = (typename TabT::acc_t)acc[k].get();
  __syncthreads();
  if (tid == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      R t = 0;
      for (int i = 0; i < kHugeWarps; ++i) t += (R)tb->red[i][k];
      tb->sum[k] = (typename TabT::acc_t)t;
    }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = (R)tb->sum[k];
  __syncthreads();
}

template <class T, class A, int DIM, bool ONE>
__global__ void __launch_bounds__(kHugeThreads, 2) k_collide_huge(StepArgs a) {
  using Acc = CellAcc<T, A>;
  constexpr bool kMixed = mixed_prec<T, A>();
  extern __shared__ __align__(16) unsigned char smem[];
  HugeTab<T, A>* tb = (HugeTab<T, A>*)smem;
  unsigned char* stage = smem + (sizeof(HugeTab<T, A>) + 15) / 16 * 16;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t step = *a.step;
  const uint32_t nb = *a.big_count;
  for (uint32_t it = blockIdx.x; it < nb; it += gridDim.x) {
    const int64_t k = (int64_t)a.big_list[it];
    const uint32_t p0 = a.start[k];
    const int N = (int)(a.start[k + 1] - p0);
    if (N <= kHugeCell) continue;  // the one-warp launch's cell
    const uint32_t inst = a.cell_inst[k];
    const InstParams& Pi = inst_params<ONE>(a, inst);
    const uint32_t kl = (uint32_t)(k - Pi.cell_off);
    // ---- staging: shared memory, else the cell's own output slots
    T *svx, *svy, *svz;
    uint32_t* sidx;
    int* stag;
    if (N <= huge_smem_cap<T>()) {
      const int cap = huge_smem_cap<T>();
      svx = (T*)stage;
      svy = svx + cap;
      svz = svy + cap;
      sidx = (uint32_t*)(svz + cap);
      stag = (int*)(sidx + cap);
    } else {
      svx = (T*)a.Bvel[0] + p0;
      svy = (T*)a.Bvel[1] + p0;
      svz = (T*)a.Bvel[2] + p0;
      sidx = a.key + p0;
      stag = (int*)((T*)a.Bpos[0] + p0);
    }
    // ---- 1. source indices (in source order when the run is reproducible)
    for (int s = tid; s < N; s += kHugeThreads) sidx[s] = a.perm[p0 + s];
    __syncthreads();
    // Bird's sub-cells (option): the slots in a stable order by sub-cell
    const int nsub = Pi.nsub;
    if (nsub > 1) {
      for (int s = tid; s < N; s += kHugeThreads) {
        T x[3] = {0, 0, 0};
        const uint32_t o = sidx[s];
#pragma unroll
        for (int d = 0; d < DIM; ++d) x[d] = ((const T*)a.Apos[d])[o];
        stag[s] = subcell_of<T, DIM>(Pi, kl, x);
      }
      __syncthreads();
      if (tid == 0) {
        int* so = tb->soff;
        for (int t = 0; t <= nsub; ++t) so[t] = 0;
        for (int s = 0; s < N; ++s) so[stag[s] + 1] += 1;
        for (int t = 0; t < nsub; ++t) so[t + 1] += so[t];
        uint32_t* tmp = (uint32_t*)svy;  // free until the gather
        for (int s = 0; s < N; ++s) tmp[so[stag[s]]++] = sidx[s];
        for (int t = nsub; t > 0; --t) so[t] = so[t - 1];
        so[0] = 0;
      }
      __syncthreads();
      for (int s = tid; s < N; s += kHugeThreads) {
        sidx[s] = ((const uint32_t*)svy)[s];
        a.perm[p0 + s] = sidx[s];  // (for the free flight)
      }
      __syncthreads();
    }
    // ---- 2. gather
    {
      const T* Av0 = (const T*)a.Avel[0];
      const T* Av1 = (const T*)a.Avel[1];
      const T* Av2 = (const T*)a.Avel[2];
      for (int s = tid; s < N; s += kHugeThreads) {
        const uint32_t o = sidx[s];
        svx[s] = Av0[o];
        svy[s] = Av1[o];
        svz[s] = Av2[o];
        stag[s] = 0x7FFFFFFF;
      }
    }
    __syncthreads();
    // ---- 3. moments: the mean, then the central sums about it
    A r1[3];
    block_sums<Acc, 3>(tb, N, r1, [&](int s, auto* v, auto* lo) {
      v[0] = svx[s];
      v[1] = svy[s];
      v[2] = svz[s];
      lo[0] = lo[1] = lo[2] = 0;
    });
    T sh[3], shl[3] = {0, 0, 0};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const A Ud = cdiv(r1[d], (A)N);
      sh[d] = (T)Ud;
      if constexpr (kMixed) shl[d] = (T)(Ud - (A)(T)Ud);
    }
    A r2[4];
    block_sums<Acc, 4>(tb, N, r2, [&](int s, auto* v, auto* lo) {
      T C0 = svx[s] - sh[0], C1 = svy[s] - sh[1], C2 = svz[s] - sh[2];
      if constexpr (kMixed) {
        C0 -= shl[0];
        C1 -= shl[1];
        C2 -= shl[2];
      }
      const T c2 = C0 * C0 + C1 * C1 + C2 * C2;
      v[0] = c2;
      v[1] = c2 * C0;
      v[2] = c2 * C1;
      v[3] = c2 * C2;
      lo[0] = lo[1] = lo[2] = lo[3] = 0;
    });
    // ---- 4. per-cell arithmetic (thread 0)
    const bool sample = (int64_t)step >= (int64_t)Pi.n_steady;
    if (tid == 0) {
      CellMath<A> cm;
      cm.clear();
      const T smaxT = (T)a.smax[k];
      cell_math<T, A>(a, Pi, k, kl, N, r1[0], r1[1], r1[2], r2[0], r2[1], r2[2], r2[3],
                      mixed_prec<T, A>() ? a.ivol[k] : a.vol[k], smaxT,
                      a.dt_cur[inst], step, cm);
      if (cm.dtbits != ~0ull) atomicMin(&a.dt_min[inst], cm.dtbits);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        tb->U[d] = (T)cm.U[d];
        tb->q[d] = (T)cm.q[d];
        tb->UA[d] = cm.U[d];
      }
      tb->TA = cm.T;
      tb->RT = (T)cm.RT;
      tb->s2RT = (T)cm.s2RT;
      tb->Amax = (T)cm.Amax;
      tb->omp = (T)cm.omp;
      tb->Pres = cm.shk ? (T)cm.Pres : (T)0;
      tb->smax = smaxT;
      tb->ncol = (int)cm.ncol;
      tb->nacc = 0;
      tb->nres = 0;
      tb->nar = 0;
      tb->ratio = (double)cm.ratio;
      tb->shk = cm.shk ? 1 : 0;
    }
    __syncthreads();
    // ---- 5. DSMC: rounds of kHugeThreads consecutive candidates
    const int ncol = tb->ncol;
    if (ncol > 0) {
      const T coef = geo<T>(Pi).sigc_coef, ex = geo<T>(Pi).sigc_exp;
      T smx = tb->smax;
      for (int base = 0; base < ncol; base += kHugeThreads) {
        const int g = base + tid;
        const bool valid = g < ncol;
        int ci = 0, cj = 0;
        NtcDraw<T> dr = {};
        if (valid) {
          dr = ntc_draw((T)0, step, kl, (uint32_t)g, Pi.key0, Pi.key1);
          select_pair(N, dr.u1, dr.u2, tb->soff, nsub, &ci, &cj);
        }
        bool pending = valid, known = false;
        T ax = 0, ay = 0, az = 0, bx = 0, by = 0, bz = 0, cr = 0, sc = (T)-1;
        NtcTest tt = {-1.0, 0.0f, false};
        for (;;) {
          if (pending) {
            atomicMin(&stag[ci], tid);
            atomicMin(&stag[cj], tid);
          }
          __syncthreads();
          const bool ev = pending && stag[ci] == tid && stag[cj] == tid;
          __syncthreads();
          if (pending) {
            stag[ci] = 0x7FFFFFFF;
            stag[cj] = 0x7FFFFFFF;
          }
          if (ev && !known) {
            ax = svx[ci]; ay = svy[ci]; az = svz[ci];
            bx = svx[cj]; by = svy[cj]; bz = svz[cj];
            const T g0 = ax - bx, g1 = ay - by, g2 = az - bz;
            if constexpr (sizeof(T) == 4) {
              cr = csqrt(g0 * g0 + g1 * g1 + g2 * g2);
              sc = coef * cpow(cr, ex);
            } else {
              tt = ntc_test(g0, g1, g2, smx, coef, ex, Pi.g32.sigc_coef, Pi.g32.sigc_exp);
              sc = tt.sc;
            }
            known = true;
          }
          // inclusive prefix over the candidates: maximum of the evaluated
          // sigma c, and whether every earlier one is evaluated
          T pm = known ? sc : (T)-1;
          int all = known || !valid;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const T y = __shfl_up_sync(kFull, pm, o);
            const int ya = __shfl_up_sync(kFull, all, o);
            if (lane >= o) {
              if (y > pm) pm = y;
              all = all && ya;
            }
          }
          if (lane == 31) {
            tb->wpm[w] = pm;
            tb->wall[w] = all;
          }
          __syncthreads();
          for (int i = 0; i < w; ++i) {
            if (tb->wpm[i] > pm) pm = tb->wpm[i];
            all = all && tb->wall[i];
          }
          const T smL = pm > smx ? pm : smx;
          bool pass;
          if constexpr (sizeof(T) == 4) pass = ev && dr.u3 * smL < sc;
          else pass = ev && ntc_pass(tt, dr, ax - bx, ay - by, az - bz, smx, smL, coef, ex);
          const bool decided = ev && (all || !pass);
          if (decided && pass) {
            atomicAdd(&tb->nacc, 1);
            T u4, u5;
            if constexpr (sizeof(T) == 4) {
              u4 = dr.u4;
              u5 = dr.u5;
            } else {
              const T g0 = ax - bx, g1 = ay - by, g2 = az - bz;
              cr = csqrt(g0 * g0 + g1 * g1 + g2 * g2);
              u4 = dr.u4();
              u5 = ntc_u5(step, kl, (uint32_t)g, Pi.key0, Pi.key1);
            }
            const T cchi = (T)2.0 * u4 - (T)1.0;
            const T schi = csqrt((T)1.0 - cchi * cchi);
            T sn, cs;
            sincos2pi(u5, &sn, &cs);
            const T w0 = cchi, w1 = schi * cs, w2 = schi * sn;
            const T q0 = ax + bx, q1 = ay + by, q2 = az + bz;
            svx[ci] = (T)0.5 * (q0 - cr * w0);
            svy[ci] = (T)0.5 * (q1 - cr * w1);
            svz[ci] = (T)0.5 * (q2 - cr * w2);
            svx[cj] = (T)0.5 * (q0 + cr * w0);
            svy[cj] = (T)0.5 * (q1 + cr * w1);
            svz[cj] = (T)0.5 * (q2 + cr * w2);
          }
          if (decided) pending = false;
          if (!__syncthreads_or(pending)) break;
        }
        // the round's candidates raise (sigma c)_max
        T mx = sc;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const T y = __shfl_xor_sync(kFull, mx, o);
          if (y > mx) mx = y;
        }
        if (lane == 0) tb->wpm[w] = mx;
        __syncthreads();
        for (int i = 0; i < kHugeWarps; ++i)
          if (tb->wpm[i] > smx) smx = tb->wpm[i];
        __syncthreads();
      }
      if (tid == 0) a.smax[k] = (double)smx;
    }
    // ---- 6. Shakhov resampling, slot by slot
    if (tb->shk) {
      const T Pres = tb->Pres;
      const T RT = tb->RT, s2RT = tb->s2RT, Amax = tb->Amax, omp = tb->omp;
      const T q0 = tb->q[0], q1 = tb->q[1], q2 = tb->q[2];
      T kA = 0, iRT = 0;
      if constexpr (sizeof(T) == 4) {
        kA = omp / ((T)5.0 * RT * RT);
        iRT = (T)1.0 / RT;
      }
      const ShakhovFilter fl = shakhov_filter(RT, Amax, omp, q0, q1, q2);
      int nres = 0, nar = 0;
      for (int s = tid; s < N; s += kHugeThreads) {
        const Uni<T> r0(step, kl, (uint32_t)s, kPurpShk << 24, Pi.key0, Pi.key1);
        Uni<T> r = r0;
        if (!(r.get(0) < Pres)) continue;
        ++nres;
        if (a.resamp) a.resamp[p0 + s] = 1;
        for (int t = 0;; ++t) {
          T C0, C1, C2;
          t = shakhov_skip(r0, t, Pi.ar_max, fl);
          const bool acc = shakhov_attempt<T>(r0, t, s2RT, Amax, omp, RT, kA, iRT, q0, q1, q2, &C0, &C1, &C2);
          if (acc || t == Pi.ar_max - 1) {
            if (!acc) atomicAdd(&a.err[kErrAr], 1ull);
            nar += t + 1;
            svx[s] = tb->U[0] + C0;
            svy[s] = tb->U[1] + C1;
            svz[s] = tb->U[2] + C2;
            break;
          }
        }
      }
      if (nres) {
        atomicAdd(&tb->nres, nres);
        atomicAdd(&tb->nar, nar);
      }
    }
    __syncthreads();
    // ---- 7. conservation rescale (as process_batch)
    const int nres = tb->nres;
    A bsq[3] = {0, 0, 0};
    bool bsq_ok = false;
    if (nres > 0) {
      if constexpr (!kMixed) {
        A u[3];
        block_sums<Acc, 3>(tb, N, u, [&](int s, auto* v, auto* lo) {
          v[0] = svx[s];
          v[1] = svy[s];
          v[2] = svz[s];
          lo[0] = lo[1] = lo[2] = 0;
        });
        const T Up0 = (T)(u[0] / (A)N), Up1 = (T)(u[1] / (A)N), Up2 = (T)(u[2] / (A)N);
        A e[1];
        block_sums<Acc, 1>(tb, N, e, [&](int s, auto* v, auto* lo) {
          const T C0 = svx[s] - Up0, C1 = svy[s] - Up1, C2 = svz[s] - Up2;
          v[0] = C0 * C0 + C1 * C1 + C2 * C2;
          lo[0] = 0;
        });
        const double Tp = (double)e[0] / (3.0 * Pi.R * (double)(N - 1));
        const T f = Tp > 0 ? (T)sqrt((double)tb->TA / Tp) : (T)-1;
        if (f > (T)0)
          for (int s = tid; s < N; s += kHugeThreads) {
            svx[s] = tb->U[0] + (svx[s] - Up0) * f;
            svy[s] = tb->U[1] + (svy[s] - Up1) * f;
            svz[s] = tb->U[2] + (svz[s] - Up2) * f;
          }
        __syncthreads();
        if constexpr (sizeof(T) == 8) {
          if (a.cons && f > (T)0) {
            double r3[4];
            block_sums<PlainSum<double>, 4>(tb, N, r3, [&](int s, double* v, double* lo) {
              v[0] = svx[s];
              v[1] = svy[s];
              v[2] = svz[s];
              v[3] = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
              lo[0] = lo[1] = lo[2] = lo[3] = 0;
            });
            if (tid == 0) record_conservation(a, k, N, Pi, tb->UA, tb->TA, r3);
          }
        }
      } else {
        A r[6];
        const T uh0 = tb->U[0], uh1 = tb->U[1], uh2 = tb->U[2];
        block_sums<Acc, 6, true>(tb, N, r, [&](int s, auto* v, auto* lo) {
          const T x[3] = {svx[s], svy[s], svz[s]};
          const T u[3] = {uh0, uh1, uh2};
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            float dl;
            const float dh = two_sum(x[d], -u[d], &dl);
            v[d] = dh;
            lo[d] = dl;
            float pe;
            v[3 + d] = two_prod(dh, dh, &pe);
            lo[3 + d] = fmaf(2.0f * dh, dl, pe);
          }
        });
        if (tid == 0) {
          A Upd[3], Sii[3], Sp = 0;
          const A iN = (A)1 / (A)N;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const A e = r[d] * iN;
            Upd[d] = (A)tb->U[d] + e;
            Sii[d] = r[3 + d] - r[d] * e;
            Sp += Sii[d];
          }
          tb->f = (T)-1;
          if (Sp > 0) {
            const A f = sqrt(tb->TA * (A)3.0 * (A)Pi.R * (A)(N - 1) / Sp);
            tb->f = (T)f;
            tb->fl = (T)(f - (A)(T)f);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const A K = tb->UA[d] - Upd[d] * f;
              tb->Kh[d] = (T)K;
              tb->Kl[d] = (T)(K - (A)(T)K);
              tb->red[0][d] = f * f * Sii[d] + (A)N * tb->UA[d] * tb->UA[d];
            }
          } else {
#pragma unroll
            for (int d = 0; d < 3; ++d) tb->red[0][d] = Sii[d] + (A)N * Upd[d] * Upd[d];
          }
        }
        __syncthreads();
#pragma unroll
        for (int d = 0; d < 3; ++d) bsq[d] = tb->red[0][d];
        bsq_ok = true;
        const T f = tb->f;
        __syncthreads();
        if (f > (T)0) {
          const T fl = tb->fl;
          if (a.cons) {
            double r3[4];
            block_sums<PlainSum<double>, 4>(tb, N, r3, [&](int s, double* v, double* lo) {
              const T x[3] = {svx[s], svy[s], svz[s]};
#pragma unroll
              for (int d = 0; d < 3; ++d) {
                float l;
                const float h = affine_ff(x[d], f, fl, tb->Kh[d], tb->Kl[d], &l);
                v[d] = (double)h + (double)l;
                lo[d] = 0;
              }
              v[3] = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
              lo[3] = 0;
            });
            if (tid == 0) record_conservation(a, k, N, Pi, tb->UA, tb->TA, r3);
          }
          for (int s = tid; s < N; s += kHugeThreads) {
            float l;
            float h = affine_ff(svx[s], f, fl, tb->Kh[0], tb->Kl[0], &l);
            svx[s] = h + l;
            h = affine_ff(svy[s], f, fl, tb->Kh[1], tb->Kl[1], &l);
            svy[s] = h + l;
            h = affine_ff(svz[s], f, fl, tb->Kh[2], tb->Kl[2], &l);
            svz[s] = h + l;
          }
        }
        __syncthreads();
      }
    }
    // ---- 8. Step 5 sums
    if (sample) {
      if (!bsq_ok) {
        block_sums<Acc, 3>(tb, N, bsq, [&](int s, auto* v, auto* lo) {
          const T x0 = svx[s], x1 = svy[s], x2 = svz[s];
          v[0] = x0 * x0;
          v[1] = x1 * x1;
          v[2] = x2 * x2;
          lo[0] = lo[1] = lo[2] = 0;
        });
      }
      if (tid == 0) {
        double* S = a.samp;
        const int64_t NC = a.NC;
        S[0 * NC + k] += (double)N;
        S[1 * NC + k] += (double)r1[0];
        S[2 * NC + k] += (double)r1[1];
        S[3 * NC + k] += (double)r1[2];
        S[4 * NC + k] += (double)bsq[0];
        S[5 * NC + k] += (double)bsq[1];
        S[6 * NC + k] += (double)bsq[2];
        S[7 * NC + k] += tb->ratio;
      }
    }
    if (tid == 0 && a.rec) {
      const int64_t NC = a.NC;
      a.rec[0 * NC + k] = tb->ncol;
      a.rec[1 * NC + k] = tb->nacc;
      a.rec[2 * NC + k] = tb->nres;
      a.rec[3 * NC + k] = tb->nar;
    }
    // ---- 9. the post-collision velocities, for the free flight
    if (N <= huge_smem_cap<T>())
      for (int s = tid; s < N; s += kHugeThreads) {
        ((T*)a.Bvel[0])[p0 + s] = svx[s];
        ((T*)a.Bvel[1])[p0 + s] = svy[s];
        ((T*)a.Bvel[2])[p0 + s] = svz[s];
      }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Free flight of the next interval (Step 2), new key and histogram: one
// thread per slot of the current cell order, kFlightPer slots per thread
// (strided by the block) whose loads are in flight together.  Its inputs are
// the source index and the post-collision velocity of the slot (coalesced)
// and the source's position (runs of neighbouring indices).  The slot's cell
// -- for the instance, the wall draws' counters and the O-grid's walk -- is
// the source's key of the last step.
// Bound by memory latency: 36 B per particle in 2-D FP32, 64 us for 6.6 M
// (3.7 TB/s); sphere, 30 M, 44 B: 315 us (4.2 TB/s); O-grid, 3.6 M: 66 us;
// FP64, 1.6 M: 75 us (206 without flight_clear).  Inside the collision kernel,
// at its 12 warps per SM, the flight was 29 % of the cylinder's, 38 % of the
// sphere's and 60 % of the O-grid's collision time (steps 0.353 -> 0.337,
// 1.92 -> 1.70, 0.31 -> 0.229 ms).  Two slots per thread and 4 blocks per SM
// measured best (1 x 6 blocks, 2 x 5, 4 x 3, 4 x 4: 0 to 5 % slower).
// ---------------------------------------------------------------------------
constexpr int kFlightThreads = 256;
template <class T>
constexpr int kFlightPer = sizeof(T) == 4 ? 2 : 1;

template <class T, int DIM, bool ONE, bool MESH>
__global__ void __launch_bounds__(kFlightThreads, sizeof(T) == 4 ? 4 : 3) k_flight(StepArgs a) {
  constexpr int R = kFlightPer<T>;
  const int64_t M = (int64_t)a.start[a.NC];
  const uint32_t step = *a.step;
  constexpr int64_t tile = (int64_t)kFlightThreads * R;
  const T dt0 = ONE ? (T)a.dt_cur[0] : (T)0;
  for (int64_t b0 = (int64_t)blockIdx.x * tile; b0 < M; b0 += (int64_t)gridDim.x * tile) {
    uint32_t og[R], cg[R];
    T xg[R][3], vg[R][3];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int64_t s = b0 + (int64_t)j * kFlightThreads + threadIdx.x;
      og[j] = s < M ? a.perm[s] : kSentinel;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        xg[j][d] = 0;
        vg[j][d] = s < M ? ((const T*)a.Bvel[d])[s] : (T)0;
      }
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      cg[j] = 0;
      if (og[j] != kSentinel) {
#pragma unroll
        for (int d = 0; d < DIM; ++d) xg[j][d] = ((const T*)a.Apos[d])[og[j]];
        if (MESH || !ONE) cg[j] = a.key_in[og[j]];
      }
    }
#pragma unroll 1
    for (int j = 0; j < R; ++j) {
      const int64_t s = b0 + (int64_t)j * kFlightThreads + threadIdx.x;
      uint32_t key = kSentinel;
      if (s < M) {
        T* x = xg[0];
        T* v = vg[0];
        const uint32_t inst = ONE ? 0u : a.cell_inst[cg[0]];
        const InstParams& P = inst_params<ONE>(a, inst);
        const T dt = ONE ? dt0 : (T)a.dt_cur[inst];
        bool hit = false;  // the velocity changed (a wall event)
        if constexpr (MESH) {
          const int64_t k0 = (int64_t)cg[0] - P.cell_off;
          int64_t kl = k0;
          const bool gone = mesh_walk<T>(P, (const T*)a.mface, a.surf, kl, x, v, dt, step, kPurpWall, (uint32_t)k0,
                                         (uint32_t)(s - a.start[cg[0]]), 0u, a.err, false);
          hit = true;
          if (!gone) key = (uint32_t)(P.cell_off + kl);
        } else {
          bool gone = false, clear = false;
          if constexpr (sizeof(T) == 8) {
            clear = flight_clear<DIM>(P, x, v, dt);
            if (clear) {
#pragma unroll
              for (int d = 0; d < DIM; ++d) x[d] += v[d] * dt;
              key = (uint32_t)P.cell_off + cell_of_clear<DIM>(P, x);
            }
          }
          if (!clear) {
            if (!flight_fast<T, DIM>(P, x, v, dt)) {
              const uint32_t c = ONE ? a.key_in[og[0]] : cg[0];
              gone = move_particle<T, DIM>(P, a.surf, x, v, dt, step, kPurpWall, (uint32_t)(c - P.cell_off),
                                           (uint32_t)(s - a.start[c]), 0u, a.err);
              hit = true;
            }
            if (!gone) key = (uint32_t)P.cell_off + cell_of<T, DIM>(P, x);
          }
        }
#pragma unroll
        for (int d = 0; d < DIM; ++d) ((T*)a.Bpos[d])[s] = x[d];
        if (hit) {
#pragma unroll
          for (int d = 0; d < 3; ++d) ((T*)a.Bvel[d])[s] = v[d];
        }
        a.key[s] = key;
      }
      warp_count(key, a.count);
#pragma unroll
      for (int i = 0; i + 1 < R; ++i) {
        og[i] = og[i + 1];
        cg[i] = cg[i + 1];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          xg[i][d] = xg[i + 1][d];
          vg[i][d] = vg[i + 1][d];
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Reservoir injection (ghost cells outside inflow faces), two passes:
// pass 0 counts survivors per ghost cell, pass 1 writes them at
// Mcur + goff[g] in (ghost cell, particle) order.
// ---------------------------------------------------------------------------
template <class T, int DIM>
__global__ void k_inject(InjectArgs a, int pass) {
  // one warp per reservoir cell; lanes take its particles m = lane, lane+32,
  // ...; survivors keep the (cell, m) order through ballot prefix counts
  const int lane = threadIdx.x & 31;
  const int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (g >= a.n_ghost) return;
  const GhostCell G = a.ghosts[g];
  const InstParams& P = a.P[G.inst];
  const uint32_t step = *a.step;
  const double dtd = a.dt_cur[G.inst];
  const T dt = (T)dtd;
  const int ax = G.face / 2, side = G.face % 2;
  const Geo<T>& GE = geo<T>(P);
  const T face = side ? GE.hi[ax] : GE.lo[ax];
  const uint32_t sb = (uint32_t)G.face * 16u;
  Uni<T> rc(step, G.gc, kSentinel, (kPurpInj << 24) | sb, P.key0, P.key1);
  const int64_t ng = (int64_t)floor(G.lam + (double)rc.get(0));
  uint32_t nsurv = 0;
  const int64_t base = pass == 1 ? (int64_t)*a.Mcur + (int64_t)a.goff[g] : 0;
  T* Bx[3] = {(T*)a.Bpos[0], (T*)a.Bpos[1], (T*)a.Bpos[2]};
  T* Bv[3] = {(T*)a.Bvel[0], (T*)a.Bvel[1], (T*)a.Bvel[2]};
  const T s2RT = (T)G.s2RT;
  T blo[3], bhi[3], u0[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    blo[d] = (T)G.blo[d];
    bhi[d] = (T)G.bhi[d];
    u0[d] = (T)G.u[d];
  }
  for (int64_t m0 = 0; m0 < ng; m0 += 32) {
    const int64_t m = m0 + lane;
    bool ok = m < ng;
    T x[3] = {0, 0, 0}, v[3] = {0, 0, 0};
    if (ok) {
      Uni<T> r(step, G.gc, (uint32_t)m, (kPurpInj << 24) | sb, P.key0, P.key1);
#pragma unroll
      for (int d = 0; d < DIM; ++d) x[d] = blo[d] + r.get(d) * (bhi[d] - blo[d]);
      const T R1 = r.get(3), R2 = r.get(4), R3 = r.get(5), R4 = r.get(6);
      const T r2 = tsqrt(-tlog(R2)), r4 = tsqrt(-tlog(R4));
      T sn3, cs3;
      sincos2pi(R3, &sn3, &cs3);
      v[0] = u0[0] + s2RT * cos2pi(R1) * r2;
      v[1] = u0[1] + s2RT * cs3 * r4;
      v[2] = u0[2] + s2RT * sn3 * r4;
      const T vn = v[ax];
      ok = side == 0 ? (vn > (T)0) : (vn < (T)0);
      T te = 0;
      if (ok) {
        te = (face - x[ax]) / vn;
        ok = te < dt;
      }
      if (ok) {
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
          if (d == ax || !ok) continue;
          T y = x[d] + v[d] * te;
          if (y < GE.lo[d]) {
            if (P.face_bc[2 * d] != 0) { ok = false; continue; }
            y = (T)2.0 * GE.lo[d] - y;
            v[d] = -v[d];
          } else if (y > GE.hi[d]) {
            if (P.face_bc[2 * d + 1] != 0) { ok = false; continue; }
            y = (T)2.0 * GE.hi[d] - y;
            v[d] = -v[d];
          }
          if (y < GE.lo[d] || y > GE.hi[d]) { ok = false; continue; }
          x[d] = y;
        }
      }
      if (ok) {
        x[ax] = face;
        if ((P.face_win >> G.face) & 1) ok = face_open<T, DIM>(GE, G.face, x);
      }
      if (ok) {
        ok = !move_particle<T, DIM>(P, a.surf, x, v, dt - te, step, kPurpInjWall, G.gc, (uint32_t)m,
                                    (uint32_t)G.face << 16, a.err);
      }
    }
    const unsigned sv = __ballot_sync(kFull, ok);
    if (pass == 1 && ok) {
      const int64_t idx = base + nsurv + __popc(sv & ((1u << lane) - 1u));
      if (idx >= a.cap) {
        atomicAdd(&a.err[kErrCapacity], 1ull);
      } else {
        const uint32_t key = (uint32_t)P.cell_off + cell_of<T, DIM>(P, x);
#pragma unroll
        for (int d = 0; d < DIM; ++d) Bx[d][idx] = x[d];
        Bv[0][idx] = v[0];
        Bv[1][idx] = v[1];
        Bv[2][idx] = v[2];
        a.key[idx] = key;
        atomicAdd(&a.count[key], 1u);
      }
    }
    nsurv += __popc(sv);
  }
  if (pass == 0 && lane == 0) a.gcount[g] = nsurv;
}

// Reservoir injection through the outer polygon of an O-grid (face 1 an
// inflow boundary), two passes as k_inject: the reservoir quadrilateral of
// ghost cell g is ring mlay beyond the outer polygon, sector msec; its
// particles are uniform in it (triangle A B C or A C D chosen by area),
// Maxwellian at the face state; one whose straight path enters the outer
// polygon within the step through one of the mnl + 1 outer edges on either
// side of its sector enters at the first crossing and walks the rest of the
// step from the boundary cell.
template <class T>
__global__ void k_inject_mesh(InjectArgs a, int pass) {
  const int lane = threadIdx.x & 31;
  const int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (g >= a.n_ghost) return;
  const GhostCell G = a.ghosts[g];
  const InstParams& P = a.P[G.inst];
  const uint32_t step = *a.step;
  const T dt = (T)a.dt_cur[G.inst];
  const int nr = P.n[0], nt = P.n[1], w = P.mnl + 1;
  const T* mface = (const T*)a.mface;
  const T* nd = (const T*)a.mnode + 2 * P.mnode_off;
  const int i0 = nr + G.mlay, j = G.msec, j1 = (j + 1) % nt;
  const T* A = nd + 2 * ((int64_t)i0 * nt + j);
  const T* B = nd + 2 * ((int64_t)(i0 + 1) * nt + j);
  const T* C = nd + 2 * ((int64_t)(i0 + 1) * nt + j1);
  const T* D = nd + 2 * ((int64_t)i0 * nt + j1);
  const double a1 = G.a1, a12 = G.a1 + G.a2;
  const uint32_t sb = (uint32_t)G.face * 16u;
  Uni<T> rc(step, G.gc, kSentinel, (kPurpInj << 24) | sb, P.key0, P.key1);
  const int64_t ng = (int64_t)floor(G.lam + (double)rc.get(0));
  uint32_t nsurv = 0;
  const int64_t base = pass == 1 ? (int64_t)*a.Mcur + (int64_t)a.goff[g] : 0;
  T* Bx[2] = {(T*)a.Bpos[0], (T*)a.Bpos[1]};
  T* Bv[3] = {(T*)a.Bvel[0], (T*)a.Bvel[1], (T*)a.Bvel[2]};
  const T s2RT = (T)G.s2RT;
  const T u0[3] = {(T)G.u[0], (T)G.u[1], (T)G.u[2]};
  for (int64_t m0 = 0; m0 < ng; m0 += 32) {
    const int64_t m = m0 + lane;
    bool ok = m < ng;
    T x[3] = {0, 0, 0}, v[3] = {0, 0, 0};
    int64_t kl = 0;
    if (ok) {
      Uni<T> r(step, G.gc, (uint32_t)m, (kPurpInj << 24) | sb, P.key0, P.key1);
      const T uu = r.get(0);
      T s = r.get(1), t = r.get(2);
      if (s + t > (T)1) {
        s = (T)1 - s;
        t = (T)1 - t;
      }
      const T* P1 = B;
      const T* P2 = C;
      if (!((double)uu * a12 < a1)) {
        P1 = C;
        P2 = D;
      }
      x[0] = A[0] + s * (P1[0] - A[0]) + t * (P2[0] - A[0]);
      x[1] = A[1] + s * (P1[1] - A[1]) + t * (P2[1] - A[1]);
      const T R1 = r.get(3), R2 = r.get(4), R3 = r.get(5), R4 = r.get(6);
      const T r2 = tsqrt(-tlog(R2)), r4 = tsqrt(-tlog(R4));
      T sn3, cs3;
      sincos2pi(R3, &sn3, &cs3);
      v[0] = u0[0] + s2RT * cos2pi(R1) * r2;
      v[1] = u0[1] + s2RT * cs3 * r4;
      v[2] = u0[2] + s2RT * sn3 * r4;
      // first crossing of an outer edge within the step
      T best = tinf<T>();
      int jb = -1;
      for (int o = -w; o <= w; ++o) {
        const int jj = ((j + o) % nt + nt) % nt;
        const T* f = mface + 12 * (P.cell_off + (nr - 1) + (int64_t)nr * jj) + 3;
        const T nvv = f[0] * v[0] + f[1] * v[1];
        if (!(nvv < (T)0)) continue;
        const T sx = f[0] * x[0] + f[1] * x[1];
        if (!(sx > f[2])) continue;
        const T te = (f[2] - sx) / nvv;
        if (!(te < dt) || !(te < best)) continue;
        const T* E0 = nd + 2 * ((int64_t)nr * nt + jj);
        const T* E1 = nd + 2 * ((int64_t)nr * nt + (jj + 1) % nt);
        const T ex = E1[0] - E0[0], ey = E1[1] - E0[1];
        const T xc = x[0] + v[0] * te, yc = x[1] + v[1] * te;
        const T u = ((xc - E0[0]) * ex + (yc - E0[1]) * ey) / (ex * ex + ey * ey);
        if (u < (T)0 || u > (T)1) continue;
        best = te;
        jb = jj;
      }
      ok = jb >= 0;
      if (ok) {
        x[0] += v[0] * best;
        x[1] += v[1] * best;
        kl = (nr - 1) + (int64_t)nr * jb;
        ok = !mesh_walk<T>(P, mface, a.surf, kl, x, v, dt - best, step, kPurpInjWall, G.gc, (uint32_t)m,
                           (uint32_t)G.face << 16, a.err, false);
      }
    }
    const unsigned sv = __ballot_sync(kFull, ok);
    if (pass == 1 && ok) {
      const int64_t idx = base + nsurv + __popc(sv & ((1u << lane) - 1u));
      if (idx >= a.cap) {
        atomicAdd(&a.err[kErrCapacity], 1ull);
      } else {
        const uint32_t key = (uint32_t)(P.cell_off + kl);
        Bx[0][idx] = x[0];
        Bx[1][idx] = x[1];
        Bv[0][idx] = v[0];
        Bv[1][idx] = v[1];
        Bv[2][idx] = v[2];
        a.key[idx] = key;
        atomicAdd(&a.count[key], 1u);
      }
    }
    nsurv += __popc(sv);
  }
  if (pass == 0 && lane == 0) a.gcount[g] = nsurv;
}

// Cell keys of uploaded particles on O-grid instances (point location by
// face crossing; outside the mesh: the sentinel), with the histogram.
template <class T>
__global__ void k_keys_mesh(const T* x0, const T* x1, int64_t M, const uint32_t* part_inst,
                            const InstParams* Ps, const T* mface, const T* mnode, const double* mrad,
                            uint32_t* key, uint32_t* count) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t k = kSentinel;
  if (i < M) {
    const InstParams& P = Ps[part_inst ? part_inst[i] : 0u];
    const T x[2] = {x0[i], x1[i]};
    const int64_t kl = mesh_locate<T>(P, mface, mnode, mrad, x);
    if (kl >= 0) k = (uint32_t)(P.cell_off + kl);
    key[i] = k;
  }
  warp_count(k, count);
}

// ---------------------------------------------------------------------------
// Observability / initialisation kernels
// ---------------------------------------------------------------------------
// Moments of the current state for cells [c0, c1), in the cells' current
// slot order, in two kernels.  k_moment_sums: kMomentLanes lanes per cell (a
// warp per dense cell of an FP64 state); lanes stride over the cell's slots, a
// butterfly combines them, and the first lane writes the cell's sums to
// sums[7][nc]: sum c (3), then sum |C|^2 and, when the fields are wanted (kQ),
// sum |C|^2 C (3) about
// the mean.  The sums use the
// collision kernel's accumulators (FP64 values in FP64 mode, FP32 terms
// carried without loss in FP32 mode, plain FP32 in the all-FP32 mode).
// With an FP32 state a sum is stored as its FP32 pair (s, e) in the 8-byte
// slot, so that this kernel issues no FP64 instruction: on GB300 one costs
// a whole warp ~67 cycles of a scheduler's FP64 unit even with one lane
// active, and a kernel with a few lanes per cell would spend most of its
// time there.  k_moment_cells: one thread per cell forms the FP64 values and
// scalars (U, n, T, q, tau, dt_c, the split ratio) from them on full warps,
// and writes the fields to out [12][nc] or, with out == nullptr, takes the
// minimum dt_c into dt_min (a warp minimum, then one atomic per warp).
// Lanes per cell: 16 with an FP32 state; 4 with an FP64 state, where the
// butterfly's additions hold the FP64 pipe as long as the terms' (2 M
// particles, 30 per cell: 221 -> 118 us with the heat flux), and 32 for its
// cells above kMomentDense particles, whose time is the gathers of one lane.
// Reads of an FP64 state with 16, 4 and these lanes: one cell of 200,000 21.1,
// 35.7 and 4.6 ms; 267 cells of 1500 240, 615 and 123 us; 2000 of 200 120, 134
// and 83 us; 5000 of 80 123, 87 and 88 us.  Four rounds of gathers are in
// flight (one: 20 to 60 % slower on dense cells; eight: 10 % slower on others).
template <class T>
constexpr int kMomentLanes = sizeof(T) == 8 ? 4 : 16;
constexpr int kMomentDense = 128;

// One cell of N particles from slot s0 on, by L neighbouring lanes of a warp
// (`lane` of L); the whole warp calls it (N = 0 where a group has no cell).
// store: write the sums to sums[..][i].
template <class T, class A, bool kQ, int L>
__device__ __forceinline__ void moment_cell(const StepArgs& a, uint32_t s0, int N, int lane, bool store, int64_t i,
                                            int64_t nc, double* sums) {
  using Acc = CellAcc<T, A>;
  constexpr bool kMixed = mixed_prec<T, A>();
  constexpr bool kPair = sizeof(T) == 4;
  const T* Av0 = (const T*)a.Avel[0];
  const T* Av1 = (const T*)a.Avel[1];
  const T* Av2 = (const T*)a.Avel[2];
  // (the FP32 state's Delta t pass is faster as the compiler unrolls it: an
  // upload of 3.2 M particles 437 us, 456 with four rounds)
  const auto each_slot = [&](auto f) {
    if constexpr (kQ || sizeof(T) == 8) {
#pragma unroll 4
      for (int s = lane; s < N; s += L) f(s);
    } else {
      for (int s = lane; s < N; s += L) f(s);
    }
  };
  Acc sx[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) sx[d].init();
  each_slot([&](int s) {
    const uint32_t o = a.perm[s0 + s];
    sx[0].add1(Av0[o]);
    sx[1].add1(Av1[o]);
    sx[2].add1(Av2[o]);
  });
#pragma unroll
  for (int m = L / 2; m > 0; m >>= 1)
#pragma unroll
    for (int d = 0; d < 3; ++d) sx[d].combine(sx[d].shfl_xor(m));
  // the shift of the central sums: the mean (FP32 state: the FP32 pair
  // U_h + U_l of the exact sum, formed without FP64 work)
  T Uh[3] = {0, 0, 0}, Ul[3] = {0, 0, 0};
  if (N > 0) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if constexpr (kMixed) {
        const float fN = (float)N, rN = 1.0f / fN;
        Uh[d] = sx[d].s * rN;
        Ul[d] = (fmaf(-Uh[d], fN, sx[d].s) + sx[d].e) * rN;
      } else if constexpr (kPair) {
        Uh[d] = sx[d].get() * (1.0f / (float)N);
      } else {
        Uh[d] = (T)((double)sx[d].get() / N);
      }
    }
  }
  // sum |C|^2, and with kQ sum |C|^2 C (the heat flux; not needed for dt_c)
  constexpr int K2 = kQ ? 4 : 1;
  Acc r[K2];
#pragma unroll
  for (int d = 0; d < K2; ++d) r[d].init();
  if (N >= 2) {
    each_slot([&](int s) {
      const uint32_t o = a.perm[s0 + s];
      T C0 = Av0[o] - Uh[0], C1 = Av1[o] - Uh[1], C2 = Av2[o] - Uh[2];
      if constexpr (kMixed) {
        C0 -= Ul[0];
        C1 -= Ul[1];
        C2 -= Ul[2];
      }
      const T c2 = C0 * C0 + C1 * C1 + C2 * C2;
      r[0].add1(c2);
      if constexpr (kQ) {
        r[1].add1(c2 * C0);
        r[2].add1(c2 * C1);
        r[3].add1(c2 * C2);
      }
    });
  }
#pragma unroll
  for (int m = L / 2; m > 0; m >>= 1)
#pragma unroll
    for (int d = 0; d < K2; ++d) r[d].combine(r[d].shfl_xor(m));
  if (lane == 0 && store) {
    if constexpr (kPair) {
      float2* sp2 = (float2*)sums;
#pragma unroll
      for (int d = 0; d < 3; ++d) sp2[d * nc + i] = acc_pair(sx[d]);
#pragma unroll
      for (int d = 0; d < K2; ++d) sp2[(3 + d) * nc + i] = acc_pair(r[d]);
    } else {
#pragma unroll
      for (int d = 0; d < 3; ++d) sums[d * nc + i] = (double)sx[d].get();
#pragma unroll
      for (int d = 0; d < K2; ++d) sums[(3 + d) * nc + i] = (double)r[d].get();
    }
  }
}

// A warp takes G cells at a time: one per group of L lanes (W), or fewer
// where dense cells (FP64 state: above kMomentDense on average) are too few
// to give every warp of the launch W of them.  Which cells share a warp does
// not change how a cell is summed.
template <class T, class A, bool kQ>
__global__ void k_moment_sums(StepArgs a, int64_t c0, int64_t c1, double* sums) {
  constexpr int L = kMomentLanes<T>, W = 32 / L;
  constexpr bool kDense = sizeof(T) == 8;
  const int64_t nc = c1 - c0, nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  int G = W;
  if (kDense && (int64_t)(a.start[c1] - a.start[c0]) > kMomentDense * nc) {
    const int64_t g = (nc + nw - 1) / nw;
    if (g < W) G = (int)g;
  }
  const int wl = threadIdx.x & 31, lane = wl & (L - 1), grp = wl / L;
  // (the same trip count for all lanes of a warp: the shuffles need them)
  for (int64_t kb = c0 + ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * G; kb < c1; kb += nw * G) {
    const int64_t k = kb + grp;
    const bool valid = grp < G && k < c1;
    const uint32_t s0 = valid ? a.start[k] : 0u;
    const int N = valid ? (int)(a.start[k + 1] - s0) : 0;
    const bool dense = kDense && N > kMomentDense;
    moment_cell<T, A, kQ, L>(a, s0, dense ? 0 : N, lane, valid && !dense, k - c0, nc, sums);
    if constexpr (kDense) {
      for (unsigned todo = __ballot_sync(kFull, dense && lane == 0); todo; todo &= todo - 1) {
        const int src = __ffs((int)todo) - 1;
        moment_cell<T, A, kQ, 32>(a, __shfl_sync(kFull, s0, src), __shfl_sync(kFull, N, src), wl, true,
                                  kb + src / L - c0, nc, sums);
      }
    }
  }
}

template <bool kPair>
__device__ __forceinline__ double moment_sum(const double* sums, int64_t idx) {
  if constexpr (kPair) {
    const float2 p = ((const float2*)sums)[idx];
    return (double)p.x + (double)p.y;
  } else {
    return sums[idx];
  }
}

// FP64 state (kPair false): the oracle's arithmetic, operation for operation,
// on sums whose order is k_moment_sums' (so Delta t and fields agree with the
// oracle's to the rounding of the sums).  FP32 state: the same quantities with
// the divisions taken as products of reciprocals (1/k from the table, 1/V, 1/L)
// and the viscosity power as tau = tau_k exp((omega - 1) ln T) / n: a few ulps
// from the quotient forms, at a third of the FP64 instructions.
template <bool kPair>
__global__ void k_moment_cells(StepArgs a, int64_t c0, int64_t c1, const double* sums, double* out) {
  const int64_t nc = c1 - c0;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = i < nc;
  const int64_t k = c0 + (valid ? i : 0);
  const int N = valid ? (int)(a.start[k + 1] - a.start[k]) : 0;
  const uint32_t inst = a.cell_inst[k];
  const InstParams& P = a.P[inst];
  CellMoments m;
  m.U[0] = m.U[1] = m.U[2] = 0;
  m.n = 0;
  m.T = 0;
  m.q[0] = m.q[1] = m.q[2] = 0;
  m.tau = __longlong_as_double(0x7FF0000000000000ll);
  m.dtc = m.tau;
  if constexpr (kPair) {
    const double iL = a.iLc ? a.iLc[k] : P.inv_Lmin;
    const auto rcp = [&](int j) { return j <= kHugeCell ? a.rcp[j] : 1.0 / (double)j; };
    if (N > 0) {
      const double rN = rcp(N);
#pragma unroll
      for (int d = 0; d < 3; ++d) m.U[d] = moment_sum<true>(sums, d * nc + i) * rN;
      m.n = (double)N * P.Fn * a.ivol[k];
    }
    if (N >= 2) {
      m.T = moment_sum<true>(sums, 3 * nc + i) * P.inv3R * rcp(N - 1);
      if (N >= 3 && out) {
        const double f = 0.5 * (double)N * rcp(N - 1) * rcp(N - 2);
#pragma unroll
        for (int d = 0; d < 3; ++d) m.q[d] = f * moment_sum<true>(sums, (4 + d) * nc + i);
      }
      const double umag = sqrt(m.U[0] * m.U[0] + m.U[1] * m.U[1] + m.U[2] * m.U[2]);
      double idtc = umag * iL;  // 1 / dt_c
      if (m.T > 0) {
        idtc = (umag + sqrt(P.gamma * P.R * m.T)) * iL;
        if (out) m.tau = P.tau_k * exp((P.omega - 1.0) * log(m.T)) / m.n;
      }
      if (idtc > 0) m.dtc = 1.0 / idtc;
      if (out) {
        double ratio = 1.0;
        if (P.mode == 2) ratio = 0.0;
        else if (P.mode != 1 && m.T > 0 && m.dtc > m.tau) ratio = m.tau * idtc;
        out[11 * nc + i] = ratio;
      }
    } else if (out && valid) {
      out[11 * nc + i] = P.mode == 2 ? 0.0 : 1.0;
    }
  } else {
    const double Lk = a.Lc ? a.Lc[k] : P.Lmin;
    if (N > 0) {
#pragma unroll
      for (int d = 0; d < 3; ++d) m.U[d] = moment_sum<false>(sums, d * nc + i) / N;
    }
    m.n = N > 0 ? (double)N * P.Fn / a.vol[k] : 0.0;
    if (N >= 2) {
      m.T = moment_sum<false>(sums, 3 * nc + i) / (3.0 * P.R * (double)(N - 1));
      if (N >= 3 && out) {
        const double f = 0.5 * (double)N / ((double)(N - 1) * (double)(N - 2));
#pragma unroll
        for (int d = 0; d < 3; ++d) m.q[d] = f * moment_sum<false>(sums, (4 + d) * nc + i);
      }
      const double umag = sqrt(m.U[0] * m.U[0] + m.U[1] * m.U[1] + m.U[2] * m.U[2]);
      if (m.T > 0) {
        if (out) {  // tau is an output field only (dt_c does not need it)
          const double p = m.n * P.m * P.R * m.T;
          m.tau = P.mu_ref * pow(m.T / P.T_ref, P.omega) / p;
        }
        m.dtc = Lk / (umag + sqrt(P.gamma * P.R * m.T));
      } else if (umag > 0) {
        m.dtc = Lk / umag;
      }
    }
    if (out && valid) out[11 * nc + i] = dsmc_ratio(P, N, m);
  }
  if (out) {
    if (valid) {
      out[0 * nc + i] = (double)N;
      out[1 * nc + i] = m.n;
      out[2 * nc + i] = m.U[0];
      out[3 * nc + i] = m.U[1];
      out[4 * nc + i] = m.U[2];
      out[5 * nc + i] = m.T;
      out[6 * nc + i] = m.q[0];
      out[7 * nc + i] = m.q[1];
      out[8 * nc + i] = m.q[2];
      out[9 * nc + i] = m.tau;
      out[10 * nc + i] = m.dtc;
    }
  } else {
    // minimum dt_c per instance: a warp minimum where the warp's cells share
    // an instance (dt_c > 0, so the bit patterns order as the values), then
    // one atomic per warp
    unsigned long long v = (N >= 2 && valid) ? (unsigned long long)__double_as_longlong(m.dtc)
                                             : 0x7FF0000000000000ull;
    const uint32_t inst0 = __shfl_sync(kFull, inst, 0);
    if (__all_sync(kFull, !valid || inst == inst0)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(kFull, v, o);
        v = w < v ? w : v;
      }
      if ((threadIdx.x & 31) == 0 && v < 0x7FF0000000000000ull) atomicMin(&a.dt_min[inst0], v);
    } else if (v < 0x7FF0000000000000ull) {
      atomicMin(&a.dt_min[inst], v);
    }
  }
}

template <class T, int DIM>
__global__ void k_keys(const T* x0, const T* x1, const T* x2, int64_t M, const uint32_t* part_inst,
                       const InstParams* Ps, uint32_t* key, uint32_t* count) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t k = kSentinel;
  if (i < M) {
    const InstParams& P = Ps[part_inst ? part_inst[i] : 0u];
    T x[3] = {x0[i], DIM > 1 ? x1[i] : (T)0, DIM > 2 ? x2[i] : (T)0};
    if constexpr (sizeof(T) == 8) k = (uint32_t)P.cell_off + cell_of_clear<DIM>(P, x);
    else k = (uint32_t)P.cell_off + cell_of<T, DIM>(P, x);
    key[i] = k;
  }
  warp_count(k, count);  // one atomic per cell per warp (input sorted by cell: few)
}

// Host-provided FP64 particles of one instance -> state buffers at offset off.
template <class T, class S>
__global__ void k_stage_in(const S* pos, const S* vel, int dim, int64_t n, T* p0, T* p1, T* p2,
                           T* v0, T* v1, T* v2, int64_t off, uint32_t* part_inst, uint32_t inst) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  T* P3[3] = {p0, p1, p2};
  for (int d = 0; d < dim; ++d) P3[d][off + j] = (T)pos[d * n + j];
  v0[off + j] = (T)vel[j];
  v1[off + j] = (T)vel[n + j];
  v2[off + j] = (T)vel[2 * n + j];
  if (part_inst) part_inst[off + j] = inst;
}

template <class T>
__global__ void k_gather(const T* p0, const T* p1, const T* p2, const T* v0, const T* v1, const T* v2,
                         int dim, const uint32_t* perm, int64_t s0, int64_t n, double* out_pos,
                         double* out_vel) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const uint32_t o = perm[s0 + j];
  const T* P3[3] = {p0, p1, p2};
  for (int d = 0; d < dim; ++d) out_pos[d * n + j] = (double)P3[d][o];
  out_vel[0 * n + j] = (double)v0[o];
  out_vel[1 * n + j] = (double)v1[o];
  out_vel[2 * n + j] = (double)v2[o];
}

}  // namespace sp
