// Shared device helpers: complex float64 arithmetic on double2, block
// reductions, and a bounded grid-wide barrier for cooperative launches.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

typedef double2 cplx;

#define HD __host__ __device__ __forceinline__
#define DV __device__ __forceinline__

HD cplx mk(double re, double im) { return make_double2(re, im); }
HD cplx cadd(cplx a, cplx b) { return mk(a.x + b.x, a.y + b.y); }
HD cplx csub(cplx a, cplx b) { return mk(a.x - b.x, a.y - b.y); }
HD cplx cscale(cplx a, double s) { return mk(a.x * s, a.y * s); }
HD cplx cconj(cplx a) { return mk(a.x, -a.y); }
HD cplx cmul(cplx a, cplx b) { return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
// conj(a) * b
HD cplx cmulc(cplx a, cplx b) { return mk(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x); }
HD double cabs2(cplx a) { return a.x * a.x + a.y * a.y; }
// a * b rounded by itself whatever stands around it: cmul's second products may
// be fused with a sum that takes its result.
DV cplx cmul_rounded(cplx a, cplx b) {
  return mk(fma(a.x, b.x, -__dmul_rn(a.y, b.y)), fma(a.x, b.y, __dmul_rn(a.y, b.x)));
}
// acc + a * b
DV cplx cfma(cplx a, cplx b, cplx acc) {
  return mk(fma(a.x, b.x, fma(-a.y, b.y, acc.x)), fma(a.x, b.y, fma(a.y, b.x, acc.y)));
}
// acc + conj(a) * b
DV cplx cfmac(cplx a, cplx b, cplx acc) {
  return mk(fma(a.x, b.x, fma(a.y, b.y, acc.x)), fma(a.x, b.y, fma(-a.y, b.x, acc.y)));
}
HD cplx cinv(cplx a) {
  double s = 1.0 / (a.x * a.x + a.y * a.y);
  return mk(a.x * s, -a.y * s);
}

// Comparisons on the bits: one on the values is an FP64 instruction, 64 cycles
// of a warp.  x == 0; x < 0; |a| < |b| (the last two not for NaN).
DV bool d_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
DV bool d_neg(double x) { return __double_as_longlong(x) < 0 && !d_zero(x); }
DV bool d_mag_less(double a, double b) {
  return (unsigned long long)__double_as_longlong(a) << 1 < (unsigned long long)__double_as_longlong(b) << 1;
}

// Reciprocal to FP64 rounding level: the hardware's 20-bit seed y and one step of
// Householder's iteration of third order for 1 / y - x, y (1 + e + e^2) with
// e = 1 - x y (error e^3): half a unit in the last place and a little.  About 230
// cycles of dependent operations against 640 measured for the IEEE division, on
// serial chains that wait for it.  |x| in [1e-290, 1e290].
DV double rcp_fast(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// 1 / sqrt(x), same range: Householder's third order for 1 / y^2 - x, the binomial
// series of (1 - e)^(-1/2) with e = 1 - x y^2 up to e^2: y (1 + e / 2 + 3 e^2 / 8)
// (error 5 e^3 / 16).  The product x y is rounded: one unit in the last place.
DV double rsqrt_fast(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}
// Householder reflector H = I - tau v v^H, v = [1; x scale], with H^H [alpha; x]
// = [beta; 0], beta real (zlarfg conventions), from alpha and |x|^2, by a whole
// warp whose lanes 0 to 3 (at least) hold the inputs; out[0..2] <- tau, scale,
// beta.  One reciprocal root and one reciprocal, issued after one another's
// inputs are known, instead of a root and two divisions; the IEEE forms where a
// square leaves the range of the fast ones.  Every FP64 instruction of a warp
// takes 64 cycles, so the four last products are one, a lane each.
DV void house_fast(cplx al, double s2, cplx* out) {
  const int lane = threadIdx.x & 31;
  const double a2 = fma(al.x, al.x, fma(al.y, al.y, s2));
  // in: a2 between 2^-928 and 2^929
  const int hi = __double2hiint(a2);
  const bool none = d_zero(s2) && d_zero(al.y), neg = d_neg(al.x), in = hi > 0x05f00000 && hi < 0x7a000000;
  const double rs = in ? rsqrt_fast(a2) : 1.0 / sqrt(a2);
  const double an = in ? a2 * rs : sqrt(a2);
  const double b = neg ? an : -an, ib = neg ? rs : -rs;
  const double dr = al.x - b, den = fma(dr, dr, al.y * al.y);
  const double id2 = in ? rcp_fast(den) : 1.0 / den;
  const double r = ((lane & 1) ? -al.y : (lane & 2) ? dr : -dr) * ((lane & 2) ? id2 : ib);
  if (lane < 4) reinterpret_cast<double*>(out)[lane] = none ? 0.0 : r;
  if (lane == 0) out[2] = mk(none ? al.x : b, 0.0);
}

// The same with IEEE root and divisions, by a whole warp whose lanes 0 and 1 (at
// least) hold the inputs; the results are theirs.  The two divisions (about 640
// cycles each, and one after the other in one lane's code) run side by side in
// the two lanes.
DV void house_warp(cplx al, double s2, cplx* tau, cplx* scale, double* beta) {
  const double an = sqrt(al.x * al.x + al.y * al.y + s2);
  const double b = d_neg(al.x) ? an : -an;
  const double dr = al.x - b, den = dr * dr + al.y * al.y;
  const double r = 1.0 / ((threadIdx.x & 1) ? den : b);
  const double ib = __shfl_sync(0xffffffffu, r, 0), id2 = __shfl_sync(0xffffffffu, r, 1);
  const bool none = d_zero(s2) && d_zero(al.y);
  *tau = none ? mk(0, 0) : mk((b - al.x) * ib, -al.y * ib);
  *scale = none ? mk(0, 0) : mk(dr * id2, -al.y * id2);
  *beta = none ? al.x : b;
}

// Single-precision complex (mixed-precision trailing updates and products).
typedef float2 cplxf;
HD cplxf mkf(float re, float im) { return make_float2(re, im); }
HD cplxf tof(cplx a) { return make_float2((float)a.x, (float)a.y); }
HD cplx tod(cplxf a) { return make_double2((double)a.x, (double)a.y); }
// acc + a * b
DV cplxf cfmaf(cplxf a, cplxf b, cplxf acc) {
  return mkf(fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y)));
}
// acc + conj(a) * b
DV cplxf cfmacf(cplxf a, cplxf b, cplxf acc) {
  return mkf(fmaf(a.x, b.x, fmaf(a.y, b.y, acc.x)), fmaf(a.x, b.y, fmaf(-a.y, b.x, acc.y)));
}

// Double-float arithmetic: a value is hi + lo with hi, lo in FP32 (about 48
// significant bits).  Used by the mixed-precision trailing updates: the FP32
// pipe is 64 times the FP64 pipe on this GPU, so ~13 FP32 operations per
// real multiply-add still beat one FP64 FMA by a wide margin.
struct df2 {   // complex double-float: (re.hi, im.hi, re.lo, im.lo)
  float rh, ih, rl, il;
};
HD df2 df_zero() { return df2{0.f, 0.f, 0.f, 0.f}; }
HD df2 df_from(cplx a) {
  const float rh = (float)a.x, ih = (float)a.y;
  return df2{rh, ih, (float)(a.x - (double)rh), (float)(a.y - (double)ih)};
}
HD cplx df_to(df2 a) { return make_double2((double)a.rh + (double)a.rl, (double)a.ih + (double)a.il); }

// Conversions between FP64 and double-float by integer arithmetic on the
// IEEE bit patterns (on this GPU an FP64 conversion, scaling or addition
// occupies the narrow FP64 pipe; these use the integer and FP32 pipes).
// (double)f * 2^E (negated if neg) from the bit pattern of f: sign, exponent
// rebiased from 127 to 1023 plus E, significand shifted into place.  Zero
// and FP32 subnormals give 0 (a subnormal low part sits below 2^-149 of its
// high part); an exponent outside the double range saturates to 0 or inf.
DV double f2d_scaled(float f, int E, int neg) {
  const unsigned int u = __float_as_uint(f);
  const unsigned int e8 = (u >> 23) & 0xFFu;
  if (e8 == 0) return 0.0;
  const long long sgn = (long long)((u >> 31) ^ (unsigned)neg) << 63;
  const int e11 = (int)e8 - 127 + 1023 + E;
  if (e11 <= 0) return 0.0;
  if (e11 >= 2047) return __longlong_as_double(sgn | (0x7FFll << 52));
  return __longlong_as_double(sgn | ((long long)e11 << 52) | ((long long)(u & 0x7FFFFFu) << 29));
}

// 2^d as a float for -126 <= d <= 127 (exact), 0 below: multiplying by it
// scales exactly while the result stays normal.
DV float pow2f(int d) { return d >= -126 ? __int_as_float((127 + d) << 23) : 0.f; }

// x 2^-E as a double-float pair (hi, lo): hi is the 53-bit significand
// rounded to 24 bits, lo the remainder (|lo| <= ulp(hi) / 2, itself rounded
// to 24 bits).  Values whose hi part would fall below the FP32 normal range
// (|x 2^-E| < 2^-126), zeros and FP64 subnormals give (0, 0).
DV void df_split_scaled(double x, int E, float& hi, float& lo) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7FF);
  const int e = ex - 1023 - E;  // |x| 2^-E = M 2^(e - 52), M in [2^52, 2^53)
  if (ex == 0 || e < -126) {
    hi = 0.f;
    lo = 0.f;
    return;
  }
  const long long M = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  long long Mh = (M + (1ll << 28)) >> 29;  // 24 bits, or 2^24 after a carry
  const int r = (int)(M - (Mh << 29));     // |r| <= 2^28
  int eh = e;
  if (Mh == (1ll << 24)) {
    Mh >>= 1;
    eh += 1;
  }
  const unsigned int sgn = (unsigned int)((unsigned long long)b >> 63) << 31;
  if (eh > 127) {  // beyond the FP32 range
    hi = __uint_as_float(sgn | 0x7F800000u);
    lo = 0.f;
    return;
  }
  hi = __uint_as_float(sgn | ((unsigned int)(eh + 127) << 23) | ((unsigned int)Mh & 0x7FFFFFu));
  // r 2^(e - 52) in two exact steps (e - 52 can be below -126)
  const int s1 = (e - 52) / 2;
  const float l = (float)r * pow2f(s1) * pow2f(e - 52 - s1);
  lo = sgn ? -l : l;
}
DV df2 df_from_scaled(cplx a, int E) {
  df2 r;
  df_split_scaled(a.x, E, r.rh, r.rl);
  df_split_scaled(a.y, E, r.ih, r.il);
  return r;
}
// (hi + lo) 2^E in FP64: the two parts converted exactly from their bits,
// one FP64 addition.
DV cplx df_to_scaled(const df2& a, int E) {
  return make_double2(f2d_scaled(a.rh, E, 0) + f2d_scaled(a.rl, E, 0), f2d_scaled(a.ih, E, 0) + f2d_scaled(a.il, E, 0));
}
// (hi, lo) += a * b for double-float reals a = (ah, al), b = (bh, bl):
// exact product of the high parts (TwoProduct with an FMA), exact sum
// (TwoSum), the low-order cross terms added to lo.
DV void df_mac(float& hi, float& lo, float ah, float al, float bh, float bl) {
  const float p = ah * bh;
  const float pe = fmaf(ah, bh, -p);
  const float cross = fmaf(ah, bl, al * bh);
  const float s = hi + p;
  const float bb = s - hi;
  const float se = (hi - (s - bb)) + (p - bb);
  hi = s;
  lo += se + pe + cross;
}
// acc += conj(a) * b
DV void df_cmac_conj(df2& acc, const df2& a, const df2& b) {
  df_mac(acc.rh, acc.rl, a.rh, a.rl, b.rh, b.rl);
  df_mac(acc.rh, acc.rl, a.ih, a.il, b.ih, b.il);
  df_mac(acc.ih, acc.il, a.rh, a.rl, b.ih, b.il);
  df_mac(acc.ih, acc.il, -a.ih, -a.il, b.rh, b.rl);
}
// acc += a * b
DV void df_cmac(df2& acc, const df2& a, const df2& b) {
  df_mac(acc.rh, acc.rl, a.rh, a.rl, b.rh, b.rl);
  df_mac(acc.rh, acc.rl, -a.ih, -a.il, b.ih, b.il);
  df_mac(acc.ih, acc.il, a.rh, a.rl, b.ih, b.il);
  df_mac(acc.ih, acc.il, a.ih, a.il, b.rh, b.rl);
}

// a + b for complex double-float values (TwoSum on each part, then
// renormalised).
DV void df_add_part(float& h, float& l, float bh, float bl) {
  const float s = h + bh;
  const float bb = s - h;
  const float e = (h - (s - bb)) + (bh - bb) + l + bl;
  h = s + e;
  l = e - (h - s);
}
DV df2 df_cadd(df2 a, const df2& b) {
  df_add_part(a.rh, a.rl, b.rh, b.rl);
  df_add_part(a.ih, a.il, b.ih, b.il);
  return a;
}

// Sum over a warp (all 32 lanes active).
DV double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// The halves of the warp take the real and the imaginary parts after the first
// exchange: five additions instead of ten (an FP64 instruction of a warp takes
// 64 cycles), in the same order.
DV cplx warp_sum(cplx v) {
  unsigned int lane;
  asm("mov.u32 %0, %%laneid;" : "=r"(lane));
  const bool im = lane & 16u;
  double s = (im ? v.y : v.x) + __shfl_xor_sync(0xffffffffu, im ? v.x : v.y, 16);
  for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return mk(__shfl_sync(0xffffffffu, s, 0), __shfl_sync(0xffffffffu, s, 16));
}
// Sum of a complex value over S >= 2 adjacent lanes (a power of two): the even
// ones return its real part, the odd ones its imaginary part, for half the
// additions of summing both.
DV double half_sum(cplx a, int S) {
  const bool im = threadIdx.x & 1;
  double h = (im ? a.y : a.x) + __shfl_xor_sync(0xffffffffu, im ? a.x : a.y, 1);
  for (int o = 2; o < S; o <<= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
  return h;
}
DV float warp_sumf(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Deterministic block sum; `red` needs blockDim.x/32 slots.  Every thread
// gets the result.
template <typename T>
DV T block_sum(T v, T* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  T s = red[0];
  for (int i = 1; i < nw; ++i) s = s + red[i];
  __syncthreads();
  return s;
}
template <>
DV cplx block_sum<cplx>(cplx v, cplx* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  cplx s = red[0];
  for (int i = 1; i < nw; ++i) s = cadd(s, red[i]);
  __syncthreads();
  return s;
}

DV uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier state (device memory).  `count` is zeroed by the host before
// every cooperative launch; `err` records an expired wait.
struct GridBar {
  unsigned int count;
  unsigned int limit_us;  // wait limit in microseconds (0: kBarrierTimeoutNs)
  int err;                // nonzero after a wait expired
  int pad;
};

// Barrier across all CTAs of a cooperative launch (co-residency guaranteed
// by cudaLaunchCooperativeKernel).  The arrival counter only grows: on its
// k-th barrier every CTA adds one and waits until the counter reaches
// k * gridDim, so no CTA has to reset anything between barriers (one atomic
// and one polled load per CTA per barrier).  Every wait is bounded: after
// kBarrierTimeoutNs of wall time (or the context's limit_us) the CTA records
// the expiry in err, and every CTA of the launch leaves (grid_sync returns
// true).
constexpr uint64_t kBarrierTimeoutNs = 4000000000ull;  // 4 s

struct GridSync {
  GridBar* bar;
  unsigned int target;  // used by thread 0 of each CTA
};

// Arrival is a release reduction (the CTA's writes, ordered before it by
// the CTA barrier, become visible with it; the arriving thread does not
// wait for a returned value), polling an acquire load: one L2 round trip
// after the last arrival instead of a fence, a returning atomic and a
// trailing fence.
DV void bar_arrive_release(unsigned int* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
DV unsigned int ld_acquire_gpu(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Set in the arrival counter by an expired wait (a launch counts far below).
constexpr unsigned int kBarFail = 0x80000000u;

// Returns true if a wait expired (to every thread of the CTA: all leave).
// The expiry travels in the arrival counter itself, so that a column of a
// factorisation waits for one L2 round trip after the last arrival and no
// more: reading the err record before arriving and after leaving cost two
// further round trips per barrier.  err is read once per launch (an expiry of
// an earlier one still ends the later ones at once).
DV void grid_arrive(GridSync& gs) {
  __syncthreads();
  if (threadIdx.x == 0) bar_arrive_release(&gs.bar->count);
}
// Work that no other CTA waits for may stand between the two halves.
DV bool grid_wait(GridSync& gs) {
  int failed = 0;
  if (threadIdx.x == 0) {
    unsigned int* cnt = &gs.bar->count;
    if (gs.target == 0u && *((volatile int*)&gs.bar->err) != 0) failed = 1;
    gs.target += gridDim.x * gridDim.y * gridDim.z;
    uint64_t t0 = 0, limit_ns = 0;
    for (unsigned int spins = 1; !failed; ++spins) {
      const unsigned int v = ld_acquire_gpu(cnt);
      if (v & kBarFail) failed = 1;
      else if (v >= gs.target) break;
      else if ((spins & 31u) == 0u) {
        const uint64_t now = global_ns();
        if (t0 == 0) {
          const unsigned int lim = *((volatile unsigned int*)&gs.bar->limit_us);
          limit_ns = lim ? (uint64_t)lim * 1000ull : kBarrierTimeoutNs;
          t0 = now;
        } else if (now - t0 > limit_ns) {
          atomicExch(&gs.bar->err, 1);
          atomicOr(cnt, kBarFail);
          failed = 1;
        } else {
          __nanosleep(32);
        }
      }
    }
  }
  return __syncthreads_or(failed) != 0;
}
DV bool grid_sync(GridSync& gs) {
  grid_arrive(gs);
  return grid_wait(gs);
}
