// Device-side helpers shared by the kernel translation units: on-the-fly
// index generation by zero-bit insertion (Sec. 2: indices generated with
// binary operations), 2x2 complex products and the fp64 block reduction.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "sv_internal.cuh"

namespace sv {

template <typename I>
struct Ins {
  int m;
  I low[40];  // low[i] = 2^p_i - 1, p_i ascending (positions in the final index)
};

template <typename I>
inline Ins<I> make_ins(std::vector<int> pos) {
  std::sort(pos.begin(), pos.end());
  Ins<I> s{};
  s.m = (int)pos.size();
  for (int i = 0; i < s.m; ++i) s.low[i] = (I(1) << pos[i]) - 1;
  return s;
}

// Insert a 0 bit at every position of `s`, lowest first.
template <typename I>
__device__ __forceinline__ I insert_zeros(I u, const Ins<I>& s) {
  for (int i = 0; i < s.m; ++i) {
    const I lm = s.low[i];
    u = ((u & ~lm) << 1) | (u & lm);
  }
  return u;
}

// 2x2 complex matrix G00, G01, G10, G11 (real and imaginary parts apart).
template <typename R>
struct M2 {
  R r[4];
  R i[4];
};

template <typename R>
inline M2<R> to_m2(const HostMatrix& G) {
  M2<R> m;
  for (int e = 0; e < 4; ++e) {
    m.r[e] = (R)G.m[e].re;
    m.i[e] = (R)G.m[e].im;
  }
  return m;
}

// Arithmetic variants of (a, b) <- G (a, b); fewer products where the
// matrix structure allows (fp64 throughput is scarce on GB300).
enum { MK_DENSE = 0, MK_DIAG = 1, MK_REAL = 2, MK_IMOFF = 3 };

template <int MK, typename R>
__device__ __forceinline__ void mv2(const M2<R>& g, R& ar, R& ai, R& br, R& bi) {
  R nar, nai, nbr, nbi;
  if (MK == MK_DENSE) {
    nar = g.r[0] * ar - g.i[0] * ai + g.r[1] * br - g.i[1] * bi;
    nai = g.r[0] * ai + g.i[0] * ar + g.r[1] * bi + g.i[1] * br;
    nbr = g.r[2] * ar - g.i[2] * ai + g.r[3] * br - g.i[3] * bi;
    nbi = g.r[2] * ai + g.i[2] * ar + g.r[3] * bi + g.i[3] * br;
  } else if (MK == MK_DIAG) {
    nar = g.r[0] * ar - g.i[0] * ai;
    nai = g.r[0] * ai + g.i[0] * ar;
    nbr = g.r[3] * br - g.i[3] * bi;
    nbi = g.r[3] * bi + g.i[3] * br;
  } else if (MK == MK_REAL) {
    nar = g.r[0] * ar + g.r[1] * br;
    nai = g.r[0] * ai + g.r[1] * bi;
    nbr = g.r[2] * ar + g.r[3] * br;
    nbi = g.r[2] * ai + g.r[3] * bi;
  } else {  // [[r0, i*i1], [i*i2, r3]]
    nar = g.r[0] * ar - g.i[1] * bi;
    nai = g.r[0] * ai + g.i[1] * br;
    nbr = g.r[3] * br - g.i[2] * ai;
    nbi = g.r[3] * bi + g.i[2] * ar;
  }
  ar = nar;
  ai = nai;
  br = nbr;
  bi = nbi;
}

// ---- complex128: rotations as shears ------------------------------------------------
// GB300 issues fp64 at 1/64 of its fp32 rate, so complex128 gates are bound by
// their fp64 instructions.  A rotation by an angle of at most pi / 4 is three
// shears, x += a y, y += b x, x += a y with a = -tan(angle / 2), b = sin(angle): three
// FMAs where the products take four instructions; whole quarter turns k come off
// first, exactly and without fp64 arithmetic.
struct Shear {
  double a, b;
  int k;
};

// (x, y) <- the rotation of (x, y); i^k by selects and sign bits, without branches
// (which would keep a thread's other units from overlapping this one's FMAs:
// 274 -> 394 us a phase kernel at n = 27 instead of 213)
__device__ __forceinline__ void shear_rot(const Shear& h, double& x, double& y) {
  const long long sx = (long long)((unsigned)(h.k + 1) & 2u) << 62, sy = (long long)(h.k & 2) << 62;
  const double u = (h.k & 1) ? y : x, v = (h.k & 1) ? x : y;
  x = __longlong_as_double(__double_as_longlong(u) ^ sx);
  y = __longlong_as_double(__double_as_longlong(v) ^ sy);
  x = fma(h.a, y, x);
  y = fma(h.b, x, y);
  x = fma(h.a, y, x);
}

// the same by the opposite angle when `odd` (0 or 1)
__device__ __forceinline__ double flip_sign(double x, int odd) {
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)odd << 63));
}
__device__ __forceinline__ void shear_rot(const Shear& h, int odd, double& x, double& y) {
  const Shear g = {flip_sign(h.a, odd), flip_sign(h.b, odd), odd ? (4 - h.k) & 3 : h.k};
  shear_rot(g, x, y);
}

// complex64: the shears of the angle that the rounded a makes, so that a and b are the
// rotation's to half an ulp of b and no scale repeats with one sign
struct ShearF {
  float a, b;
  int k;
};
template <typename R>
struct ShearOf {
  typedef Shear T;
};
template <>
struct ShearOf<float> {
  typedef ShearF T;
};
__device__ __forceinline__ float flip_sign(float x, int odd) {
  return __uint_as_float(__float_as_uint(x) ^ ((unsigned)odd << 31));
}
inline ShearF round_shear(const Shear& h) {
  const float a = (float)h.a;
  return {a, (float)(-2.0 * a / (1.0 + (double)a * a)), h.k};
}
__device__ __forceinline__ void shear_rot(const ShearF& h, int odd, float& x, float& y) {
  const int k = odd ? (4 - h.k) & 3 : h.k;
  const unsigned s = (unsigned)odd << 31;
  const unsigned sx = ((unsigned)(k + 1) & 2u) << 30, sy = ((unsigned)k & 2u) << 30;
  const float u = (k & 1) ? y : x, v = (k & 1) ? x : y;
  const float a = __uint_as_float(__float_as_uint(h.a) ^ s);
  const float b = __uint_as_float(__float_as_uint(h.b) ^ s);
  x = __uint_as_float(__float_as_uint(u) ^ sx);
  y = __uint_as_float(__float_as_uint(v) ^ sy);
  x = fmaf(a, y, x);
  y = fmaf(b, x, y);
  x = fmaf(a, y, x);
}

// (a, b) <- G (a, b) for the 2x2s that are rotations: SK_REAL [[c, -s], [s, c]]
// (h[0]; refl: of (a, -b), as H), SK_IMOFF [[c, i s], [i s, c]] (h[0], RX), SK_PHASES
// diag(e^{i f}, e^{i g}) (h[0], h[1], RZ).  SK_NONE: none of them.
enum { SK_NONE = 0, SK_REAL = 1, SK_IMOFF = 2, SK_PHASES = 3 };
struct Shear2 {
  int kind, refl;
  Shear h[2];
};

template <int SK>
__device__ __forceinline__ void shear2(const Shear2& g, double& ar, double& ai, double& br,
                                       double& bi) {
  if (SK == SK_REAL) {
    // sign bits, not negations (which would go through the fp64 pipe)
    const long long sg = (long long)g.refl << 63;
    br = __longlong_as_double(__double_as_longlong(br) ^ sg);
    bi = __longlong_as_double(__double_as_longlong(bi) ^ sg);
    shear_rot(g.h[0], ar, br);
    shear_rot(g.h[0], ai, bi);
  } else if (SK == SK_IMOFF) {
    shear_rot(g.h[0], ar, bi);
    shear_rot(g.h[0], br, ai);
  } else {
    shear_rot(g.h[0], ar, ai);
    shear_rot(g.h[1], br, bi);
  }
}

// The shears of cos + i sin; false unless it has modulus 1 to fp64 rounding.
inline bool make_shear(double c, double s, Shear* h) {
  if (!(std::fabs(c * c + s * s - 1.0) < 4e-15)) return false;
  int k = 0;  // (c, s) = i^k (c', s') with c' >= |s'|
  while (k < 4 && !(c > 0 && c >= std::fabs(s))) {
    const double t = c;  // times -i
    c = s;
    s = -t;
    ++k;
  }
  *h = {-s / (1.0 + c), s, k & 3};
  return k < 4;
}

// The shear form of a 2x2, kind SK_NONE if it has none.
inline Shear2 make_shear2(const HostMatrix& G) {
  Shear2 g{};
  const cd u = G.at(0, 0), v = G.at(0, 1), w = G.at(1, 0), x = G.at(1, 1);
  const bool real = u.im == 0 && v.im == 0 && w.im == 0 && x.im == 0;
  if (v.re == 0 && v.im == 0 && w.re == 0 && w.im == 0) {
    if (make_shear(u.re, u.im, &g.h[0]) && make_shear(x.re, x.im, &g.h[1])) g.kind = SK_PHASES;
  } else if (real && v.re == -w.re && u.re == x.re) {
    if (make_shear(u.re, w.re, &g.h[0])) g.kind = SK_REAL;
  } else if (real && v.re == w.re && u.re == -x.re) {
    g.refl = 1;
    if (make_shear(u.re, w.re, &g.h[0])) g.kind = SK_REAL;
  } else if (u.im == 0 && x.im == 0 && v.re == 0 && w.re == 0 && u.re == x.re && v.im == w.im) {
    if (make_shear(u.re, v.im, &g.h[0])) g.kind = SK_IMOFF;
  }
  return g;
}

// ---- complex64: dithered rounding ---------------------------------------------
// Round-to-nearest errors of identical inputs are identical.  In states with
// many equal amplitudes (uniform superpositions, the iterates of Grover's
// search) every amplitude of such a class makes the same rounding error at
// every gate, and ||psi||^2 moves by the same relative amount each time: a
// drift linear in the gate count (measured 3e-8 per Grover iteration at
// n = 20).  Complex64 gate kernels therefore add, inside each output's
// fused multiply-add chain before its final rounding, a pseudo-random term
// rho (|a| + |b|) with |rho| <= 2^-24 and zero mean, keyed by the amplitude
// index and a per-launch seed: the final rounding becomes dithered (its
// error random, with zero mean, from amplitude to amplitude) and equal
// amplitudes leave the gate distinct in their last bit, so later roundings
// are uncorrelated as well.  The added error is of the size of one rounding.
//
// mix32: the "lowbias32" integer hash (C. Wellons, hash-prospector, 2018).
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

// byte i of h as an odd integer in -255..255 times 2^-32 (|rho| < 2^-24,
// mean 0 over uniform bytes)
__device__ __forceinline__ float dither_rho(uint32_t h, int i) {
  const int b = (int)(int8_t)(h >> (8 * i));
  return (float)(2 * b + 1) * 2.3283064365386963e-10f;
}

// (a, b) <- G (a, b) in fp32 with the final rounding of each of the four
// outputs dithered by rho_i (|a| + |b|) of its own component.
template <int MK>
__device__ __forceinline__ void mv2_dither(const M2<float>& g, float& ar, float& ai, float& br,
                                           float& bi, uint32_t h) {
  const float dr0 = dither_rho(h, 0) * (fabsf(ar) + fabsf(br));
  const float di0 = dither_rho(h, 1) * (fabsf(ai) + fabsf(bi));
  const float dr1 = dither_rho(h, 2) * (fabsf(ar) + fabsf(br));
  const float di1 = dither_rho(h, 3) * (fabsf(ai) + fabsf(bi));
  float nar, nai, nbr, nbi;
  if (MK == MK_DENSE) {
    nar = fmaf(g.r[0], ar, fmaf(-g.i[0], ai, fmaf(g.r[1], br, fmaf(-g.i[1], bi, dr0))));
    nai = fmaf(g.r[0], ai, fmaf(g.i[0], ar, fmaf(g.r[1], bi, fmaf(g.i[1], br, di0))));
    nbr = fmaf(g.r[2], ar, fmaf(-g.i[2], ai, fmaf(g.r[3], br, fmaf(-g.i[3], bi, dr1))));
    nbi = fmaf(g.r[2], ai, fmaf(g.i[2], ar, fmaf(g.r[3], bi, fmaf(g.i[3], br, di1))));
  } else if (MK == MK_DIAG) {
    nar = fmaf(g.r[0], ar, fmaf(-g.i[0], ai, dr0));
    nai = fmaf(g.r[0], ai, fmaf(g.i[0], ar, di0));
    nbr = fmaf(g.r[3], br, fmaf(-g.i[3], bi, dr1));
    nbi = fmaf(g.r[3], bi, fmaf(g.i[3], br, di1));
  } else if (MK == MK_REAL) {
    nar = fmaf(g.r[0], ar, fmaf(g.r[1], br, dr0));
    nai = fmaf(g.r[0], ai, fmaf(g.r[1], bi, di0));
    nbr = fmaf(g.r[2], ar, fmaf(g.r[3], br, dr1));
    nbi = fmaf(g.r[2], ai, fmaf(g.r[3], bi, di1));
  } else {  // [[r0, i*i1], [i*i2, r3]]
    nar = fmaf(g.r[0], ar, fmaf(-g.i[1], bi, dr0));
    nai = fmaf(g.r[0], ai, fmaf(g.i[1], br, di0));
    nbr = fmaf(g.r[3], br, fmaf(-g.i[2], ai, dr1));
    nbi = fmaf(g.r[3], bi, fmaf(g.i[2], ar, di1));
  }
  ar = nar;
  ai = nai;
  br = nbr;
  bi = nbi;
}

// A pair of fp32 lanes in one 64-bit register: the arithmetic below stays on
// these from load to store, so that every step is one paired instruction
// (float2 values assembled from parts were split into scalar FMAs and moves).
typedef unsigned long long Pair;

__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
  Pair d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ Pair pair_of(float x, float y) {
  Pair d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ float2 lanes_of(Pair p) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ Pair pair_both(float x) { return pair_of(x, x); }
__device__ __forceinline__ Pair pair_swap(Pair p) {
  const float2 v = lanes_of(p);
  return pair_of(v.y, v.x);
}
// p += a q
__device__ __forceinline__ void pair_add(Pair& p, Pair a, Pair q) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(p) : "l"(a), "l"(q));
}

// A thread's running sum: compensated (Kahan) in fp32 for complex64 kernels
// (GB300 issues fp64 at a small fraction of the fp32 rate, so the per-unit
// additions stay in fp32 and s - c meets the fp64 block sum once), plain fp64
// for complex128.
template <typename R>
struct CompSum {
  R s = 0, c = 0;
  __device__ __forceinline__ void add(R x) {
    if constexpr (sizeof(R) == 4) {
      const R y = x - c;
      const R t = s + y;
      c = (t - s) - y;
      s = t;
    } else {
      s += x;
    }
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// Sum over the block (fixed order); the result is valid in thread 0.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double ws[32];
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) ws[w] = v;
  __syncthreads();
  if (w == 0) {
    v = lane < (int)(blockDim.x >> 5) ? ws[lane] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  return v;
}

bool use_32bit_index(int n, sv_dtype dt);

// ---- dependent launches ----------------------------------------------------------
// A kernel launched by launch_dependent may have its blocks set up while the
// stream's previous kernel drains; it calls grid_dependency_wait before its
// first access to device memory, which returns once everything earlier on the
// stream has finished and is visible.  No kernel signals its dependents early,
// so a block never occupies an SM that the previous kernel still needs.
// Measured on GB300 for chains of one-gate kernels, against plain launches:
// n = 12 complex128 (831 launches) 3.41 -> 1.62 ms, n = 18 complex64 5.13 ->
// 2.47 ms, the QFT at n = 20 0.91 -> 0.43 ms and at n = 26 21.9 -> 20.9 ms.
// The passes, sweeps and reductions: HEA gradient gate by gate at n = 14 2.51
// -> 1.37 ms (complex128 3.79 -> 2.08), Trotter at n = 16 0.77 -> 0.48 ms.
// (Signalling dependents at a kernel's start, so that their blocks also wait
// on the SMs: no faster, and the n = 22 QAOA gradient 4.39 -> 4.74 ms.)
__device__ __forceinline__ void grid_dependency_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... KArgs>
inline cudaError_t launch_dependent(void (*kern)(KArgs...), unsigned grid, unsigned threads,
                                    size_t smem, cudaStream_t st,
                                    const std::common_type_t<KArgs>&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  void* p[] = {const_cast<void*>(static_cast<const void*>(&args))...};
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kern), p);
}

}  // namespace sv
