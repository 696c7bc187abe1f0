// Pauli-string rotations and Trotterized time evolution (Sec. 3: Hamiltonian
// objects with a time-evolution solver using the Trotter decomposition; the
// same rotations build QAOA-style layers).
//
// For a Pauli string P with masks (xm, zm): P^2 = I, so
//     exp(-i a P) psi = cos(a) psi - i sin(a) P psi,
//     (P psi)_x = i^{#Y} (-1)^{popcount((x ^ xm) & zm)} psi_{x ^ xm}.
// Off-diagonal strings (xm != 0) update the pairs (x, x ^ xm) together (x
// with the highest bit of xm clear).  Diagonal strings (xm = 0) multiply
// psi_x by exp(-i a s(x)), s(x) = (-1)^{popcount(x & zm)}; a run of
// consecutive diagonal terms commutes, so one pass applies the whole run:
// psi_x *= exp(-i sum_k a_k s_k(x)).
//
// A run of diagonal strings goes through kdiag_run (and kadj_diag in reverse
// sweeps).  What bounds it is the work per amplitude and term, not HBM, so a
// thread takes a register tile of amplitudes that differ in a few bits: with
// z_k split into its part on the tile bits (rho_k) and the rest, the tile's
// angles are the Walsh-Hadamard transform of v[rho] = sum over the terms with
// rho_k = rho of +-a_k - one sign per term and tile instead of one per term
// and amplitude.  Angles are fixed-point fractions of a turn (32 bits for
// complex64, 64 for complex128), scaled up by the power of two that the sum of
// their magnitudes leaves room for (see angle_shift): sums and differences are
// exact, where an fp32 sum of k angles loses log2(k) + log2(sum) bits, and small
// angles keep their relative accuracy.
#include <cmath>
#include <vector>

#include "sv_device.cuh"

namespace sv {
namespace {

constexpr int kEThreads = 256;
constexpr int kMaxDiag = 64;

struct DiagRun {
  int nt;
  uint64_t zm[kMaxDiag];
  double a[kMaxDiag];
};

// the 16-byte vector of a state: two complex64 amplitudes or one complex128
template <typename R>
struct TurnVec;
template <>
struct TurnVec<float> {
  typedef float4 T;
};
template <>
struct TurnVec<double> {
  typedef double2 T;
};

// The general diagonal kernels: states of less than a tile per warp (under
// kRunMinQubits qubits) and angles that have no fixed-point form (not finite,
// or beyond 2^50).
// complex64 vectors (2 amplitudes), phases from an fp32 angle sum
__global__ void __launch_bounds__(kEThreads)
    kdiag_c64(float4* __restrict__ psi, uint64_t nvec, const __grid_constant__ DiagRun D) {
  grid_dependency_wait();
  constexpr int IT = 8;
  const uint64_t base = (uint64_t)blockIdx.x * (kEThreads * IT) + threadIdx.x;
  float4 v[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t i = base + (uint64_t)it * kEThreads;
    if (i < nvec) v[it] = psi[i];
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t i = base + (uint64_t)it * kEThreads;
    if (i >= nvec) continue;
    float ph0 = 0.f, ph1 = 0.f;  // angle sums for amplitudes 2i and 2i+1
    for (int k = 0; k < D.nt; ++k) {
      const uint64_t z = D.zm[k];
      const float a = (float)D.a[k];
      const int p0 = __popcll((2 * i) & z) & 1;
      ph0 += p0 ? -a : a;
      const int p1 = p0 ^ (int)(z & 1);
      ph1 += p1 ? -a : a;
    }
    float s0, c0, s1, c1;
    sincosf(ph0, &s0, &c0);
    sincosf(ph1, &s1, &c1);
    float4 x = v[it];
    // multiply by exp(-i ph) = c - i s
    const float r0 = c0 * x.x + s0 * x.y, i0 = c0 * x.y - s0 * x.x;
    const float r1 = c1 * x.z + s1 * x.w, i1 = c1 * x.w - s1 * x.z;
    psi[i] = make_float4(r0, i0, r1, i1);
  }
}

__global__ void __launch_bounds__(kEThreads)
    kdiag_c128(double2* __restrict__ psi, uint64_t dim, const __grid_constant__ DiagRun D) {
  grid_dependency_wait();
  constexpr int IT = 8;
  const uint64_t base = (uint64_t)blockIdx.x * (kEThreads * IT) + threadIdx.x;
  double2 v[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t i = base + (uint64_t)it * kEThreads;
    if (i < dim) v[it] = psi[i];
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t i = base + (uint64_t)it * kEThreads;
    if (i >= dim) continue;
    double ph = 0.0;
    for (int k = 0; k < D.nt; ++k) ph += (__popcll(i & D.zm[k]) & 1) ? -D.a[k] : D.a[k];
    double s, c;
    sincos(ph, &s, &c);
    const double2 x = v[it];
    psi[i] = make_double2(c * x.x + s * x.y, c * x.y - s * x.x);
  }
}

// complex128, a few strings: one rotation after the other as three FMAs an amplitude
// (see Shear), where the angle sum's fp64 sine and cosine alone take about 40
// instructions.  n = 20, one string: 73 -> 12 us, eight 89 -> 53 (n = 25: 2110 -> 1302),
// 6 us each: up to kShearTerms of them, short of where the two cost the same.
constexpr int kShearTerms = 12;
struct DiagShears {
  int nt;
  uint64_t zm[kShearTerms];
  Shear h[kShearTerms];
};
__global__ void __launch_bounds__(kEThreads)
    kdiag_shears(double2* __restrict__ psi, uint64_t dim, const __grid_constant__ DiagShears D) {
  grid_dependency_wait();
  constexpr int IT = 4;
  const uint64_t base = (uint64_t)blockIdx.x * (kEThreads * IT) + threadIdx.x;
  double2 v[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t i = base + (uint64_t)it * kEThreads;
    if (i < dim) v[it] = psi[i];
  }
  for (int k = 0; k < D.nt; ++k) {
    const uint64_t z = D.zm[k];
    const Shear h = D.h[k];
#pragma unroll
    for (int it = 0; it < IT; ++it)
      shear_rot(h, __popcll((base + (uint64_t)it * kEThreads) & z) & 1, v[it].x, v[it].y);
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t i = base + (uint64_t)it * kEThreads;
    if (i < dim) psi[i] = v[it];
  }
}

// complex64, up to kShearTermsF strings: the sine and cosine of one angle are rounded
// alike on every amplitude, and a circuit that repeats it (QAOA's edges, gate by
// gate) repeats their scale; shears have none.  QAOA, n = 14..20, energies and
// gradients against 64 bits: 0.8..3.6e-6 before, 4.0..6.6e-7 now, with as little work.
constexpr int kShearTermsF = 4;
struct DiagShearsF {
  int nt;
  uint64_t zm[kShearTermsF];
  ShearF h[kShearTermsF];
};
__global__ void __launch_bounds__(kEThreads)
    kdiag_shears_f(float4* __restrict__ psi, uint64_t nvec, const __grid_constant__ DiagShearsF D) {
  grid_dependency_wait();
  constexpr int IT = 4;
  const uint64_t base = (uint64_t)blockIdx.x * (kEThreads * IT) + threadIdx.x;
  float4 v[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t i = base + (uint64_t)it * kEThreads;
    if (i < nvec) v[it] = psi[i];
  }
  for (int k = 0; k < D.nt; ++k) {
    const uint64_t z = D.zm[k];
    const ShearF h = D.h[k];
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int odd = __popcll((2 * (base + (uint64_t)it * kEThreads)) & z) & 1;
      shear_rot(h, odd, v[it].x, v[it].y);
      shear_rot(h, odd ^ (int)(z & 1), v[it].z, v[it].w);
    }
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t i = base + (uint64_t)it * kEThreads;
    if (i < nvec) psi[i] = v[it];
  }
}

// ---- runs of diagonal strings --------------------------------------------------------
constexpr int kRunTerms = 256;  // terms of one kdiag_run launch
constexpr int kAdjTerms = 128;  // terms of one kadj_diag launch

// a turn in 2^32 (complex64) or 2^64 (complex128) steps
template <typename R>
struct Turn;
template <>
struct Turn<float> {
  typedef uint32_t T;
};
template <>
struct Turn<double> {
  typedef uint64_t T;
};

// Tiles of NT amplitudes: the in-vector bit (complex64) and the top three bits
// of the vector index; the other bits are the thread index, so that a warp's
// 16-byte loads are contiguous.  Terms sorted by rho: [start[r], start[r + 1])
// have z pattern r on the tile bits and zt on the thread bits.  unit: half turns
// of one step of a; half and mask: what takes the nearest quarter turn off an
// angle of whole turns, 0 for scaled ones.
template <typename R, int CAP>
struct DiagTiles {
  static constexpr int NT = sizeof(R) == 4 ? 16 : 8;
  typename Turn<R>::T half, mask;
  R unit;
  uint16_t start[NT + 1];
  uint32_t zt[CAP];
  typename Turn<R>::T a[CAP];
};

// the tile's angles: angle of amplitude r = sum_rho (-1)^{popcount(r & rho)} v[rho]
template <typename R, int CAP, int NT>
__device__ __forceinline__ void tile_angles(const DiagTiles<R, CAP>& D, uint32_t t,
                                            typename Turn<R>::T (&v)[NT]) {
  typedef typename Turn<R>::T F;
#pragma unroll
  for (int r = 0; r < NT; ++r) {
    F x = 0;
    for (int k = D.start[r]; k < D.start[r + 1]; ++k) {
      const F a = D.a[k];
      x += (__popc(t & D.zt[k]) & 1) ? F(0) - a : a;
    }
    v[r] = x;
  }
#pragma unroll
  for (int i = 0; (1 << i) < NT; ++i)
#pragma unroll
    for (int r = 0; r < NT; ++r) {
      if (r & (1 << i)) continue;
      const F x = v[r], y = v[r | (1 << i)];
      v[r] = x + y;
      v[r | (1 << i)] = x - y;
    }
}

// sine and cosine of a fixed-point angle of D: the nearest quarter turn comes off
// in integers, so that the remainder (at most an eighth of a turn) converts to
// R with an error below 2^-28 (2^-57) turns; a scaled angle is below an eighth
template <int CAP>
__device__ __forceinline__ void turn_sincos(const DiagTiles<float, CAP>& D, uint32_t f, float* s,
                                            float* c) {
  const uint32_t q = (f + D.half) & D.mask;
  const int rem = (int)(f - q);
  float sn, cs;
  sincospif((float)rem * D.unit, &sn, &cs);
  const float x = (q & 0x40000000u) ? sn : cs, y = (q & 0x40000000u) ? cs : sn;
  *c = ((q >> 31) ^ ((q >> 30) & 1)) ? -x : x;
  *s = (q >> 31) ? -y : y;
}

template <int CAP>
__device__ __forceinline__ void turn_sincos(const DiagTiles<double, CAP>& D, uint64_t f, double* s,
                                            double* c) {
  const uint64_t q = (f + D.half) & D.mask;
  const long long rem = (long long)(f - q);
  double sn, cs;
  sincospi((double)rem * D.unit, &sn, &cs);
  const uint32_t h = (uint32_t)(q >> 32);
  const double x = (h & 0x40000000u) ? sn : cs, y = (h & 0x40000000u) ? cs : sn;
  *c = ((h >> 31) ^ ((h >> 30) & 1)) ? -x : x;
  *s = (h >> 31) ? -y : y;
}

// re + i im <- (c - i s)(re + i im)
template <typename R>
__device__ __forceinline__ void turn_back(R c, R s, R& re, R& im) {
  const R r = c * re + s * im;
  im = c * im - s * re;
  re = r;
}

// psi_x *= exp(-i angle(x)), one tile per thread (T = 2^n / NT threads, a
// multiple of the block size).  complex64, n = 26, the 25 ZZ strings of a
// chain: 1359 us with one sign per amplitude and term, 174 us so (the HBM read
// and write: 160 us).
template <typename R>
__global__ void __launch_bounds__(kEThreads)
    kdiag_run(typename TurnVec<R>::T* __restrict__ psi, uint32_t T,
              const __grid_constant__ DiagTiles<R, kRunTerms> D) {
  grid_dependency_wait();
  constexpr int NT = DiagTiles<R, kRunTerms>::NT;
  typedef typename TurnVec<R>::T V;
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  V x[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) x[u] = psi[(uint64_t)T * u + t];
  typename Turn<R>::T v[NT];
  tile_angles<R, kRunTerms, NT>(D, t, v);
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    R s, c;
    if constexpr (sizeof(R) == 4) {
      turn_sincos(D, v[2 * u], &s, &c);
      turn_back<R>(c, s, x[u].x, x[u].y);
      turn_sincos(D, v[2 * u + 1], &s, &c);
      turn_back<R>(c, s, x[u].z, x[u].w);
    } else {
      turn_sincos(D, v[u], &s, &c);
      turn_back<R>(c, s, x[u].x, x[u].y);
    }
    psi[(uint64_t)T * u + t] = x[u];
  }
}

// The gradients of a run's rotations exp(-i theta_k P_k / 2): terms sorted by
// gradient slot, [sstart[j], sstart[j + 1]) belong to slot[j].
struct DiagGrads {
  int ns;
  int slot[kAdjTerms];
  uint16_t sstart[kAdjTerms + 1];
  uint8_t rho[kAdjTerms];
  uint32_t zt[kAdjTerms];
};

// to (lane 0's) += the sum of the lanes' g, each step's rounding error carried along
__device__ __forceinline__ void warp_add(const CompSum<float>& g, CompSum<float>& to, int lane) {
  float s = g.s, e = -g.c;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const float x = __shfl_xor_sync(0xffffffffu, s, o);
    e += __shfl_xor_sync(0xffffffffu, e, o);
    const float t = s + x, b = t - s;
    e += (s - (t - b)) + (x - b);
    s = t;
  }
  if (lane == 0) {
    to.add(s);
    to.add(e);
  }
}
__device__ __forceinline__ void warp_add(const CompSum<double>& g, CompSum<double>& to, int lane) {
  double s = g.s;
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) to.add(s);
}

// Reverse-sweep step of a run of diagonal rotations: all commute, so every
// gradient Im<lambda|P_k|psi> = sum_x s_k(x) Im(conj(lambda_x) psi_x) comes
// from the states before the run is un-applied.  The Walsh-Hadamard transform
// of a tile's Im(conj(lambda) psi) gives each term's tile sum; the terms of a
// slot (gates that share a parameter) add up in the thread before one warp
// sum.  Past the tile's transform (four additions) every sum is compensated (fp64
// for complex128): the terms of a thread, the warp's and the warp's tiles; per block
// fp64 into partials[slot * pstride + blockIdx.x].  With plain sums of the terms 127
// equal ones were up to 32 * 2^-24 off.  QAOA on a 3-regular graph, n = 22, 33 ZZ gates
// per layer on one parameter: 33 launches of 16.5 us before, one of 35 us.
template <typename R>
__global__ void __launch_bounds__(kEThreads, 2)
    kadj_diag(typename TurnVec<R>::T* __restrict__ psi, typename TurnVec<R>::T* __restrict__ lam,
              uint32_t T, const __grid_constant__ DiagTiles<R, kAdjTerms> D,
              const __grid_constant__ DiagGrads G, double* __restrict__ partials, int pstride) {
  grid_dependency_wait();
  constexpr int NT = DiagTiles<R, kAdjTerms>::NT;
  typedef typename TurnVec<R>::T V;
  extern __shared__ __align__(16) unsigned char smem[];
  R* sw = reinterpret_cast<R*>(smem);  // [NT][blockDim.x]
  CompSum<R>* gw = reinterpret_cast<CompSum<R>*>(sw + NT * blockDim.x);  // [warp][slot]
  const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < nw * G.ns; i += blockDim.x) gw[i] = CompSum<R>();
  __syncthreads();
  for (uint32_t t0 = blockIdx.x * blockDim.x; t0 < T; t0 += gridDim.x * blockDim.x) {
    const uint32_t t = t0 + threadIdx.x;
    V x[8], l[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      x[u] = psi[(uint64_t)T * u + t];
      l[u] = lam[(uint64_t)T * u + t];
    }
    if (G.ns) {
      R w[NT];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if constexpr (sizeof(R) == 4) {
          w[2 * u] = l[u].x * x[u].y - l[u].y * x[u].x;
          w[2 * u + 1] = l[u].z * x[u].w - l[u].w * x[u].z;
        } else {
          w[u] = l[u].x * x[u].y - l[u].y * x[u].x;
        }
      }
#pragma unroll
      for (int i = 0; (1 << i) < NT; ++i)
#pragma unroll
        for (int r = 0; r < NT; ++r) {
          if (r & (1 << i)) continue;
          const R a = w[r], b = w[r | (1 << i)];
          w[r] = a + b;
          w[r | (1 << i)] = a - b;
        }
      // each thread reads back only its own column: no barrier
#pragma unroll
      for (int r = 0; r < NT; ++r) sw[r * blockDim.x + threadIdx.x] = w[r];
      for (int j = 0; j < G.ns; ++j) {
        CompSum<R> g;
        for (int k = G.sstart[j]; k < G.sstart[j + 1]; ++k) {
          const R a = sw[G.rho[k] * blockDim.x + threadIdx.x];
          g.add((__popc(t & G.zt[k]) & 1) ? -a : a);
        }
        warp_add(g, gw[warp * G.ns + j], lane);
      }
    }
    typename Turn<R>::T v[NT];
    tile_angles<R, kAdjTerms, NT>(D, t, v);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      R s, c;
      if constexpr (sizeof(R) == 4) {
        turn_sincos(D, v[2 * u], &s, &c);
        turn_back<R>(c, s, x[u].x, x[u].y);
        turn_back<R>(c, s, l[u].x, l[u].y);
        turn_sincos(D, v[2 * u + 1], &s, &c);
        turn_back<R>(c, s, x[u].z, x[u].w);
        turn_back<R>(c, s, l[u].z, l[u].w);
      } else {
        turn_sincos(D, v[u], &s, &c);
        turn_back<R>(c, s, x[u].x, x[u].y);
        turn_back<R>(c, s, l[u].x, l[u].y);
      }
      psi[(uint64_t)T * u + t] = x[u];
      lam[(uint64_t)T * u + t] = l[u];
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < G.ns; j += blockDim.x) {
    double e = 0.0;
    for (int w = 0; w < nw; ++w) e += gw[w * G.ns + j].value();
    partials[(size_t)G.slot[j] * pstride + blockIdx.x] = e;
  }
}

// off-diagonal string: pairs (x, y = x ^ xm), x with bit h = top bit of xm clear.
// coef = -i sin(a) i^{#Y}; (x', y') = (c x + coef sy y, c y + coef sx x),
// sy = (-1)^{popcount(y & zm)}, sx = (-1)^{popcount(x & zm)}.
template <typename R, typename T2>
__global__ void __launch_bounds__(kEThreads)
    kpair(T2* __restrict__ psi, uint64_t npairs, uint64_t lowmask, uint64_t xm, uint64_t zm,
          R c, R kr, R ki) {
  grid_dependency_wait();
  constexpr int IT = 8;
  const uint64_t base = (uint64_t)blockIdx.x * (kEThreads * IT) + threadIdx.x;
  uint64_t xs[IT];
  T2 a[IT], b[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t u = base + (uint64_t)it * kEThreads;
    if (u < npairs) {
      xs[it] = ((u & ~lowmask) << 1) | (u & lowmask);
      a[it] = psi[xs[it]];
      b[it] = psi[xs[it] ^ xm];
    }
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t u = base + (uint64_t)it * kEThreads;
    if (u >= npairs) continue;
    const uint64_t x = xs[it], y = x ^ xm;
    const R sx = (__popcll(x & zm) & 1) ? R(-1) : R(1);
    const R sy = (__popcll(y & zm) & 1) ? R(-1) : R(1);
    const T2 p = a[it], q = b[it];
    T2 np, nq;
    // coef * sy * q and coef * sx * p with coef = kr + i ki
    np.x = c * p.x + sy * (kr * q.x - ki * q.y);
    np.y = c * p.y + sy * (kr * q.y + ki * q.x);
    nq.x = c * q.x + sx * (kr * p.x - ki * p.y);
    nq.y = c * q.y + sx * (kr * p.y + ki * p.x);
    psi[x] = np;
    psi[y] = nq;
  }
}

// A Pauli-string rotation c I + coef P of complex128 states as shears: with P's
// i^{ny} and the strings' signs, even ny rotates (re x, im y) and (re y, im x) by
// one angle, odd ny (re x, re y) and (im x, im y), with the angle's sign by
// parity(y & zm) ^ (ny >> 1).  Six FMAs an amplitude pair where the products take 24
// and more fp64 instructions: n = 20 25 -> 12.4 us.
template <bool ODD, typename H, typename T2>
__device__ __forceinline__ void shear_pair(const H& h, int sign, T2& x, T2& y) {
  if (ODD) {
    shear_rot(h, sign, x.x, y.x);
    shear_rot(h, sign, x.y, y.y);
  } else {
    shear_rot(h, sign, x.x, y.y);
    shear_rot(h, sign, y.x, x.y);
  }
}

template <bool ODD>
__global__ void __launch_bounds__(kEThreads)
    kpair_c128(double2* __restrict__ psi, uint64_t npairs, uint64_t lowmask, uint64_t xm,
               uint64_t zm, int neg, Shear h) {
  grid_dependency_wait();
  constexpr int IT = 4;
  const uint64_t base = (uint64_t)blockIdx.x * (kEThreads * IT) + threadIdx.x;
  double2 a[IT], b[IT];
  uint64_t xs[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t u = base + (uint64_t)it * kEThreads;
    xs[it] = ((u & ~lowmask) << 1) | (u & lowmask);
    if (u < npairs) {
      a[it] = psi[xs[it]];
      b[it] = psi[xs[it] ^ xm];
    }
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const uint64_t u = base + (uint64_t)it * kEThreads;
    if (u >= npairs) continue;
    const uint64_t y = xs[it] ^ xm;
    shear_pair<ODD>(h, (__popcll(y & zm) & 1) ^ neg, a[it], b[it]);
    psi[xs[it]] = a[it];
    psi[y] = b[it];
  }
}

// the rotated state: device data, precision, qubits, stream and the
// complex64 rounding feedback (see feedback_round)
struct Target {
  void* data;
  sv_dtype dt;
  int n;
  cudaStream_t stream;
  RoundCtx* rc;
};

// Adjoint step of a Pauli-string rotation U = exp(-i theta P / 2) in a
// reverse sweep (P = i^{ny} X^xm Z^zm up to the sign convention above): each
// unit first adds its part of Im<lambda|P|psi> (the gradient of theta) and
// then un-applies U^dagger on psi and lambda, as shears.  KIND 0 (xm = 0): a unit
// is one amplitude, (P v)_x = s(x) v_x; otherwise (KIND 1 even ny, 2 odd ny) a unit
// is the pair (x, y = x ^ xm) with bit h = top bit of xm clear in x and
// (P v)_x = i^{ny} s(y) v_y, (P v)_y = i^{ny} s(x) v_x, s(v) =
// (-1)^{popcount(v & zm)}, s(x) = s(y) (-1)^{ny}.  Per-thread sums: compensated in
// fp32 for complex64, fp64 for complex128; the block's fp64 sum goes to
// partials[blockIdx.x] (grid-stride loop, every block writes its slot).
// complex128 is bound by fp64 issue: a diagonal string takes 9 instructions an
// amplitude of psi and lambda where the products take 14, the others 17 a unit in
// place of 50: n = 20 42.7 -> 25 us (HBM and L2: 32 MiB of states read and written).
// complex64 loses no norm (see kdiag_shears_f); its time is the states' traffic.
template <typename R, typename T2, int KIND>
__global__ void __launch_bounds__(kEThreads)
    kadj_pauli(T2* __restrict__ psi, T2* __restrict__ lam, uint64_t units, uint64_t lowmask,
               uint64_t xm, uint64_t zm, int neg, typename ShearOf<R>::T h,
               double* __restrict__ partials) {
  grid_dependency_wait();
  CompSum<R> acc;
  for (uint64_t u = (uint64_t)blockIdx.x * kEThreads + threadIdx.x; u < units;
       u += (uint64_t)gridDim.x * kEThreads) {
    if (KIND == 0) {
      T2 p = psi[u], l = lam[u];
      const int odd = __popcll(u & zm) & 1;
      acc.add(flip_sign(l.x * p.y - l.y * p.x, odd));
      shear_rot(h, odd, p.x, p.y);
      shear_rot(h, odd, l.x, l.y);
      psi[u] = p;
      lam[u] = l;
    } else {
      const uint64_t x = ((u & ~lowmask) << 1) | (u & lowmask), y = x ^ xm;
      T2 px = psi[x], py = psi[y], lx = lam[x], ly = lam[y];
      const int sign = (__popcll(y & zm) & 1) ^ neg;
      if (KIND == 1)
        acc.add(flip_sign(lx.x * py.y - lx.y * py.x + ly.x * px.y - ly.y * px.x, sign));
      else
        acc.add(flip_sign(lx.x * py.x + lx.y * py.y - ly.x * px.x - ly.y * px.y, sign));
      shear_pair<KIND == 2>(h, sign, px, py);
      shear_pair<KIND == 2>(h, sign, lx, ly);
      psi[x] = px;
      psi[y] = py;
      lam[x] = lx;
      lam[y] = ly;
    }
  }
  const double t = block_sum(acc.value());
  if (threadIdx.x == 0 && partials) partials[blockIdx.x] = t;
}

sv_status run_diag(const Target& s, const DiagRun& D) {
  if (D.nt == 0) return SV_OK;
  ProfScope prof(s.stream, s.dt == SV_C64 ? "kdiag_c64" : "kdiag_c128");
  if (s.dt == SV_C64) {
    const uint64_t nvec = uint64_t(1) << (s.n - 1);
    const unsigned g = (unsigned)((nvec + kEThreads * 8 - 1) / (kEThreads * 8));
    launch_dependent(kdiag_c64, g, kEThreads, 0, s.stream, (float4*)s.data, nvec, D);
  } else {
    const uint64_t dim = uint64_t(1) << s.n;
    const unsigned g = (unsigned)((dim + kEThreads * 8 - 1) / (kEThreads * 8));
    launch_dependent(kdiag_c128, g, kEThreads, 0, s.stream, (double2*)s.data, dim, D);
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return check_launch("diagonal rotation kernel");
}

// States of at least kRunMinQubits qubits have a tile for every lane of a warp.
constexpr int kRunMinQubits = 9;

// angle / (2 pi) modulo 1 in 2^64 steps: the product with 1 / (2 pi) as a sum
// of two doubles (104 bits), whole turns removed before it is scaled
constexpr double kTurnHi = 0.15915494309189535, kTurnLo = -9.839338337591243e-18;  // 1 / (2 pi)
uint64_t turns64(double a) {
  const double hi = a * kTurnHi;
  const double lo = std::fma(a, kTurnHi, -hi) + a * kTurnLo;
  const double frac = (hi - std::rint(hi)) + lo;  // |frac| <= 1/2 and a little
  return (uint64_t)std::llrint(frac * 4611686018427387904.0) << 2;  // 2^62, then 2^2
}

// The angle in steps of 2^-(32 + shift) (complex128: 2^-(64 + shift)) turns.
template <typename R>
typename Turn<R>::T turns(double a, int shift) {
  if (shift) {
    const double hi = a * kTurnHi;
    const double lo = std::fma(a, kTurnHi, -hi) + a * kTurnLo;
    const int bits = 8 * (int)sizeof(R) + shift;
    if constexpr (sizeof(R) == 4) return (uint32_t)std::llrint(std::ldexp(hi + lo, bits));
    return (typename Turn<R>::T)(std::llrint(std::ldexp(hi, bits)) + std::llrint(std::ldexp(lo, bits)));
  }
  const uint64_t f = turns64(a);
  if constexpr (sizeof(R) == 4)
    return (uint32_t)((f + 0x80000000ull) >> 32);
  else
    return f;
}

// How far the angles of one launch are scaled up: a step of 2^-32 turns is an error of
// up to 7e-10 rad an angle however small the angle is, the same in every step of a
// time evolution.  With the sum of the magnitudes below 2^-(1 + shift) turns no sum
// of scaled angles wraps; from 2 on (below an eighth of a turn) no quarter turn
// has to come off before the sine and cosine.  The rms error of 25 equal angles' sum: at
// 10^-4 rad 4e-9 in steps of 2^-32 turns, 6e-11 in fp32 and below that so; over 5 to
// 256 strings of 10^-6 to 10 rad below the fp32 sum's throughout.
int angle_shift(const double* a, int cnt) {
  double sum = 0.0;
  for (int k = 0; k < cnt; ++k) sum += std::fabs(a[k]);
  sum = sum * kTurnHi * 1.000001;  // and the roundings of cnt angles
  if (!(sum > 0.0)) return 0;
  const int shift = std::min(-1 - (int)std::ceil(std::log2(sum)), 60);
  return shift >= 2 ? shift : 0;
}

bool fixed_point_angle(double a) { return std::isfinite(a) && std::fabs(a) < 1.125899906842624e15; }

// z mask -> tile pattern and thread part (see DiagTiles)
template <typename R>
void split_mask(int n, uint64_t zm, int* rho, uint32_t* zt) {
  const int tb = n - (sizeof(R) == 4 ? 4 : 3);  // thread bits
  if (sizeof(R) == 4) {
    *rho = (int)((zm & 1) | (((zm >> (tb + 1)) & 7) << 1));
    *zt = (uint32_t)((zm >> 1) & ((uint64_t(1) << tb) - 1));
  } else {
    *rho = (int)((zm >> tb) & 7);
    *zt = (uint32_t)(zm & ((uint64_t(1) << tb) - 1));
  }
}

// exp(-i a_k P_k) for the diagonal strings zm[0..cnt) as tiles
template <typename R, int CAP>
void fill_tiles(int n, const uint64_t* zm, const double* a, int cnt, DiagTiles<R, CAP>* D) {
  constexpr int NT = DiagTiles<R, CAP>::NT;
  typedef typename Turn<R>::T F;
  const int shift = angle_shift(a, cnt);
  D->half = shift ? 0 : F(1) << (8 * sizeof(R) - 3);
  D->mask = shift ? 0 : F(3) << (8 * sizeof(R) - 2);
  D->unit = (R)std::ldexp(1.0, 1 - 8 * (int)sizeof(R) - shift);
  int pos = 0;
  for (int r = 0; r < NT; ++r) {
    D->start[r] = (uint16_t)pos;
    for (int k = 0; k < cnt; ++k) {
      int rho;
      uint32_t zt;
      split_mask<R>(n, zm[k], &rho, &zt);
      if (rho != r) continue;
      D->zt[pos] = zt;
      D->a[pos++] = turns<R>(a[k], shift);
    }
  }
  D->start[NT] = (uint16_t)pos;
}

template <typename R>
void run_tiles(const Target& s, const uint64_t* zm, const double* a, int cnt) {
  DiagTiles<R, kRunTerms> D;
  fill_tiles<R, kRunTerms>(s.n, zm, a, cnt, &D);
  const uint32_t T = uint32_t(1) << (s.n - (sizeof(R) == 4 ? 4 : 3));
  const unsigned threads = std::min<uint32_t>(T, kEThreads);
  launch_dependent(kdiag_run<R>, T / threads, threads, 0, s.stream,
                   (typename TurnVec<R>::T*)s.data, T, D);
}

// A run of commuting diagonal rotations exp(-i a_k P_k).
sv_status run_diags(const Target& s, const std::vector<uint64_t>& zm, const std::vector<double>& a) {
  if (zm.empty()) return SV_OK;
  if (zm.size() <= (size_t)(s.dt == SV_C64 ? kShearTermsF : kShearTerms)) {
    Shear h[kShearTerms];
    size_t k = 0;  // stops at an angle that is not finite
    while (k < zm.size() && make_shear(std::cos(a[k]), -std::sin(a[k]), &h[k])) ++k;
    if (k == zm.size()) {
      const uint64_t vecs = uint64_t(1) << (s.dt == SV_C64 ? s.n - 1 : s.n);
      const unsigned grid = (unsigned)((vecs + kEThreads * 4 - 1) / (kEThreads * 4));
      ProfScope prof(s.stream, s.dt == SV_C64 ? "kdiag_shears_c64" : "kdiag_shears_c128");
      if (s.dt == SV_C64) {
        DiagShearsF D{};
        for (; D.nt < (int)k; ++D.nt) {
          D.zm[D.nt] = zm[D.nt];
          D.h[D.nt] = round_shear(h[D.nt]);
        }
        launch_dependent(kdiag_shears_f, grid, kEThreads, 0, s.stream, (float4*)s.data, vecs, D);
      } else {
        DiagShears D{};
        for (; D.nt < (int)k; ++D.nt) {
          D.zm[D.nt] = zm[D.nt];
          D.h[D.nt] = h[D.nt];
        }
        launch_dependent(kdiag_shears, grid, kEThreads, 0, s.stream, (double2*)s.data, vecs, D);
      }
      g_launches.fetch_add(1, std::memory_order_relaxed);
      return check_launch("diagonal rotations kernel");
    }
  }
  bool tiles = s.n >= kRunMinQubits;
  for (double x : a) tiles = tiles && fixed_point_angle(x);
  if (!tiles) {
    DiagRun D{};
    for (size_t k = 0; k < zm.size(); ++k) {
      D.zm[D.nt] = zm[k];
      D.a[D.nt++] = a[k];
      if (D.nt == kMaxDiag || k + 1 == zm.size()) {
        sv_status st = run_diag(s, D);
        if (st) return st;
        D.nt = 0;
      }
    }
    return SV_OK;
  }
  for (size_t k = 0; k < zm.size(); k += kRunTerms) {
    const int cnt = (int)std::min<size_t>(kRunTerms, zm.size() - k);
    ProfScope prof(s.stream, s.dt == SV_C64 ? "kdiag_run_c64" : "kdiag_run_c128");
    if (s.dt == SV_C64)
      run_tiles<float>(s, zm.data() + k, a.data() + k, cnt);
    else
      run_tiles<double>(s, zm.data() + k, a.data() + k, cnt);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    sv_status st = check_launch("diagonal run kernel");
    if (st) return st;
  }
  return SV_OK;
}

template <typename R>
void run_adj_tiles(void* psi, void* lam, int n, cudaStream_t st, const DiagGate* g, int cnt,
                   double* partials, int pstride) {
  DiagTiles<R, kAdjTerms> D;
  uint64_t zm[kAdjTerms];
  double a[kAdjTerms];
  for (int k = 0; k < cnt; ++k) {
    zm[k] = g[k].zm;
    a[k] = -0.5 * g[k].theta;  // un-apply: exp(+i theta P / 2)
  }
  fill_tiles<R, kAdjTerms>(n, zm, a, cnt, &D);
  DiagGrads G;
  G.ns = 0;
  int pos = 0;
  for (int k = 0; k < cnt; ++k) {  // the first gate of every parameter, then its other gates
    bool first = g[k].slot >= 0;
    for (int j = 0; j < k && first; ++j) first = g[j].slot < 0 || g[j].param != g[k].param;
    if (!first) continue;
    G.slot[G.ns] = g[k].slot;
    G.sstart[G.ns++] = (uint16_t)pos;
    for (int j = k; j < cnt; ++j) {
      if (g[j].slot < 0 || g[j].param != g[k].param) continue;
      int rho;
      split_mask<R>(n, zm[j], &rho, &G.zt[pos]);
      G.rho[pos++] = (uint8_t)rho;
    }
  }
  G.sstart[G.ns] = (uint16_t)pos;
  constexpr int NT = DiagTiles<R, kAdjTerms>::NT;
  const uint32_t T = uint32_t(1) << (n - (sizeof(R) == 4 ? 4 : 3));
  const unsigned threads = std::min<uint32_t>(T, kEThreads);
  // two resident blocks per SM, several tiles per thread on larger states
  const unsigned grid = std::min({T / threads, 304u, (unsigned)pstride});
  const size_t smem = sizeof(R) * NT * threads + sizeof(CompSum<R>) * (threads / 32) * G.ns;
  launch_dependent(kadj_diag<R>, grid, threads, smem, st, (typename TurnVec<R>::T*)psi,
                   (typename TurnVec<R>::T*)lam, T, D, G, partials, pstride);
}

sv_status run_pair(const Target& s, uint64_t xm, uint64_t zm, double a) {
  int h = 63;
  while (!((xm >> h) & 1)) --h;
  const uint64_t lowmask = (uint64_t(1) << h) - 1;
  const uint64_t npairs = uint64_t(1) << (s.n - 1);
  const int ny = __builtin_popcountll(xm & zm) & 3;
  // coef = -i sin(a) i^{ny}
  const double sa = std::sin(a), ca = std::cos(a);
  double kr = 0, ki = 0;
  switch (ny) {
    case 0: ki = -sa; break;        // -i s
    case 1: kr = sa; break;         // -i s * i = s
    case 2: ki = sa; break;         // -i s * -1 = i s
    default: kr = -sa; break;       // -i s * -i = -s
  }
  const unsigned g = (unsigned)((npairs + kEThreads * 8 - 1) / (kEThreads * 8));
  ProfScope prof(s.stream, s.dt == SV_C64 ? "kpair_c64" : "kpair_c128");
  if (s.dt == SV_C64) {
    // c I + k P with P^2 = I scales ||psi||^2 by |c|^2 + |k|^2 on every
    // state: round with the state's error feedback
    double c32 = ca;
    cd k32{kr, ki};
    feedback_round_pair(&c32, &k32, s.rc ? &s.rc->drift : nullptr);
    launch_dependent(kpair<float, float2>, g, kEThreads, 0, s.stream, (float2*)s.data, npairs,
                     lowmask, xm, zm, (float)c32, (float)k32.re, (float)k32.im);
  } else {
    Shear h;
    if (!make_shear(ca, -sa, &h)) h = {ca, -sa, 0};  // not finite, and so the result
    const unsigned g4 = (unsigned)((npairs + kEThreads * 4 - 1) / (kEThreads * 4));
    launch_dependent((ny & 1) ? kpair_c128<true> : kpair_c128<false>, g4, kEThreads, 0, s.stream,
                     (double2*)s.data, npairs, lowmask, xm, zm, ny >> 1, h);
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return check_launch("pair rotation kernel");
}

// A run of single-qubit X and Y rotations as fused passes: up to 13 bits a
// pass instead of one.  Measured on the TFIM's transverse field (n rotations,
// 5 steps, complex64): n = 10 112 -> 72 us, n = 20 379 -> 147 us, n = 26 21.7 ->
// 4.8 ms; complex128 n = 22 8.9 -> 4.9 ms; below 10 qubits a pass has no
// bulk-copy geometry, and a run of one or two rotations is cheaper alone.
constexpr int kRunPassQubits = 10;
constexpr size_t kRunPassGates = 3;

sv_status run_1q(const Target& s, const std::vector<uint64_t>& xm, const std::vector<uint64_t>& zm,
                 const std::vector<double>& a, size_t k0, size_t k1) {
  std::vector<Gate1q> gates;
  for (size_t k = k0; k < k1; ++k) {
    const double c = std::cos(a[k]), sn = std::sin(a[k]);
    Gate1q g{__builtin_ctzll(xm[k]), {{c, 0}, {0, -sn}, {0, -sn}, {c, 0}}};  // c I - i s X
    if (zm[k]) {                                                            // c I - i s Y
      g.m[1] = {-sn, 0};
      g.m[2] = {sn, 0};
    }
    gates.push_back(g);
  }
  std::vector<FusionItem> plan;
  plan_fusion_1q(s.n, gates, fusion_config(s.n, s.dt, 4), &plan);
  for (FusionItem& it : plan) {
    it.pass.lift = true;
    sv_status st = launch_fused_pass(s.data, s.dt, s.n, s.stream, it.pass, s.rc);
    if (st) return st;
  }
  return SV_OK;
}

// Applies exp(-i a_k P_k) for the sequence (xm, zm, a): runs of consecutive
// diagonal strings in one pass, runs of single-qubit strings in fused passes,
// every other string in a pass of its own.
sv_status run_sequence(const Target& s, const std::vector<uint64_t>& xm,
                       const std::vector<uint64_t>& zm, const std::vector<double>& a) {
  const size_t K = xm.size();
  auto one_qubit = [&](size_t k) {
    return xm[k] && !(xm[k] & (xm[k] - 1)) && !(zm[k] & ~xm[k]) && std::isfinite(a[k]);
  };
  for (size_t k = 0; k < K;) {
    size_t e = k;
    sv_status st;
    if (xm[k] == 0) {
      while (e < K && xm[e] == 0) ++e;
      st = run_diags(s, {zm.begin() + k, zm.begin() + e}, {a.begin() + k, a.begin() + e});
    } else {
      while (s.n >= kRunPassQubits && e < K && one_qubit(e)) ++e;
      if (e - k >= kRunPassGates) {
        st = run_1q(s, xm, zm, a, k, e);
      } else {
        e = k + 1;
        st = run_pair(s, xm[k], zm[k], a[k]);
      }
    }
    if (st) return st;
    k = e;
  }
  return SV_OK;
}

}  // namespace

sv_status launch_pauli_rotation(void* data, sv_dtype dt, int n, cudaStream_t st, uint64_t xm,
                                uint64_t zm, double a, RoundCtx* rc) {
  return run_sequence({data, dt, n, st, rc}, {xm}, {zm}, {a});
}

sv_status launch_diag_rotations(void* data, sv_dtype dt, int n, cudaStream_t st,
                                const std::vector<uint64_t>& zm, const std::vector<double>& a) {
  return run_diags({data, dt, n, st, nullptr}, zm, a);
}

bool adjoint_diag_ok(int n, double theta) { return n >= kRunMinQubits && fixed_point_angle(theta); }

sv_status launch_adjoint_diag(void* psi, void* lam, sv_dtype dt, int n, cudaStream_t st,
                              const std::vector<DiagGate>& g, double* partials, int pstride) {
  for (size_t k = 0; k < g.size(); k += kAdjTerms) {
    const int cnt = (int)std::min<size_t>(kAdjTerms, g.size() - k);
    ProfScope prof(st, dt == SV_C64 ? "kadj_diag_c64" : "kadj_diag_c128");
    if (dt == SV_C64)
      run_adj_tiles<float>(psi, lam, n, st, g.data() + k, cnt, partials, pstride);
    else
      run_adj_tiles<double>(psi, lam, n, st, g.data() + k, cnt, partials, pstride);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    sv_status r = check_launch("adjoint diagonal run kernel");
    if (r) return r;
  }
  return SV_OK;
}

sv_status launch_adjoint_pauli(void* psi, void* lam, sv_dtype dt, int n, cudaStream_t st,
                               uint64_t xm, uint64_t zm, double theta, double* partials,
                               int* nparts) {
  // the same fixed grid as the 1-qubit adjoint kernels: every gate writes
  // the same number of partials
  const int grid = red_blocks(uint64_t(1) << (n >= 2 ? n - 2 : 0));
  const int ny = __builtin_popcountll(xm & zm) & 3;
  const double c = std::cos(0.5 * theta), sn = std::sin(0.5 * theta);
  const bool diag = xm == 0;
  uint64_t units = uint64_t(1) << n, lowmask = 0;
  if (!diag) {
    int h = 63;
    while (!((xm >> h) & 1)) --h;
    lowmask = (uint64_t(1) << h) - 1;
    units >>= 1;
  }
  ProfScope prof(st, dt == SV_C64 ? "kadj_pauli_c64" : "kadj_pauli_c128");
  // c I + i sin i^{ny} P: the un-applied rotation's angle is +theta / 2
  Shear h;
  if (!make_shear(c, sn, &h)) h = {c, sn, 0};  // not finite, and so the result
  if (dt == SV_C64) {
    const auto kern = diag       ? kadj_pauli<float, float2, 0>
                      : (ny & 1) ? kadj_pauli<float, float2, 2>
                                 : kadj_pauli<float, float2, 1>;
    launch_dependent(kern, grid, kEThreads, 0, st, (float2*)psi, (float2*)lam, units, lowmask, xm,
                     zm, ny >> 1, round_shear(h), partials);
  } else {
    const auto kern = diag       ? kadj_pauli<double, double2, 0>
                      : (ny & 1) ? kadj_pauli<double, double2, 2>
                                 : kadj_pauli<double, double2, 1>;
    launch_dependent(kern, grid, kEThreads, 0, st, (double2*)psi, (double2*)lam, units, lowmask, xm,
                     zm, ny >> 1, h, partials);
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if (nparts) *nparts = grid;
  return check_launch("adjoint Pauli rotation kernel");
}

}  // namespace sv

using namespace sv;

extern "C" {

sv_status sv_pauli_rotation(sv_state s, uint64_t xmask, uint64_t zmask, double theta) {
  if (!s || !s->data) {
    set_error("sv_pauli_rotation: null state");
    return SV_ERR_INVALID;
  }
  const uint64_t lim = (uint64_t(1) << s->n) - 1;
  if ((xmask | zmask) & ~lim || !std::isfinite(theta)) {
    set_error("sv_pauli_rotation: mask bits beyond %d qubits or non-finite angle", s->n);
    return SV_ERR_INVALID;
  }
  return run_sequence({s->data, s->dt, s->n, s->stream, &s->rc}, {xmask}, {zmask}, {theta});
}

sv_status sv_trotter(sv_state s, const sv_pauli_sum* H, double t, int steps, int order) {
  if (!s || !s->data || !H || H->n_terms < 0 || H->n_terms > SV_MAX_PAULI_TERMS ||
      (H->n_terms > 0 && (!H->xmask || !H->zmask || !H->coeff)) || steps < 1 ||
      (order != 1 && order != 2) || !std::isfinite(t)) {
    set_error("sv_trotter: bad arguments (steps >= 1, order 1 or 2)");
    return SV_ERR_INVALID;
  }
  const uint64_t lim = (uint64_t(1) << s->n) - 1;
  for (int k = 0; k < H->n_terms; ++k)
    if ((H->xmask[k] | H->zmask[k]) & ~lim) {
      set_error("sv_trotter: term %d has mask bits beyond %d qubits", k, s->n);
      return SV_ERR_INVALID;
    }
  const double dt = t / steps;
  std::vector<uint64_t> xm, zm;
  std::vector<double> a;
  for (int step = 0; step < steps; ++step) {
    if (order == 1) {
      for (int k = 0; k < H->n_terms; ++k) {
        xm.push_back(H->xmask[k]);
        zm.push_back(H->zmask[k]);
        a.push_back(H->coeff[k] * dt);
      }
    } else {
      for (int k = 0; k < H->n_terms; ++k) {
        xm.push_back(H->xmask[k]);
        zm.push_back(H->zmask[k]);
        a.push_back(0.5 * H->coeff[k] * dt);
      }
      for (int k = H->n_terms - 1; k >= 0; --k) {
        xm.push_back(H->xmask[k]);
        zm.push_back(H->zmask[k]);
        a.push_back(0.5 * H->coeff[k] * dt);
      }
    }
  }
  return run_sequence({s->data, s->dt, s->n, s->stream, &s->rc}, xm, zm, a);
}

}  // extern "C"
