// Batched energies and adjoint gradients in one persistent launch.
//
// Many small variational circuits (Sec. 3: variational layers, VQE) are
// evaluated together: thread blocks pull items (a circuit, its parameters and
// its Pauli-sum Hamiltonian) from an atomic queue and run each item to the
// end inside the block - the forward pass from |0...0>, lambda = H psi and
// E = <psi|lambda>, then the adjoint reverse sweep (dE/dtheta_j =
// Im<lambda|P_j|psi> before U_j is un-applied on both states).  The states
// stay in shared memory - small items side by side in one block, large ones over
// a cluster - or in the block's workspace slot of two states (2 x 2^nmax complex64),
// small enough to stay in L1/L2 while the block works on it.
//
// Gates are applied in register groups: the host list-schedules each
// circuit's gates into groups of at most k qubits; a thread pulls the 2^k
// amplitudes of a sub-block into registers, applies the group's gates in
// order (backward: their adjoints in reverse order) and writes them back, so
// the block synchronises once per group instead of once per gate.
//
// Precision: states and gate arithmetic in fp32; gate matrices from fp64
// sincos; the energy and every gradient accumulate per thread / per warp in
// compensated fp32 sums and across warps in fp64 (fixed order, so results
// repeat bit for bit; the two-block cluster kernel keeps fp64 slots).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include <cooperative_groups.h>

#include "sv_device.cuh"

namespace sv {
namespace {

constexpr int kBMaxGates = 480;    // gates of one circuit (static smem stays < 48 KB)
constexpr int kBMaxParams = 256;   // parameters of one circuit
constexpr int kBMaxTerms = 64;     // Pauli terms of one Hamiltonian
static_assert(SV_BATCH_MAX_QUBITS < 31, "term masks are packed in 31 bits");

struct BCirc {
  int n, ngates, gate0, ngroups, group0, nparams, nterms, term0;
  int ndiag;  // terms[term0 .. term0 + ndiag) are diagonal (no X or Y factor)
  // the single-block kernels' sign patterns rsigns[sign0 .. sign0 + nsign), rotations
  // rots[rot0 .. rot0 + nrot) and other gates gens[gen0 .. gen0 + ngen)
  int nsign, sign0, nrot, rot0, ngen, gen0;
};
struct BGateDesc {
  int kind;   // SV_GATE_* (1-qubit kinds)
  int param;  // -1: fixed angle
  double angle;
  int free_rot;  // RX, RY or RZ without controls
};
struct BRot {  // a rotation without controls in the single-block kernels' lists
  int kind, param;
  double angle;
};
// One size class of items: teams of `ts` threads, 512 / ts of them in a block at once,
// each with `stride` bytes of shared memory (byte offsets o_*, see BSmem).
struct BPhase {
  int first, count;  // items order[first .. first + count)
  int ts, stride;
  int o_mats, o_wpart, o_ops, o_grp, o_term, o_tcoef, o_sign, o_state;
  int pstride;       // gradient partials of one warp
  int state_floats;  // floats of state memory from o_state
};
constexpr int kBPhases = 4;
struct alignas(16) BGroup {
  uint8_t k, bits[5];
  int32_t op0, op1;
};
struct alignas(8) BOp {
  uint8_t b0;     // group-local target index
  uint8_t cm;     // group-local control mask
  uint8_t pauli;  // generator for gradients: 0 none, 1 X, 2 Y, 3 Z
  uint8_t cls;    // arithmetic class of the 2x2 matrix (BC_*)
  int16_t param;  // parameter index or -1
  int16_t gi;     // gate index within the circuit (matrix table slot)
};
struct BTerm {
  uint64_t xm, zm;
  double cre, cim;  // coefficient times i^{#Y}
};

struct BatchArgs {
  const BCirc* circs;
  const BGateDesc* gates;
  const BGroup* groups;
  const BOp* ops;
  const BTerm* terms;
  const BGroup* rgroups;   // the same groups over rops: the single-block kernels' lists
  const BOp* rops;
  const uint32_t* rsigns;
  const BRot* rots;
  const BGateDesc* gens;
  const int* order;      // items, longest first
  const int* item_circ;  // circuit of each item
  const int* theta_off;  // parameter offset of each item
  int n_items, nmax;
  const double* theta;
  double* energy;
  double* grad;
  float2* work;          // gridDim.x slots of 2 x 2^nmax amplitudes
  int* queue;
  int n_phases;
  BPhase phase[kBPhases], wide;  // queue[0 .. kBPhases), and queue[kBPhases] for the wide items
};

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__host__ __device__ constexpr int lowbit_b(int r) { return (r & 1) ? 0 : 1 + lowbit_b(r >> 1); }

// Compensated (Kahan) fp32 sum: GB300 issues fp64 instructions at a small
// fraction of the fp32 rate, so per-operation and per-amplitude additions
// stay in fp32 and only s - c enters the fp64 totals.
__device__ __forceinline__ void ksum_add(float2& a, float x) {  // a = (s, c)
  const float y = x - a.y;
  const float t = a.x + y;
  a.y = (t - a.x) - y;
  a.x = t;
}
__device__ __forceinline__ double ksum_value(float2 a) { return (double)a.x - (double)a.y; }

// Arithmetic classes of a gate's 2x2 matrix: the work per pair drops from 16
// multiply-adds (dense) to 8 (real: H, X, RY; imaginary off-diagonal: Y, RX;
// diagonal: RZ), to 4 on one amplitude (phase: U1) or to a sign flip (Z, CZ).
// The single-block kernels' lists also have BC_SIGN (a run of sign flips as one
// pattern, gi its index) and BC_RUN (cm rotations without controls from rotation gi on,
// bit 3 b + 0, 1, 2 of param for an RX, RY, RZ on group bit b, in that order).
enum { BC_DENSE = 0, BC_REAL = 1, BC_IMOFF = 2, BC_DIAG = 3, BC_PHASE = 4, BC_NEG = 5,
       BC_SIGN = 6, BC_RUN = 7 };

// (a, b) <- M (a, b) for every register pair on group bit B (with controls cm
// when CTRL).
template <int K, int B, int CLS, bool CTRL>
__device__ __forceinline__ void pair_apply_c(const float* M, int cm, float (&re)[1 << K],
                                             float (&im)[1 << K]) {
  const float g0r = M[0], g0i = M[1], g1r = M[2], g1i = M[3];
  const float g2r = M[4], g2i = M[5], g3r = M[6], g3i = M[7];
#pragma unroll
  for (int r = 0; r < (1 << K); ++r) {
    if (r & (1 << B)) continue;
    if (CTRL && (r & cm) != cm) continue;
    const int r1 = r | (1 << B);
    const float ar = re[r], ai = im[r], br = re[r1], bi = im[r1];
    if (CLS == BC_NEG) {
      re[r1] = -br;
      im[r1] = -bi;
    } else if (CLS == BC_PHASE) {
      re[r1] = g3r * br - g3i * bi;
      im[r1] = g3r * bi + g3i * br;
    } else if (CLS == BC_DIAG) {
      re[r] = g0r * ar - g0i * ai;
      im[r] = g0r * ai + g0i * ar;
      re[r1] = g3r * br - g3i * bi;
      im[r1] = g3r * bi + g3i * br;
    } else if (CLS == BC_REAL) {
      re[r] = g0r * ar + g1r * br;
      im[r] = g0r * ai + g1r * bi;
      re[r1] = g2r * ar + g3r * br;
      im[r1] = g2r * ai + g3r * bi;
    } else if (CLS == BC_IMOFF) {
      re[r] = g0r * ar - g1i * bi;
      im[r] = g0r * ai + g1i * br;
      re[r1] = g3r * br - g2i * ai;
      im[r1] = g3r * bi + g2i * ar;
    } else {
      re[r] = g0r * ar - g0i * ai + g1r * br - g1i * bi;
      im[r] = g0r * ai + g0i * ar + g1r * bi + g1i * br;
      re[r1] = g2r * ar - g2i * ai + g3r * br - g3i * bi;
      im[r1] = g2r * ai + g2i * ar + g3r * bi + g3i * br;
    }
  }
}

// controlled phase / sign flip with the control mask CM fixed at compile time
// (no per-register mask tests)
template <int K, int B, int CLS, int CM>
__device__ __forceinline__ void pair_apply_cm(const float* M, float (&re)[1 << K],
                                              float (&im)[1 << K]) {
  if constexpr ((CM >> B) & 1) {
    return;  // a mask holding the target bit selects no pair (as the runtime test)
  } else {
    const float g3r = M[6], g3i = M[7];
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) {
      if (r & (1 << B)) continue;
      if ((r & CM) != CM) continue;
      const int r1 = r | (1 << B);
      const float br = re[r1], bi = im[r1];
      if (CLS == BC_NEG) {
        re[r1] = -br;
        im[r1] = -bi;
      } else {
        re[r1] = g3r * br - g3i * bi;
        im[r1] = g3r * bi + g3i * br;
      }
    }
  }
}

template <int K, int B, int CLS>
__device__ __forceinline__ void pair_apply_ctrl(const float* M, int cm, float (&re)[1 << K],
                                                float (&im)[1 << K]) {
#define SV_CM_CASE(v)                                                       \
  case v:                                                                   \
    if constexpr (v < (1 << K)) pair_apply_cm<K, B, CLS, v>(M, re, im);     \
    break;
  switch (cm) {
    SV_CM_CASE(1) SV_CM_CASE(2) SV_CM_CASE(3) SV_CM_CASE(4) SV_CM_CASE(5)
    SV_CM_CASE(6) SV_CM_CASE(7) SV_CM_CASE(8) SV_CM_CASE(9) SV_CM_CASE(10)
    SV_CM_CASE(11) SV_CM_CASE(12) SV_CM_CASE(13) SV_CM_CASE(14) SV_CM_CASE(15)
    default: pair_apply_c<K, B, CLS, true>(M, cm, re, im); break;
  }
#undef SV_CM_CASE
}

template <int K, int B>
__device__ __forceinline__ void pair_apply(int cls, const float* M, int cm, float (&re)[1 << K],
                                           float (&im)[1 << K]) {
  if (cm) {
    switch (cls) {
      case BC_PHASE: pair_apply_ctrl<K, B, BC_PHASE>(M, cm, re, im); break;
      case BC_NEG: pair_apply_ctrl<K, B, BC_NEG>(M, cm, re, im); break;
      default: pair_apply_c<K, B, BC_DENSE, true>(M, cm, re, im); break;
    }
  } else {
    switch (cls) {
      case BC_REAL: pair_apply_c<K, B, BC_REAL, false>(M, 0, re, im); break;
      case BC_IMOFF: pair_apply_c<K, B, BC_IMOFF, false>(M, 0, re, im); break;
      case BC_DIAG: pair_apply_c<K, B, BC_DIAG, false>(M, 0, re, im); break;
      case BC_PHASE: pair_apply_c<K, B, BC_PHASE, false>(M, 0, re, im); break;
      case BC_NEG: pair_apply_c<K, B, BC_NEG, false>(M, 0, re, im); break;
      default: pair_apply_c<K, B, BC_DENSE, false>(M, 0, re, im); break;
    }
  }
}

// the adjoint of M (same arithmetic class) applied to the pairs
template <int K, int B>
__device__ __forceinline__ void pair_apply_dag(int cls, const float* M, int cm,
                                               float (&re)[1 << K], float (&im)[1 << K]) {
  // M^dagger = [[conj g0, conj g2], [conj g1, conj g3]]
  const float h[8] = {M[0], -M[1], M[4], -M[5], M[2], -M[3], M[6], -M[7]};
  pair_apply<K, B>(cls, h, cm, re, im);
}

// sum over the pairs of Im( conj(l0) (P p)_0 + conj(l1) (P p)_1 )
template <int K, int B, int PAULI, bool CTRL>
__device__ __forceinline__ float pair_grad_c(int cm, const float (&pr)[1 << K],
                                             const float (&pi)[1 << K], const float (&lr)[1 << K],
                                             const float (&li)[1 << K]) {
  float acc = 0.f;
#pragma unroll
  for (int r = 0; r < (1 << K); ++r) {
    if (r & (1 << B)) continue;
    const int r1 = r | (1 << B);
    if (CTRL && (r & cm) != cm) continue;
    const float p0r = pr[r], p0i = pi[r], p1r = pr[r1], p1i = pi[r1];
    const float l0r = lr[r], l0i = li[r], l1r = lr[r1], l1i = li[r1];
    if (PAULI == 1)
      acc += (l0r * p1i - l0i * p1r) + (l1r * p0i - l1i * p0r);
    else if (PAULI == 2)
      acc += -(l0r * p1r + l0i * p1i) + (l1r * p0r + l1i * p0i);
    else
      acc += (l0r * p0i - l0i * p0r) - (l1r * p1i - l1i * p1r);
  }
  return acc;
}

template <int K, int B>
__device__ __forceinline__ float pair_grad(int pauli, int cm, const float (&pr)[1 << K],
                                           const float (&pi)[1 << K], const float (&lr)[1 << K],
                                           const float (&li)[1 << K]) {
  if (cm) {
    switch (pauli) {
      case 1: return pair_grad_c<K, B, 1, true>(cm, pr, pi, lr, li);
      case 2: return pair_grad_c<K, B, 2, true>(cm, pr, pi, lr, li);
      default: return pair_grad_c<K, B, 3, true>(cm, pr, pi, lr, li);
    }
  }
  switch (pauli) {
    case 1: return pair_grad_c<K, B, 1, false>(0, pr, pi, lr, li);
    case 2: return pair_grad_c<K, B, 2, false>(0, pr, pi, lr, li);
    default: return pair_grad_c<K, B, 3, false>(0, pr, pi, lr, li);
  }
}

#define SV_BIT_SWITCH(B, CALL) \
  switch (B) {                 \
    case 0: CALL(0); break;    \
    case 1: CALL(1); break;    \
    case 2: CALL(2); break;    \
    default: CALL(3); break;   \
  }

template <int K>
__device__ void group_offsets(const BGroup& g, int (&off)[1 << K], int (&lm)[K]) {
  off[0] = 0;
#pragma unroll
  for (int r = 1; r < (1 << K); ++r) off[r] = off[r & (r - 1)] | (1 << g.bits[lowbit_b(r)]);
#pragma unroll
  for (int i = 0; i < K; ++i) lm[i] = (1 << g.bits[i]) - 1;
}

template <int K>
__device__ __forceinline__ int sub_base(int s, const int (&lm)[K], int kk) {
  int b = s;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (i < kk) b = ((b & ~lm[i]) << 1) | (b & lm[i]);
  return b;
}

template <int I, int N, typename F>
__device__ __forceinline__ void static_for(const F& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>());
    static_for<I + 1, N>(f);
  }
}

// Byte offsets and masks of a state split over a cluster carry the block's rank from here.
constexpr int kRankShift = 28;

// Slices of the index range that one thread of apply_terms takes.
__device__ __forceinline__ int term_slices(int n) { return n >= 10 ? 8 : 2; }

// ---- single-block items ------------------------------------------------------------
// An item's state is one plane of 2^n real parts and, when CX, a second plane of
// imaginary parts.  Batches made of real gates and terms run with one plane: H, X, Z, RY
// and their controlled forms map |0...0> to real states, and a Hamiltonian whose
// terms are real matrices (coefficient times i^{#Y} real, as for the
// transverse-field Ising model) maps a real state to a real lambda = H psi.  That
// is half the bytes and half the multiply-adds, and both states of an n = 14
// item (2 x 64 KiB) in shared memory.
//
// Storage order: amplitude x of a plane lives at swzr(x) = x ^ ((x >> 5) & 31),
// which spreads the 32 values of a 128-byte row over the row by the next five
// index bits (a bijection of [0, 2^n), linear over XOR): a warp whose lanes step
// over a register group's low bits reaches 32 banks.
//
// Register tile: pairs of group bit 0's values (group indices 2 p and 2 p + 1), so
// that the operations on the other bits are paired fp32 instructions whatever the
// group's place in memory.  A rotation without controls is three shears in place:
// RY x += a y, y += b x, x += a y with a = -tan(angle / 4) and b = sin(angle / 2), and
// RX the same between a and i b; the half angle is taken modulo pi (a sign of the
// whole state, which neither the energy nor a gradient sees) so that |a| <= 1.  RZ
// is the one phase e^{i angle} on the upper half (a phase of the whole state
// dropped).  A run of CZs is one multiplication by its sign pattern.  Per tile of 16 or
// 32 amplitudes a rotation costs 24 paired FMAs in place of 64 (RX, RY) or 128 (RZ)
// single ones: 768 parameter sets of the n = 11, 6-layer random layered circuit and 192
// mixed items 0.85 -> 0.66 ms, 1024 sets of the n = 14 real ansatz (10 layers) 3.3 -> 2.34.
__device__ __forceinline__ int swzr(int x) { return x ^ ((x >> 5) & 31); }

template <int K, bool CX>
struct Tile {
  Pair r[1 << (K - 1)], i[CX ? 1 << (K - 1) : 1];
};

// (a, b) <- [[g0, g1], [g2, g3]] (a, b) on the pairs of group bit B (inside the
// group-local control mask cm when CTRL); NEG: b <- -b
template <int K, int B, bool NEG, bool CTRL>
__device__ __forceinline__ void re_pairs(float g0, float g1, float g2, float g3, int cm,
                                         float (&v)[1 << K]) {
#pragma unroll
  for (int r = 0; r < (1 << K); ++r) {
    if (r & (1 << B)) continue;
    if (CTRL && (r & cm) != cm) continue;
    const int r1 = r | (1 << B);
    if (NEG) {
      v[r1] = -v[r1];
    } else {
      const float a = v[r], b = v[r1];
      v[r] = g0 * a + g1 * b;
      v[r1] = g2 * a + g3 * b;
    }
  }
}

// operation (cls BC_REAL or BC_NEG) with matrix M (8 floats, re/im) or, when
// DAG, its transpose
template <int K, int B, bool DAG>
__device__ __forceinline__ void re_apply(const BOp& op, const float* M, float (&v)[1 << K]) {
  if (op.cls == BC_NEG) {
    re_pairs<K, B, true, true>(0.f, 0.f, 0.f, 0.f, op.cm, v);
    return;
  }
  const float g0 = M[0], g1 = DAG ? M[4] : M[2], g2 = DAG ? M[2] : M[4], g3 = M[6];
  if (op.cm)
    re_pairs<K, B, false, true>(g0, g1, g2, g3, op.cm, v);
  else
    re_pairs<K, B, false, false>(g0, g1, g2, g3, 0, v);
}

template <int K, int B>
__device__ __forceinline__ float re_grad(int cm, const float (&p)[1 << K], const float (&l)[1 << K]) {
  float acc = 0.f;
#pragma unroll
  for (int r = 0; r < (1 << K); ++r) {
    if (r & (1 << B)) continue;
    if ((r & cm) != cm) continue;
    const int r1 = r | (1 << B);
    acc = fmaf(l[r1], p[r], acc);
    acc = fmaf(-l[r], p[r1], acc);
  }
  return acc;
}

template <int K>
__device__ __forceinline__ void unpack(const Pair (&v)[1 << (K - 1)], float (&w)[1 << K]) {
#pragma unroll
  for (int p = 0; p < (1 << (K - 1)); ++p) {
    const float2 x = lanes_of(v[p]);
    w[2 * p] = x.x;
    w[2 * p + 1] = x.y;
  }
}
template <int K>
__device__ __forceinline__ void repack(const float (&w)[1 << K], Pair (&v)[1 << (K - 1)]) {
#pragma unroll
  for (int p = 0; p < (1 << (K - 1)); ++p) v[p] = pair_of(w[2 * p], w[2 * p + 1]);
}

// x += a y, y += b x, x += a y on group bit B of one plane
template <int K, int B>
__device__ __forceinline__ void plane_rot(float a, float b, Pair (&v)[1 << (K - 1)]) {
  if constexpr (B == 0) {
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
      float2 x = lanes_of(v[p]);
      x.x = fmaf(a, x.y, x.x);
      x.y = fmaf(b, x.x, x.y);
      x.x = fmaf(a, x.y, x.x);
      v[p] = pair_of(x.x, x.y);
    }
  } else {
    const Pair pa = pair_both(a), pb = pair_both(b);
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
      if (p & (1 << (B - 1))) continue;
      const int q = p | (1 << (B - 1));
      pair_add(v[p], pa, v[q]);
      pair_add(v[q], pb, v[p]);
      pair_add(v[p], pa, v[q]);
    }
  }
}

// RX: the shears between a and y = i b, (re y, im y) = (-im b, re b)
template <int K, int B>
__device__ __forceinline__ void rx_rot(float a, float b, Tile<K, true>& t) {
  if constexpr (B == 0) {
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
      float2 r = lanes_of(t.r[p]), i = lanes_of(t.i[p]);
      r.x = fmaf(-a, i.y, r.x);
      i.x = fmaf(a, r.y, i.x);
      i.y = fmaf(-b, r.x, i.y);
      r.y = fmaf(b, i.x, r.y);
      r.x = fmaf(-a, i.y, r.x);
      i.x = fmaf(a, r.y, i.x);
      t.r[p] = pair_of(r.x, r.y);
      t.i[p] = pair_of(i.x, i.y);
    }
  } else {
    const Pair pa = pair_both(a), na = pair_both(-a), pb = pair_both(b), nb = pair_both(-b);
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
      if (p & (1 << (B - 1))) continue;
      const int q = p | (1 << (B - 1));
      pair_add(t.r[p], na, t.i[q]);
      pair_add(t.i[p], pa, t.r[q]);
      pair_add(t.i[q], nb, t.r[p]);
      pair_add(t.r[q], pb, t.i[p]);
      pair_add(t.r[p], na, t.i[q]);
      pair_add(t.i[p], pa, t.r[q]);
    }
  }
}

// RZ up to a phase of the whole state: the upper half times c + i s
template <int K, int B>
__device__ __forceinline__ void rz_rot(float c, float s, Tile<K, true>& t) {
  if constexpr (B == 0) {
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
      float2 r = lanes_of(t.r[p]), i = lanes_of(t.i[p]);
      const float u = c * r.y;
      const float w = c * i.y;
      i.y = fmaf(s, r.y, w);
      r.y = fmaf(-s, lanes_of(t.i[p]).y, u);
      t.r[p] = pair_of(r.x, r.y);
      t.i[p] = pair_of(i.x, i.y);
    }
  } else {
    const Pair pc = pair_both(c), ps = pair_both(s), ns = pair_both(-s);
#pragma unroll
    for (int q = 0; q < (1 << (K - 1)); ++q) {
      if (!(q & (1 << (B - 1)))) continue;
      const Pair r = t.r[q], i = t.i[q];
      t.r[q] = pair_mul(pc, r);
      pair_add(t.r[q], ns, i);
      t.i[q] = pair_mul(pc, i);
      pair_add(t.i[q], ps, r);
    }
  }
}

// Im <l|P|p> over the tile for a generator without controls: Y on one plane, and X
// and Z (and the other plane's part of Y) with both
template <int K, int B, bool CX>
__device__ __forceinline__ float tile_grad_y(const Tile<K, CX>& p, const Tile<K, CX>& l) {
  if constexpr (B == 0) {
    float x = 0.f, y = 0.f;
#pragma unroll
    for (int k = 0; k < (1 << (K - 1)); ++k) {
      const float2 u = lanes_of(p.r[k]), w = lanes_of(l.r[k]);
      x = fmaf(w.y, u.x, x);
      y = fmaf(w.x, u.y, y);
      if constexpr (CX) {
        const float2 v = lanes_of(p.i[k]), z = lanes_of(l.i[k]);
        x = fmaf(z.y, v.x, x);
        y = fmaf(z.x, v.y, y);
      }
    }
    return x - y;
  } else {
    Pair x = 0, y = 0;
#pragma unroll
    for (int k = 0; k < (1 << (K - 1)); ++k) {
      if (k & (1 << (B - 1))) continue;
      const int q = k | (1 << (B - 1));
      pair_add(x, l.r[q], p.r[k]);
      pair_add(y, l.r[k], p.r[q]);
      if constexpr (CX) {
        pair_add(x, l.i[q], p.i[k]);
        pair_add(y, l.i[k], p.i[q]);
      }
    }
    const float2 u = lanes_of(x), w = lanes_of(y);
    return (u.x - w.x) + (u.y - w.y);
  }
}
template <int K, int B>
__device__ __forceinline__ float tile_grad_x(const Tile<K, true>& p, const Tile<K, true>& l) {
  if constexpr (B == 0) {
    float x = 0.f, y = 0.f;
#pragma unroll
    for (int k = 0; k < (1 << (K - 1)); ++k) {
      const float2 pr = lanes_of(p.r[k]), pi = lanes_of(p.i[k]);
      const float2 lr = lanes_of(l.r[k]), li = lanes_of(l.i[k]);
      x = fmaf(lr.x, pi.y, x);
      y = fmaf(li.x, pr.y, y);
      x = fmaf(lr.y, pi.x, x);
      y = fmaf(li.y, pr.x, y);
    }
    return x - y;
  } else {
    Pair x = 0, y = 0;
#pragma unroll
    for (int k = 0; k < (1 << (K - 1)); ++k) {
      if (k & (1 << (B - 1))) continue;
      const int q = k | (1 << (B - 1));
      pair_add(x, l.r[k], p.i[q]);
      pair_add(y, l.i[k], p.r[q]);
      pair_add(x, l.r[q], p.i[k]);
      pair_add(y, l.i[q], p.r[k]);
    }
    const float2 u = lanes_of(x), w = lanes_of(y);
    return (u.x - w.x) + (u.y - w.y);
  }
}
template <int K, int B>
__device__ __forceinline__ float tile_grad_z(const Tile<K, true>& p, const Tile<K, true>& l) {
  // x: l_r p_i, y: l_i p_r, the lower half's minus the upper half's
  Pair x0 = 0, y0 = 0, x1 = 0, y1 = 0;
#pragma unroll
  for (int k = 0; k < (1 << (K - 1)); ++k) {
    const bool up = B > 0 && (k & (1 << (B > 0 ? B - 1 : 0)));
    pair_add(up ? x1 : x0, l.r[k], p.i[k]);
    pair_add(up ? y1 : y0, l.i[k], p.r[k]);
  }
  const float2 a = lanes_of(x0), b = lanes_of(y0);
  if constexpr (B == 0) {
    return (a.x - b.x) - (a.y - b.y);
  } else {
    const float2 c = lanes_of(x1), d = lanes_of(y1);
    return ((a.x - b.x) + (a.y - b.y)) - ((c.x - d.x) + (c.y - d.y));
  }
}

// Four (eight) values summed over the warp with 6 (9) shuffles in place of 20 (40): a
// lane ends with the sum of value lane >> 3 (lane >> 2).
__device__ __forceinline__ float reduce2(float c0, float c1, int lane, int bit) {
  const bool up = lane & bit;
  return (up ? c1 : c0) + __shfl_xor_sync(0xffffffffu, up ? c0 : c1, bit);
}
__device__ __forceinline__ float reduce4(float c0, float c1, float c2, float c3, int lane) {
  float v = reduce2(reduce2(c0, c2, lane, 16), reduce2(c1, c3, lane, 16), lane, 8);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v + __shfl_xor_sync(0xffffffffu, v, 1);
}
// A run of rotations R[0 .. ), (a, b, parameter) each, in order (bit, kind) as `mask` says:
// straight-line code with a skip per absent one, in place of a dispatch, a jump
// and a warp sum of its own for each.
template <int K, bool CX>
__device__ __forceinline__ void run_fwd(const float4* R, int mask, Tile<K, CX>& t) {
  static_for<0, K>([&](auto bb) {
    constexpr int B = decltype(bb)::value;
    if constexpr (CX) {
      if ((mask >> (3 * B)) & 1) {
        const float2 r = *reinterpret_cast<const float2*>(R++);
        rx_rot<K, B>(r.x, r.y, t);
      }
    }
    if ((mask >> (3 * B + 1)) & 1) {
      const float2 r = *reinterpret_cast<const float2*>(R++);
      plane_rot<K, B>(r.x, r.y, t.r);
      if constexpr (CX) plane_rot<K, B>(r.x, r.y, t.i);
    }
    if constexpr (CX) {
      if ((mask >> (3 * B + 2)) & 1) {
        const float2 r = *reinterpret_cast<const float2*>(R++);
        rz_rot<K, B>(r.x, r.y, t);
      }
    }
  });
}

// Backward over the same run (R one past its last): each rotation's gradient, added to
// this warp's partials, then its inverse on both tiles.  No parameter occurs
// twice in a run, so the lanes add to different partials.
template <int K, bool CX>
__device__ __forceinline__ void run_bwd(const float4* R, int mask, Tile<K, CX>& p, Tile<K, CX>& l,
                                        float2* part) {
  const int lane = threadIdx.x & 31;
  const auto add = [&](const float4* r, float c) {
    const int param = __float_as_int(r->z);
    if (param >= 0) ksum_add(part[param], c);
  };
  static_for<0, K>([&](auto bb) {
    constexpr int B = K - 1 - decltype(bb)::value;
    if constexpr (CX) {
      const int m = (mask >> (3 * B)) & 7;
      if (m) {
        float x = 0.f, y = 0.f, z = 0.f;
        if (m & 4) {
          const float2 r = *reinterpret_cast<const float2*>(--R);
          z = tile_grad_z<K, B>(p, l);
          rz_rot<K, B>(r.x, -r.y, p);
          rz_rot<K, B>(r.x, -r.y, l);
        }
        if (m & 2) {
          const float2 r = *reinterpret_cast<const float2*>(--R);
          y = tile_grad_y<K, B, CX>(p, l);
          plane_rot<K, B>(-r.x, -r.y, p.r);
          plane_rot<K, B>(-r.x, -r.y, p.i);
          plane_rot<K, B>(-r.x, -r.y, l.r);
          plane_rot<K, B>(-r.x, -r.y, l.i);
        }
        if (m & 1) {
          const float2 r = *reinterpret_cast<const float2*>(--R);
          x = tile_grad_x<K, B>(p, l);
          rx_rot<K, B>(-r.x, -r.y, p);
          rx_rot<K, B>(-r.x, -r.y, l);
        }
        const float v = reduce4(x, y, z, 0.f, lane);
        const int k = lane >> 3;
        if ((lane & 7) == 0 && ((m >> k) & 1)) add(R + __popc(m & ((1 << k) - 1)), v);
      }
    } else {
      if ((mask >> (3 * B + 1)) & 1) {
        const float2 r = *reinterpret_cast<const float2*>(--R);
        float c = tile_grad_y<K, B, CX>(p, l);
        c = warp_sum_f(c);
        plane_rot<K, B>(-r.x, -r.y, p.r);
        plane_rot<K, B>(-r.x, -r.y, l.r);
        if (lane == 0) add(R, c);
      }
    }
  });
}

template <int K, bool CX>
__device__ __forceinline__ void tile_signs(const float* sg, Tile<K, CX>& t) {
  const Pair* s = reinterpret_cast<const Pair*>(sg);
#pragma unroll
  for (int p = 0; p < (1 << (K - 1)); ++p) {
    t.r[p] = pair_mul(s[p], t.r[p]);
    if constexpr (CX) t.i[p] = pair_mul(s[p], t.i[p]);
  }
}
template <int K, bool CX>
__device__ __forceinline__ void tile_signs2(const float* sg, Tile<K, CX>& t, Tile<K, CX>& u) {
  const Pair* s = reinterpret_cast<const Pair*>(sg);
#pragma unroll
  for (int p = 0; p < (1 << (K - 1)); ++p) {
    const Pair x = s[p];
    t.r[p] = pair_mul(x, t.r[p]);
    u.r[p] = pair_mul(x, u.r[p]);
    if constexpr (CX) {
      t.i[p] = pair_mul(x, t.i[p]);
      u.i[p] = pair_mul(x, u.i[p]);
    }
  }
}

#define SV_TILE_BITS(B, CALL) \
  switch (B) {                \
    case 0: CALL(0); break;   \
    case 1: CALL(1); break;   \
    case 2: CALL(2); break;   \
    case 3: CALL(3); break;   \
    default: CALL(4); break;  \
  }

// any other operation, on the tile as single values
template <int K, bool CX, bool DAG>
__device__ __forceinline__ void tile_other(const BOp& op, const float* M, Tile<K, CX>& t) {
  float w[1 << K];
  unpack<K>(t.r, w);
  if constexpr (CX) {
    float u[1 << K];
    unpack<K>(t.i, u);
#define SV_OTHER(BB)                                                   \
  if constexpr (BB < K) {                                              \
    if constexpr (DAG)                                                 \
      pair_apply_dag<K, BB>(op.cls, M, op.cm, w, u);                   \
    else                                                               \
      pair_apply<K, BB>(op.cls, M, op.cm, w, u);                       \
  }
    SV_TILE_BITS(op.b0, SV_OTHER)
#undef SV_OTHER
    repack<K>(u, t.i);
  } else {
#define SV_OTHER(BB) \
  if constexpr (BB < K) re_apply<K, BB, DAG>(op, M, w)
    SV_TILE_BITS(op.b0, SV_OTHER)
#undef SV_OTHER
  }
  repack<K>(w, t.r);
}

// the gradient of a controlled rotation
template <int K, bool CX>
__device__ __forceinline__ float tile_other_grad(const BOp& op, const Tile<K, CX>& p,
                                                 const Tile<K, CX>& l) {
  float u[1 << K], w[1 << K], c = 0.f;
  unpack<K>(p.r, u);
  unpack<K>(l.r, w);
  if constexpr (CX) {
    float v[1 << K], z[1 << K];
    unpack<K>(p.i, v);
    unpack<K>(l.i, z);
#define SV_OTHER(BB) \
  if constexpr (BB < K) c = pair_grad<K, BB>(op.pauli, op.cm, u, v, w, z)
    SV_TILE_BITS(op.b0, SV_OTHER)
#undef SV_OTHER
  } else {
#define SV_OTHER(BB) \
  if constexpr (BB < K) c = re_grad<K, BB>(op.cm, u, w)
    SV_TILE_BITS(op.b0, SV_OTHER)
#undef SV_OTHER
  }
  return c;
}

// A group's places: pl.step[i] the byte offset of its bit i in storage order (XORed), pl.low
// the bits' low masks.
template <int K>
struct Places {
  int step[K], low[K];
};
template <int K>
__device__ __forceinline__ Places<K> group_places(const BGroup& g) {
  Places<K> pl;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    pl.step[i] = swzr(1 << g.bits[i]) * (int)sizeof(float);
    pl.low[i] = (1 << g.bits[i]) - 1;
  }
  return pl;
}

// Tile s of the group, in Gray-code order: one XOR an address, and no table of
// 2^K offsets to keep in registers across the operations.
template <int K, bool CX>
__device__ __forceinline__ void tile_load(const float* st, int s, const Places<K>& pl, int plane,
                                          Tile<K, CX>& t) {
  int b = swzr(sub_base<K>(s, pl.low, K)) * (int)sizeof(float);
  const char* re = reinterpret_cast<const char*>(st);
  const char* im = reinterpret_cast<const char*>(st + plane);
#pragma unroll
  for (int k = 0; k < (1 << (K - 1)); ++k) {
    const int p = k ^ (k >> 1);
    if (k) b ^= pl.step[1 + lowbit_b(k)];
    const int c = b ^ pl.step[0];
    t.r[p] = pair_of(*reinterpret_cast<const float*>(re + b), *reinterpret_cast<const float*>(re + c));
    if constexpr (CX)
      t.i[p] =
          pair_of(*reinterpret_cast<const float*>(im + b), *reinterpret_cast<const float*>(im + c));
  }
}
template <int K, bool CX>
__device__ __forceinline__ void tile_store(float* st, int s, const Places<K>& pl, int plane,
                                           const Tile<K, CX>& t) {
  int b = swzr(sub_base<K>(s, pl.low, K)) * (int)sizeof(float);
  char* re = reinterpret_cast<char*>(st);
  char* im = reinterpret_cast<char*>(st + plane);
#pragma unroll
  for (int k = 0; k < (1 << (K - 1)); ++k) {
    const int p = k ^ (k >> 1);
    if (k) b ^= pl.step[1 + lowbit_b(k)];
    const int c = b ^ pl.step[0];
    const float2 v = lanes_of(t.r[p]);
    *reinterpret_cast<float*>(re + b) = v.x;
    *reinterpret_cast<float*>(re + c) = v.y;
    if constexpr (CX) {
      const float2 w = lanes_of(t.i[p]);
      *reinterpret_cast<float*>(im + b) = w.x;
      *reinterpret_cast<float*>(im + c) = w.y;
    }
  }
}

// The threads that run one item: all of the block, or a power of two of its warps.
struct Team {
  int tid, n, bar;  // thread of the team, threads, named barrier
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(n) : "memory");
  }
};

// Per team: the item's rotations, gate matrices, operations, groups, terms and sign
// patterns, and per-warp gradient sums, in dynamic shared memory sized by the
// phase's items.
struct BSmem {
  unsigned char* mem;
  const BPhase& P;
  // (a, b, parameter)
  __device__ __forceinline__ float4* rot() const { return reinterpret_cast<float4*>(mem); }
  // 8 floats a gate
  __device__ __forceinline__ float* mats() const { return at<float>(P.o_mats); }
  // per warp and parameter: (sum, compensation)
  __device__ __forceinline__ float2* wpart() const { return at<float2>(P.o_wpart); }
  __device__ __forceinline__ BOp* ops() const { return at<BOp>(P.o_ops); }
  __device__ __forceinline__ BGroup* grp() const { return at<BGroup>(P.o_grp); }
  // (swzr(x mask's local bits) | the others << kRankShift, z mask | (an odd number of Y) << 31)
  __device__ __forceinline__ int2* term() const { return at<int2>(P.o_term); }
  // 8 a term: the coefficient times the sign of slice j's high bits
  __device__ __forceinline__ float* tcoef() const { return at<float>(P.o_tcoef); }
  // patterns of 2^K values
  __device__ __forceinline__ float* sign() const { return at<float>(P.o_sign); }
  template <typename T>
  __device__ __forceinline__ T* at(int o) const {
    return reinterpret_cast<T*>(mem + o);
  }
};

// the group's operations on a tile; backward, on both tiles, each after its gradient
template <int K, bool CX>
__device__ __forceinline__ void tile_fwd(const BGroup& g, const BSmem& S, Tile<K, CX>& t) {
  for (int o = g.op0; o < g.op1; ++o) {
    const BOp op = S.ops()[o];
    if (op.cls == BC_RUN)
      run_fwd<K, CX>(S.rot() + op.gi, op.param, t);
    else if (op.cls == BC_SIGN)
      tile_signs<K, CX>(S.sign() + (op.gi << K), t);
    else
      tile_other<K, CX, false>(op, S.mats() + 8 * op.gi, t);
  }
}
template <int K, bool CX>
__device__ __forceinline__ void tile_bwd(const BGroup& g, const BSmem& S, float2* part,
                                         Tile<K, CX>& p, Tile<K, CX>& l) {
  const int lane = threadIdx.x & 31;
  for (int o = g.op1 - 1; o >= g.op0; --o) {
    const BOp op = S.ops()[o];
    if (op.cls == BC_RUN) {
      run_bwd<K, CX>(S.rot() + op.gi + op.cm, op.param, p, l, part);
    } else if (op.cls == BC_SIGN) {
      tile_signs2<K, CX>(S.sign() + (op.gi << K), p, l);
    } else {
      if (op.pauli) {
        const float c = warp_sum_f(tile_other_grad<K, CX>(op, p, l));
        if (lane == 0) ksum_add(part[op.param], c);
      }
      tile_other<K, CX, true>(op, S.mats() + 8 * op.gi, p);
      tile_other<K, CX, true>(op, S.mats() + 8 * op.gi, l);
    }
    __syncwarp();  // a warp's next partials may be another lane's
  }
}

// forward: psi <- group ops in order
template <int K, bool CX>
__device__ __forceinline__ void group_fwd(float* psi, int np, const BGroup& g, const BSmem& S,
                                          const Team& T) {
  const int nsub = 1 << (np - K);
  for (int s = T.tid; s < nsub; s += T.n) {
    Tile<K, CX> t;
    tile_load<K, CX>(psi, s, group_places<K>(g), 1 << np, t);
    tile_fwd<K, CX>(g, S, t);
    asm volatile("" ::: "memory");  // the places are read again, not kept
    tile_store<K, CX>(psi, s, group_places<K>(g), 1 << np, t);
  }
}

// backward: for ops in reverse, gradient contribution then un-apply on both
template <int K, bool CX>
__device__ __forceinline__ void group_bwd(float* psi, float* lam, int np, int pstride,
                                          const BGroup& g, const BSmem& S, const Team& T) {
  const int nsub = 1 << (np - K);
  const int lane = T.tid & 31;
  float2* const part = S.wpart() + (T.tid >> 5) * pstride;
  // every lane of a warp runs the same number of iterations (warp sums)
  for (int s0 = T.tid - lane; s0 < nsub; s0 += T.n) {
    const int s = s0 + lane;
    const bool live = s < nsub;
    Tile<K, CX> p, l;
    if (live) {
      const Places<K> pl = group_places<K>(g);
      tile_load<K, CX>(psi, s, pl, 1 << np, p);
      tile_load<K, CX>(lam, s, pl, 1 << np, l);
    } else {
      p = {};
      l = {};
    }
    tile_bwd<K, CX>(g, S, part, p, l);
    asm volatile("" ::: "memory");  // the places are read again, not kept
    if (live) {
      const Places<K> pl = group_places<K>(g);
      tile_store<K, CX>(psi, s, pl, 1 << np, p);
      tile_store<K, CX>(lam, s, pl, 1 << np, l);
    }
  }
}

// lambda = H psi and this thread's part of E = Re <psi|lambda>.  A thread takes the J
// amplitudes x0 + j 2^n / J, so that a term's sign is one parity of x0 times
// a sign of j that the whole block shares (in tcoef): 2^14 amplitudes with
// 27 terms took about a fifth of a real item's instructions with a parity per
// amplitude and term.
// SPLIT: psi and lam are rank `rank`'s quarter of a cluster's states, nloc = n - 2.
template <int J, bool CX, bool SPLIT = false>
__device__ __forceinline__ void apply_terms(const float* psi, float* lam, const BCirc& C, int nloc,
                                            int np, int rank, const BSmem& S, const Team& T,
                                            float2& ek) {
  const int d = (1 << nloc) / J, plane = 1 << np;
  int off[J];
#pragma unroll
  for (int j = 0; j < J; ++j) off[j] = swzr(j * d);
  for (int x0 = T.tid; x0 < d; x0 += T.n) {
    const int p0 = swzr(x0);
    Pair dg[J / 2], ar[J / 2], ai[CX ? J / 2 : 1], sr[J / 2], si[CX ? J / 2 : 1];
#pragma unroll
    for (int k = 0; k < J / 2; ++k) {
      dg[k] = 0;
      const float* x = psi + (p0 ^ off[2 * k]);
      const float* y = psi + (p0 ^ off[2 * k + 1]);
      ar[k] = pair_of(*x, *y);
      if constexpr (CX) ai[k] = pair_of(x[plane], y[plane]);
    }
    for (int t = 0; t < C.ndiag; ++t) {
      const Pair sg = pair_both(__popc((x0 | (rank << nloc)) & S.term()[t].y) & 1 ? -1.f : 1.f);
      const Pair* cf = reinterpret_cast<const Pair*>(S.tcoef() + 8 * t);
#pragma unroll
      for (int k = 0; k < J / 2; ++k) pair_add(dg[k], sg, cf[k]);
    }
#pragma unroll
    for (int k = 0; k < J / 2; ++k) {
      sr[k] = pair_mul(dg[k], ar[k]);
      if constexpr (CX) si[k] = pair_mul(dg[k], ai[k]);
    }
    for (int t = C.ndiag; t < C.nterms; ++t) {
      const int2 q = S.term()[t];
      const int odd = __popc((x0 | (rank << nloc)) & q.y) & 1;
      const Pair sg = pair_both(odd ? -1.f : 1.f);
      const Pair* cf = reinterpret_cast<const Pair*>(S.tcoef() + 8 * t);
      const int pt = p0 ^ (q.x & ((1 << kRankShift) - 1));
      const float* from = psi;
      if constexpr (SPLIT) {
        const int flip = q.x >> kRankShift;
        if (flip)
          from = cooperative_groups::this_cluster().map_shared_rank(const_cast<float*>(psi),
                                                                    rank ^ flip);
      }
#pragma unroll
      for (int k = 0; k < J / 2; ++k) {
        const Pair w = pair_mul(sg, cf[k]);
        const float* x = from + (pt ^ off[2 * k]);
        const float* y = from + (pt ^ off[2 * k + 1]);
        const Pair br = pair_of(*x, *y);
        if constexpr (CX) {
          const Pair bi = pair_of(x[plane], y[plane]);
          if (q.y < 0) {  // an odd number of Y factors: i times real
            pair_add(sr[k], pair_mul(pair_both(-1.f), w), bi);
            pair_add(si[k], w, br);
          } else {
            pair_add(sr[k], w, br);
            pair_add(si[k], w, bi);
          }
        } else {
          pair_add(sr[k], w, br);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < J / 2; ++k) {
      float* x = lam + (p0 ^ off[2 * k]);
      float* y = lam + (p0 ^ off[2 * k + 1]);
      const float2 o = lanes_of(sr[k]), a = lanes_of(ar[k]);
      *x = o.x;
      *y = o.y;
      float e0 = a.x * o.x, e1 = a.y * o.y;
      if constexpr (CX) {
        const float2 oi = lanes_of(si[k]), aa = lanes_of(ai[k]);
        x[plane] = oi.x;
        y[plane] = oi.y;
        e0 = fmaf(aa.x, oi.x, e0);
        e1 = fmaf(aa.y, oi.y, e1);
      }
      ksum_add(ek, e0);
      ksum_add(ek, e1);
    }
  }
}

// forward pass, lambda and the reverse sweep of one item; returns this thread's energy
template <int K, bool CX>
__device__ __forceinline__ double run_item(float* psi, float* lam, const BCirc& C, int pstride,
                                           const BSmem& S, const Team& T) {
  const int np = max(C.n, K);
  // |0...0>: swzr(0) = 0 and swzr maps every other index to a nonzero one
  for (int x = T.tid; x < ((CX ? 2 : 1) << np); x += T.n) psi[x] = x == 0 ? 1.f : 0.f;
  if (C.n < K)  // the tile is wider than the state: what lies beyond stays zero
    for (int x = T.tid; x < ((CX ? 2 : 1) << np); x += T.n) lam[x] = 0.f;
  T.sync();
  for (int gg = 0; gg < C.ngroups; ++gg) {
    group_fwd<K, CX>(psi, np, S.grp()[gg], S, T);
    T.sync();
  }
  float2 ek = make_float2(0.f, 0.f);
  if (term_slices(C.n) == 8)
    apply_terms<8, CX>(psi, lam, C, C.n, np, 0, S, T, ek);
  else
    apply_terms<2, CX>(psi, lam, C, C.n, np, 0, S, T, ek);
  T.sync();
  for (int gg = C.ngroups - 1; gg >= 0; --gg) {
    group_bwd<K, CX>(psi, lam, np, pstride, S.grp()[gg], S, T);
    T.sync();
  }
  return ksum_value(ek);
}

// An item's rotations, matrices, lists and terms into the team's shared memory, and its
// partials to zero.  nloc: qubits of the state that one block holds.
template <int K>
__device__ __forceinline__ void load_item(const BatchArgs& A, const BPhase& P, const BCirc& C,
                                          const double* th, int nloc, const BSmem& S,
                                          const Team& T) {
  // rotations and gate matrices (fp64 trigonometry, rounded once), zero partials
  for (int i = T.tid; i < C.nrot; i += T.n) {
    const BRot d = A.rots[C.rot0 + i];
    const double a = d.param >= 0 ? th[d.param] : d.angle;
    double s, c;
    sincos(d.kind == SV_GATE_RZ ? a : 0.5 * a, &s, &c);
    if (d.kind == SV_GATE_RZ) {
      S.rot()[i] = make_float4((float)c, (float)s, __int_as_float(d.param), 0.f);
    } else {
      if (c < 0) {
        c = -c;
        s = -s;
      }
      S.rot()[i] = make_float4((float)(-s / (1.0 + c)), (float)s, __int_as_float(d.param), 0.f);
    }
  }
  for (int i = T.tid; i < C.ngen; i += T.n) {
    const BGateDesc d = A.gens[C.gen0 + i];
    const double a = d.param >= 0 ? th[d.param] : d.angle;
    double s, c;
    sincos(d.kind == SV_GATE_U1 ? a : 0.5 * a, &s, &c);
    double m[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const double r2 = 0.70710678118654752440;
    switch (d.kind) {
      case SV_GATE_H: m[0] = r2; m[2] = r2; m[4] = r2; m[6] = -r2; break;
      case SV_GATE_X: m[2] = 1; m[4] = 1; break;
      case SV_GATE_Y: m[3] = -1; m[5] = 1; break;
      case SV_GATE_Z: m[0] = 1; m[6] = -1; break;
      case SV_GATE_RX: m[0] = c; m[3] = -s; m[5] = -s; m[6] = c; break;
      case SV_GATE_RY: m[0] = c; m[2] = -s; m[4] = s; m[6] = c; break;
      case SV_GATE_RZ: m[0] = c; m[1] = -s; m[6] = c; m[7] = s; break;
      default: m[0] = 1; m[6] = c; m[7] = s;  // U1: diag(1, e^{ia})
    }
    for (int e = 0; e < 8; ++e) S.mats()[8 * i + e] = (float)m[e];
  }
  for (int i = T.tid; i < (T.n >> 5) * P.pstride; i += T.n) S.wpart()[i] = make_float2(0.f, 0.f);
  {  // this item's groups and operations, operation indices rebased to the cache
    const int ng = C.ngroups;
    const int op_base = ng ? A.rgroups[C.group0].op0 : 0;
    const int nops = ng ? A.rgroups[C.group0 + ng - 1].op1 - op_base : 0;
    for (int i = T.tid; i < nops; i += T.n) S.ops()[i] = A.rops[op_base + i];
    for (int i = T.tid; i < (C.nsign << K); i += T.n)
      S.sign()[i] = (A.rsigns[C.sign0 + (i >> K)] >> (i & ((1 << K) - 1))) & 1 ? -1.f : 1.f;
    for (int i = T.tid; i < ng; i += T.n) {
      BGroup G = A.rgroups[C.group0 + i];
      G.op0 -= op_base;
      G.op1 -= op_base;
      for (int k = G.k; k < K; ++k) G.bits[k] = (uint8_t)k;  // n < K: the group is the state
      S.grp()[i] = G;
    }
    const int js = term_slices(nloc), dlog = nloc - (js == 8 ? 3 : 1);
    for (int t = T.tid; t < C.nterms; t += T.n) {
      const BTerm M = A.terms[C.term0 + t];
      const int xm = (int)M.xm, zm = (int)M.zm;  // n <= SV_BATCH_MAX_QUBITS < 30
      const bool imag = __popc(xm & zm) & 1;     // i^{#Y} imaginary
      S.term()[t] = make_int2(swzr(xm & ((1 << nloc) - 1)) | ((xm >> nloc) << kRankShift),
                              (int)((unsigned)zm | ((unsigned)imag << 31)));
      // sign at x: the parity of (x ^ xm) & zm
      const float c = (float)(imag ? -M.cim : M.cre);
      for (int j = 0; j < 8; ++j)
        S.tcoef()[8 * t + j] = __popc((j << dlog) & zm) & 1 ? -c : c;
    }
  }
}

// SMS: one block of 512 threads an SM that works through the size classes from
// the largest.  2^K amplitudes a thread make a group of an n-qubit item one round of
// 2^(n - K) threads: items of that size class run side by side in teams of as many,
// each with its own barrier, and 512 threads' tiles of two states just fill
// 128 KiB of shared memory whatever the size.  With one team of 256 threads an item
// of 11 qubits left half of its warps at the barriers (4 of 11 stalled cycles
// an instruction): 768 items of 11 qubits and 192 mixed 0.66 -> 0.41 ms, 740 of 10
// qubits and 40 mixed 0.51 -> 0.22 ms.  Otherwise one size class and one team, states in global memory.
template <int K, int MAXT, int MINB, bool CX, bool SMS>
__global__ void __launch_bounds__(MAXT, MINB) kbatch(const BatchArgs A) {
  __shared__ double red[MAXT / 32];
  __shared__ int s_item[8];
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* const gpsi = reinterpret_cast<float*>(A.work + (size_t)blockIdx.x * (size_t(2) << A.nmax));
  float* const glam = gpsi + (size_t(2) << A.nmax);
  for (int ph = 0; ph < A.n_phases; ++ph) {
    const BPhase& P = A.phase[ph];
    const int team = (int)threadIdx.x / P.ts;
    const Team T = {(int)threadIdx.x - team * P.ts, P.ts, 1 + team};
    unsigned char* const mem = dyn_smem + team * P.stride;
    const BSmem S = {mem, P};
    float* const dyn_state = reinterpret_cast<float*>(mem + P.o_state);
    const int nwarps = P.ts >> 5;
    while (true) {
      if (T.tid == 0) s_item[team] = atomicAdd(A.queue + ph, 1);
      T.sync();
      const int slot = s_item[team];
      if (slot >= P.count) break;
      const int item = A.order[P.first + slot];
      const BCirc C = A.circs[A.item_circ[item]];
      const double* th = A.theta + A.theta_off[item];
      load_item<K>(A, P, C, th, C.n, S, T);
      const int size = (CX ? 2 : 1) << max(C.n, K);  // floats of one state
      double e;
      if constexpr (SMS) {
        if (2 * size <= P.state_floats)
          e = run_item<K, CX>(dyn_state, dyn_state + size, C, P.pstride, S, T);
        else
          e = run_item<K, CX>(size <= P.state_floats ? dyn_state : gpsi, glam, C, P.pstride, S, T);
      } else {
        e = run_item<K, CX>(gpsi, glam, C, P.pstride, S, T);
      }
      e = warp_sum_d(e);
      if (lane == 0) red[warp] = e;
      T.sync();
      const int toff = A.theta_off[item];
      for (int p = T.tid; p < C.nparams; p += T.n) {
        double g = 0.0;
        for (int w = 0; w < nwarps; ++w) g += ksum_value(S.wpart()[w * P.pstride + p]);
        A.grad[toff + p] = g;
      }
      if (T.tid == 0) {
        double E = 0.0;
        for (int w = 0; w < nwarps; ++w) E += red[warp + w];
        A.energy[item] = E;
      }
      T.sync();
    }
    __syncthreads();  // the next size class lays the shared memory out anew
  }
  grid_dependency_wait();  // the wide items, which this launch may overlap: done before it is
}

// ---- wide items: states in the shared memory of four blocks ------------------------
// An item of 2 more qubits than one block's shared memory holds (real: 15 and 16, complex: 14
// and 15) split by its two top bits over a cluster.  A group of lower bits runs in each
// block on its own quarter; the tiles of the others are shared out and read
// and written across the cluster.  From the global workspace one block took 3.1
// ms for an n = 16 real item of 10 layers (0.9 ms for n = 15), the time of a whole batch of
// smaller ones: its strided tiles do not fit the L1 beside the other items'
// shared memory.  On four it takes 0.49 ms; 857 parameter sets of the n = 11, 8-layer
// ansatz with 129 mixed items of 8 to 16 qubits 2.34 -> 0.53 ms.

// Element `at` (see kRankShift) of a plane at shared address `base`.
__device__ __forceinline__ float wide_load(unsigned base, int at) {
  float v;
  asm volatile(
      "{\n .reg .u32 a;\n mapa.shared::cluster.u32 a, %1, %2;\n"
      " ld.shared::cluster.f32 %0, [a];\n}"
      : "=f"(v)
      : "r"(base + (at & ((1 << kRankShift) - 1))), "r"(at >> kRankShift));
  return v;
}
__device__ __forceinline__ void wide_store(unsigned base, int at, float v) {
  asm volatile(
      "{\n .reg .u32 a;\n mapa.shared::cluster.u32 a, %0, %1;\n"
      " st.shared::cluster.f32 [a], %2;\n}" ::"r"(base + (at & ((1 << kRankShift) - 1))),
      "r"(at >> kRankShift), "f"(v)
      : "memory");
}

// steps of a split group, and the place of its tile s
template <int K>
__device__ __forceinline__ Places<K> wide_places(const BGroup& g, int nloc) {
  Places<K> pl;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const int bit = g.bits[i];
    pl.step[i] = bit >= nloc ? 1 << (kRankShift + bit - nloc) : swzr(1 << bit) * (int)sizeof(float);
    pl.low[i] = (1 << bit) - 1;
  }
  return pl;
}
template <int K>
__device__ __forceinline__ int wide_base(int s, const Places<K>& pl, int nloc) {
  const int x = sub_base<K>(s, pl.low, K);
  return ((x >> nloc) << kRankShift) | (swzr(x & ((1 << nloc) - 1)) * (int)sizeof(float));
}
template <int K, bool CX>
__device__ __forceinline__ void wide_tile_load(unsigned re, int s, const Places<K>& pl, int nloc,
                                               Tile<K, CX>& t) {
  const unsigned im = re + (unsigned)(sizeof(float) << nloc);
  int b = wide_base<K>(s, pl, nloc);
#pragma unroll
  for (int k = 0; k < (1 << (K - 1)); ++k) {
    const int p = k ^ (k >> 1);
    if (k) b ^= pl.step[1 + lowbit_b(k)];
    const int c = b ^ pl.step[0];
    t.r[p] = pair_of(wide_load(re, b), wide_load(re, c));
    if constexpr (CX) t.i[p] = pair_of(wide_load(im, b), wide_load(im, c));
  }
}
template <int K, bool CX>
__device__ __forceinline__ void wide_tile_store(unsigned re, int s, const Places<K>& pl, int nloc,
                                                const Tile<K, CX>& t) {
  const unsigned im = re + (unsigned)(sizeof(float) << nloc);
  int b = wide_base<K>(s, pl, nloc);
#pragma unroll
  for (int k = 0; k < (1 << (K - 1)); ++k) {
    const int p = k ^ (k >> 1);
    if (k) b ^= pl.step[1 + lowbit_b(k)];
    const int c = b ^ pl.step[0];
    const float2 v = lanes_of(t.r[p]);
    wide_store(re, b, v.x);
    wide_store(re, c, v.y);
    if constexpr (CX) {
      const float2 w = lanes_of(t.i[p]);
      wide_store(im, b, w.x);
      wide_store(im, c, w.y);
    }
  }
}

constexpr int kWide = 4;  // blocks of a cluster

template <int K, bool CX>
__global__ void __cluster_dims__(kWide, 1, 1) __launch_bounds__(512, 1)
    kbatch_wide(const BatchArgs A) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double red[16];
  __shared__ int s_item;
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  asm volatile("griddepcontrol.launch_dependents;");  // the other items run beside these
  const int rank = (int)cluster.block_rank();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const BPhase& P = A.wide;
  const Team T = {(int)threadIdx.x, 512, 1};
  const BSmem S = {dyn_smem, P};
  cluster.sync();  // block 0 stores into the others' shared memory: they have to have started
  while (true) {
    if (rank == 0 && threadIdx.x == 0) {
      const int v = atomicAdd(A.queue + kBPhases, 1);
      for (int r = 0; r < kWide; ++r) *cluster.map_shared_rank(&s_item, r) = v;
    }
    cluster.sync();
    const int slot = s_item;
    if (slot >= P.count) break;
    const int item = A.order[P.first + slot];
    const BCirc C = A.circs[A.item_circ[item]];
    const int nloc = C.n - 2, size = (CX ? 2 : 1) << nloc;
    float* const psi = reinterpret_cast<float*>(dyn_smem + P.o_state);
    float* const lam = psi + size;
    const unsigned upsi = (unsigned)__cvta_generic_to_shared(psi);
    const unsigned ulam = upsi + (unsigned)(sizeof(float) * size);
    load_item<K>(A, P, C, A.theta + A.theta_off[item], nloc, S, T);
    for (int x = T.tid; x < size; x += T.n) psi[x] = rank == 0 && x == 0 ? 1.f : 0.f;
    cluster.sync();
    bool synced = true;  // right after a cluster barrier
    const auto split = [&](const BGroup& g) { return (int)g.bits[K - 1] >= nloc; };  // bits ascend
    const auto done = [&](bool sp) {
      if (sp)
        cluster.sync();
      else
        T.sync();
      synced = sp;
    };
    const int nsub = 1 << (nloc - K);  // a block's share of the tiles
    for (int gg = 0; gg < C.ngroups; ++gg) {
      const BGroup& g = S.grp()[gg];
      const bool sp = split(g);
      if (sp) {
        if (!synced) cluster.sync();
        for (int s = T.tid; s < nsub; s += T.n) {
          Tile<K, CX> t;
          wide_tile_load<K, CX>(upsi, s + rank * nsub, wide_places<K>(g, nloc), nloc, t);
          tile_fwd<K, CX>(g, S, t);
          asm volatile("" ::: "memory");
          wide_tile_store<K, CX>(upsi, s + rank * nsub, wide_places<K>(g, nloc), nloc, t);
        }
      } else {
        group_fwd<K, CX>(psi, nloc, g, S, T);
      }
      done(sp);
    }
    if (!synced) cluster.sync();
    float2 ek = make_float2(0.f, 0.f);
    apply_terms<8, CX, true>(psi, lam, C, nloc, nloc, rank, S, T, ek);
    cluster.sync();  // lambda complete; nobody still reads another's psi
    synced = true;
    for (int gg = C.ngroups - 1; gg >= 0; --gg) {
      const BGroup& g = S.grp()[gg];
      const bool sp = split(g);
      if (sp) {
        if (!synced) cluster.sync();
        float2* const part = S.wpart() + warp * P.pstride;
        for (int s = T.tid; s < nsub; s += T.n) {  // nsub is a multiple of 32
          Tile<K, CX> p, l;
          {
            const Places<K> pl = wide_places<K>(g, nloc);
            wide_tile_load<K, CX>(upsi, s + rank * nsub, pl, nloc, p);
            wide_tile_load<K, CX>(ulam, s + rank * nsub, pl, nloc, l);
          }
          tile_bwd<K, CX>(g, S, part, p, l);
          asm volatile("" ::: "memory");
          const Places<K> pl = wide_places<K>(g, nloc);
          wide_tile_store<K, CX>(upsi, s + rank * nsub, pl, nloc, p);
          wide_tile_store<K, CX>(ulam, s + rank * nsub, pl, nloc, l);
        }
      } else {
        group_bwd<K, CX>(psi, lam, nloc, P.pstride, g, S, T);
      }
      done(sp);
    }
    const double e = warp_sum_d(ksum_value(ek));
    if (lane == 0) red[warp] = e;
    cluster.sync();  // every block's partials final
    if (rank == 0) {
      const int toff = A.theta_off[item];
      for (int p = threadIdx.x; p < C.nparams; p += 512) {
        double g = 0.0;
        for (int r = 0; r < kWide; ++r) {
          const float2* w = cluster.map_shared_rank(S.wpart(), r);
          for (int i = 0; i < 16; ++i) g += ksum_value(w[i * P.pstride + p]);
        }
        A.grad[toff + p] = g;
      }
      if (threadIdx.x == 0) {
        double E = 0.0;
        for (int r = 0; r < kWide; ++r) {
          const double* d = cluster.map_shared_rank(red, r);
          for (int i = 0; i < 16; ++i) E += d[i];
        }
        A.energy[item] = E;
      }
    }
    // the next item's barrier orders block 0's reads before the others reuse their partials
  }
}

// ---- two-block clusters: each item's states split over the pair ----------------------
// A cluster of two blocks (one per SM) runs one item at a time.  Block c
// holds the amplitudes whose top bit (n - 1) is c, of both psi and lambda: in
// its shared memory when n <= kClSmemQubits (2 x 64 KiB at n = 14), else in
// the cluster's global workspace slot.  A register group that does not touch
// bit n - 1 runs on each block's own half; a group that does ("split") gives
// each block half of the sub-blocks and reaches the partner's half through
// distributed shared memory (or global memory), with cluster barriers before
// and after.  Energy and gradient partials are summed per block, then block 0
// adds the partner's partials in a fixed order.
constexpr int kClSmemQubits = 14;
constexpr int kClThreads = 512;

// amplitude x of the whole state: its block's half, offset inside the half
struct Halves {
  float2* h0;
  float2* h1;
  int hn;  // qubits per half (n - 1)
  __device__ __forceinline__ float2& at(int x) const {
    return ((x >> hn) ? h1 : h0)[x & ((1 << hn) - 1)];
  }
};

template <int K>
__device__ __forceinline__ void cl_group_fwd(const Halves& P, float2* own, int rank, int n,
                                             bool split, const BGroup& g, const BOp* ops,
                                             const float* mats) {
  int off[1 << K], lm[K];
  group_offsets<K>(g, off, lm);
  const int kk = g.k, width = 1 << kk;
  if (!split) {
    const int nsub = 1 << (P.hn - kk);
    for (int s = threadIdx.x; s < nsub; s += kClThreads) {
      const int b = sub_base<K>(s, lm, kk);
      float re[1 << K], im[1 << K];
#pragma unroll
      for (int r = 0; r < (1 << K); ++r)
        if (r < width) {
          const float2 v = own[b | off[r]];
          re[r] = v.x;
          im[r] = v.y;
        }
      for (int o = g.op0; o < g.op1; ++o) {
        const BOp op = ops[o];
        const float* M = mats + 8 * op.gi;
#define SV_FWD(BB) \
  if constexpr (BB < K) pair_apply<K, BB>(op.cls, M, op.cm, re, im)
        SV_BIT_SWITCH(op.b0, SV_FWD)
#undef SV_FWD
      }
#pragma unroll
      for (int r = 0; r < (1 << K); ++r)
        if (r < width) own[b | off[r]] = make_float2(re[r], im[r]);
    }
  } else {
    const int nsub = 1 << (n - kk);  // sub-blocks s = rank, rank + 2, ...
    for (int s = rank + 2 * (int)threadIdx.x; s < nsub; s += 2 * kClThreads) {
      const int b = sub_base<K>(s, lm, kk);
      float re[1 << K], im[1 << K];
#pragma unroll
      for (int r = 0; r < (1 << K); ++r)
        if (r < width) {
          const float2 v = P.at(b | off[r]);
          re[r] = v.x;
          im[r] = v.y;
        }
      for (int o = g.op0; o < g.op1; ++o) {
        const BOp op = ops[o];
        const float* M = mats + 8 * op.gi;
#define SV_FWD(BB) \
  if constexpr (BB < K) pair_apply<K, BB>(op.cls, M, op.cm, re, im)
        SV_BIT_SWITCH(op.b0, SV_FWD)
#undef SV_FWD
      }
#pragma unroll
      for (int r = 0; r < (1 << K); ++r)
        if (r < width) P.at(b | off[r]) = make_float2(re[r], im[r]);
    }
  }
}

template <int K, bool split>
__device__ __forceinline__ void cl_group_bwd(const Halves& Pp, const Halves& Pl, float2* ownp,
                                             float2* ownl, int rank, int n, const BGroup& g,
                                             const BOp* ops, const float* mats, double* wpart) {
  int off[1 << K], lm[K];
  group_offsets<K>(g, off, lm);
  const int kk = g.k, width = 1 << kk;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nsub = split ? 1 << (n - kk) : 1 << (Pp.hn - kk);
  const int first = split ? rank : 0, step = split ? 2 : 1;
  // every lane of a warp runs the same number of iterations (warp sums)
  const int mine = split ? (nsub - rank + 1) / 2 : nsub;
  const int iters = (mine + kClThreads - 1) / kClThreads;
  for (int it = 0; it < iters; ++it) {
    const int t = threadIdx.x + it * kClThreads;
    const bool live = t < mine;
    const int s = first + step * t;
    const int b = live ? sub_base<K>(s, lm, kk) : 0;
    float pr[1 << K], pi[1 << K], lr[1 << K], li[1 << K];
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) {
      pr[r] = pi[r] = lr[r] = li[r] = 0.f;
      if (live && r < width) {
        const int x = b | off[r];
        float2 v, w;
        if constexpr (split) {
          v = Pp.at(x);
          w = Pl.at(x);
        } else {
          v = ownp[x];
          w = ownl[x];
        }
        pr[r] = v.x;
        pi[r] = v.y;
        lr[r] = w.x;
        li[r] = w.y;
      }
    }
    for (int o = g.op1 - 1; o >= g.op0; --o) {
      const BOp op = ops[o];
      const float* M = mats + 8 * op.gi;
      if (op.pauli) {
        float c = 0.f;
#define SV_GRAD(BB) \
  if constexpr (BB < K) c = pair_grad<K, BB>(op.pauli, op.cm, pr, pi, lr, li)
        SV_BIT_SWITCH(op.b0, SV_GRAD)
#undef SV_GRAD
        c = warp_sum_f(c);
        if (lane == 0) wpart[warp * kBMaxParams + op.param] += (double)c;
      }
#define SV_BWD(BB)                                   \
  if constexpr (BB < K) {                            \
    pair_apply_dag<K, BB>(op.cls, M, op.cm, pr, pi); \
    pair_apply_dag<K, BB>(op.cls, M, op.cm, lr, li); \
  }
      SV_BIT_SWITCH(op.b0, SV_BWD)
#undef SV_BWD
    }
    if (live) {
#pragma unroll
      for (int r = 0; r < (1 << K); ++r)
        if (r < width) {
          const int x = b | off[r];
          if constexpr (split) {
            Pp.at(x) = make_float2(pr[r], pi[r]);
            Pl.at(x) = make_float2(lr[r], li[r]);
          } else {
            ownp[x] = make_float2(pr[r], pi[r]);
            ownl[x] = make_float2(lr[r], li[r]);
          }
        }
    }
  }
}

__device__ __forceinline__ bool group_is_split(const BGroup& g, int hn) {
  if (hn < g.k) return true;
  for (int i = 0; i < g.k; ++i)
    if (g.bits[i] == hn) return true;
  return false;
}

// Dynamic shared memory: psi half, lambda half (2^13 amplitudes each), gate
// matrices, per-warp gradient partials.
constexpr size_t kClSmemBytes = (sizeof(float2) << kClSmemQubits) + sizeof(float) * 8 * kBMaxGates +
                                sizeof(double) * (kClThreads / 32) * kBMaxParams;

template <int K>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kClThreads, 1)
    kbatch_cl(const BatchArgs A) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char cl_smem[];
  float2* sh_psi = reinterpret_cast<float2*>(cl_smem);
  float2* sh_lam = sh_psi + (1 << (kClSmemQubits - 1));
  float* mats = reinterpret_cast<float*>(sh_lam + (1 << (kClSmemQubits - 1)));
  double* wpart = reinterpret_cast<double*>(mats + 8 * kBMaxGates);
  __shared__ double red[kClThreads / 32];
  __shared__ int s_item;
  const int rank = (int)cluster.block_rank();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int nwarps = kClThreads / 32;
  const size_t cid = blockIdx.x / 2;
  float2* gw = A.work + cid * (size_t(2) << A.nmax);  // global slot: psi, then lambda
  int* partner_item = cluster.map_shared_rank(&s_item, 1);
  cluster.sync();  // block 0 stores into its partner's shared memory: it has to have started
  while (true) {
    if (rank == 0 && threadIdx.x == 0) {
      const int v = atomicAdd(A.queue, 1);
      s_item = v;
      *partner_item = v;
    }
    cluster.sync();
    const int slot = s_item;
    if (slot >= A.n_items) break;
    const int item = A.order[slot];
    const BCirc C = A.circs[A.item_circ[item]];
    const double* th = A.theta + A.theta_off[item];
    const int n = C.n, hn = n - 1, hdim = 1 << hn;
    const bool in_smem = n <= kClSmemQubits;
    Halves Pp, Pl;
    Pp.hn = Pl.hn = hn;
    if (in_smem) {
      Pp.h0 = cluster.map_shared_rank(sh_psi, 0);
      Pp.h1 = cluster.map_shared_rank(sh_psi, 1);
      Pl.h0 = cluster.map_shared_rank(sh_lam, 0);
      Pl.h1 = cluster.map_shared_rank(sh_lam, 1);
    } else {
      Pp.h0 = gw;
      Pp.h1 = gw + hdim;
      Pl.h0 = gw + (size_t(1) << A.nmax);
      Pl.h1 = Pl.h0 + hdim;
    }
    float2* ownp = in_smem ? sh_psi : (rank ? Pp.h1 : Pp.h0);
    float2* ownl = in_smem ? sh_lam : (rank ? Pl.h1 : Pl.h0);
    for (int gi = threadIdx.x; gi < C.ngates; gi += kClThreads) {
      const BGateDesc d = A.gates[C.gate0 + gi];
      const double a = d.param >= 0 ? th[d.param] : d.angle;
      double sn, cs;
      sincos(0.5 * a, &sn, &cs);
      double m[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      const double r2 = 0.70710678118654752440;
      switch (d.kind) {
        case SV_GATE_H: m[0] = r2; m[2] = r2; m[4] = r2; m[6] = -r2; break;
        case SV_GATE_X: m[2] = 1; m[4] = 1; break;
        case SV_GATE_Y: m[3] = -1; m[5] = 1; break;
        case SV_GATE_Z: m[0] = 1; m[6] = -1; break;
        case SV_GATE_RX: m[0] = cs; m[3] = -sn; m[5] = -sn; m[6] = cs; break;
        case SV_GATE_RY: m[0] = cs; m[2] = -sn; m[4] = sn; m[6] = cs; break;
        case SV_GATE_RZ: m[0] = cs; m[1] = -sn; m[6] = cs; m[7] = sn; break;
        default: {  // U1: diag(1, e^{ia})
          double sa, ca;
          sincos(a, &sa, &ca);
          m[0] = 1; m[6] = ca; m[7] = sa;
        }
      }
      for (int e = 0; e < 8; ++e) mats[8 * gi + e] = (float)m[e];
    }
    for (int x = threadIdx.x; x < hdim; x += kClThreads)
      ownp[x] = make_float2(rank == 0 && x == 0 ? 1.f : 0.f, 0.f);
    for (int i = threadIdx.x; i < nwarps * kBMaxParams; i += kClThreads) wpart[i] = 0.0;
    __syncthreads();
    // forward
    bool synced = false;  // true right after a cluster barrier
    for (int gg = 0; gg < C.ngroups; ++gg) {
      const BGroup G = A.groups[C.group0 + gg];
      const bool split = group_is_split(G, hn);
      if (split && !synced) cluster.sync();
      cl_group_fwd<K>(Pp, ownp, rank, n, split, G, A.ops, mats);
      if (split) {
        cluster.sync();
        synced = true;
      } else {
        __syncthreads();
        synced = false;
      }
    }
    if (!synced) cluster.sync();
    // lambda = H psi on this block's half, E = Re <psi|lambda>
    double e = 0.0;
    for (int xl = threadIdx.x; xl < hdim; xl += kClThreads) {
      const int x = (rank << hn) | xl;
      float orr = 0.f, oi = 0.f;
      for (int t = 0; t < C.nterms; ++t) {
        const BTerm T = A.terms[C.term0 + t];
        const float2 b = Pp.at(x ^ (int)T.xm);
        const float cr = (float)T.cre, ci = (float)T.cim;
        const float sr = cr * b.x - ci * b.y, si = cr * b.y + ci * b.x;
        if (__popcll(((uint64_t)x ^ T.xm) & T.zm) & 1) {
          orr -= sr;
          oi -= si;
        } else {
          orr += sr;
          oi += si;
        }
      }
      ownl[xl] = make_float2(orr, oi);
      const float2 a = ownp[xl];
      e += (double)(a.x * orr + a.y * oi);
    }
    e = warp_sum_d(e);
    if (lane == 0) red[warp] = e;
    cluster.sync();  // lambda complete; nobody still reads the partner's psi
    // reverse sweep
    synced = true;
    for (int gg = C.ngroups - 1; gg >= 0; --gg) {
      const BGroup G = A.groups[C.group0 + gg];
      const bool split = group_is_split(G, hn);
      if (split && !synced) cluster.sync();
      if (split)
        cl_group_bwd<K, true>(Pp, Pl, ownp, ownl, rank, n, G, A.ops, mats, wpart);
      else
        cl_group_bwd<K, false>(Pp, Pl, ownp, ownl, rank, n, G, A.ops, mats, wpart);
      if (split) {
        cluster.sync();
        synced = true;
      } else {
        __syncthreads();
        synced = false;
      }
    }
    cluster.sync();  // both blocks' partials final
    if (rank == 0) {
      const double* pw = cluster.map_shared_rank(wpart, 1);
      const double* pred = cluster.map_shared_rank(red, 1);
      const int toff = A.theta_off[item];
      for (int p = threadIdx.x; p < C.nparams; p += kClThreads) {
        double g = 0.0;
        for (int w = 0; w < nwarps; ++w) g += wpart[w * kBMaxParams + p];
        for (int w = 0; w < nwarps; ++w) g += pw[w * kBMaxParams + p];
        A.grad[toff + p] = g;
      }
      if (threadIdx.x == 0) {
        double E = 0.0;
        for (int w = 0; w < nwarps; ++w) E += red[w];
        for (int w = 0; w < nwarps; ++w) E += pred[w];
        A.energy[item] = E;
      }
    }
    // the next item's barrier orders block 0's reads before block 1 reuses its partials
  }
}

}  // namespace
}  // namespace sv

// ---- host side: descriptors, autotuner, launches ---------------------------------
struct sv_batch_s {
  int n_items = 0, nmax = 0, total_params = 0;
  int k = 4, threads = 256, blocks = 0;  // chosen tile
  bool cluster = false;                  // two-block cluster kernel
  bool smem_states = false;              // single-block kernel with states in shared memory
  bool real = false;                     // real amplitudes (kbatch with one plane)
  int sms = 152;
  // device buffers
  sv::BCirc* circs = nullptr;
  sv::BGateDesc* gates = nullptr;
  sv::BGroup* groups = nullptr;
  sv::BOp* ops = nullptr;
  sv::BTerm* terms = nullptr;
  sv::BGroup* rgroups = nullptr;  // the single-block kernels' lists
  sv::BOp* rops = nullptr;
  uint32_t* rsigns = nullptr;
  sv::BRot* rots = nullptr;
  sv::BGateDesc* gens = nullptr;
  int* order = nullptr;
  int* item_circ = nullptr;
  int* theta_off = nullptr;
  int* queue = nullptr;
  float2* work = nullptr;
  size_t work_slots = 0;
  std::vector<sv::BCirc> h_circs;       // of the chosen group width, with
  std::vector<int> h_ops;               // the single-block kernels' operations of each
  std::vector<int> h_order, h_item_circ;
  int n_phases = 0;                     // of the chosen tile
  sv::BPhase phase[sv::kBPhases], wide;
  size_t smem = 0;
  // captured graph
  cudaGraphExec_t gexec = nullptr;
  const void* g_key[4] = {nullptr, nullptr, nullptr, nullptr};
};

namespace sv {
namespace {

struct HostPlan {
  std::vector<BCirc> circs;
  std::vector<BGateDesc> gates;
  std::vector<BGroup> groups;
  std::vector<BOp> ops;
  std::vector<BTerm> terms;
  std::vector<BGroup> rgroups;  // filled by tile_lists
  std::vector<BOp> rops;
  std::vector<uint32_t> rsigns;
  std::vector<BRot> rots;
  std::vector<BGateDesc> gens;
};

int popc64(uint64_t x) { return __builtin_popcountll(x); }

// List-schedule one circuit's gates (1-qubit kinds with controls) into groups
// of at most k qubits, as the fused pass planner does, without merging gates
// (every parameter keeps its own gate for the gradient).
bool plan_circuit(const sv_circuit* c, const sv_pauli_sum* H, int k, HostPlan* P) {
  const int n = c->n_qubits;
  BCirc C{};
  C.n = n;
  C.ngates = c->n_gates;
  C.gate0 = (int)P->gates.size();
  C.group0 = (int)P->groups.size();
  C.nparams = c->n_params;
  C.nterms = H->n_terms;
  C.term0 = (int)P->terms.size();
  std::vector<uint64_t> qm(c->n_gates);
  for (int i = 0; i < c->n_gates; ++i) {
    const sv_gate& g = c->gates[i];
    const bool rot = g.kind == SV_GATE_RX || g.kind == SV_GATE_RY || g.kind == SV_GATE_RZ;
    BGateDesc d{g.kind, g.param, g.angle, rot && g.n_ctrl == 0};
    P->gates.push_back(d);
    uint64_t m = uint64_t(1) << (n - 1 - g.targets[0]);
    for (int j = 0; j < g.n_ctrl; ++j) m |= uint64_t(1) << (n - 1 - g.controls[j]);
    qm[i] = m;
  }
  std::vector<int> pending(c->n_gates);
  for (int i = 0; i < c->n_gates; ++i) pending[i] = i;
  while (!pending.empty()) {
    if (popc64(qm[pending[0]]) > k) return false;  // a gate wider than a group
    uint64_t gq = qm[pending[0]], acc = 0;
    std::vector<int> members, rest;
    for (int j : pending) {
      if (!(qm[j] & acc) && popc64(gq | qm[j]) <= k) {
        gq |= qm[j];
        members.push_back(j);
      } else {
        acc |= qm[j];
        rest.push_back(j);
      }
    }
    BGroup G{};
    int bits[64], nb = 0;
    for (int b = 0; b < n; ++b)
      if ((gq >> b) & 1) bits[nb++] = b;
    // pad narrow groups with free bits so every group has exactly min(k, n) bits
    for (int b = 0; b < n && nb < std::min(k, n); ++b)
      if (!((gq >> b) & 1)) {
        gq |= uint64_t(1) << b;
        bits[nb++] = b;
      }
    std::sort(bits, bits + nb);
    G.k = (uint8_t)nb;
    for (int i = 0; i < nb; ++i) G.bits[i] = (uint8_t)bits[i];
    G.op0 = (int32_t)P->ops.size();
    for (int j : members) {
      const sv_gate& g = c->gates[j];
      auto local = [&](int bit) {
        for (int i = 0; i < nb; ++i)
          if (bits[i] == bit) return i;
        return 0;
      };
      BOp op{};
      op.b0 = (uint8_t)local(n - 1 - g.targets[0]);
      for (int t = 0; t < g.n_ctrl; ++t) op.cm |= (uint8_t)(1 << local(n - 1 - g.controls[t]));
      op.pauli = g.param >= 0 ? (g.kind == SV_GATE_RX ? 1 : g.kind == SV_GATE_RY ? 2 : 3) : 0;
      switch (g.kind) {
        case SV_GATE_H: case SV_GATE_X: case SV_GATE_RY: op.cls = BC_REAL; break;
        case SV_GATE_Y: case SV_GATE_RX: op.cls = BC_IMOFF; break;
        case SV_GATE_RZ: op.cls = BC_DIAG; break;
        case SV_GATE_Z: op.cls = BC_NEG; break;
        case SV_GATE_U1: op.cls = BC_PHASE; break;
        default: op.cls = BC_DENSE;
      }
      op.param = (int16_t)g.param;
      op.gi = (int16_t)j;
      P->ops.push_back(op);
    }
    G.op1 = (int32_t)P->ops.size();
    P->groups.push_back(G);
    pending.swap(rest);
  }
  C.ngroups = (int)P->groups.size() - C.group0;
  // diagonal terms first: their coefficients combine per amplitude before
  // the one product with psi_x
  C.ndiag = 0;
  for (int pass = 0; pass < 2; ++pass)
    for (int t = 0; t < H->n_terms; ++t) {
      const uint64_t xm = H->xmask[t], zm = H->zmask[t];
      if ((xm == 0) != (pass == 0)) continue;
      const int ny = popc64(xm & zm) & 3;
      const double cf = H->coeff[t];
      P->terms.push_back({xm, zm, ny == 0 ? cf : ny == 2 ? -cf : 0.0,
                          ny == 1 ? cf : ny == 3 ? -cf : 0.0});
      if (pass == 0) ++C.ndiag;
    }
  P->circs.push_back(C);
  return P->ops.size() < (size_t)0x7fffffff;
}

// A circuit with more patterns keeps its single flips.
constexpr int kBMaxSigns = 96;

// The single-block kernels' lists of every circuit of P.  Rotations without controls join
// the group's last run while none of their qubit's later operations stand between, in
// the order (qubit, X < Y < Z), no parameter twice; each run of sign flips with
// no other than diagonal operations on their bits in between is one pattern
// over the group's 2^k indices.
void tile_lists(HostPlan* P) {
  for (BCirc& C : P->circs) {
    C.gen0 = (int)P->gens.size();
    C.rot0 = (int)P->rots.size();
    for (int merge = 1; merge >= 0; --merge) {
      const size_t o0 = P->rops.size(), s0 = P->rsigns.size(), g0 = P->rgroups.size();
      for (int g = C.group0; g < C.group0 + C.ngroups; ++g) {
        BGroup G = P->groups[g];
        const int a = G.op0, b = G.op1;
        G.op0 = (int32_t)P->rops.size();
        int open = -1, dirty = 0;     // the last pattern, and bits touched since
        int run = -1, since = 0;      // the last run, and bits touched since
        std::vector<std::pair<int, BRot>> rots;  // its rotations by 3 bit + kind
        auto close = [&] {
          if (run < 0) return;
          std::sort(rots.begin(), rots.end(),
                    [](const auto& x, const auto& y) { return x.first < y.first; });
          BOp& r = P->rops[run];
          r.gi = (int16_t)(P->rots.size() - C.rot0);
          r.cm = (uint8_t)rots.size();
          for (const auto& x : rots) {
            r.param = (int16_t)(r.param | (1 << x.first));
            P->rots.push_back(x.second);
          }
          rots.clear();
          run = -1;
          since = 0;
        };
        for (int o = a; o < b; ++o) {
          BOp op = P->ops[o];
          const int bits = op.cm | (1 << op.b0);
          if (op.cls == BC_NEG && merge) {
            if (open < 0 || (bits & dirty)) {
              open = (int)P->rsigns.size();
              dirty = 0;
              P->rsigns.push_back(0);
              BOp sg{};
              sg.cls = BC_SIGN;
              sg.param = -1;
              sg.gi = (int16_t)(open - (int)s0);
              P->rops.push_back(sg);
            }
            since |= bits;
            for (int r = 0; r < (1 << G.k); ++r)
              if ((r & bits) == bits) P->rsigns[open] ^= 1u << r;
            continue;
          }
          if (op.cls != BC_DIAG && op.cls != BC_PHASE) dirty |= bits;
          const BGateDesc& d = P->gates[C.gate0 + op.gi];
          if (d.free_rot) {
            const int at = 3 * op.b0 + (d.kind == SV_GATE_RX ? 0 : d.kind == SV_GATE_RY ? 1 : 2);
            bool join = run >= 0 && !(since & bits);
            for (const auto& x : rots)
              if ((x.first / 3 == op.b0 && x.first >= at) ||
                  (d.param >= 0 && x.second.param == d.param))
                join = false;
            if (!join) {
              close();
              run = (int)P->rops.size();
              BOp r{};
              r.cls = BC_RUN;
              P->rops.push_back(r);
            }
            rots.push_back({at, BRot{d.kind, d.param, d.angle}});
            continue;
          }
          since |= bits;
          op.gi = (int16_t)(P->gens.size() - C.gen0);
          P->gens.push_back(d);
          P->rops.push_back(op);
        }
        close();
        G.op1 = (int32_t)P->rops.size();
        P->rgroups.push_back(G);
      }
      C.sign0 = (int)s0;
      C.nsign = (int)(P->rsigns.size() - s0);
      C.nrot = (int)P->rots.size() - C.rot0;
      C.ngen = (int)P->gens.size() - C.gen0;
      if (C.nsign <= kBMaxSigns) break;
      P->rops.resize(o0);
      P->rsigns.resize(s0);
      P->rgroups.resize(g0);
      P->rots.resize(C.rot0);
      P->gens.resize(C.gen0);
    }
  }
}

template <typename T>
sv_status upload(T** dst, const std::vector<T>& v) {
  const size_t bytes = std::max<size_t>(1, v.size()) * sizeof(T);
  SV_CUDA_TRY(cudaMalloc((void**)dst, bytes));
  if (!v.empty()) SV_CUDA_TRY(cudaMemcpy(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
  return SV_OK;
}

void free_batch(sv_batch b) {
  void* ptrs[] = {b->circs, b->gates, b->groups, b->ops, b->terms, b->rgroups,
                  b->rops, b->rsigns, b->rots, b->gens, b->order, b->item_circ, b->theta_off, b->queue, b->work};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
}

typedef void (*BatchKernel)(const BatchArgs);
// Kernel variants by group width (and threads per block, resident blocks per SM).
BatchKernel real_kernel_for(int k) {
  return k <= 3   ? kbatch<3, 512, 1, false, true>
         : k == 4 ? kbatch<4, 512, 1, false, true>
                  : kbatch<5, 512, 1, false, true>;
}
BatchKernel wide_kernel_for(int k, bool re) {
  if (re)
    return k <= 3 ? kbatch_wide<3, false> : k == 4 ? kbatch_wide<4, false> : kbatch_wide<5, false>;
  return k == 2 ? kbatch_wide<2, true> : k == 3 ? kbatch_wide<3, true> : kbatch_wide<4, true>;
}
BatchKernel smem_kernel_for(int k) {
  return k == 2   ? kbatch<2, 512, 1, true, true>
         : k == 3 ? kbatch<3, 512, 1, true, true>
                  : kbatch<4, 512, 1, true, true>;
}
// states in the global workspace
BatchKernel kernel_for(int k, int threads, int per_sm) {
  if (threads <= 128) return k == 2 ? kbatch<2, 128, 8, true, false> : kbatch<3, 128, 8, true, false>;
  if (per_sm >= 4) return k == 2 ? kbatch<2, 256, 4, true, false> : kbatch<3, 256, 4, true, false>;
  return k == 2   ? kbatch<2, 256, 2, true, false>
         : k == 3 ? kbatch<3, 256, 2, true, false>
                  : kbatch<4, 256, 2, true, false>;
}

// register groups of 2 or 3 qubits (4 would spill at 512 threads per block)
BatchKernel cluster_kernel_for(int k) { return k == 2 ? kbatch_cl<2> : kbatch_cl<3>; }

// The shared memory of one team (see BSmem) that runs `items`, with a state memory of a
// power of two floats that the budget leaves, no more than the largest item wants.
// Wide: a quarter of the states.
void team_smem(sv_batch b, const std::vector<int>& items, int k, bool re, size_t budget, bool wide,
               BPhase* P) {
  int rots = 1, gens = 1, params = 1, ops = 1, groups = 1, terms = 1, signs = 1, n = k;
  for (int i : items) {
    const BCirc& C = b->h_circs[b->h_item_circ[i]];
    rots = std::max(rots, C.nrot);
    gens = std::max(gens, C.ngen);
    params = std::max(params, C.nparams);
    ops = std::max(ops, b->h_ops[b->h_item_circ[i]]);
    groups = std::max(groups, C.ngroups);
    terms = std::max(terms, C.nterms);
    signs = std::max(signs, C.nsign);
    n = std::max(n, C.n);
  }
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t o = at;
    at += (bytes + 15) & ~size_t(15);
    return (int)o;
  };
  take(sizeof(float4) * rots);
  P->o_mats = take(sizeof(float) * 8 * gens);
  P->o_wpart = take(sizeof(float2) * (P->ts / 32) * params);
  P->o_ops = take(sizeof(BOp) * ops);
  P->o_grp = take(sizeof(BGroup) * groups);
  P->o_term = take(sizeof(int2) * terms);
  P->o_tcoef = take(sizeof(float) * 8 * terms);
  P->o_sign = take((sizeof(float) << k) * signs);
  P->o_state = (int)at;
  P->pstride = params;
  const size_t want = size_t(re ? 2 : 4) << (wide ? n - 2 : n);
  size_t f = 0;
  for (size_t c = 64; c <= want && at + sizeof(float) * c <= budget; c *= 2) f = c;
  P->state_floats = (int)f;
  P->stride = (int)(at + sizeof(float) * f);
  P->count = (int)items.size();
}

// The size classes of the batch for a tile, and the items' order by them.  A class of
// teams smaller than the block holds both states of its items in shared memory;
// items whose states do not fit go to larger teams.
sv_status set_phases(sv_batch b, int k, int threads, bool states, bool re) {
  const size_t budget = (size_t)227 * 1024 - 512;  // 512: the static variables
  std::vector<int> order;
  std::vector<char> carried(b->n_items, 0), taken(b->n_items, 0);
  std::vector<std::vector<int>> lists;
  b->n_phases = 0;
  b->smem = 0;
  b->wide = BPhase{};
  if (!states) {
    BPhase P{};
    P.ts = threads;
    team_smem(b, b->h_order, k, re, 0, false, &P);
    b->phase[b->n_phases++] = P;
    order = b->h_order;
    b->smem = P.stride;
  } else {
    // Wide items: more than one block's 512 tiles, no more than four.  Those of twice 512 cost
    // 1.7 SM-milliseconds on a cluster and 0.93 in one block (n = 15, 10 layers, real,
    // where n = 14 costs 0.33), but take 0.42 and 0.93 ms: they go to clusters where one in
    // a block would outlast half of the batch, and where they are an eighth of it or
    // less (1024 items of n = 14 and 256 of 8 to 16: 2.86 ms in blocks, 2.76 wide;
    // 152 items of n = 15: 0.93 in blocks, 1.76 wide).
    double total = 0, twice = 0;
    const auto cost = [&](int i) {
      const BCirc& C = b->h_circs[b->h_item_circ[i]];
      return (C.n == k + 10 ? 1.4 : 1.0) * C.ngates * (double)(1 << C.n);
    };
    for (int i : b->h_order) {
      total += cost(i);
      if (b->h_circs[b->h_item_circ[i]].n == k + 10) twice += cost(i);
    }
    std::vector<int> wide;
    for (int i : b->h_order) {
      const int n = b->h_circs[b->h_item_circ[i]].n;
      if (n == k + 11 || (n == k + 10 && (8 * twice <= total || cost(i) * b->sms > 2 * total)))
        wide.push_back(i);
    }
    if (!wide.empty()) {
      b->wide.ts = 512;
      team_smem(b, wide, k, re, budget, true, &b->wide);
      int n = 0;
      for (int i : wide) n = std::max(n, b->h_circs[b->h_item_circ[i]].n);
      if ((size_t)b->wide.state_floats < size_t(re ? 2 : 4) << (n - 2)) {
        b->wide = BPhase{};
        wide.clear();
      }
    }
    for (int i : wide) taken[i] = 1;
    order = wide;
    std::vector<BPhase> phases;  // from the smallest teams
    for (int ts = 64; ts <= 512; ts *= 2) {
      std::vector<int> mine;  // keeps h_order's order: longest first
      for (int i : b->h_order) {
        const int n = std::max(b->h_circs[b->h_item_circ[i]].n, k);
        const int tiles = 1 << (n - k);
        const bool fits = ts == 64 ? tiles <= 64 : ts == 512 ? tiles >= 512 : tiles == ts;
        if ((fits && !taken[i]) || carried[i]) mine.push_back(i);
        carried[i] = 0;
      }
      if (mine.empty()) continue;
      BPhase P{};
      P.ts = ts;
      team_smem(b, mine, k, re, budget / (512 / ts) & ~size_t(15), false, &P);
      int n = k;
      for (int i : mine) n = std::max(n, b->h_circs[b->h_item_circ[i]].n);
      if (ts < 512 && (size_t)P.state_floats < size_t(re ? 2 : 4) << n) {
        for (int i : mine) carried[i] = 1;  // to the next class
        continue;
      }
      b->smem = std::max(b->smem, (size_t)P.stride * (512 / ts));
      phases.push_back(P);
      lists.push_back(mine);
    }
    for (size_t i = phases.size(); i-- > 0;) {
      phases[i].first = (int)order.size();
      order.insert(order.end(), lists[i].begin(), lists[i].end());
      b->phase[b->n_phases++] = phases[i];
    }
  }
  SV_CUDA_TRY(cudaMemcpy(b->order, order.data(), order.size() * sizeof(int), cudaMemcpyHostToDevice));
  return SV_OK;
}

sv_status launch_batch(sv_batch b, const double* theta, double* energy, double* grad,
                       cudaStream_t st, int k, int threads, int blocks, bool cl, bool sms,
                       bool re) {
  BatchArgs A;
  A.circs = b->circs;
  A.gates = b->gates;
  A.groups = b->groups;
  A.ops = b->ops;
  A.terms = b->terms;
  A.rgroups = b->rgroups;
  A.rops = b->rops;
  A.rsigns = b->rsigns;
  A.rots = b->rots;
  A.gens = b->gens;
  A.n_phases = b->n_phases;
  for (int i = 0; i < b->n_phases; ++i) A.phase[i] = b->phase[i];
  A.wide = b->wide;
  A.order = b->order;
  A.item_circ = b->item_circ;
  A.theta_off = b->theta_off;
  A.n_items = b->n_items;
  A.nmax = std::max(b->nmax, 5);  // a tile of 2^k amplitudes at least
  A.theta = theta;
  A.energy = energy;
  A.grad = grad;
  A.work = b->work;
  A.queue = b->queue;
  SV_CUDA_TRY(cudaMemsetAsync(b->queue, 0, (kBPhases + 1) * sizeof(int), st));
  if (cl) {
    BatchKernel kern = cluster_kernel_for(k);
    static bool attr[5] = {false, false, false, false, false};
    if (!attr[k]) {
      SV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kClSmemBytes));
      attr[k] = true;
    }
    ProfScope prof(st, "kbatch_cl");
    kern<<<blocks, kClThreads, kClSmemBytes, st>>>(A);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return check_launch("batch cluster kernel");
  }
  const int per_sm = std::max(1, blocks / std::max(1, b->sms));
  BatchKernel kern = re    ? real_kernel_for(k)
                     : sms ? smem_kernel_for(k)
                           : kernel_for(k, threads, per_sm);
  // opt in to more than the default 48 KiB, to the most any batch has asked for
  const auto allow = [](BatchKernel kern, size_t smem) -> sv_status {
    static std::mutex mu;
    static std::vector<std::pair<BatchKernel, size_t>> done;
    std::lock_guard<std::mutex> lk(mu);
    auto it = std::find_if(done.begin(), done.end(), [&](const auto& d) { return d.first == kern; });
    if (it == done.end() || it->second < smem) {
      SV_CUDA_TRY(
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      if (it == done.end())
        done.push_back({kern, smem});
      else
        it->second = smem;
    }
    return SV_OK;
  };
  ProfScope prof(st, re ? "kbatch_real" : sms ? "kbatch_smem" : "kbatch");
  sv_status s = allow(kern, b->smem);
  if (s) return s;
  if (b->wide.count > 0) {
    BatchKernel wide = wide_kernel_for(k, re);
    s = allow(wide, b->wide.stride);
    if (s) return s;
    const int clusters = std::min(b->wide.count, std::max(1, b->sms / kWide));
    wide<<<clusters * kWide, 512, b->wide.stride, st>>>(A);
    s = check_launch("batch kernel (wide items)");
    if (s) return s;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (b->n_phases == 0) return SV_OK;
    launch_dependent(kern, blocks, threads, b->smem, st, A);
  } else {
    kern<<<blocks, threads, b->smem, st>>>(A);
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return check_launch("batch kernel");
}

}  // namespace
}  // namespace sv

using namespace sv;

// Checks every circuit and Hamiltonian against the batch kernel's limits;
// returns the largest qubit count and the widest gate (target + controls).
static sv_status validate_batch(const char* who, const sv_circuit* circuits,
                                const sv_pauli_sum* hamiltonians, int n_circuits, int* nmax_out,
                                int* width_out) {
  if (!circuits || !hamiltonians || n_circuits < 1) {
    set_error("%s: bad arguments", who);
    return SV_ERR_INVALID;
  }
  int nmax = 1, width = 1;  // widest gate: target plus controls
  for (int c = 0; c < n_circuits; ++c) {
    const sv_circuit& C = circuits[c];
    const sv_pauli_sum& H = hamiltonians[c];
    if (C.n_qubits < 1 || C.n_qubits > SV_BATCH_MAX_QUBITS || C.n_gates < 0 ||
        C.n_gates > kBMaxGates || C.n_params < 0 || C.n_params > kBMaxParams ||
        (C.n_gates > 0 && !C.gates)) {
      set_error("%s: circuit %d outside the batch limits (qubits <= %d, gates <= %d,"
                " parameters <= %d)", who, c, SV_BATCH_MAX_QUBITS, kBMaxGates, kBMaxParams);
      return SV_ERR_INVALID;
    }
    if (H.n_terms < 0 || H.n_terms > kBMaxTerms || (H.n_terms > 0 && (!H.xmask || !H.zmask || !H.coeff))) {
      set_error("%s: Hamiltonian %d must have 0..%d terms", who, c, kBMaxTerms);
      return SV_ERR_INVALID;
    }
    const uint64_t lim = (uint64_t(1) << C.n_qubits) - 1;
    for (int t = 0; t < H.n_terms; ++t)
      if ((H.xmask[t] | H.zmask[t]) & ~lim) {
        set_error("%s: Hamiltonian %d term %d has bits beyond %d qubits", who, c, t, C.n_qubits);
        return SV_ERR_INVALID;
      }
    for (int i = 0; i < C.n_gates; ++i) {
      const sv_gate& g = C.gates[i];
      const bool onequbit = g.kind >= SV_GATE_H && g.kind <= SV_GATE_U1 && g.n_tar == 1;
      bool ok = onequbit && g.n_ctrl >= 0 && g.n_ctrl <= 3 && g.param >= -1 && g.param < C.n_params;
      if (g.param >= 0 && g.kind != SV_GATE_RX && g.kind != SV_GATE_RY && g.kind != SV_GATE_RZ) ok = false;
      uint64_t seen = 0;
      for (int j = 0; ok && j < 1 + g.n_ctrl; ++j) {
        const int q = j == 0 ? g.targets[0] : g.controls[j - 1];
        if (q < 0 || q >= C.n_qubits || ((seen >> q) & 1)) ok = false;
        else seen |= uint64_t(1) << q;
      }
      if (!ok) {
        set_error("%s: circuit %d gate %d: the batch kernel takes 1-qubit kinds "
                  "(H X Y Z RX RY RZ U1) with up to 3 controls; parameters on RX/RY/RZ only", who, c, i);
        return SV_ERR_INVALID;
      }
    }
    nmax = std::max(nmax, C.n_qubits);
    for (int i = 0; i < C.n_gates; ++i) width = std::max(width, 1 + C.gates[i].n_ctrl);
  }
  *nmax_out = nmax;
  *width_out = width;
  return SV_OK;
}

extern "C" {

sv_status sv_batch_plan(const sv_circuit* circuits, const sv_pauli_sum* hamiltonians,
                        int n_circuits, int k, int32_t* groups_per_circuit) {
  int nmax = 0, width = 0;
  sv_status st = validate_batch("sv_batch_plan", circuits, hamiltonians, n_circuits, &nmax, &width);
  if (st) return st;
  if (k < 2 || k > 5 || k < width || !groups_per_circuit) {
    set_error("sv_batch_plan: group width %d must be in max(2, widest gate %d)..5", k, width);
    return SV_ERR_INVALID;
  }
  HostPlan P;
  for (int c = 0; c < n_circuits; ++c) {
    const size_t g0 = P.groups.size();
    if (!plan_circuit(&circuits[c], &hamiltonians[c], k, &P)) {
      set_error("sv_batch_plan: circuit %d does not fit groups of %d qubits", c, k);
      return SV_ERR_INVALID;
    }
    groups_per_circuit[c] = (int32_t)(P.groups.size() - g0);
  }
  return SV_OK;
}

sv_status sv_batch_create(const sv_circuit* circuits, const sv_pauli_sum* hamiltonians,
                          int n_circuits, const int32_t* item_circuit, int n_items, int tune,
                          sv_batch* out) {
  if (!item_circuit || !out || n_items < 1 || tune < 0 || tune > 4) {
    set_error("sv_batch_create: bad arguments");
    return SV_ERR_INVALID;
  }
  int nmax = 1, width = 1;
  {
    sv_status vs = validate_batch("sv_batch_create", circuits, hamiltonians, n_circuits, &nmax,
                                  &width);
    if (vs) return vs;
  }
  std::vector<int> ic(item_circuit, item_circuit + n_items), toff(n_items);
  int total = 0;
  for (int i = 0; i < n_items; ++i) {
    if (ic[i] < 0 || ic[i] >= n_circuits) {
      set_error("sv_batch_create: item %d names circuit %d of %d", i, ic[i], n_circuits);
      return SV_ERR_INVALID;
    }
    toff[i] = total;
    total += circuits[ic[i]].n_params;
  }
  sv_batch b = new sv_batch_s();
  b->n_items = n_items;
  b->nmax = nmax;
  b->total_params = total;
  // batch packing: longest items first (work ~ gates x 2^n)
  std::vector<int> order(n_items);
  for (int i = 0; i < n_items; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
    const sv_circuit& A = circuits[ic[a]];
    const sv_circuit& C = circuits[ic[c]];
    return (double)A.n_gates * (1 << A.n_qubits) > (double)C.n_gates * (1 << C.n_qubits);
  });
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = 152;
  // candidates: group width k, threads per block, blocks per SM
  struct Cand {
    int k, threads, per_sm;
    bool cl;          // two-block clusters (per_sm = 1, threads = kClThreads)
    bool sms = false; // states in shared memory as far as they fit
    bool re = false;  // real amplitudes
  };
  // real batch: every gate real (H, X, Z, RY, with controls) and every term a
  // real matrix (an even number of Y factors)
  bool all_real = true;
  for (int c = 0; c < n_circuits && all_real; ++c) {
    for (int i = 0; i < circuits[c].n_gates; ++i) {
      const int kd = circuits[c].gates[i].kind;
      if (kd != SV_GATE_H && kd != SV_GATE_X && kd != SV_GATE_Z && kd != SV_GATE_RY) all_real = false;
    }
    for (int t = 0; t < hamiltonians[c].n_terms; ++t)
      if (popc64(hamiltonians[c].xmask[t] & hamiltonians[c].zmask[t]) & 1) all_real = false;
  }
  std::vector<Cand> cands;
  if (tune == 4) {
    if (!all_real) {
      set_error("sv_batch_create: tune = 4 (real amplitudes) needs every gate real (H X Z RY)"
                " and every term with an even number of Y factors");
      delete b;
      return SV_ERR_INVALID;
    }
    cands.push_back({std::max(4, width), 512, 1, false, true, true});
  } else if (tune == 1) {
    const Cand all[] = {{3, 512, 1, false, true, true}, {4, 512, 1, false, true, true},
                        {5, 512, 1, false, true, true},
                        {2, 512, 1, false, true}, {3, 512, 1, false, true}, {4, 512, 1, false, true},
                        {2, kClThreads, 1, true}, {3, kClThreads, 1, true},
                        {2, 256, 2, false}, {3, 256, 2, false}, {4, 256, 2, false},
                        {2, 256, 4, false}, {3, 256, 4, false}, {2, 128, 8, false},
                        {3, 128, 8, false}};
    for (const Cand& c : all)
      if (c.k >= width && (!c.re || all_real)) cands.push_back(c);
  } else if (tune == 2 && width <= 3) {
    cands.push_back({3, kClThreads, 1, true});
  } else if (tune == 3) {
    cands.push_back({std::max(4, width), 512, 1, false, true});
  } else {
    cands.push_back({std::max(4, width), 256, 2, false});
  }
  int max_per = 1;
  for (auto& c : cands) max_per = std::max(max_per, c.per_sm);
  b->work_slots = (size_t)sms * max_per;
  b->sms = sms;
  sv_status st = SV_OK;
  // plans per k are built on demand; start with the device buffers that do not depend on k
  b->h_order = order;
  b->h_item_circ = ic;
  st = upload(&b->order, order);
  if (!st) st = upload(&b->item_circ, ic);
  if (!st) st = upload(&b->theta_off, toff);
  if (!st) {
    cudaError_t e = cudaMalloc(&b->queue, (kBPhases + 1) * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&b->work, b->work_slots * (sizeof(float2) << (std::max(nmax, 5) + 1)));
    if (e != cudaSuccess) {
      set_error("sv_batch_create: %s", cudaGetErrorString(e));
      st = e == cudaErrorMemoryAllocation ? SV_ERR_OOM : SV_ERR_CUDA;
    }
  }
  auto build_for_k = [&](int k) -> sv_status {
    HostPlan P;
    for (int c = 0; c < n_circuits; ++c)
      if (!plan_circuit(&circuits[c], &hamiltonians[c], k, &P)) {
        set_error("sv_batch_create: a gate does not fit a register group of %d qubits", k);
        return SV_ERR_INVALID;
      }
    tile_lists(&P);
    b->h_circs = P.circs;
    b->h_ops.clear();
    for (const BCirc& C : P.circs)
      b->h_ops.push_back(C.ngroups ? P.rgroups[C.group0 + C.ngroups - 1].op1 - P.rgroups[C.group0].op0
                                   : 0);
    void* olds[] = {b->circs, b->gates, b->groups, b->ops, b->terms, b->rgroups, b->rops, b->rsigns,
                    b->rots, b->gens};
    for (void* p : olds)
      if (p) cudaFree(p);
    b->circs = nullptr; b->gates = nullptr; b->groups = nullptr; b->ops = nullptr; b->terms = nullptr;
    b->rgroups = nullptr; b->rops = nullptr; b->rsigns = nullptr; b->rots = nullptr; b->gens = nullptr;
    sv_status s2 = upload(&b->circs, P.circs);
    if (!s2) s2 = upload(&b->gates, P.gates);
    if (!s2) s2 = upload(&b->groups, P.groups);
    if (!s2) s2 = upload(&b->ops, P.ops);
    if (!s2) s2 = upload(&b->terms, P.terms);
    if (!s2) s2 = upload(&b->rgroups, P.rgroups);
    if (!s2) s2 = upload(&b->rops, P.rops);
    if (!s2) s2 = upload(&b->rsigns, P.rsigns);
    if (!s2) s2 = upload(&b->rots, P.rots);
    if (!s2) s2 = upload(&b->gens, P.gens);
    return s2;
  };
  double* th = nullptr;
  double* en = nullptr;
  double* gr = nullptr;
  if (!st && cands.size() > 1) {
    // autotune on the real batch with arbitrary parameters (timing does not depend on them)
    std::vector<double> tv(std::max(1, total));
    for (size_t i = 0; i < tv.size(); ++i) tv[i] = 0.001 * (double)(i % 997);
    cudaError_t e = cudaMalloc(&th, tv.size() * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&en, n_items * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&gr, tv.size() * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpy(th, tv.data(), tv.size() * sizeof(double), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
      set_error("sv_batch_create: tuning buffers: %s", cudaGetErrorString(e));
      st = SV_ERR_CUDA;
    }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int built = -1;
    for (const Cand& c : cands) {
      if (st) break;
      if (c.k != built) {
        st = build_for_k(c.k);
        built = c.k;
        if (st) break;
      }
      const int blocks = c.cl ? 2 * (sms / 2) : sms * c.per_sm;
      st = set_phases(b, c.k, c.threads, c.sms || c.re, c.re);
      if (st) break;
      st = launch_batch(b, th, en, gr, 0, c.k, c.threads, blocks, c.cl, c.sms, c.re);  // warm-up
      if (st) break;
      cudaEventRecord(e0, 0);
      st = launch_batch(b, th, en, gr, 0, c.k, c.threads, blocks, c.cl, c.sms, c.re);
      cudaEventRecord(e1, 0);
      if (cudaEventSynchronize(e1) != cudaSuccess) {
        set_error("sv_batch_create: tuning run failed: %s", cudaGetErrorString(cudaGetLastError()));
        st = SV_ERR_CUDA;
        break;
      }
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (ms < best) {
        best = ms;
        b->k = c.k;
        b->threads = c.threads;
        b->blocks = blocks;
        b->cluster = c.cl;
        b->smem_states = c.sms;
        b->real = c.re;
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
  } else if (!st) {
    b->k = cands[0].k;
    b->threads = cands[0].threads;
    b->cluster = cands[0].cl;
    b->smem_states = cands[0].sms;
    b->real = cands[0].re;
    b->blocks = cands[0].cl ? 2 * (sms / 2) : sms * cands[0].per_sm;
  }
  if (th) cudaFree(th);
  if (en) cudaFree(en);
  if (gr) cudaFree(gr);
  if (!st) st = build_for_k(b->k);
  if (!st) st = set_phases(b, b->k, b->threads, b->smem_states || b->real, b->real);
  if (!st) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
      set_error("sv_batch_create: %s", cudaGetErrorString(e));
      st = SV_ERR_CUDA;
    }
  }
  if (st) {
    free_batch(b);
    delete b;
    return st;
  }
  *out = b;
  return SV_OK;
}

sv_status sv_batch_info(sv_batch b, int* k, int* threads, int* blocks, int* total_params) {
  if (!b) {
    set_error("sv_batch_info: null batch");
    return SV_ERR_INVALID;
  }
  if (k) *k = b->k;
  if (threads) *threads = b->threads;
  if (blocks) *blocks = b->blocks;
  if (total_params) *total_params = b->total_params;
  return SV_OK;
}

sv_status sv_batch_kernel(sv_batch b, int* cluster_size, int* smem_states, int* real_states) {
  if (!b || !cluster_size || !smem_states || !real_states) {
    set_error("sv_batch_kernel: bad arguments");
    return SV_ERR_INVALID;
  }
  *cluster_size = b->cluster ? 2 : 1;
  *smem_states = (b->cluster || b->smem_states || b->real) ? 1 : 0;
  *real_states = b->real ? 1 : 0;
  return SV_OK;
}

sv_status sv_batch_run(sv_batch b, const double* dev_theta, double* dev_energy, double* dev_grad,
                       void* cuda_stream) {
  if (!b || !dev_theta || !dev_energy || !dev_grad) {
    set_error("sv_batch_run: bad arguments");
    return SV_ERR_INVALID;
  }
  return launch_batch(b, dev_theta, dev_energy, dev_grad, (cudaStream_t)cuda_stream, b->k,
                      b->threads, b->blocks, b->cluster, b->smem_states, b->real);
}

sv_status sv_batch_run_graph(sv_batch b, const double* dev_theta, double* dev_energy,
                             double* dev_grad, void* cuda_stream) {
  if (!b || !dev_theta || !dev_energy || !dev_grad) {
    set_error("sv_batch_run_graph: bad arguments");
    return SV_ERR_INVALID;
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const void* key[4] = {dev_theta, dev_energy, dev_grad, cuda_stream};
  if (!b->gexec || memcmp(key, b->g_key, sizeof(key)) != 0) {
    if (b->gexec) {
      cudaGraphExecDestroy(b->gexec);
      b->gexec = nullptr;
    }
    cudaStream_t cap = nullptr;
    SV_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    sv_status s2 = SV_OK;
    if (e == cudaSuccess) {
      s2 = launch_batch(b, dev_theta, dev_energy, dev_grad, cap, b->k, b->threads, b->blocks,
                        b->cluster, b->smem_states, b->real);
      e = cudaStreamEndCapture(cap, &g);
    }
    if (e == cudaSuccess && s2 == SV_OK) e = cudaGraphInstantiate(&b->gexec, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cap);
    if (e != cudaSuccess || s2 != SV_OK) {
      if (e != cudaSuccess) set_error("sv_batch_run_graph: capture: %s", cudaGetErrorString(e));
      b->gexec = nullptr;
      return s2 != SV_OK ? s2 : SV_ERR_CUDA;
    }
    memcpy(b->g_key, key, sizeof(key));
  }
  SV_CUDA_TRY(cudaGraphLaunch(b->gexec, st));
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return SV_OK;
}

sv_status sv_batch_grad(const sv_circuit* circuits, const sv_pauli_sum* hamiltonians,
                        int n_circuits, const int32_t* item_circuit, int n_items,
                        const double* theta, void* cuda_stream, double* energies, double* grads) {
  if (!theta || !energies || !grads) {
    set_error("sv_batch_grad: null host arrays");
    return SV_ERR_INVALID;
  }
  sv_batch b = nullptr;
  sv_status st = sv_batch_create(circuits, hamiltonians, n_circuits, item_circuit, n_items, 0, &b);
  if (st) return st;
  const size_t np = std::max(1, b->total_params);
  double *th = nullptr, *en = nullptr, *gr = nullptr;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaMalloc(&th, np * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&en, n_items * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&gr, np * sizeof(double));
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(th, theta, b->total_params * sizeof(double), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    st = sv_batch_run(b, th, en, gr, cuda_stream);
    if (!st) {
      e = cudaMemcpyAsync(energies, en, n_items * sizeof(double), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(grads, gr, b->total_params * sizeof(double), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
  }
  if (e != cudaSuccess && !st) {
    set_error("sv_batch_grad: %s", cudaGetErrorString(e));
    st = e == cudaErrorMemoryAllocation ? SV_ERR_OOM : SV_ERR_CUDA;
  }
  if (th) cudaFree(th);
  if (en) cudaFree(en);
  if (gr) cudaFree(gr);
  sv_batch_free(b);
  return st;
}

sv_status sv_batch_free(sv_batch b) {
  if (!b) return SV_OK;
  cudaDeviceSynchronize();
  free_batch(b);
  delete b;
  return SV_OK;
}

}  // extern "C"
