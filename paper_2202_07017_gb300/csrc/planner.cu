// Gate-fusion planner (host, fp64).
//
// The paper applies a circuit gate by gate (Sec. 2, Eq. 1), one pass over
// the 2^n-amplitude state per gate.  Here consecutive gates are grouped
// into passes: a pass stages m amplitude-index bits S (the L lowest bits,
// giving contiguous runs, plus high bits) so that each thread block loads
// one 2^m-amplitude slice into shared memory, applies every gate of the
// pass whose qubits lie in S, and writes the slice back: one HBM round
// trip for many gates.  Gates on disjoint qubits commute, so any order
// that keeps, for every qubit, the circuit order of the gates touching it
// computes the same product.
//
// Planning steps:
//   1. gates become FGates (1-qubit dense with controls, phase on an
//      all-ones subspace, SWAP with controls, or "alone" for anything else
//      or anything wider than fuse_k qubits); consecutive uncontrolled
//      1-qubit gates on one qubit are multiplied into one 2x2 in fp64;
//   2. a pass's S is grown greedily from the earliest remaining gate (unused
//      places filled with the lowest free bits, for longer contiguous runs), or
//      is the low run plus a contiguous window of high bits, whichever takes more
//      gates: every remaining gate whose qubits lie in S and that no skipped
//      earlier gate overlaps;
//   3. the pass's gates are list-scheduled into register groups of at
//      most fuse_k qubits (a gate joins the open group when every earlier
//      unscheduled gate it overlaps is scheduled and the union stays within
//      fuse_k qubits).
#include <algorithm>
#include <cmath>

#include "sv_internal.cuh"

namespace sv {
namespace {

int popc(uint64_t x) { return __builtin_popcountll(x); }

bool is_zero(cd z) { return z.re == 0.0 && z.im == 0.0; }
bool is_one(cd z) { return z.re == 1.0 && z.im == 0.0; }

// a := b * a (2x2 complex, row-major)
void mul2_left(const cd* b, cd* a) {
  cd r[4];
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      double re = 0, im = 0;
      for (int k = 0; k < 2; ++k) {
        const cd x = b[i * 2 + k], y = a[k * 2 + j];
        re += x.re * y.re - x.im * y.im;
        im += x.re * y.im + x.im * y.re;
      }
      r[i * 2 + j] = {re, im};
    }
  for (int e = 0; e < 4; ++e) a[e] = r[e];
}

// The FGate of circuit gate g (index i) with matrix G, in bit positions.
FGate classify(const sv_gate& g, int i, int n, const HostMatrix& G, int kmax) {
  FGate f;
  f.orig = i;
  f.origs.push_back(i);
  int tp[SV_MAX_TARGETS];
  uint64_t cm = 0;
  for (int j = 0; j < g.n_tar; ++j) {
    tp[j] = n - 1 - g.targets[j];
    f.qmask |= uint64_t(1) << tp[j];
  }
  for (int j = 0; j < g.n_ctrl; ++j) cm |= uint64_t(1) << (n - 1 - g.controls[j]);
  f.qmask |= cm;
  const int k = g.n_tar, d = 1 << k;
  bool diag = true, ones = true;
  for (int r = 0; r < d; ++r)
    for (int q = 0; q < d; ++q)
      if (r != q && !is_zero(G.at(r, q))) diag = false;
  for (int r = 0; r + 1 < d; ++r)
    if (!is_one(G.at(r, r))) ones = false;
  bool swap = k == 2;
  if (swap) {
    static const int perm[4] = {0, 2, 1, 3};
    for (int r = 0; r < 4; ++r)
      for (int q = 0; q < 4; ++q)
        if (q == perm[r] ? !is_one(G.at(r, q)) : !is_zero(G.at(r, q))) swap = false;
  }
  f.diag = diag;
  if (diag && ones) {
    f.type = FG_PHASE;
    f.cmask = f.qmask;
    f.m[0] = G.at(d - 1, d - 1);
  } else if (swap) {
    f.type = FG_SWAP;
    f.a = tp[0];
    f.b = tp[1];
    f.cmask = cm;
  } else if (k == 1) {
    f.type = FG_1Q;
    f.t = tp[0];
    f.cmask = cm;
    for (int e = 0; e < 4; ++e) f.m[e] = G.m[e];
  } else {
    f.type = FG_ALONE;
  }
  if (popc(f.qmask) > kmax) f.type = FG_ALONE;
  // a multi-qubit Pauli string runs as one rotation pass of its own
  if (g.kind == SV_GATE_PAULI && k > 1) f.type = FG_ALONE;
  return f;
}

// Appends f, multiplying an uncontrolled 1-qubit gate into the previous
// operation on its qubit when that is an uncontrolled 1-qubit gate.
void push_fgate(FGate f, std::vector<int>* last, std::vector<FGate>* out) {
  if (f.type == FG_1Q && f.cmask == 0) {
    const int p = (*last)[f.t];
    if (p >= 0 && (*out)[p].type == FG_1Q && (*out)[p].cmask == 0 && (*out)[p].t == f.t) {
      mul2_left(f.m, (*out)[p].m);
      for (int o : f.origs) (*out)[p].origs.push_back(o);
      (*out)[p].orig = f.orig;
      return;
    }
  }
  out->push_back(std::move(f));
  for (uint64_t q = out->back().qmask; q; q &= q - 1)
    (*last)[__builtin_ctzll(q)] = (int)out->size() - 1;
}

// 2x2 complex products (row-major)
void mul2(const cd* a, const cd* b, cd* out) {  // out = a b
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      double re = 0, im = 0;
      for (int k = 0; k < 2; ++k) {
        const cd x = a[i * 2 + k], y = b[k * 2 + j];
        re += x.re * y.re - x.im * y.im;
        im += x.re * y.im + x.im * y.re;
      }
      out[i * 2 + j] = {re, im};
    }
}

// (a, d, re b, im b) of an FG_GRAD's generator [[a, b], [conj b, d]]
void generator_of(const FGate& g, double* out) {
  static const double kPauli[4][4] = {{0, 0, 0, 0}, {0, 0, 1, 0}, {0, 0, 0, -1}, {1, -1, 0, 0}};
  if (g.pauli) {
    for (int e = 0; e < 4; ++e) out[e] = kPauli[g.pauli][e];
  } else {
    out[0] = g.m[0].re;
    out[1] = g.m[3].re;
    out[2] = g.m[1].re;
    out[3] = g.m[1].im;
  }
}

bool is_unitary2(const cd* u) {
  for (int i = 0; i < 2; ++i)
    for (int j = i; j < 2; ++j) {
      double re = 0, im = 0;
      for (int r = 0; r < 2; ++r) {  // (U^dagger U)_ij
        const cd x = u[r * 2 + i], y = u[r * 2 + j];
        re += x.re * y.re + x.im * y.im;
        im += x.re * y.im - x.im * y.re;
      }
      if (std::fabs(re - (i == j ? 1.0 : 0.0)) > 1e-12 || std::fabs(im) > 1e-12) return false;
    }
  return true;
}

// Input phases moved back.  A rotation U = A S B between diagonals (see
// rotation_form in fused_kernels.cu) needs B applied before S: as the first gate of a
// register group that is a diagonal of its own over the whole state.  B
// commutes with the diagonal gates between U and the previous uncontrolled
// 1-qubit gate V on the qubit, so V takes it: V <- diag(1, beta) V, U <- U
// diag(1, 1 / beta), beta = -u01 conj(u00) / |u01 u00|, whatever pass V is in.
// Generators of gradients on the qubit in between are carried over.  A register
// group then starts with a diagonal only for a qubit's first gate: random layered
// circuit, n = 28, depth 30 (159 groups of 442 layers), 1255 -> 1211 us a pass.
void move_input_phases(std::vector<FGate>* F) {
  struct Before {
    int gate = -1;           // the previous uncontrolled 1-qubit gate on the bit
    std::vector<int> grads;  // gradients on the bit since
  };
  std::vector<Before> before(64);
  for (int j = 0; j < (int)F->size(); ++j) {
    FGate& f = (*F)[j];
    if (f.type == FG_GRAD && f.cmask == 0) {
      before[f.t].grads.push_back(j);
      continue;
    }
    if (f.type == FG_1Q && f.cmask == 0 && !(is_zero(f.m[1]) && is_zero(f.m[2]))) {
      Before& b = before[f.t];
      const cd u = f.m[0], w = f.m[1];
      const double d = std::sqrt((u.re * u.re + u.im * u.im) * (w.re * w.re + w.im * w.im));
      const cd beta{-(w.re * u.re + w.im * u.im) / d, -(w.im * u.re - w.re * u.im) / d};
      if (b.gate >= 0 && d > 1e-10 && is_unitary2(f.m) && !is_one(beta)) {
        const cd in[4] = {{1, 0}, {0, 0}, {0, 0}, beta};
        const cd out[4] = {{1, 0}, {0, 0}, {0, 0}, {beta.re, -beta.im}};
        mul2_left(in, (*F)[b.gate].m);
        cd r[4];
        mul2(f.m, out, r);
        for (int e = 0; e < 4; ++e) f.m[e] = r[e];
        for (int g : b.grads) {
          FGate& h = (*F)[g];
          if (h.ng == 1) generator_of(h, h.gen[0]);
          for (int i = 0; i < h.ng; ++i) {  // off-diagonal times conj(beta)
            double* q = h.gen[i];
            const double re = q[2] * beta.re + q[3] * beta.im, im = q[3] * beta.re - q[2] * beta.im;
            q[2] = re;
            q[3] = im;
          }
          if (h.ng == 1) {
            const double* q = h.gen[0];
            h.pauli = 0;
            h.m[0] = {q[0], 0};
            h.m[1] = {q[2], q[3]};
            h.m[2] = {q[2], -q[3]};
            h.m[3] = {q[1], 0};
          }
        }
      }
      b.gate = j;
      b.grads.clear();
      continue;
    }
    if (f.diag || (f.type == FG_1Q && f.cmask == 0)) continue;  // commutes
    for (uint64_t q = f.qmask; q; q &= q - 1) {
      Before& b = before[__builtin_ctzll(q)];
      b.gate = -1;
      b.grads.clear();
    }
  }
}

bool to_fgates(const sv_circuit* c, const double* theta, int kmax, std::vector<FGate>* out) {
  const int n = c->n_qubits;
  std::vector<int> last(64, -1);
  HostMatrix G;
  for (int i = 0; i < c->n_gates; ++i) {
    const sv_gate& g = c->gates[i];
    if (!gate_matrix(g, theta, c->mat_pool, &G)) {
      set_error("gate %d: cannot build matrix", i);
      return false;
    }
    push_fgate(classify(g, i, n, G, kmax), &last, out);
  }
  return true;
}

// Reverse sweep over [lo, hi): gate hi-1 first, each as its adjoint, a
// parameterised gate preceded by its FG_GRAD.  Uncontrolled 1-qubit
// adjoints are kept pending per qubit (their product W, not yet applied)
// until another kind of gate touches the qubit; a gradient met while W is
// pending is evaluated on the untransformed states with the generator
// W^dagger P W (Im<W lambda|P|W psi> = Im<lambda|W^dagger P W|psi>), so a
// run RZ, RY, RX on one qubit costs one un-apply.  Gradients on one qubit with
// nothing else touching it in between share one FG_GRAD (up to kGradPerOp):
// the ops between them act on other qubits, commute with the generator and
// leave the inner product unchanged.  A parameterised gate
// wider than kmax stays unfused with its gradient.
bool to_fgates_reverse(const sv_circuit* c, const double* theta, int lo, int hi,
                       const std::vector<int>& slot_of, int kmax, std::vector<FGate>* out) {
  const int n = c->n_qubits;
  std::vector<int> last(64, -1);
  struct Pend {
    bool on = false;
    cd W[4];
    int orig = -1;
    std::vector<int> origs;  // every circuit gate folded into W
  };
  std::vector<Pend> pend(64);
  auto flush = [&](int t) {
    if (!pend[t].on) return;
    FGate f;
    f.type = FG_1Q;
    f.t = t;
    f.qmask = uint64_t(1) << t;
    f.cmask = 0;
    for (int e = 0; e < 4; ++e) f.m[e] = pend[t].W[e];
    f.orig = pend[t].orig;
    f.origs.swap(pend[t].origs);
    push_fgate(std::move(f), &last, out);
    pend[t].on = false;
  };
  HostMatrix G, D;
  for (int i = hi - 1; i >= lo; --i) {
    const sv_gate& g = c->gates[i];
    if (!gate_matrix(g, theta, c->mat_pool, &G)) {
      set_error("gate %d: cannot build matrix", i);
      return false;
    }
    const int d = 1 << G.k;
    D.k = G.k;
    for (int r = 0; r < d; ++r)
      for (int q = 0; q < d; ++q) {
        const cd z = G.at(q, r);
        D.m[r * d + q] = {z.re, -z.im};
      }
    FGate f = classify(g, i, n, D, kmax);
    if (f.type == FG_PHASE && G.k == 1 && g.n_ctrl == 0) {  // Z, U1: a 1-qubit adjoint too
      f.type = FG_1Q;
      f.t = n - 1 - g.targets[0];
      f.cmask = 0;
      for (int e = 0; e < 4; ++e) f.m[e] = D.m[e];
    }
    // generator of a parameterised gate: 1 X, 2 Y, 3 Z on its target; a
    // multi-qubit PAULI string (4) stays unfused with its own adjoint kernel
    int pauli = 0;
    if (g.param >= 0) {
      if (g.kind == SV_GATE_PAULI)
        pauli = g.n_tar == 1 ? (g.paulis & 3) : 4;
      else
        pauli = g.kind == SV_GATE_RX ? 1 : g.kind == SV_GATE_RY ? 2 : 3;
    }
    if (g.kind == SV_GATE_PAULI && g.n_tar > 1) f.type = FG_ALONE;
    if (f.type == FG_1Q && f.cmask == 0) {
      const int t = f.t;
      if (pauli) {
        FGate gr;
        gr.type = FG_GRAD;
        gr.qmask = uint64_t(1) << t;
        gr.t = t;
        gr.cmask = 0;
        gr.pauli = pauli;
        gr.slot = slot_of[i];
        gr.orig = i;
        if (pend[t].on) {  // generator W^dagger P W, stored as a Hermitian 2x2
          static const cd PX[4] = {{0, 0}, {1, 0}, {1, 0}, {0, 0}};
          static const cd PY[4] = {{0, 0}, {0, -1}, {0, 1}, {0, 0}};
          static const cd PZ[4] = {{1, 0}, {0, 0}, {0, 0}, {-1, 0}};
          const cd* P = pauli == 1 ? PX : pauli == 2 ? PY : PZ;
          const cd* W = pend[t].W;
          const cd Wd[4] = {{W[0].re, -W[0].im}, {W[2].re, -W[2].im},
                            {W[1].re, -W[1].im}, {W[3].re, -W[3].im}};
          cd PW[4], M[4];
          mul2(P, W, PW);
          mul2(Wd, PW, M);
          gr.pauli = 0;  // general generator in m
          for (int e = 0; e < 4; ++e) gr.m[e] = M[e];
        }
        // nothing has touched t since a gradient on t: evaluate this one there
        const int p = last[t];
        if (p >= 0 && (*out)[p].type == FG_GRAD && (*out)[p].cmask == 0 && (*out)[p].t == t &&
            (*out)[p].ng < kGradPerOp) {
          FGate& h = (*out)[p];
          if (h.ng == 1) {
            generator_of(h, h.gen[0]);
            h.gslots[0] = h.slot;
          }
          generator_of(gr, h.gen[h.ng]);
          h.gslots[h.ng++] = gr.slot;
        } else {
          push_fgate(std::move(gr), &last, out);
        }
      }
      if (pend[t].on) {
        cd r[4];
        mul2(f.m, pend[t].W, r);  // this adjoint acts after the pending product
        for (int e = 0; e < 4; ++e) pend[t].W[e] = r[e];
      } else {
        pend[t].on = true;
        for (int e = 0; e < 4; ++e) pend[t].W[e] = f.m[e];
      }
      pend[t].orig = i;
      pend[t].origs.push_back(i);
      continue;
    }
    for (uint64_t q = f.qmask; q; q &= q - 1) flush(__builtin_ctzll(q));
    if (pauli) {
      if (f.type == FG_ALONE) {
        f.pauli = pauli;
        f.slot = slot_of[i];
      } else {
        FGate gr;
        gr.type = FG_GRAD;
        gr.qmask = f.qmask;
        gr.t = n - 1 - g.targets[0];
        gr.cmask = f.qmask & ~(uint64_t(1) << gr.t);
        gr.pauli = pauli;
        gr.slot = slot_of[i];
        gr.orig = i;
        push_fgate(std::move(gr), &last, out);
      }
    }
    push_fgate(std::move(f), &last, out);
  }
  for (int b = 0; b < 64; ++b) flush(b);
  return true;
}

int local_of(const std::vector<int>& S, int bit) {
  return (int)(std::lower_bound(S.begin(), S.end(), bit) - S.begin());
}

}  // namespace

FusionConfig fusion_config(int n, sv_dtype dt, int fuse_k) {
  FusionConfig c;
  c.fuse_k = std::min(fuse_k, 4);  // the pass kernel holds register groups of <= 4 qubits
  int m = std::min(n, dt == SV_C64 ? 13 : 12);
  // keep at least 2^8 blocks for mid-size states, down to 2^10 amplitudes
  if (n > 10) m = std::max(std::min(m, n - 8), std::min(n, 10));
  c.m = m;
  // 12288 bytes of coefficients and 128 layers a pass; a layer of 4 qubits has 40 fp32 (on planes)
  // or 36 fp64 coefficients, one of 3 with dithered rounding 40, one of 2 at most 24.  Groups
  // of 2 in passes of up to 124 layers in place of 72: QFT, n = 10 52.5 -> 48.2 us, n = 12
  // 77.1 -> 72.9; complex128 the same either way (n = 10 layered -4 %, n = 14 QFT +2 %).
  c.max_layers = dt == SV_C64 ? (c.fuse_k <= 2 ? 124 : 72) : 40;
  c.L = std::min(dt == SV_C64 ? 5 : 4, m);
  if (c.m - c.L < fuse_k) c.L = std::max(1, c.m - fuse_k);
  return c;
}

FusionConfig fusion_config_reverse(int n, sv_dtype dt, int fuse_k) {
  // two 2^k tiles per thread: up to 4 qubits for complex64, 3 for complex128
  FusionConfig c = fusion_config(n, dt, std::min(fuse_k, dt == SV_C64 ? 4 : 3));
  // complex128 sweeps run gate lists, where moved phases make dense matrices of RX and RY
  // and general generators of single letters (n = 18: HEA 3.18 ms without, 3.33 with,
  // QAOA 2.04 and 2.30; gradients at n = 12 off by 1.8e-15 and 3.9e-15)
  c.move_phases = dt == SV_C64;
  // only 4-qubit groups on planes are layer programs: gate lists have no layers to run out
  // of (HEA n = 12, 10 layers, complex128, groups of 2: 1469 -> 1376 us a gradient)
  if (dt != SV_C64 || c.fuse_k < 4) c.max_layers = 1 << 20;
  if (c.m > 10) {
    c.m -= 1;
    if (c.m - c.L < c.fuse_k) c.L = std::max(1, c.m - c.fuse_k);
  }
  return c;
}

namespace {

// Passes (steps 2 and 3 of the planning) over the operation list F, whose operations
// move into them.  The searches read 16 bytes of an operation, side by side in
// the order of the remaining ones, instead of the operation itself: planning
// both sweeps of the 10-layer HEA at n = 20 is a third of its gradient's time on the
// host: 1.47 -> 1.37 ms a step (the plans themselves 1.6 times as fast).
void form_passes(std::vector<FGate>& F, int n, const FusionConfig& cfg,
                 std::vector<FusionItem>* out) {
  struct Brief {
    uint64_t qmask;
    int id;
    uint8_t type, ng;
  };
  const uint64_t lowL = (cfg.L >= 64) ? ~uint64_t(0) : ((uint64_t(1) << cfg.L) - 1);
  uint64_t active = 0;
  for (const FGate& f : F) active |= f.qmask;
  std::vector<Brief> rem(F.size());  // operations not yet planned, in order
  for (size_t j = 0; j < F.size(); ++j)
    rem[j] = {F[j].qmask, (int)j, (uint8_t)F[j].type, (uint8_t)F[j].ng};
  size_t head = 0;  // rem[0..head) are planned
  out->clear();
  // The operations of a pass that stages S, in order: those inside S that no
  // skipped earlier one overlaps; at most `scan` operations looked at.  grow: S
  // takes the bits of every operation met, up to m.
  auto collect = [&](uint64_t* S, bool grow, size_t scan, std::vector<int>* take) {
    uint64_t blocked = 0;
    int nS = popc(*S), ngrads = 0, ops = 0, count = 0;
    for (size_t i = head; i < rem.size() && scan > 0; ++i, --scan) {
      const Brief f = rem[i];
      bool ok = f.type != FG_ALONE && !(f.qmask & blocked) && count < cfg.max_ops &&
                (f.type != FG_GRAD || ngrads + f.ng <= cfg.max_grads);
      if (ok) {
        const uint64_t need = f.qmask & ~*S;
        if (need && (!grow || nS + popc(need) > cfg.m)) {
          ok = false;
        } else {
          *S |= need;
          nS += popc(need);
        }
      }
      if (ok) {
        ++count;
        if (take) take->push_back((int)i);
        if (f.type == FG_GRAD) ngrads += f.ng; else ++ops;
      } else {
        blocked |= f.qmask;
        if (!(active & ~blocked & (grow && nS < cfg.m ? ~uint64_t(0) : *S))) break;
      }
    }
    return ops;
  };
  while (head < rem.size()) {
    const FGate& f0 = F[rem[head].id];
    if (f0.type == FG_ALONE || popc(f0.qmask & ~lowL) > cfg.m - cfg.L) {
      for (int o : f0.origs) {
        FusionItem it;
        it.gate = o;
        it.pauli = f0.pauli;
        it.slot = f0.slot;
        out->push_back(it);
      }
      ++head;
      continue;
    }
    // 2. the staged set: grown greedily from the earliest remaining operation,
    // or the contiguous window of high bits that takes more operations.  On
    // circuits of neighbouring gates a greedy set spreads over many short runs of
    // qubits, whose light cones close after a layer or two: a random layered
    // circuit of depth 30 on 28 qubits takes 49 passes, with windows 23.
    uint64_t S = lowL;
    int best = n > cfg.m ? collect(&S, true, F.size(), nullptr) : 0;  // or every qubit
    for (int b = 0; b < n && popc(S) < cfg.m; ++b) S |= uint64_t(1) << b;
    const int w = cfg.m - cfg.L;
    for (int lo = cfg.L; lo + w <= n && n > cfg.m; ++lo) {
      uint64_t W = lowL | (((uint64_t(1) << w) - 1) << lo);
      const int ops = collect(&W, false, 2048, nullptr);
      if (ops > best) {
        best = ops;
        S = W;
      }
    }
    std::vector<int> take;
    collect(&S, false, F.size(), &take);
    // 3. register groups by list scheduling
    std::vector<int> pending = take;
    std::vector<FusedGroup> groups;
    std::vector<int> placed;
    FusionItem item;
    item.is_pass = true;
    FusedPass& P = item.pass;
    for (int b = 0; b < n; ++b)
      if ((S >> b) & 1) P.S.push_back(b);
    P.L = 0;
    while (P.L < (int)P.S.size() && P.S[P.L] == P.L) ++P.L;
    int layers = 0;
    while (!pending.empty() && (int)groups.size() < cfg.max_groups) {
      uint64_t gq = rem[pending[0]].qmask, acc = 0;
      std::vector<int> members, rest;
      for (int j : pending) {
        const uint64_t q = rem[j].qmask;
        if (!(q & acc) && popc(gq | q) <= cfg.fuse_k) {
          gq |= q;
          members.push_back(j);
        } else {
          acc |= q;
          rest.push_back(j);
        }
      }
      // a pass holds so many layers' coefficients; the rest waits for the next.  Layers of
      // the group as a layer program: a 1-qubit gate or gradient on a bit that a diagonal
      // of the layer has touched starts the next.
      int count = 1;
      uint64_t touched = 0;
      for (int j : members) {
        const Brief& f = rem[j];
        if (f.type != FG_1Q && f.type != FG_GRAD) {
          touched |= f.qmask;
        } else if (touched & f.qmask) {
          ++count;
          touched = 0;
        }
      }
      layers += count + 1;  // and one for input phases
      if (layers > cfg.max_layers && !groups.empty()) break;
      // pad every group to the same width (one kernel instantiation per
      // pass; padded bits only widen the thread's tile)
      const int width = std::min<int>(cfg.fuse_k, (int)P.S.size());
      for (int b : P.S) {
        if (popc(gq) >= width) break;
        gq |= uint64_t(1) << b;
      }
      FusedGroup grp;
      for (int b = 0; b < n; ++b)
        if ((gq >> b) & 1) grp.bits[grp.k++] = local_of(P.S, b);
      for (int j : members) {
        grp.ops.push_back((int)P.gates.size());
        P.gates.push_back(std::move(F[rem[j].id]));
        placed.push_back(j);
      }
      groups.push_back(grp);
      pending.swap(rest);
    }
    P.groups = groups;
    // drop the placed operations; the others up to the last one move up to head's side
    std::sort(placed.begin(), placed.end());
    size_t q = placed.size();
    size_t dst = placed.empty() ? head : (size_t)placed.back() + 1;
    for (size_t i = dst; i-- > head;) {
      if (q > 0 && (size_t)placed[q - 1] == i) {
        --q;
        continue;
      }
      rem[--dst] = rem[i];
    }
    head = dst;
    out->push_back(std::move(item));
  }
}

}  // namespace

bool plan_fusion(const sv_circuit* c, const double* theta, const FusionConfig& cfg,
                 std::vector<FusionItem>* out) {
  std::vector<FGate> F;
  F.reserve(c->n_gates);
  if (!to_fgates(c, theta, std::min(cfg.fuse_k, cfg.m), &F)) return false;
  if (cfg.move_phases) move_input_phases(&F);
  form_passes(F, c->n_qubits, cfg, out);
  return true;
}

void plan_fusion_1q(int n, const std::vector<Gate1q>& gates, const FusionConfig& cfg,
                    std::vector<FusionItem>* out) {
  std::vector<FGate> F;
  std::vector<int> last(64, -1);
  for (size_t i = 0; i < gates.size(); ++i) {
    FGate f;
    f.type = FG_1Q;
    f.t = gates[i].bit;
    f.qmask = uint64_t(1) << f.t;
    f.orig = (int)i;
    f.origs.push_back((int)i);
    for (int e = 0; e < 4; ++e) f.m[e] = gates[i].m[e];
    push_fgate(std::move(f), &last, &F);
  }
  form_passes(F, n, cfg, out);
}

bool plan_fusion_reverse(const sv_circuit* c, const double* theta, int lo, int hi,
                         const std::vector<int>& slot_of, const FusionConfig& cfg,
                         std::vector<FusionItem>* out) {
  std::vector<FGate> F;
  F.reserve(2 * (size_t)(hi - lo));
  if (!to_fgates_reverse(c, theta, lo, hi, slot_of, std::min(cfg.fuse_k, cfg.m), &F))
    return false;
  if (cfg.move_phases) move_input_phases(&F);
  form_passes(F, c->n_qubits, cfg, out);
  return true;
}

}  // namespace sv
