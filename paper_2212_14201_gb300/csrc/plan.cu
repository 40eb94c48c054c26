// Fusion plans (Fusion.aggregate_operations; Section "Quantum circuit fusion").
//
// The paper merges local sub-circuits into unitary blocks before the run.  Here a
// plan partitions the program into passes, each one sweep of the state:
//   PASS_GATE  one op, plain per-gate kernel;
//   PASS_TILE  a qubit set Q (m <= 12 qubits incl. 0..2) and the gates that run
//              inside shared-memory tiles of Q in one HBM round trip.
// Greedy construction (mode GREEDY): scan the remaining gates in program order,
// growing Q with each non-diagonal target until Q is full; a gate joins the pass
// unless it must wait for a gate already deferred.  Commutation is tracked per
// qubit: a gate touches its target "non-diagonally" unless the gate is diagonal,
// and its controls (and a diagonal gate's target) "diagonally"; two gates on a
// common qubit commute when both touch it diagonally.  Diagonal gates join any
// pass (their target may lie outside Q: a per-tile scalar).
#include <math.h>
#include <stddef.h>

#include <string.h>

#include <algorithm>
#include <functional>
#include <memory>
#include <new>
#include <vector>

#include "q60pair.cuh"
#include "tile.h"

using namespace qs;

enum PassKind { PASS_GATE = 0, PASS_TILE = 1 };

struct PlanPass {
  int kind = PASS_GATE;
  uint64_t qmask = 0;
  std::vector<uint32_t> gates;
};

struct qs_plan {
  int n = 0;
  int mode = 0;
  bool learned_fallback = false;  // a learned plan that kept the greedy passes
  int kmax = 1;
  int m = TILE_DEFAULT_M;
  size_t ng = 0;
  uint64_t fingerprint = 0;
  std::vector<PlanPass> passes;
  double est_seconds = 0.0;
  int64_t n_tile = 0;
  // Every gate as its own op with its own matrix: no products of matrices or phases,
  // which would add double rounding of their own (see plan_implicit).
  bool direct = false;
};

namespace {

// Structure of a record that the plan depends on (not its angles).
uint64_t fingerprint(const qs_gate* g, size_t ng) {
  uint64_t h = 1469598103934665603ull;
  auto mix = [&](uint64_t v) {
    h ^= v;
    h *= 1099511628211ull;
  };
  for (size_t k = 0; k < ng; ++k) {
    mix((uint64_t)(uint32_t)g[k].type);
    mix((uint64_t)(uint32_t)g[k].q0);
    mix((uint64_t)(uint32_t)g[k].q1);
    mix(g[k].ctrl_mask);
    mix((uint64_t)(g[k].dagger != 0));
  }
  return h;
}

// Cost model of the greedy planner (seconds): a pass costs the larger of its HBM
// time and its arithmetic time.  Rates of the Q60 engine measured at n=30: a
// tile pass runs ~5.2e12 limb products per second, a per-gate kernel streams at
// ~60 % of HBM.  (kFp64FlopPerS serves the FP64 estimate of PLAIN plans.)
constexpr double kHbmBytesPerS = 6.6e12;
constexpr double kFp64FlopPerS = 1.0e12;
constexpr double kTileLimbPerS = 5.2e12;
constexpr double kPlainHbmFraction = 0.6;

// Limb products per touched amplitude of a gate inside a tile pass, by type.
static double op_q60_per_amp(int type) {
  switch (type) {
    case QS_U3: case QS_RX: return 18.0;
    case QS_H: case QS_RY: case QS_RZ: return 12.0;
    case QS_T: case QS_P: case QS_CR: return 12.0;
    default: return 0.0;
  }
}

double op_flops_per_amp(int type) {
  switch (type) {
    case QS_U3: case QS_RX: return 14.0;
    case QS_H: case QS_RY: return 6.0;
    case QS_RZ: return 6.0;
    case QS_T: case QS_P: case QS_CR: return 3.0;
    default: return 0.0;
  }
}

// Q60 tile engine: limb products (3 per real product) per touched amplitude; a
// general 2x2 row takes its complex products in three real products (Gauss).
double op_int_ops_per_amp(const Op1& op) {
  switch (op.cls) {
    case OP_GENERAL: return 18.0;
    case OP_REAL: return 12.0;
    case OP_PHASE1: return op.code1 == U_GENERAL ? 12.0 : 0.0;
    default: return 6.0 * ((op.code0 == U_GENERAL ? 1.0 : 0.0) + (op.code1 == U_GENERAL ? 1.0 : 0.0));
  }
}

double op_touch_fraction(const qs_gate& g, uint64_t cmask) {
  double f = 1.0 / (double)(1ull << __builtin_popcountll(cmask));
  if (g.type == QS_Z || g.type == QS_S || g.type == QS_T || g.type == QS_P || g.type == QS_CZ || g.type == QS_CR)
    f *= 0.5;
  return f;
}

}  // namespace

namespace qs {

// Whether a record is diagonal for every angle: Z, S, T, RZ, P, CZ, CR (and I).
bool structurally_diagonal(int type) {
  return type == QS_I || type == QS_Z || type == QS_S || type == QS_T || type == QS_RZ || type == QS_P ||
         type == QS_CZ || type == QS_CR;
}

}  // namespace qs

namespace qs {

// Class-based figures of a resolved (possibly merged) op, per touched amplitude:
// FP64 flops and Q60 limb products, and the fraction of amplitudes it touches.
static double class_flops_per_amp(const Op1& op) {
  const int g0 = op.code0 == U_GENERAL, g1 = op.code1 == U_GENERAL;
  switch (op.cls) {
    case OP_GENERAL: return 14.0;
    case OP_REAL: return 6.0;
    case OP_PHASE1: return g1 ? 6.0 : 0.0;
    default: return 3.0 * (g0 + g1);  // DIAG / ANTI: a complex multiply on the general half
  }
}

static double class_touch_fraction(const Op1& op) {
  const double f = 1.0 / (double)(1ull << __builtin_popcountll(op.cmask));
  return op.cls == OP_PHASE1 ? 0.5 * f : f;
}

// Work of one op inside a tile pass in limb products per amplitude, plus the
// fixed cost of one more op (its shared-memory sweep, barrier and limb splits),
// in the same units: the yardstick of the merge rule below.
constexpr double kOpOverheadPerAmp = 6.0;

static Mat2 mat_mul(const Mat2& a, const Mat2& b) {  // a * b
  Mat2 r;
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const C2 x = a.m[2 * i], y = b.m[j], u = a.m[2 * i + 1], v = b.m[2 + j];
      r.m[2 * i + j] = {x.re * y.re - x.im * y.im + u.re * v.re - u.im * v.im,
                        x.re * y.im + x.im * y.re + u.re * v.im + u.im * v.re};
    }
  return r;
}

static bool is_diagonal(const Op1& op) { return op.cls == OP_PHASE1 || op.cls == OP_DIAG || op.cls == OP_IDENTITY; }

// Aggregation of a pass's gates into fewer unitaries (the paper's
// Fusion.aggregate_operations, Section "Quantum circuit fusion").  A one-qubit
// gate g (target t, controls C) is multiplied into an earlier op p of the pass
// with the same target and controls when every op between them commutes with g:
//   - an op that touches none of t and C commutes;
//   - if g is diagonal, so does an op that is diagonal itself or whose target is
//     not among t and C (it uses them as controls only: block-diagonal there);
// and the product costs no more limb products per amplitude than the two ops did,
// plus one op's overhead.  g then moves back to p (past ops it commutes with) and
// p becomes g * p.  Ops stay in pass order; an identity product is dropped.
static int aggregate_pass(int n, const PlanPass& ps, const qs_gate* gates, const double* params,
                          std::vector<Op1>* out, int* merged) {
  std::vector<Op1>& ops = *out;
  ops.clear();
  *merged = 0;
  (void)n;
  for (uint32_t k : ps.gates) {
    int t;
    uint64_t cm;
    Mat2 mat;
    QS_TRY(gate_qubits(gates[k], n, &t, &cm));
    QS_TRY(gate_matrix(gates[k], params, &mat));
    const Op1 op = classify(t, cm, mat);
    if (op.cls == OP_IDENTITY) continue;
    const uint64_t touch = cm | (1ull << t);
    const bool diag = is_diagonal(op);
    int p = -1;
    for (int j = (int)ops.size() - 1; j >= 0; --j) {
      const Op1& o = ops[j];
      const uint64_t otouch = o.cmask | (1ull << o.target);
      if (!(otouch & touch)) continue;
      if (o.target == t && o.cmask == cm) {
        p = j;
        break;
      }
      if (diag && (is_diagonal(o) || !((touch >> o.target) & 1))) continue;
      break;
    }
    if (p >= 0) {
      const Op1 mo = classify(t, cm, mat_mul(mat, ops[p].m));
      const double before = op_int_ops_per_amp(ops[p]) * class_touch_fraction(ops[p]) +
                            op_int_ops_per_amp(op) * class_touch_fraction(op) + kOpOverheadPerAmp;
      const double after = mo.cls == OP_IDENTITY ? 0.0 : op_int_ops_per_amp(mo) * class_touch_fraction(mo);
      if (after <= before) {
        ops[p] = mo;
        ++*merged;
        continue;
      }
    }
    ops.push_back(op);
  }
  return QS_OK;
}

// ---- phase tables ----------------------------------------------------------------
// An uncontrolled general one-qubit unitary U = [[a, b], [c, d]] factors exactly
// as diag(p1, p2) R diag(1, q2), R = [[cs, -sn], [sn, cs]] real (the ZYZ Euler
// form): a = p1 cs, c = p2 sn, d = p2 cs q2, b = -p1 sn q2, with p1, p2, q2 unit
// phases.  Rounding can leave entries that are zero in exact arithmetic at 1e-17
// (and differently on platforms that fuse multiply-adds), so every phase is
// taken from an entry that is large where it matters: cs, sn from the averaged
// moduli, q2 from d when |d| >= |b|, else from -b; a noisy p1 (tiny |a|) or p2
// (tiny |c|) only multiplies a tiny entry.
// Diagonals commute with each other, with diagonal gates and with gates that use
// their qubit only as a control, so within a tile pass the phases of many qubits,
// and the controlled diagonal gates (CZ, CR, ...) among the tile's qubits, collect
// into one diagonal over the tile, applied as one table op a_j *= T[j] (one
// complex product per amplitude, T in global memory and shared by every tile), and
// the general ops shrink to real rotations (12 instead of 18 limb products per
// amplitude).  A flush emits the pending diagonals before an op that does not
// commute with them, pulling forward the right factors of the next general op of
// every qubit (and the plain diagonal gates before it); it builds a table when the
// general ops made real, the pending phases and the controlled diagonal gates it
// absorbs outweigh the table op, else the pending phase of the op's qubit is
// folded into that op (or emitted as a diagonal op) and the pending controlled
// diagonal gates on that qubit are emitted as they are.
// Gains and costs in units of one uncontrolled general op over the tile (est_op).
constexpr double kTableCost = 0.62;  // a table op
constexpr double kPullGain = 0.33;   // a general op made real
constexpr double kPhaseGain = 0.5;   // a pending phase that needs no op of its own
static bool g_phase_tables = true;

extern "C" int qs_set_phase_tables(int on) {
  g_phase_tables = on != 0;
  return QS_OK;
}

// Estimated time of an op on the Q60 tile engine, in units of one uncontrolled
// general op over the tile (measured at n=24: a real rotation 0.67, a
// general-phase diagonal 0.78); used to decide on tables and to keep the phase
// table rewrite only for passes it makes cheaper.
constexpr int kTableMark = 100;
static double est_op(const Op1& o) {
  if (o.cls == kTableMark) return kTableCost;
  const double f = 1.0 / (double)(1ull << __builtin_popcountll(o.cmask));
  const int g0 = o.code0 == U_GENERAL, g1 = o.code1 == U_GENERAL;
  double c;
  switch (o.cls) {
    case OP_GENERAL: c = 1.0; break;
    case OP_REAL: c = 0.67; break;
    case OP_DIAG: c = 0.2 + 0.29 * (g0 + g1); break;
    case OP_PHASE1: c = g1 ? 0.45 : 0.15; break;
    case OP_ANTI: c = 0.2 + 0.2 * (g0 + g1); break;
    default: c = 0.0; break;
  }
  return 0.05 + c * f;
}

static double est_ops(const std::vector<Op1>& ops) {
  double t = 0.0;
  for (const Op1& o : ops)
    if (o.cls != OP_IDENTITY) t += est_op(o);
  return t;
}

static C2 cmul2(C2 x, C2 y) { return {x.re * y.re - x.im * y.im, x.re * y.im + x.im * y.re}; }
static C2 cconj2(C2 x) { return {x.re, -x.im}; }
static C2 phase_of(C2 x) {
  const double r = std::hypot(x.re, x.im);
  return r > 0.0 ? C2{x.re / r, x.im / r} : C2{1.0, 0.0};
}

struct Zyz {
  C2 p1, p2, q2;
  Mat2 R;
};

static Zyz zyz(const Mat2& U) {
  Zyz z;
  const C2 a = U.m[0], b = U.m[1], c = U.m[2], d = U.m[3];
  const double na = std::hypot(a.re, a.im), nb = std::hypot(b.re, b.im);
  const double nc = std::hypot(c.re, c.im), nd = std::hypot(d.re, d.im);
  double cs = 0.5 * (na + nd), sn = 0.5 * (nb + nc);
  const double r = std::hypot(cs, sn);
  cs /= r;
  sn /= r;
  z.p1 = phase_of(a);
  z.p2 = phase_of(c);
  z.q2 = nd >= nb ? cmul2(phase_of(d), cconj2(z.p2)) : cmul2(phase_of({-b.re, -b.im}), cconj2(z.p1));
  z.R.m[0] = {cs, 0.0};
  z.R.m[1] = {-sn, 0.0};
  z.R.m[2] = {sn, 0.0};
  z.R.m[3] = {cs, 0.0};
  return z;
}

// A controlled diagonal gate among the tile's bits: where every bit of lmask is
// set, diag(e0, e1) on tile bit tb.
struct TableTerm {
  uint32_t lmask;
  int tb;
  C2 e0, e1;
};

// A diagonal over the tile as a product: entry j (bit b of j = tile bit b) is the
// product over the tile bits of d0 or d1 and over the terms, times a sign per
// tile: (-1)^(x_q j_t) for each (q, t) in signs (a CZ between the qubit q outside
// the tile and the tile bit t; x_q is the tile's own bit q).
struct PhaseTable {
  int m = 0;
  std::vector<C2> d0, d1;
  std::vector<TableTerm> terms;
  std::vector<std::pair<int, int>> signs;  // (global qubit outside the tile, tile bit)
};

// Its 2^m entries (the kernels get theirs from k_phase_tables).
static std::vector<C2> table_entries(const PhaseTable& pt) {
  std::vector<C2> t((size_t)1 << pt.m, C2{1.0, 0.0});
  // product over tile bits, doubling the filled prefix once per bit
  for (int b = 0; b < pt.m; ++b) {
    const size_t h = (size_t)1 << b;
    for (size_t j = 0; j < h; ++j) {
      t[j + h] = cmul2(t[j], pt.d1[b]);
      t[j] = cmul2(t[j], pt.d0[b]);
    }
  }
  for (const TableTerm& tm : pt.terms)
    for (size_t j = 0; j < t.size(); ++j)
      if ((j & tm.lmask) == tm.lmask) t[j] = cmul2(t[j], ((j >> tm.tb) & 1) ? tm.e1 : tm.e0);
  return t;
}

// A diagonal op that is a CZ between a tile bit and a qubit outside the tile:
// diag(1, -1) on its target with exactly one control, one of the two qubits
// inside the tile.  Returns the tile bit and the outside qubit.
static bool cz_across(const Op1& o, const int* local, int* tile_bit, int* outside) {
  if (__builtin_popcountll(o.cmask) != 1 || o.code1 != U_MINUS_ONE) return false;
  if (!(o.cls == OP_PHASE1 || (o.cls == OP_DIAG && o.code0 == U_ONE))) return false;
  const int c = __builtin_ctzll(o.cmask);
  const int lt = local[o.target], lc = local[c];
  if (lt >= 0 && lc < 0) {
    *tile_bit = lt;
    *outside = c;
    return true;
  }
  if (lt < 0 && lc >= 0) {
    *tile_bit = lc;
    *outside = o.target;
    return true;
  }
  return false;
}

// Rewrites ops (one pass, pass order) into real rotations, phase-table markers
// (cls = kTableMark, target = table index) and the other ops unchanged.
static bool diag_cls(int c) { return c == OP_DIAG || c == OP_PHASE1 || c == OP_IDENTITY; }

static void extract_phases(const std::vector<Op1>& ops, const int* local, int n, int m, std::vector<Op1>* out,
                           std::vector<PhaseTable>* tables) {
  const size_t N = ops.size();
  out->clear();
  std::vector<char> consumed(N, 0), pulled(N, 0);
  std::vector<Zyz> z(N);
  std::vector<char> elig(N, 0);
  for (size_t i = 0; i < N; ++i)
    if (ops[i].cls == OP_GENERAL && ops[i].cmask == 0 && local[ops[i].target] >= 0) {
      elig[i] = 1;
      z[i] = zyz(ops[i].m);
    }
  C2 d0[TILE_MAX_M], d1[TILE_MAX_M];
  bool has[TILE_MAX_M];
  int gq[TILE_MAX_M];  // tile bit -> global qubit (local[] is defined for qubits 0..n-1)
  for (int b = 0; b < TILE_MAX_M; ++b) gq[b] = 0;
  for (int b = 0; b < n; ++b)
    if (local[b] >= 0 && local[b] < m) gq[local[b]] = b;
  // pending controlled diagonal gates with every qubit in the tile
  struct Term {
    uint32_t touch;  // tile bits of its controls and target
    uint32_t lmask;  // tile bits of its controls
    int tb;          // tile bit of its target
    C2 e0, e1;
    Op1 op;
  };
  std::vector<Term> terms;
  // pending CZs between a tile bit and a qubit outside the tile (sign terms of
  // the next table; ops of their own if no table is built)
  struct XTerm {
    int tb, q;
    Op1 op;
  };
  std::vector<XTerm> xterms;
  auto reset = [&](int b) {
    d0[b] = {1.0, 0.0};
    d1[b] = {1.0, 0.0};
    has[b] = false;
  };
  for (int b = 0; b < m; ++b) reset(b);
  auto absorb = [&](int b, C2 e0, C2 e1) {
    d0[b] = cmul2(d0[b], e0);
    d1[b] = cmul2(d1[b], e1);
    has[b] = true;
  };
  auto diag_of = [&](const Op1& o, C2* e0, C2* e1) {
    *e0 = o.cls == OP_PHASE1 ? C2{1.0, 0.0} : o.m.m[0];
    *e1 = o.m.m[3];
  };
  auto emit_diag = [&](int b) {
    if (!has[b]) return;
    Mat2 M;
    M.m[0] = d0[b];
    M.m[1] = {0.0, 0.0};
    M.m[2] = {0.0, 0.0};
    M.m[3] = d1[b];
    const Op1 o = classify(gq[b], 0, M);
    if (o.cls != OP_IDENTITY) out->push_back(o);
    reset(b);
  };
  // the pending controlled diagonal gates on tile bit b, as they are
  auto emit_terms = [&](int b) {
    size_t k = 0;
    for (size_t i = 0; i < terms.size(); ++i) {
      if ((terms[i].touch >> b) & 1) out->push_back(terms[i].op);
      else terms[k++] = terms[i];
    }
    terms.resize(k);
    k = 0;
    for (size_t i = 0; i < xterms.size(); ++i) {
      if (xterms[i].tb == b) out->push_back(xterms[i].op);
      else xterms[k++] = xterms[i];
    }
    xterms.resize(k);
  };
  // candidate pulls for a flush before op i: per tile bit, the diagonal gates
  // before its next general op, and that op
  struct Pull {
    std::vector<size_t> diags;
    std::vector<size_t> xs;  // CZs across the tile boundary on this tile bit before its next general op
    long gen = -1;
    size_t stop = 0;         // the first op that acts non-diagonally on this tile bit (N if none)
  };
  // in-tile controlled diagonal gates ahead of every non-diagonal op on their
  // qubits: they commute back to the table and join it
  std::vector<size_t> tpull;
  auto plan_pulls = [&](size_t i, Pull* P) {
    int count = 0;
    for (int b = 0; b < m; ++b) {
      P[b] = Pull();
      P[b].stop = N;
      const int q = gq[b];
      for (size_t j = i; j < N; ++j) {
        if (consumed[j] || ops[j].cls == OP_IDENTITY) continue;
        const Op1& o = ops[j];
        int xtb, xq;
        if (cz_across(o, local, &xtb, &xq)) {  // diagonal: commutes up to here; a sign term if on b
          if (xtb == b) P[b].xs.push_back(j);
          continue;
        }
        if (o.target != q) continue;  // untouched, or q only a control: commutes
        if (diag_cls(o.cls)) {
          if (o.cmask == 0) P[b].diags.push_back(j);
          continue;
        }
        if (elig[j] && !pulled[j]) {
          P[b].gen = (long)j;
          ++count;
        }
        P[b].stop = j;
        break;
      }
    }
    tpull.clear();
    for (size_t j = i; j < N; ++j) {
      if (consumed[j] || ops[j].cls == OP_IDENTITY || !diag_cls(ops[j].cls) || ops[j].cmask == 0) continue;
      const Op1& o = ops[j];
      const uint64_t qs = o.cmask | (1ull << o.target);
      bool ok = true;
      for (uint64_t c = qs; c && ok; c &= c - 1) {
        const int bq = local[__builtin_ctzll(c)];
        ok = bq >= 0 && j < P[bq].stop;
      }
      if (ok) tpull.push_back(j);
    }
    return count;
  };
  // applies every pending diagonal (and the pulls): one table if two or more
  // things are pending, else each as its own op
  auto commit = [&](Pull* P) {
    // CZs across the boundary ahead of each tile bit's next general op join the
    // table's sign terms (as far as the table has room for them)
    size_t room = tables->size() < (size_t)TILE_MAX_SIGNED_TABLES ? (size_t)TILE_MAX_SIGNS : 0;
    room = room > xterms.size() ? room - xterms.size() : 0;
    for (int b = 0; b < m && room; ++b)
      for (size_t j : P[b].xs) {
        if (!room) break;
        int xtb, xq;
        cz_across(ops[j], local, &xtb, &xq);
        xterms.push_back(XTerm{xtb, xq, ops[j]});
        consumed[j] = 1;
        --room;
      }
    for (size_t j : tpull) {
      const Op1& o = ops[j];
      C2 e0, e1;
      diag_of(o, &e0, &e1);
      uint32_t lm = 0;
      for (uint64_t c = o.cmask; c; c &= c - 1) lm |= 1u << local[__builtin_ctzll(c)];
      const int tb = local[o.target];
      terms.push_back(Term{lm | (1u << tb), lm, tb, e0, e1, o});
      consumed[j] = 1;
    }
    tpull.clear();
    for (int b = 0; b < m; ++b) {
      for (size_t j : P[b].diags) {
        C2 e0, e1;
        diag_of(ops[j], &e0, &e1);
        absorb(b, e0, e1);
        consumed[j] = 1;
      }
      if (P[b].gen >= 0) {
        absorb(b, {1.0, 0.0}, z[P[b].gen].q2);
        pulled[P[b].gen] = 1;
      }
    }
    int cnt = (int)terms.size() + (int)xterms.size();
    for (int b = 0; b < m; ++b) cnt += has[b];
    if (cnt < 2) {
      for (int b = 0; b < m; ++b) {
        emit_diag(b);
        emit_terms(b);
      }
      return;
    }
    PhaseTable t;
    t.m = m;
    t.d0.assign(d0, d0 + m);
    t.d1.assign(d1, d1 + m);
    for (const Term& tm : terms) t.terms.push_back(TableTerm{tm.lmask, tm.tb, tm.e0, tm.e1});
    terms.clear();
    // sign terms: a table of a pass may carry TILE_MAX_SIGNS of them, and only the
    // first TILE_MAX_SIGNED_TABLES tables of a pass carry any; the rest stay ops
    for (const XTerm& x : xterms) {
      if (tables->size() < (size_t)TILE_MAX_SIGNED_TABLES && t.signs.size() < (size_t)TILE_MAX_SIGNS)
        t.signs.push_back({x.q, x.tb});
      else
        out->push_back(x.op);
    }
    xterms.clear();
    Op1 mark{};
    mark.cls = kTableMark;
    mark.target = (int)tables->size();
    tables->push_back(std::move(t));
    out->push_back(mark);
    for (int b = 0; b < m; ++b) reset(b);
  };
  std::vector<Pull> P(m);
  for (size_t i = 0; i < N; ++i) {
    if (consumed[i] || ops[i].cls == OP_IDENTITY) continue;
    const Op1& o = ops[i];
    const int b = local[o.target];
    int xtb = -1, xq = -1;
    if (cz_across(o, local, &xtb, &xq)) {  // a CZ across the tile boundary: pending sign term
      xterms.push_back(XTerm{xtb, xq, o});
      continue;
    }
    if (b < 0) {  // diagonal on a qubit outside the tile: commutes with every table
      out->push_back(o);
      continue;
    }
    if (diag_cls(o.cls)) {
      C2 e0, e1;
      diag_of(o, &e0, &e1);
      uint32_t lm = 0;
      bool inside = true;
      for (uint64_t c = o.cmask; c; c &= c - 1) {
        const int q = __builtin_ctzll(c);
        if (local[q] < 0) inside = false;
        else lm |= 1u << local[q];
      }
      if (o.cmask == 0) absorb(b, e0, e1);
      else if (inside) terms.push_back(Term{lm | (1u << b), lm, b, e0, e1, o});
      else out->push_back(o);  // a control outside the tile: stays an op (it commutes with the pending ones)
      continue;
    }
    if (elig[i] && pulled[i]) {  // its right factor is already in a table
      emit_diag(b);                // (nothing is pending here: a pull takes every diagonal before it)
      emit_terms(b);
      out->push_back(classify(o.target, 0, z[i].R));
      absorb(b, z[i].p1, z[i].p2);
      continue;
    }
    // o does not commute with the pending diagonals on its target.  A table now
    // pays for itself through the general ops it turns real, the pending phases
    // that would otherwise become separate diagonal ops (qubits whose next
    // non-commuting op is not a general op, like this one) and the pending
    // controlled diagonal gates it absorbs.
    const int pulls = plan_pulls(i, P.data());
    int lone = 0;
    for (int bb = 0; bb < m; ++bb)
      if (has[bb] && P[bb].gen < 0) ++lone;
    double term_gain = 0.0;
    for (const Term& tm : terms) term_gain += est_op(tm.op);
    for (const XTerm& x : xterms) term_gain += est_op(x.op);
    for (int bb = 0; bb < m; ++bb)
      for (size_t j : P[bb].xs) term_gain += est_op(ops[j]);
    for (size_t j : tpull) term_gain += est_op(ops[j]);
    if (kPullGain * pulls + kPhaseGain * lone + term_gain < kTableCost) tpull.clear();  // no table now
    if (kPullGain * pulls + kPhaseGain * lone + term_gain >= kTableCost) {
      commit(P.data());
      if (elig[i]) {  // pulled by the commit
        out->push_back(classify(o.target, 0, z[i].R));
        absorb(b, z[i].p1, z[i].p2);
        continue;
      }
      out->push_back(o);
      continue;
    }
    emit_terms(b);
    if (has[b] && elig[i]) {  // fold the pending phase into the op: U diag(d0, d1)
      Mat2 M = o.m;
      M.m[0] = cmul2(M.m[0], d0[b]);
      M.m[2] = cmul2(M.m[2], d0[b]);
      M.m[1] = cmul2(M.m[1], d1[b]);
      M.m[3] = cmul2(M.m[3], d1[b]);
      reset(b);
      out->push_back(classify(o.target, o.cmask, M));
      continue;
    }
    emit_diag(b);
    out->push_back(o);
  }
  // what is left at the end of the pass
  std::vector<Pull> none(m);
  tpull.clear();
  commit(none.data());
}

GateQueue gate_queue(const std::vector<int>& tgt, const std::vector<uint64_t>& cms) {
  GateQueue q;
  q.end = (uint32_t)tgt.size();
  for (size_t k = 0; k < tgt.size(); ++k) q.used |= cms[k] | (1ull << tgt[k]);
  return q;
}

uint64_t greedy_pass(const qs_gate* gates, const std::vector<int>& tgt, const std::vector<uint64_t>& cms,
                     const GateQueue& in, int m, uint64_t low, int max_ops, std::vector<uint32_t>& pass,
                     GateQueue& rest) {
  return greedy_pass_from(gates, tgt, cms, in, m, low, max_ops, pass, rest);
}

// Qubits to start a pass with, from the remaining gates' targets: the target of
// the first gate that can run, then the most frequent targets among the next
// `window` gates that commute back to the start of the pass (earlier first on
// ties), up to m qubits with `low`.  A pass that starts from them keeps the
// qubits most gates act on, where the greedy scan takes targets in program order.
uint64_t seed_qubits(const qs_gate* gates, const std::vector<int>& tgt, const std::vector<uint64_t>& cms,
                     const GateQueue& in, int m, uint64_t low, int window) {
  uint64_t blockedN = 0, blockedD = 0;
  int count[64] = {0}, first_seen[64];
  for (int b = 0; b < 64; ++b) first_seen[b] = 1 << 30;
  uint64_t Q = low;
  int seen = 0, order = 0, left = 0;
  const size_t nl = in.left.size(), total = nl + (in.end - in.next);
  for (size_t i = 0; i < total && left < PASS_SCAN_LEFT && (blockedN & in.used) != in.used; ++i) {
    const uint32_t k = i < nl ? in.left[i] : in.next + (uint32_t)(i - nl);
    const bool diag = structurally_diagonal(gates[k].type);
    const uint64_t Nm = diag ? 0 : (1ull << tgt[k]);
    const uint64_t Dm = (diag ? (1ull << tgt[k]) : 0) | cms[k];
    const bool blocked = (Nm & (blockedN | blockedD)) || (Dm & blockedN);
    if (blocked) {
      blockedN |= Nm;
      blockedD |= Dm;
      ++left;
      continue;
    }
    if (!Nm) continue;
    if (Q == low && !(Q & Nm)) Q |= Nm;  // the first gate that can run
    ++count[tgt[k]];
    if (first_seen[tgt[k]] > order) first_seen[tgt[k]] = order;
    ++order;
    if (++seen >= window) break;
  }
  while (__builtin_popcountll(Q) < m) {
    int best = -1;
    for (int b = 0; b < 64; ++b)
      if (!((Q >> b) & 1) && count[b] > 0 &&
          (best < 0 || count[b] > count[best] || (count[b] == count[best] && first_seen[b] < first_seen[best])))
        best = b;
    if (best < 0) break;
    Q |= 1ull << best;
  }
  return Q;
}

uint64_t greedy_pass_from(const qs_gate* gates, const std::vector<int>& tgt, const std::vector<uint64_t>& cms,
                          const GateQueue& in, int m, uint64_t init, int max_ops, std::vector<uint32_t>& pass,
                          GateQueue& rest, uint64_t forbid) {
  uint64_t Q = init;
  uint64_t blockedN = 0, blockedD = 0;
  pass.clear();
  rest.left.clear();
  rest.end = in.end;
  rest.used = in.used;
  int nops = 0;
  const size_t nl = in.left.size(), total = nl + (in.end - in.next);
  size_t i = 0;
  // (past a full pass, or once every used qubit is blocked, each gate would be left)
  for (; i < total && nops < max_ops && (blockedN & in.used) != in.used && rest.left.size() < PASS_SCAN_LEFT; ++i) {
    const uint32_t k = i < nl ? in.left[i] : in.next + (uint32_t)(i - nl);
    const bool diag = structurally_diagonal(gates[k].type);
    const uint64_t Nm = diag ? 0 : (1ull << tgt[k]);
    const uint64_t Dm = (diag ? (1ull << tgt[k]) : 0) | cms[k];
    bool conflict = (Nm & (blockedN | blockedD)) || (Dm & blockedN);
    if (!conflict && Nm && !(Q & Nm)) {
      if (__builtin_popcountll(Q) < m && !(Nm & forbid)) Q |= Nm;
      else conflict = true;
    }
    if (conflict) {
      rest.left.push_back(k);
      blockedN |= Nm;
      blockedD |= Dm;
    } else {
      pass.push_back(k);
      ++nops;
    }
  }
  if (i < nl) rest.left.insert(rest.left.end(), in.left.begin() + (ptrdiff_t)i, in.left.end());
  rest.next = in.next + (uint32_t)(i < nl ? 0 : i - nl);
  return Q;
}

}  // namespace qs

// One tile pass over the queue `in` at width m, padded to the full width:
//   strategy 0  greedy: targets taken in program order;
//   strategy 1  seeded: the scan starts from seed_qubits;
//   strategy 2  lookahead: the greedy pass, or a variant of it that never takes
//               one of the qubits the greedy scan added, whichever absorbs the
//               most gates together with the greedy pass that follows it.
// A greedy tile closes over the first m targets in program order; a target whose
// gates soon wait on qubits outside the tile (the edge of a brickwork wavefront)
// can hold a slot that another qubit would fill with more gates, and the pass
// after it can start further along.  `forbid` (strategy 0) keeps the scan off
// those qubits.  A pass of diagonal gates needs few tile qubits, but a narrow
// tile means many small tiles (a CTA pass and a barrier per op for a few
// amplitudes); qubits the pass's gates touch come first in the padding (their
// diagonal ops and controls become in-tile), then the lowest.
static uint64_t low_qubits(int n) { return (1ull << std::min(n, TILE_LOW)) - 1; }
constexpr int kPassMaxGates = TILE_MAX_OPS - 32;  // op slots left for the phase tables a pass may gain

static void pad_pass(PlanPass& ps, const std::vector<int>& tgt, const std::vector<uint64_t>& cms, int n, int m) {
  uint64_t touched = 0;
  for (uint32_t k : ps.gates) touched |= cms[k] | (1ull << tgt[k]);
  for (int b = 0; b < n && __builtin_popcountll(ps.qmask) < m; ++b)
    if (((touched >> b) & 1) && !((ps.qmask >> b) & 1)) ps.qmask |= 1ull << b;
  for (int b = 0; b < n && __builtin_popcountll(ps.qmask) < m; ++b) ps.qmask |= 1ull << b;
}

// Gates the greedy pass at width m would absorb from `rest`.
static size_t greedy_absorbed(const qs_gate* gates, const std::vector<int>& tgt, const std::vector<uint64_t>& cms,
                              const GateQueue& rest, int n, int m) {
  if (rest.empty()) return 0;
  std::vector<uint32_t> p2;
  GateQueue r2;
  greedy_pass_from(gates, tgt, cms, rest, m, low_qubits(n), kPassMaxGates, p2, r2);
  return p2.size();
}

static PlanPass make_pass(const qs_gate* gates, const std::vector<int>& tgt, const std::vector<uint64_t>& cms,
                          const GateQueue& in, int n, int m, int strategy, GateQueue& rest, uint64_t forbid = 0,
                          uint64_t* grown = nullptr) {
  const uint64_t low = low_qubits(n);
  PlanPass ps;
  ps.kind = PASS_TILE;
  if (strategy == 2) {
    uint64_t g0 = 0;
    ps = make_pass(gates, tgt, cms, in, n, m, 0, rest, 0, &g0);
    size_t best = ps.gates.size() + greedy_absorbed(gates, tgt, cms, rest, n, m);
    GateQueue r;
    for (uint64_t c = g0; c; c &= c - 1) {
      PlanPass v = make_pass(gates, tgt, cms, in, n, m, 0, r, c & (~c + 1));
      const size_t a = v.gates.size() + greedy_absorbed(gates, tgt, cms, r, n, m);
      if (a > best) {
        best = a;
        ps = std::move(v);
        std::swap(rest, r);
      }
    }
    return ps;
  }
  const uint64_t init = strategy == 1 ? seed_qubits(gates, tgt, cms, in, m, low, 4 * m) : low;
  ps.qmask = greedy_pass_from(gates, tgt, cms, in, m, init, kPassMaxGates, ps.gates, rest, forbid);
  if (grown) *grown = ps.qmask & ~low;
  pad_pass(ps, tgt, cms, n, m);
  return ps;
}

static int plan_build(int n, const qs_gate* gates, size_t ng, int mode, int kmax, int mtile, qs_plan** out,
                      int strategy = 0, bool few_launches = false) {
  if (!out) return fail(QS_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (n < 1 || n > QS_MAX_QUBITS) return fail(QS_ERR_INVALID_ARG, "n out of range");
  if (kmax < 1 || kmax > 5) return fail(QS_ERR_INVALID_ARG, "kmax outside 1..5");
  if (ng && !gates) return fail(QS_ERR_INVALID_ARG, "gates is NULL");
  if (mode != QS_PLAN_PLAIN && mode != QS_PLAN_GREEDY)
    return fail(QS_ERR_UNSUPPORTED, "plan mode %d needs a trained cost model", mode);
  std::vector<int> tgt(ng);
  std::vector<uint64_t> cms(ng);
  for (size_t k = 0; k < ng; ++k) {
    int t;
    uint64_t cm;
    int rc = gate_qubits(gates[k], n, &t, &cm);
    if (rc) return fail(rc, "gate %zu: %s", k, qs_last_error());
    tgt[k] = t;
    cms[k] = cm;
  }
  qs_plan* p = new (std::nothrow) qs_plan;
  if (!p) return fail(QS_ERR_OOM, "host allocation failed");
  p->n = n;
  p->mode = mode;
  p->kmax = kmax;
  p->ng = ng;
  p->fingerprint = fingerprint(gates, ng);
  p->m = std::min(n, mtile);
  const double N = (double)(1ull << n);
  const double pass_bytes = 32.0 * N;

  if (mode == QS_PLAN_PLAIN) {
    for (size_t k = 0; k < ng; ++k) {
      PlanPass ps;
      ps.kind = PASS_GATE;
      ps.qmask = 1ull << tgt[k];
      ps.gates.push_back((uint32_t)k);
      p->passes.push_back(std::move(ps));
      double f = op_touch_fraction(gates[k], cms[k]);
      p->est_seconds += std::max(pass_bytes * f / kHbmBytesPerS, N * f * op_flops_per_amp(gates[k].type) / kFp64FlopPerS);
    }
    *out = p;
    return QS_OK;
  }

  GateQueue remaining = gate_queue(tgt, cms), rest;
  while (!remaining.empty()) {
    PlanPass ps = make_pass(gates, tgt, cms, remaining, n, p->m, strategy, rest);
    // Cost: a tile pass sweeps the whole state once and is bound by its limb
    // products; a per-gate kernel touches only the amplitudes it changes and is
    // bound by HBM.  A lone gate, or a pass of cheap data-movement gates (CZ,
    // CNOT), can be cheaper gate by gate.
    double limbs = 0.0, plain = 0.0;
    for (uint32_t k : ps.gates) {
      const double f = op_touch_fraction(gates[k], cms[k]);
      limbs += N * f * op_q60_per_amp(gates[k].type);
      plain += pass_bytes * f / (kPlainHbmFraction * kHbmBytesPerS);
    }
    const double tile_cost = std::max(pass_bytes / kHbmBytesPerS, limbs / kTileLimbPerS);
    if (!few_launches && (ps.gates.size() == 1 || plain <= tile_cost)) {
      for (uint32_t k : ps.gates) {
        PlanPass g1;
        g1.kind = PASS_GATE;
        g1.qmask = 1ull << tgt[k];
        g1.gates.push_back(k);
        p->passes.push_back(std::move(g1));
      }
      p->est_seconds += plain;
    } else {
      p->passes.push_back(std::move(ps));
      p->est_seconds += tile_cost;
      ++p->n_tile;
    }
    std::swap(remaining, rest);
  }
  *out = p;
  return QS_OK;
}

// The plan of a qs_apply without one.  Below 24 qubits the passes run every gate with
// its own matrix: a fused pass's products of matrices and phases round to double, and
// on amplitudes that large this error exceeds the 2^-60 resolution of the arithmetic
// (relative error of 300 random gates at n = 12: per gate 8.4e-16, so 7.2e-16, fused
// 1.8e-15; at n = 24 6.3e-15, 5.8e-15, 4.9e-15).  Tiles are narrow on small states, so
// that several SMs share a pass (one SM takes 1 us for a gate on 2^12 amplitudes and a
// launch 4 us).  complex64 states gain from fusion at any size.
int plan_implicit(int n, int prec, const qs_gate* gates, size_t ng, qs_plan** out) {
  if (n >= 24 || prec == 64) return plan_build(n, gates, ng, QS_PLAN_GREEDY, 5, TILE_DEFAULT_M, out);
  const int m = n <= 10 ? n : std::min(TILE_DEFAULT_M, std::max(9, n - 6));
  // (below 20 qubits a launch costs more than any sweep it saves: no per-gate passes)
  QS_TRY(plan_build(n, gates, ng, QS_PLAN_GREEDY, 5, m, out, 0, n < 20));
  (*out)->direct = true;
  return QS_OK;
}

extern "C" int qs_plan_create(int n, const qs_gate* gates, size_t ng, int mode, int kmax, qs_plan** out) {
  clear_error();
  return plan_build(n, gates, ng, mode, kmax, TILE_DEFAULT_M, out);
}

extern "C" int qs_plan_create_tiled(int n, const qs_gate* gates, size_t ng, int tile_qubits, qs_plan** out) {
  clear_error();
  if (tile_qubits < TILE_LOW + 1 || tile_qubits > TILE_MAX_M)
    return fail(QS_ERR_INVALID_ARG, "tile_qubits=%d outside %d..%d", tile_qubits, TILE_LOW + 1, TILE_MAX_M);
  return plan_build(n, gates, ng, QS_PLAN_GREEDY, 5, tile_qubits, out);
}

// Structural class of a record (valid for every angle): 0 general, 1 real,
// 2 general diagonal, 3 unit factors only (swaps, sign flips).
static int structural_class(int type) {
  switch (type) {
    case QS_H: case QS_RY: return 1;
    case QS_RZ: case QS_T: case QS_P: case QS_CR: return 2;
    case QS_X: case QS_Y: case QS_Z: case QS_S: case QS_CNOT: case QS_CZ: case QS_I: return 3;
    default: return 0;  // RX, U3
  }
}

static int tile_pass_profile(int n, const PlanPass& ps, const qs_gate* gates, const double* params,
                             int64_t* counts, double* int_ops_per_amp);

// The program as the planner sees it: a parametrised record (param_idx >= 0) takes
// fixed generic angles, so that the rewrite of a pass into kernel ops (which
// depends on the matrices only through their structure for generic angles) can
// run before the parameters are known.
static std::vector<qs_gate> structural_program(const qs_gate* gates, size_t ng) {
  std::vector<qs_gate> g(gates, gates + ng);
  for (qs_gate& r : g)
    if (r.param_idx >= 0) {
      r.param_idx = -1;
      r.p[0] = 0.7;
      r.p[1] = 0.3;
      r.p[2] = 0.5;
    }
  return g;
}

// Features of one pass for the cost model (QS_PASS_FEATURES values):
//   0 tile pass (1) or one plain gate (0); 1 tile qubits / 13; 2 state qubits / 34;
//   3 qubits outside the tile / 34; 4..7 gates by structural class (general, real,
//   general diagonal, unit factors) / 64; 8 controlled gates / 64; 9 diagonal gates
//   whose target lies outside the tile / 64; 10 distinct non-diagonal targets / 13;
//   11 gates that start a run (not right after a gate on the same target with the
//   same controls: the ops left after aggregation) / 64; 12 controlled
//   non-diagonal gates / 64; 13 log2(1 + gates) / 8;
// and for a tile pass the kernel ops the Q60 engine runs (tile_pass_profile):
//   14 limb products per amplitude / 256; 15 phase tables / 16; 16, 17, 18 groups
//   of four, three, two real rotations / 16; 19 single real rotations / 16;
//   20 general 2x2 ops / 16; 21 phase and diagonal ops / 16; 22 anti-diagonal ops
//   / 16; 23 per-tile scalars / 16; 24 kernel ops (shared-memory sweeps) / 64.
// `gates` is the structural program (structural_program).
static int pass_features(int n, const PlanPass& ps, const qs_gate* gates, double* f) {
  const int m = ps.kind == PASS_TILE ? __builtin_popcountll(ps.qmask) : 1;
  for (int i = 0; i < QS_PASS_FEATURES; ++i) f[i] = 0.0;
  f[0] = ps.kind == PASS_TILE ? 1.0 : 0.0;
  f[1] = m / 13.0;
  f[2] = n / 34.0;
  f[3] = (n - m) / 34.0;
  uint64_t targets = 0;
  int prev_t = -1;
  uint64_t prev_c = 0;
  for (uint32_t k : ps.gates) {
    int t;
    uint64_t cm;
    gate_qubits(gates[k], n, &t, &cm);
    const int cls = structural_class(gates[k].type);
    const bool diag = structurally_diagonal(gates[k].type);
    f[4 + cls] += 1.0 / 64.0;
    if (cm) f[8] += 1.0 / 64.0;
    if (ps.kind == PASS_TILE && !((ps.qmask >> t) & 1)) f[9] += 1.0 / 64.0;
    if (!diag) targets |= 1ull << t;
    if (!(t == prev_t && cm == prev_c)) f[11] += 1.0 / 64.0;
    if (!diag && cm) f[12] += 1.0 / 64.0;
    prev_t = t;
    prev_c = cm;
  }
  f[10] = __builtin_popcountll(targets) / 13.0;
  f[13] = std::log2(1.0 + (double)ps.gates.size()) / 8.0;
  if (ps.kind == PASS_TILE && !ps.gates.empty()) {
    int64_t c[QS_KOP_KINDS];
    double ipa = 0.0;
    QS_TRY(tile_pass_profile(n, ps, gates, nullptr, c, &ipa));
    f[14] = ipa / 256.0;
    f[15] = c[TOP_DTABLE] / 16.0;
    f[16] = c[TOP_REAL4] / 16.0;
    f[17] = c[TOP_REAL3] / 16.0;
    f[18] = c[TOP_REAL2] / 16.0;
    f[19] = c[TOP_REAL] / 16.0;
    f[20] = c[TOP_GENERAL] / 16.0;
    f[21] = (c[TOP_PHASE1] + c[TOP_DIAG]) / 16.0;
    f[22] = c[TOP_ANTI] / 16.0;
    f[23] = c[TOP_SCALAR] / 16.0;
    int64_t sweeps = -c[0];  // tables run inside a rotation group's loop take no sweep of their own
    for (int k = 1; k < QS_KOP_KINDS; ++k) sweeps += c[k];
    f[24] = sweeps / 64.0;
  }
  return QS_OK;
}

extern "C" int qs_plan_features(const qs_plan* p, const qs_gate* gates, size_t ng, double* out) {
  clear_error();
  if (!p || !out || (ng && !gates)) return fail(QS_ERR_INVALID_ARG, "NULL argument");
  if (p->ng != ng || p->fingerprint != fingerprint(gates, ng))
    return fail(QS_ERR_INVALID_ARG, "plan does not match the program");
  const std::vector<qs_gate> sg = structural_program(gates, ng);
  for (size_t i = 0; i < p->passes.size(); ++i)
    QS_TRY(pass_features(p->n, p->passes[i], sg.data(), out + i * QS_PASS_FEATURES));
  return QS_OK;
}

extern "C" int qs_plan_create_variant(int n, const qs_gate* gates, size_t ng, int tile_qubits, int strategy,
                                      qs_plan** out) {
  clear_error();
  if (tile_qubits < TILE_LOW + 1 || tile_qubits > TILE_MAX_M)
    return fail(QS_ERR_INVALID_ARG, "tile_qubits=%d outside %d..%d", tile_qubits, TILE_LOW + 1, TILE_MAX_M);
  if (strategy < 0 || strategy > 2) return fail(QS_ERR_INVALID_ARG, "strategy %d: use 0, 1 or 2", strategy);
  return plan_build(n, gates, ng, QS_PLAN_GREEDY, 5, tile_qubits, out, strategy);
}

// Learned plan (the cost model chooses the groupings).  Pass by pass, candidate
// tile passes over the remaining gates are built at widths 11 and 12: the greedy
// pass, the seeded pass, and the greedy pass kept off each one of the qubits the
// greedy scan added (strategy 2's variants).  The model predicts each
// candidate's time as one tile pass and as plain per-gate kernels, and the time
// of the greedy pass that would follow it; the candidate with the least
// predicted time per unit of work over the two passes (their gates' touched
// fractions of the state, a sweep each) is taken, as a tile pass or gate by gate,
// whichever the model predicts cheaper.  The greedy plan at width 12 is the
// fallback and the judge: the learned plan is kept only if the model predicts it
// faster overall by more than 5 %.  (Width 13 is left out: one 512-thread CTA per
// SM runs the tile ops slower than the widths' fewer passes save, and the model
// did not learn that from its training passes.)
using PassScorer = std::function<int(const double* x, size_t B, double* y)>;
constexpr double kLearnedMargin = 0.05;

static int plan_build_learned(int n, const qs_gate* gates, size_t ng, const PassScorer& score, qs_plan** out) {
  *out = nullptr;
  if (n < 1 || n > QS_MAX_QUBITS) return fail(QS_ERR_INVALID_ARG, "n out of range");
  if (ng && !gates) return fail(QS_ERR_INVALID_ARG, "gates is NULL");
  std::vector<int> tgt(ng);
  std::vector<uint64_t> cms(ng);
  for (size_t k = 0; k < ng; ++k) {
    int t;
    uint64_t cm;
    int rc = gate_qubits(gates[k], n, &t, &cm);
    if (rc) return fail(rc, "gate %zu: %s", k, qs_last_error());
    tgt[k] = t;
    cms[k] = cm;
  }
  qs_plan* greedy = nullptr;
  QS_TRY(plan_build(n, gates, ng, QS_PLAN_GREEDY, 5, TILE_DEFAULT_M, &greedy));
  std::unique_ptr<qs_plan> gp(greedy);
  const std::vector<qs_gate> sg = structural_program(gates, ng);
  auto predict_plan = [&](const qs_plan* pl, double* total) -> int {
    std::vector<double> x(pl->passes.size() * QS_PASS_FEATURES), y(pl->passes.size());
    for (size_t i = 0; i < pl->passes.size(); ++i)
      QS_TRY(pass_features(n, pl->passes[i], sg.data(), x.data() + i * QS_PASS_FEATURES));
    if (!y.empty()) QS_TRY(score(x.data(), y.size(), y.data()));
    *total = 0.0;
    for (double v : y) *total += std::exp(v) * 1e-3;
    return QS_OK;
  };
  std::unique_ptr<qs_plan> lp(new (std::nothrow) qs_plan);
  if (!lp) return fail(QS_ERR_OOM, "host allocation failed");
  lp->n = n;
  lp->mode = QS_PLAN_LEARNED;
  lp->kmax = 5;
  lp->ng = ng;
  lp->fingerprint = fingerprint(gates, ng);
  lp->m = 0;
  GateQueue remaining = gate_queue(tgt, cms);
  struct Cand {
    PlanPass ps;
    GateQueue rest;
    PlanPass next;  // the greedy pass that would follow (no gates at the end)
  };
  std::vector<Cand> cands;
  std::vector<double> x, y;
  double learned_total = 0.0;
  auto add_cand = [&](Cand&& c) {
    if (c.ps.gates.empty()) return;
    for (const Cand& o : cands)
      if (o.ps.qmask == c.ps.qmask && o.ps.gates == c.ps.gates) return;
    if (!c.rest.empty()) {
      GateQueue r2;
      c.next = make_pass(gates, tgt, cms, c.rest, n, std::min(n, TILE_DEFAULT_M), 0, r2);
    }
    cands.push_back(std::move(c));
  };
  while (!remaining.empty()) {
    cands.clear();
    for (int m = 11; m <= TILE_DEFAULT_M; ++m) {
      const int mm = std::min(n, m);
      uint64_t grown = 0;
      for (int strategy = 0; strategy < 2; ++strategy) {
        Cand c;
        c.ps = make_pass(gates, tgt, cms, remaining, n, mm, strategy, c.rest, 0, strategy == 0 ? &grown : nullptr);
        add_cand(std::move(c));
      }
      for (uint64_t b = grown; b; b &= b - 1) {
        Cand c;
        c.ps = make_pass(gates, tgt, cms, remaining, n, mm, 0, c.rest, b & (~b + 1));
        add_cand(std::move(c));
      }
      if (mm < m) break;
    }
    // rows: each candidate as a tile pass, then each of its gates as a plain pass,
    // then the pass after it
    x.clear();
    std::vector<size_t> first(cands.size());
    for (size_t c = 0; c < cands.size(); ++c) {
      first[c] = x.size() / QS_PASS_FEATURES;
      x.resize(x.size() + QS_PASS_FEATURES * (2 + cands[c].ps.gates.size()));
      double* row = x.data() + first[c] * QS_PASS_FEATURES;
      QS_TRY(pass_features(n, cands[c].ps, sg.data(), row));
      for (size_t i = 0; i < cands[c].ps.gates.size(); ++i) {
        PlanPass g1;
        g1.kind = PASS_GATE;
        g1.qmask = 1ull << tgt[cands[c].ps.gates[i]];
        g1.gates.push_back(cands[c].ps.gates[i]);
        QS_TRY(pass_features(n, g1, sg.data(), row + (1 + i) * QS_PASS_FEATURES));
      }
      QS_TRY(pass_features(n, cands[c].next, sg.data(), row + (1 + cands[c].ps.gates.size()) * QS_PASS_FEATURES));
    }
    y.assign(x.size() / QS_PASS_FEATURES, 0.0);
    QS_TRY(score(x.data(), y.size(), y.data()));
    size_t best = 0;
    bool best_tile = true;
    double best_rate = 1e300, best_time = 0.0;
    for (size_t c = 0; c < cands.size(); ++c) {
      const size_t ngc = cands[c].ps.gates.size();
      const double t_tile = std::exp(y[first[c]]);
      double t_gates = 0.0, work = 0.0, work_next = 0.0;
      for (size_t i = 0; i < ngc; ++i) {
        const uint32_t k = cands[c].ps.gates[i];
        t_gates += std::exp(y[first[c] + 1 + i]);
        work += op_touch_fraction(gates[k], cms[k]);
      }
      for (uint32_t k : cands[c].next.gates) work_next += op_touch_fraction(gates[k], cms[k]);
      const double t_next = cands[c].next.gates.empty() ? 0.0 : std::exp(y[first[c] + 1 + ngc]);
      const bool tile = ngc > 1 && t_tile <= t_gates;
      const double t = tile ? t_tile : t_gates;
      const double rate = (t + t_next) / std::max(work + work_next, 1e-9);
      if (rate < best_rate) {
        best_rate = rate;
        best = c;
        best_tile = tile;
        best_time = t;
      }
    }
    Cand& c = cands[best];
    learned_total += best_time * 1e-3;
    if (best_tile) {
      lp->m = std::max(lp->m, __builtin_popcountll(c.ps.qmask));
      lp->passes.push_back(c.ps);
      ++lp->n_tile;
    } else {
      for (uint32_t k : c.ps.gates) {
        PlanPass g1;
        g1.kind = PASS_GATE;
        g1.qmask = 1ull << tgt[k];
        g1.gates.push_back(k);
        lp->passes.push_back(std::move(g1));
      }
    }
    std::swap(remaining, c.rest);
  }
  if (lp->m == 0) lp->m = std::min(n, TILE_DEFAULT_M);
  double greedy_total = 0.0;
  QS_TRY(predict_plan(gp.get(), &greedy_total));
  QS_TRY(predict_plan(lp.get(), &learned_total));
  // the judge: the greedy plan unless the model predicts the learned plan faster by
  // more than its typical error on a plan's total (kLearnedMargin)
  if (learned_total > (1.0 - kLearnedMargin) * greedy_total) {
    gp->mode = QS_PLAN_LEARNED;
    gp->learned_fallback = true;
    gp->est_seconds = greedy_total;
    *out = gp.release();
    return QS_OK;
  }
  lp->est_seconds = learned_total;
  *out = lp.release();
  return QS_OK;
}

extern "C" int qs_plan_create_learned(int n, const qs_gate* gates, size_t ng, qs_mlp* model, qs_plan** out) {
  clear_error();
  if (!out) return fail(QS_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (!model) return fail(QS_ERR_UNSUPPORTED, "a learned plan needs a trained cost model");
  if (mlp_inputs(model) != QS_PASS_FEATURES)
    return fail(QS_ERR_INVALID_ARG, "the cost model takes %d inputs, a pass has %d features", mlp_inputs(model),
                QS_PASS_FEATURES);
  PassScorer score = [model](const double* x, size_t B, double* y) { return qs_mlp_forward(model, x, B, y); };
  return plan_build_learned(n, gates, ng, score, out);
}

extern "C" int qs_plan_create_scored(int n, const qs_gate* gates, size_t ng, qs_pass_scorer score, void* ctx,
                                     qs_plan** out) {
  clear_error();
  if (!out) return fail(QS_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (!score) return fail(QS_ERR_INVALID_ARG, "score is NULL");
  PassScorer sc = [score, ctx](const double* x, size_t B, double* y) {
    const int rc = score(ctx, x, B, y);
    return rc ? fail(QS_ERR_INVALID_ARG, "the pass scorer returned %d", rc) : QS_OK;
  };
  return plan_build_learned(n, gates, ng, sc, out);
}

extern "C" int qs_plan_free(qs_plan* p) {
  delete p;
  return QS_OK;
}

extern "C" int qs_plan_get_stats(const qs_plan* p, qs_plan_stats* out) {
  if (!p || !out) return fail(QS_ERR_INVALID_ARG, "NULL argument");
  out->n_gates = (int64_t)p->ng;
  out->n_passes = (int64_t)p->passes.size();
  out->n_tile_passes = p->n_tile;
  out->n_dense = 0;
  out->tile_qubits = p->m;
  out->learned_fallback = p->learned_fallback ? 1 : 0;
  out->est_seconds = p->est_seconds;
  return QS_OK;
}

extern "C" int qs_plan_pass_info(const qs_plan* p, size_t pass, int* kind, uint64_t* qmask, uint32_t* gates,
                                 size_t cap, size_t* ngates) {
  if (!p || !kind || !qmask || !ngates || (cap && !gates)) return fail(QS_ERR_INVALID_ARG, "NULL argument");
  if (pass >= p->passes.size()) return fail(QS_ERR_INVALID_ARG, "pass %zu of %zu", pass, p->passes.size());
  const PlanPass& ps = p->passes[pass];
  *kind = ps.kind;
  *qmask = ps.qmask;
  *ngates = ps.gates.size();
  for (size_t i = 0; i < ps.gates.size() && i < cap; ++i) gates[i] = ps.gates[i];
  return QS_OK;
}

static int build_pass_ops(int n, const PlanPass& ps, const qs_gate* gates, const double* params, bool tables_ok,
                          std::vector<Op1>* rops, std::vector<PhaseTable>* ptables, int* local, int* m_out,
                          bool direct = false);

extern "C" int qs_plan_pass_ops(const qs_plan* p, size_t pass, const qs_gate* gates, size_t ng, const double* params,
                                int q60, qs_pass_op* ops, size_t cap, size_t* count, double* tables,
                                size_t table_cap, size_t* ntables) {
  clear_error();
  if (!p || !count || !ntables || (cap && !ops) || (table_cap && !tables))
    return fail(QS_ERR_INVALID_ARG, "NULL argument");
  if (pass >= p->passes.size()) return fail(QS_ERR_INVALID_ARG, "pass %zu of %zu", pass, p->passes.size());
  if (p->ng != ng || p->fingerprint != fingerprint(gates, ng)) return fail(QS_ERR_INVALID_ARG, "plan does not match the program");
  QS_TRY(validate_gates(gates, ng, p->n, params));
  const PlanPass& ps = p->passes[pass];
  std::vector<Op1> rops;
  std::vector<PhaseTable> pt;
  int local[64];
  int m = 0;
  if (ps.kind == PASS_TILE) {
    QS_TRY(build_pass_ops(p->n, ps, gates, params, q60 != 0, &rops, &pt, local, &m));
  } else {
    int t;
    uint64_t cm;
    Mat2 mat;
    QS_TRY(gate_qubits(gates[ps.gates[0]], p->n, &t, &cm));
    QS_TRY(gate_matrix(gates[ps.gates[0]], params, &mat));
    rops.push_back(classify(t, cm, mat));
  }
  *count = rops.size();
  *ntables = pt.size();
  for (size_t i = 0; i < rops.size() && i < cap; ++i) {
    qs_pass_op& o = ops[i];
    memset(&o, 0, sizeof o);
    if (rops[i].cls == kTableMark) {
      o.kind = 1;
      o.table = rops[i].target;
      const PhaseTable& tb = pt[rops[i].target];
      o.bits = tb.m;
      o.nsigns = (int32_t)tb.signs.size();
      for (size_t k = 0; k < tb.signs.size() && k < 16; ++k) {
        o.sign_q[k] = (uint8_t)tb.signs[k].first;
        // the tile bit back to its qubit
        int q = 0;
        for (int b = 0; b < p->n; ++b)
          if (local[b] == tb.signs[k].second) q = b;
        o.sign_t[k] = (uint8_t)q;
      }
      continue;
    }
    o.kind = 0;
    o.target = rops[i].target;
    o.ctrl_mask = rops[i].cmask;
    for (int e = 0; e < 4; ++e) {
      o.m[2 * e] = rops[i].m.m[e].re;
      o.m[2 * e + 1] = rops[i].m.m[e].im;
    }
  }
  for (size_t t = 0; t < pt.size() && t < table_cap; ++t) {
    const std::vector<C2> e = table_entries(pt[t]);
    double* d = tables + t * 2 * e.size();
    for (size_t k = 0; k < e.size(); ++k) {
      d[2 * k] = e[k].re;
      d[2 * k + 1] = e[k].im;
    }
  }
  return QS_OK;
}

static bool g_aggregate = true;
static bool g_rotation_pairs = true;
static bool g_fuse_tables = true;

static bool g_rotation_triples = true;
static bool g_rotation_quads = true;

extern "C" int qs_set_rotation_pairs(int on) {
  g_rotation_pairs = on != 0;
  g_fuse_tables = on > 0 && on != 2;
  g_rotation_triples = on == 1 || on == 4;
  g_rotation_quads = on == 1;
  return QS_OK;
}

extern "C" int qs_set_aggregate(int on) {
  g_aggregate = on != 0;
  return QS_OK;
}


// Builds a pass's phase tables in the state's table buffer: their factors travel as
// kernel parameters and k_phase_tables multiplies them out there (on the host the
// 2^m entries of 25 tables took 0.6 ms of the 0.61 ms that 300 random gates on 20
// qubits needed, and an upload had to wait for the pass before it).  They stay in
// the workspace, which no other call uses while a pass runs (152 tables of 4096
// entries fit); more than that, or wider ones, in a buffer of their own.  Either is
// rewritten in stream order, after the previous pass's kernel.
static size_t tables_bytes(const std::vector<PhaseTable>& pt, bool f32) {
  return pt.empty() ? 0 : (pt.size() << pt[0].m) * (f32 ? sizeof(float2) : 2 * sizeof(QL));
}
static int build_tables(qs_state* s, const std::vector<PhaseTable>& pt, const QL** dev, bool f32) {
  const int m = pt[0].m;
  const size_t bytes = tables_bytes(pt, f32), per = bytes / pt.size();
  if (s->ws_bytes < bytes && s->tables_bytes < bytes) {
    if (s->tables) {
      QS_CUDA(cudaStreamSynchronize(s->stream));
      cudaFree(s->tables);
    }
    s->tables = nullptr;
    s->tables_bytes = 0;
    QS_CUDA(dmalloc(&s->tables, bytes));
    s->tables_bytes = bytes;
  }
  char* buf = (char*)(s->ws_bytes < bytes ? s->tables : s->ws);
  std::unique_ptr<TableArgs> g(new (std::nothrow) TableArgs);
  if (!g) return fail(QS_ERR_OOM, "host allocation failed");
  for (size_t t = 0; t < pt.size();) {
    g->m = m;
    g->f32 = f32;
    g->ntab = 0;
    int used = 0;
    const size_t first = t;
    for (; t < pt.size() && g->ntab < TABLE_ARGS_MAX; ++t) {
      const PhaseTable& p = pt[t];
      // a CZ is a sign where both bits are set; the others multiply
      auto is_cz = [](const TableTerm& x) {
        return unit_code(x.e0) == U_ONE && unit_code(x.e1) == U_MINUS_ONE;
      };
      int ns = 0;
      for (const TableTerm& x : p.terms) ns += is_cz(x);
      const int nt = (int)p.terms.size() - ns, need = 4 * m + ns + 5 * nt;
      if (used + need > TABLE_ARGS_WORDS) break;
      const int k = g->ntab++;
      g->off[k] = (uint16_t)used;
      g->ns[k] = (uint16_t)ns;
      g->nt[k] = (uint16_t)nt;
      double* w = g->w + used;
      for (int b = 0; b < m; ++b) {
        *w++ = p.d0[b].re;
        *w++ = p.d0[b].im;
        *w++ = p.d1[b].re;
        *w++ = p.d1[b].im;
      }
      for (const TableTerm& x : p.terms)
        if (is_cz(x)) *w++ = (double)(x.lmask | (1u << x.tb));
      for (const TableTerm& x : p.terms)
        if (!is_cz(x)) {
          *w++ = (double)((uint64_t)x.lmask * 32 + (uint64_t)x.tb);
          *w++ = x.e0.re;
          *w++ = x.e0.im;
          *w++ = x.e1.re;
          *w++ = x.e1.im;
        }
      used += need;
    }
    if (t == first) return fail(QS_ERR_UNSUPPORTED, "phase table of %zu terms", pt[t].terms.size());
    QS_TRY(launch_tables(s, *g, buf + first * per));
  }
  *dev = (const QL*)buf;
  return QS_OK;
}

// The host op list of one tile pass (shared by the kernel path and
// qs_plan_pass_ops): the pass's gates aggregated into fewer unitaries, then (Q60
// engine) general ops split into real rotations and phase tables.  local[b] is
// the tile bit of qubit b (-1 outside the tile), *m the tile width.
static int build_pass_ops(int n, const PlanPass& ps, const qs_gate* gates, const double* params, bool tables_ok,
                          std::vector<Op1>* rops, std::vector<PhaseTable>* ptables, int* local, int* m_out,
                          bool direct) {
  int m = 0;
  for (int b = 0; b < 64; ++b) local[b] = -1;
  for (int b = 0; b < n; ++b)
    if ((ps.qmask >> b) & 1) local[b] = m++;
  *m_out = m;
  rops->clear();
  ptables->clear();
  int merged = 0;
  if (g_aggregate && !direct) {
    QS_TRY(aggregate_pass(n, ps, gates, params, rops, &merged));
  } else {
    for (uint32_t k : ps.gates) {
      int t;
      uint64_t cm;
      Mat2 mat;
      QS_TRY(gate_qubits(gates[k], n, &t, &cm));
      QS_TRY(gate_matrix(gates[k], params, &mat));
      const Op1 op = classify(t, cm, mat);
      if (op.cls != OP_IDENTITY) rops->push_back(op);
    }
  }
  if (tables_ok && g_aggregate && g_phase_tables && !direct) {
    std::vector<Op1> x;
    std::vector<PhaseTable> t;
    extract_phases(*rops, local, n, m, &x, &t);
    // keep the rewrite where it is estimated cheaper (and fits the op table)
    if (x.size() <= (size_t)TILE_MAX_OPS && est_ops(x) < 0.98 * est_ops(*rops)) {
      rops->swap(x);
      ptables->swap(t);
    }
  }
  return QS_OK;
}

// The kernel arguments of one tile pass on an n-qubit state of precision `prec`
// (128 complex128, 64 complex64), host only: the op slots in `g`, the phase
// tables in `ptables` (not yet on the device), and the pass's FP64 flops and Q60
// limb products.
static int build_tile_args(int n, int prec, const PlanPass& ps, const qs_gate* gates, const double* params,
                           bool fixed, int io, TileArgs* g, std::vector<PhaseTable>& ptables, double* flops_out,
                           double* int_ops_out, bool direct = false) {
  const uint64_t Q = ps.qmask;
  int local[64];
  int m = 0;
  std::vector<Op1> rops;
  const bool f32 = prec == 64;  // complex64 state: FP32 engine
  int rc = build_pass_ops(n, ps, gates, params, (fixed && prec == 128) || f32, &rops, &ptables, local, &m, direct);
  int L = 0;
  while (L < n && ((Q >> L) & 1)) ++L;
  g->n = n;
  g->m = m;
  g->ntiles = 1ull << (n - m);
  g->nhigh = 0;
  for (int b = L; b < n; ++b)
    if ((Q >> b) & 1) g->qhigh[g->nhigh++] = b;
  g->nout = 0;
  for (int b = 0; b < n; ++b)
    if (!((Q >> b) & 1)) g->outpos[g->nout++] = b;
  g->nops = 0;
  g->io = (fixed && prec == 128) ? io : 0;
  g->tables = nullptr;
  double flops = 0.0, int_ops = 0.0;
  const double N = (double)(1ull << n);
  const bool pairs = ((fixed && prec == 128) || f32) && g_rotation_pairs && !direct;
  const bool triples = g_rotation_triples;
  const bool quads = g_rotation_quads;
  auto in_tile_real = [&](const Op1& o) { return o.cls == OP_REAL && o.cmask == 0 && local[o.target] >= 0; };
  if (rc == QS_OK && pairs && quads) {
    // Within each run of consecutive real rotations on distinct tile qubits (they
    // commute), order them by (tile bit mod 3, tile bit): the groups of four then
    // mix low and high bits, so a group's 16 amplitudes per lane pair never span
    // only tile bits 4 and up of the lanes' addresses (shared-memory bank spread).
    for (size_t i = 0; i < rops.size();) {
      if (!in_tile_real(rops[i])) {
        ++i;
        continue;
      }
      size_t e = i;
      uint32_t seen = 0;
      while (e < rops.size() && in_tile_real(rops[e]) && !((seen >> local[rops[e].target]) & 1)) {
        seen |= 1u << local[rops[e].target];
        ++e;
      }
      if (e - i >= 5)
        std::stable_sort(rops.begin() + i, rops.begin() + e, [&](const Op1& x, const Op1& y) {
          const int bx = local[x.target], by = local[y.target];
          return bx % 3 != by % 3 ? bx % 3 < by % 3 : bx < by;
        });
      i = e;
    }
  }
  for (size_t i = 0; rc == QS_OK && i < rops.size(); ++i) {
    const Op1& op = rops[i];
    if (pairs && quads && f32 && i + 3 < rops.size() && in_tile_real(op) && in_tile_real(rops[i + 1]) &&
        in_tile_real(rops[i + 2]) && in_tile_real(rops[i + 3])) {
      const uint32_t tm = (1u << local[op.target]) | (1u << local[rops[i + 1].target]) |
                          (1u << local[rops[i + 2].target]) | (1u << local[rops[i + 3].target]);
      if (__builtin_popcount(tm) == 4) {
        // FP32: four real rotations on 16 amplitudes in registers (one slot), a
        // phase table just before them applied in the same loop
        int tab = -1;
        if (g_fuse_tables && i > 0 && rops[i - 1].cls == kTableMark && g->nops > 0 &&
            g->ops[g->nops - 1].kind == TOP_DTABLE && g->ops[g->nops - 1].lcmask < 128) {
          --g->nops;
          tab = (int)g->ops[g->nops].lcmask;
        }
        TileOp& t0 = g->ops[g->nops];
        memset(&t0, 0, sizeof t0);
        t0.kind = TOP_REAL4;
        t0.tb = (int8_t)local[op.target];
        t0.code0 = (int8_t)local[rops[i + 1].target];
        t0.code1 = (int8_t)tab;
        t0.lcmask = ((uint32_t)local[rops[i + 2].target] << 8) | ((uint32_t)local[rops[i + 3].target] << 16);
        float* f = reinterpret_cast<float*>(t0.q);
        for (int q = 0; q < 4; ++q)
          for (int e = 0; e < 4; ++e) f[4 * q + e] = (float)rops[i + q].m.m[e].re;
        flops += N * 24.0;  // per rotation and amplitude: two components x (1 mul + 1 fma)
        g->nops += 1;
        i += 3;
        continue;
      }
    }
    // A run of r >= 5 rotations on distinct tile qubits right after a phase table
    // (not the pass's first op, which runs in the tile's load loop) starts with a
    // triple (r = 4k + 1 or 4k + 3) or a pair (r = 4k + 2): the group takes the
    // table into its loop, and the run still takes as many sweeps as groups of
    // four first would (r = 9: triple, four, pair against four, four, single).
    int lead = 0;
    if (pairs && quads && triples && g_fuse_tables && !f32 && in_tile_real(op) && i > 0 &&
        rops[i - 1].cls == kTableMark && g->nops >= 2 && g->ops[g->nops - 1].kind == TOP_DTABLE &&
        g->ops[g->nops - 1].lcmask < 128) {
      size_t e = i;
      uint32_t seen = 0;
      while (e < rops.size() && in_tile_real(rops[e]) && !((seen >> local[rops[e].target]) & 1)) {
        seen |= 1u << local[rops[e].target];
        ++e;
      }
      const size_t r = e - i;
      if (r >= 5 && r % 4 != 0) lead = r % 4 == 2 ? 2 : 3;
    }
    if (lead == 0 && pairs && quads && !f32 && i + 3 < rops.size() && g->nops + 2 <= TILE_MAX_OPS && in_tile_real(op) &&
        in_tile_real(rops[i + 1]) && in_tile_real(rops[i + 2]) && in_tile_real(rops[i + 3])) {
      const uint32_t tm = (1u << local[op.target]) | (1u << local[rops[i + 1].target]) |
                          (1u << local[rops[i + 2].target]) | (1u << local[rops[i + 3].target]);
      if (__builtin_popcount(tm) == 4) {
        // four real rotations on different tile qubits: one op on one component of
        // 16 amplitudes at a time (two slots); a table before it stays its own op
        TileOp* t = &g->ops[g->nops];
        memset(t, 0, 2 * sizeof(TileOp));
        t[0].kind = TOP_REAL4;
        t[0].tb = (int8_t)local[op.target];
        t[0].code0 = (int8_t)local[rops[i + 1].target];
        t[0].code1 = -1;
        t[1].kind = TOP_CONT;
        double mr[4][4];
        for (int q = 0; q < 4; ++q)
          for (int e = 0; e < 4; ++e) mr[q][e] = rops[i + q].m.m[e].re;
        QW G[24];
        int flags = 0;
        q60_quad4_gauss_coef(mr[0], mr[1], mr[2], mr[3], G, &flags);
        for (int e = 0; e < 24; ++e) reinterpret_cast<QW*>(t[e / 12].q)[e % 12] = G[e];
        t[0].lcmask = (uint32_t)flags | ((uint32_t)local[rops[i + 2].target] << 8) |
                      ((uint32_t)local[rops[i + 3].target] << 16);
        int_ops += N * 12.0;  // as four real products a complex product (the planner's unit)
        g->nops += 2;
        i += 3;
        continue;
      }
    }
    if (lead != 2 && pairs && triples && !f32 && i + 2 < rops.size() && in_tile_real(op) && in_tile_real(rops[i + 1]) &&
        in_tile_real(rops[i + 2]) && rops[i + 1].target != op.target && rops[i + 2].target != op.target &&
        rops[i + 2].target != rops[i + 1].target) {
      // three real rotations on different tile qubits: one op on octets
      int tab = -1;
      if (g_fuse_tables && i > 0 && rops[i - 1].cls == kTableMark && g->nops > 0 &&
          g->ops[g->nops - 1].kind == TOP_DTABLE && g->ops[g->nops - 1].lcmask < 128) {
        --g->nops;
        tab = (int)g->ops[g->nops].lcmask;
      }
      TileOp& t0 = g->ops[g->nops];
      memset(&t0, 0, sizeof t0);
      t0.kind = TOP_REAL3;
      t0.tb = (int8_t)local[op.target];
      t0.code0 = (int8_t)local[rops[i + 1].target];
      t0.code1 = (int8_t)tab;
      double m0[4], m1[4], m2[4];
      for (int e = 0; e < 4; ++e) {
        m0[e] = op.m.m[e].re;
        m1[e] = rops[i + 1].m.m[e].re;
        m2[e] = rops[i + 2].m.m[e].re;
      }
      int flags = 0;
      q60_triple_gauss_coef(m0, m1, m2, reinterpret_cast<QW*>(t0.q), &flags);
      t0.lcmask = (uint32_t)flags | ((uint32_t)local[rops[i + 2].target] << 8);
      int_ops += N * 12.0;  // as four real products a complex product
      g->nops += 1;
      i += 2;
      continue;
    }
    if (pairs && i + 1 < rops.size() && in_tile_real(op) && in_tile_real(rops[i + 1]) &&
        rops[i + 1].target != op.target) {
      // two real rotations on different tile qubits: one 4x4 op on quads (two slots)
      const Mat2& ra = op.m;
      const Mat2& rb = rops[i + 1].m;
      // a phase table op just before the pair runs inside the pair's quad loop
      int tab = -1;
      if (g_fuse_tables && i > 0 && rops[i - 1].cls == kTableMark && g->nops > 0 &&
          g->ops[g->nops - 1].kind == TOP_DTABLE && g->ops[g->nops - 1].lcmask < 128) {
        --g->nops;
        tab = (int)g->ops[g->nops].lcmask;
      }
      TileOp& t0 = g->ops[g->nops];
      TileOp& t1 = g->ops[g->nops + 1];
      memset(&t0, 0, sizeof t0);
      memset(&t1, 0, sizeof t1);
      t0.kind = TOP_REAL2;
      t0.tb = (int8_t)local[op.target];
      t0.code0 = (int8_t)local[rops[i + 1].target];
      t0.code1 = (int8_t)tab;
      t1.kind = TOP_CONT;
      float* f0 = reinterpret_cast<float*>(t0.f);
      float* f1 = reinterpret_cast<float*>(t1.f);
      if (f32) {
        for (int k = 0; k < 4; ++k)
          for (int c = 0; c < 4; ++c) {
            const double v = rb.m[2 * (k >> 1) + (c >> 1)].re * ra.m[2 * (k & 1) + (c & 1)].re;
            const int e = 4 * k + c;
            (e < 8 ? f0[e] : f1[e - 8]) = (float)v;
          }
        flops += N * 16.0;  // 4 real multiply-adds per output component, 2 components, per 4 amplitudes x 4 outputs
      } else {
        // two complex products on the quad (q60pair.cuh), reflection flags in lcmask
        double m0[4], m1[4];
        for (int e = 0; e < 4; ++e) {
          m0[e] = ra.m[e].re;
          m1[e] = rb.m[e].re;
        }
        int flags = 0;
        q60_pair_gauss_coef(m0, m1, reinterpret_cast<QP*>(t0.q), &flags);
        t0.lcmask = (uint32_t)flags;
        int_ops += N * 12.0;  // as four real products a complex product
      }
      g->nops += 2;
      ++i;
      continue;
    }
    if (op.cls == kTableMark) {
      TileOp& to = g->ops[g->nops];
      to.kind = TOP_DTABLE;
      to.tb = (int8_t)ptables[op.target].m;
      to.lcmask = (uint32_t)op.target;
      to.ext_cmask = 0;
      to.code0 = to.code1 = U_GENERAL;
      if (f32) flops += N * 6.0;  // one complex product per amplitude
      else int_ops += N * 12.0;   // one complex product (counted as four real ones) per amplitude
      ++g->nops;
      continue;
    }
    if (op.cls == OP_IDENTITY) continue;
    const Mat2& mat = op.m;
    const int t = op.target;
    const uint64_t cm = op.cmask;
    TileOp& to = g->ops[g->nops];
    if (prec == 64)
      for (int e = 0; e < 4; ++e) to.f[e] = make_float2((float)mat.m[e].re, (float)mat.m[e].im);
    else if (fixed && op.cls == OP_REAL)  // c + i s, or a reflection's after the flip of its bit-1 half
      to.q[0] = qc_make_gauss(mat.m[0].re, mat.m[2].re);
    else if (fixed)
      for (int e = 0; e < 4; ++e) to.q[e] = qc_make_gauss(mat.m[e].re, mat.m[e].im);
    else
      for (int e = 0; e < 4; ++e) to.m[e] = make_double2(mat.m[e].re, mat.m[e].im);
    to.code0 = (int8_t)op.code0;
    to.code1 = (int8_t)op.code1;
    if (op.cls == OP_REAL) to.code1 = mat.m[0].re * mat.m[3].re - mat.m[1].re * mat.m[2].re < 0.0;
    uint32_t lcm = 0;
    uint64_t ext = 0;
    for (int b = 0; b < n; ++b)
      if ((cm >> b) & 1) {
        if (local[b] >= 0) lcm |= 1u << local[b];
        else ext |= 1ull << b;
      }
    to.lcmask = lcm;
    to.ext_cmask = ext;
    if (local[t] >= 0) {
      to.kind = (int8_t)op.cls;
      to.tb = (int8_t)local[t];
    } else {
      if (op.cls != OP_PHASE1 && op.cls != OP_DIAG) {
        rc = fail(QS_ERR_INVALID_ARG, "plan does not match the program (non-diagonal op on qubit %d outside its tile)", t);
        break;
      }
      to.kind = TOP_SCALAR;
      to.tb = (int8_t)t;
    }
    flops += N * class_touch_fraction(op) * class_flops_per_amp(op);
    int_ops += N * class_touch_fraction(op) * op_int_ops_per_amp(op);
    ++g->nops;
  }
  // Q60 engine: a phase table that opens or closes the pass runs inside the tile's
  // load or store loop (no shared-memory sweep and barrier of its own).
  if (rc == QS_OK && fixed && prec == 128 && g_fuse_tables) {
    auto table_op = [&](const TileOp& o) {
      return o.kind == TOP_DTABLE && o.lcmask < ptables.size() && o.lcmask < 255 && o.tb == m;
    };
    if (g->nops > 0 && table_op(g->ops[0])) {
      g->io |= (int)(g->ops[0].lcmask + 1) << 8;
      memmove(&g->ops[0], &g->ops[1], sizeof(TileOp) * (size_t)(g->nops - 1));
      --g->nops;
    }
    if (g->nops > 0 && table_op(g->ops[g->nops - 1])) {
      g->io |= (int)(g->ops[g->nops - 1].lcmask + 1) << 16;
      --g->nops;
    }
  }
  for (int k = 0; rc == QS_OK && k < g->nops; ++k) {
    const TileOp& o = g->ops[k];
    if (o.kind == TOP_DTABLE && (o.lcmask >= ptables.size() || o.tb != m || ptables[o.lcmask].m != m))
      rc = fail(QS_ERR_INVALID_ARG, "internal: malformed phase-table op");
    if ((o.kind == TOP_REAL2 || o.kind == TOP_REAL3) && o.code1 >= 0 && (size_t)o.code1 >= ptables.size())
      rc = fail(QS_ERR_INVALID_ARG, "internal: malformed rotation-group op");
    if (o.kind == TOP_REAL2 && (k + 1 >= g->nops || g->ops[k + 1].kind != TOP_CONT))
      rc = fail(QS_ERR_INVALID_ARG, "internal: malformed rotation-pair op");
  }
  for (int t = 0; t < TILE_MAX_SIGNED_TABLES; ++t) g->signs[t].n = 0;
  for (size_t t = 0; rc == QS_OK && t < ptables.size(); ++t) {
    const auto& sg = ptables[t].signs;
    if (sg.empty()) continue;
    if (t >= (size_t)TILE_MAX_SIGNED_TABLES || sg.size() > (size_t)TILE_MAX_SIGNS) {
      rc = fail(QS_ERR_INVALID_ARG, "internal: phase table %zu with %zu sign terms", t, sg.size());
      break;
    }
    g->signs[t].n = (uint8_t)sg.size();
    for (size_t k = 0; k < sg.size(); ++k) {
      g->signs[t].q[k] = (uint8_t)sg[k].first;
      g->signs[t].t[k] = (uint8_t)sg[k].second;
    }
  }
  *flops_out = flops;
  *int_ops_out = int_ops;
  return rc;
}

// io: TileArgs::io (Q60 engine only); *launched: whether the pass's kernel was queued,
// also when the call fails (a pass whose ops all cancel launches nothing).
static int run_tile_pass(qs_state* s, const PlanPass& ps, const qs_gate* gates, const double* params, bool fixed,
                         int io, bool* launched, bool direct) {
  *launched = false;
  TileArgs* g = new (std::nothrow) TileArgs;
  if (!g) return fail(QS_ERR_OOM, "host allocation failed");
  std::vector<PhaseTable> ptables;
  double flops = 0.0, int_ops = 0.0;
  int rc = build_tile_args(s->n, s->prec, ps, gates, params, fixed, io, g, ptables, &flops, &int_ops, direct);
  if (rc == QS_OK && (g->nops > 0 || (g->io >> 8) != 0)) {
    // one record of the timing log for the pass: its tables, then its tile kernel
    KTimer kt(s, QS_K_TILE, g->m, (int)ps.gates.size(), ps.qmask, 0, (double)(1ull << g->n), fixed ? 0.0 : flops,
              fixed ? int_ops : 0.0);
    if (!ptables.empty()) rc = build_tables(s, ptables, &g->tables, s->prec == 64);
    if (rc == QS_OK) rc = launch_tile(s, *g, fixed, launched);
  }
  delete g;
  return rc;
}

// Kernel ops of one tile pass by kind (host only; the Q60 engine on a complex128
// state): counts[k] for TileOpKind k (continuation slots not counted; phase tables
// that run inside a rotation group's loop counted in counts[TOP_DTABLE] and again
// in counts[0]), and the pass's limb products per amplitude.
static int tile_pass_profile(int n, const PlanPass& ps, const qs_gate* gates, const double* params,
                             int64_t* counts, double* int_ops_per_amp) {
  for (int k = 0; k < QS_KOP_KINDS; ++k) counts[k] = 0;
  *int_ops_per_amp = 0.0;
  if (ps.kind != PASS_TILE) return QS_OK;
  std::unique_ptr<TileArgs> g(new (std::nothrow) TileArgs);
  if (!g) return fail(QS_ERR_OOM, "host allocation failed");
  std::vector<PhaseTable> ptables;
  double flops = 0.0, int_ops = 0.0;
  QS_TRY(build_tile_args(n, 128, ps, gates, params, true, 0, g.get(), ptables, &flops, &int_ops));
  if ((g->io >> 8) & 255) ++counts[TOP_DTABLE], ++counts[0];   // tables run in the load or store loop
  if ((g->io >> 16) & 255) ++counts[TOP_DTABLE], ++counts[0];
  for (int k = 0; k < g->nops; ++k) {
    const int kind = g->ops[k].kind;
    if (kind == TOP_CONT) continue;
    if (kind >= 0 && kind < QS_KOP_KINDS) ++counts[kind];
    if ((kind == TOP_REAL2 || kind == TOP_REAL3 || kind == TOP_REAL4) && g->ops[k].code1 >= 0) {
      ++counts[TOP_DTABLE];  // a table fused into the group's loop
      ++counts[0];
    }
  }
  *int_ops_per_amp = int_ops / (double)(1ull << n);
  return QS_OK;
}

extern "C" int qs_plan_pass_kernel_ops(const qs_plan* p, size_t pass, const qs_gate* gates, size_t ng,
                                       const double* params, int64_t* counts, double* int_ops_per_amp) {
  clear_error();
  if (!p || !counts || !int_ops_per_amp || (ng && !gates)) return fail(QS_ERR_INVALID_ARG, "NULL argument");
  if (p->ng != ng || p->fingerprint != fingerprint(gates, ng))
    return fail(QS_ERR_INVALID_ARG, "plan does not match the program");
  if (pass >= p->passes.size()) return fail(QS_ERR_INVALID_ARG, "pass %zu of %zu", pass, p->passes.size());
  return tile_pass_profile(p->n, p->passes[pass], gates, params, counts, int_ops_per_amp);
}

// The passes of a plan.  Between consecutive Q60 tile passes the buffer keeps the Q60
// integers (the same 16 bytes per amplitude): no conversion to complex128 and back, and
// no rounding to double in between.  *held: whether it holds them now, also after an
// error; last_held: it may hold them at the end.
static int run_passes(qs_state* s, const qs_gate* gates, const double* params, const qs_plan* plan, bool fixed,
                      bool last_held, bool* held_out) {
  const bool q60 = fixed && s->prec == 128;
  bool& held = *held_out;
  for (size_t i = 0; i < plan->passes.size(); ++i) {
    const PlanPass& ps = plan->passes[i];
    if (ps.kind == PASS_GATE) {
      if (held) QS_TRY(launch_q60_release(s, &held));
      const qs_gate& g = gates[ps.gates[0]];
      int t;
      uint64_t cm;
      Mat2 m;
      QS_TRY(gate_qubits(g, s->n, &t, &cm));
      QS_TRY(gate_matrix(g, params, &m));
      QS_TRY(launch_op1(s, classify(t, cm, m), fixed));
    } else {
      const bool last = i + 1 == plan->passes.size();
      const bool next_tile = q60 && (last ? last_held : plan->passes[i + 1].kind == PASS_TILE);
      bool launched = false;
      const int rc = run_tile_pass(s, ps, gates, params, fixed, (held ? 1 : 0) | (next_tile ? 2 : 0), &launched,
                                   plan->direct);
      if (launched) held = next_tile;
      if (rc != QS_OK) return rc;
    }
  }
  return QS_OK;
}

int qs_apply_plan(qs_state* s, const qs_gate* gates, size_t ng, const double* params, const qs_plan* plan,
                  bool fixed, bool* held_out) {
  if (plan->n != s->n || plan->ng != ng || plan->fingerprint != fingerprint(gates, ng))
    return fail(QS_ERR_INVALID_ARG, "plan does not match the program");
  bool held = false;
  int rc = run_passes(s, gates, params, plan, fixed, held_out != nullptr, &held);
  if (held && (rc != QS_OK || !held_out)) {  // integers would be read as doubles
    const int rc2 = launch_q60_release(s, &held);
    if (rc == QS_OK) rc = rc2;
  }
  if (rc != QS_OK) s->bound = 0;  // a kernel may be missing: the next call looks at the norm again
  if (held_out) *held_out = held;
  return rc;
}
