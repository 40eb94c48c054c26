// Shared Q60 tile machinery of the batched and the single-state adjoint passes:
// op descriptors in global memory, tile ops on int64 (Q60) amplitude pairs, and the
// generator inner product Im <lambda| G |psi> over a tile.
#pragma once

#include <string.h>

#include <algorithm>
#include <utility>

#include <vector>

#include "fixed.h"
#include "internal.h"
#include "q60pair.cuh"

namespace qs {

constexpr int BT_THREADS = 256;
constexpr int BT_M = 11;          // tile qubits: psi and lambda tiles of 2^11 x 16 B
constexpr int BT_MAX_OPS = 128;   // gates (and gradient slots) per pass
constexpr int BT_MAX_N = 24;
constexpr int BT_OFFS = 1 << (BT_M - 3);  // high-bit offset table: tiles hold qubits 0..2 (or all of n < 3)

// BK_DGROUP: a group of up to four uncontrolled diagonal gates on distinct tile
// qubits, run as one op: amplitude j gets E[idx], idx = the member target bits
// of j (member m at bit m), E = the product of the members' diagonals (16 entries
// per group, Gauss form).  The members follow the head as BK_MEMBER records
// (nothing to run on their own) and keep their generator slots.
// BK_RPAIR: two uncontrolled real rotations on distinct tile qubits a (first member)
// and b, run as two complex products on one component of the quads (j, j|a, j|b,
// j|a|b) at a time (q60pair.cuh; 2 coefficients per pair, gate = pair index); in the
// backward sweep the op also takes both members' generator terms from the basis
// that the products run in.
// BK_PERM: a run of X and CNOT gates without a gradient, run as one permutation of
// the tile (nmem members follow).
enum : int8_t { BK_SCALAR = 9, BK_DGROUP = 10, BK_MEMBER = 11, BK_RPAIR = 12, BK_PERM = 13 };
constexpr int BT_DG_MAX = 4;  // members per group
enum : int8_t { BG_NONE = 0, BG_X = 1, BG_Y = 2, BG_Z = 3, BG_P = 4 };

struct BPass {
  int m, nhigh, nout, op_begin, op_end, nslots;
  int dg_begin, dg_end, rp_begin, rp_end;  // its diagonal groups and real pairs
  int qhigh[16];
  int outpos[32];
};

struct BOp {
  uint64_t ext;     // controls outside the tile
  uint32_t lcm;     // controls inside the tile (local bits)
  int gate;         // global gate index (matrix tables)
  int param;        // global parameter index, or -1
  double gsign;     // generator sign (-1 for a dagger record)
  int16_t slot;     // gradient slot within the pass, or -1
  int8_t kf, kb;    // op class forward / adjoint
  int8_t tb;        // local target bit (global target bit for SCALAR)
  int8_t gen;
  int8_t c0f, c1f, c0b, c1b;
  int8_t nmem;      // group heads: members following it (gate = group index)
  int8_t rot;       // a real rotation (determinant +1) for every angle
};

// Diagonal group (see BK_DGROUP): a_j *= E[idx(j)].
static __device__ void bt_apply_dgroup(longlong2* tile, uint32_t TS, const BOp* mem, int nm, const QC* E) {
  int tbs[BT_DG_MAX];
#pragma unroll
  for (int m = 0; m < BT_DG_MAX; ++m) tbs[m] = m < nm ? mem[m].tb : 0;
  for (uint32_t j = threadIdx.x; j < TS; j += BT_THREADS) {
    uint32_t idx = 0;
#pragma unroll
    for (int m = 0; m < BT_DG_MAX; ++m)
      if (m < nm) idx |= ((j >> tbs[m]) & 1u) << m;
    const QC u = E[idx];
    const longlong2 a = tile[j];
    int64_t re, im;
    q60_gauss_mul(u, q60_split(a.x), q60_split(a.y), q60_split(a.x + a.y), &re, &im);
    tile[j] = make_longlong2(re, im);
  }
}

// Generator term of one pair (amplitudes 0 and 1 of the pair) for generator `gen`,
// as the signed products of bt_gen_partial, exactly in Q60 units.
__device__ __forceinline__ int64_t bt_pair_gen(int gen, QL l0x, QL l0y, QL l1x, QL l1y, QL p0x, QL p0y, QL p1x,
                                               QL p1y) {
  QAccF pos{0, 0, 0}, neg{0, 0, 0};
  switch (gen) {
    case BG_X:  // l0x p1y - l0y p1x + l1x p0y - l1y p0x
      qaccf_add(pos, l0x, p1y); qaccf_add(neg, l0y, p1x); qaccf_add(pos, l1x, p0y); qaccf_add(neg, l1y, p0x);
      break;
    case BG_Y:  // -l0x p1x - l0y p1y + l1x p0x + l1y p0y
      qaccf_add(neg, l0x, p1x); qaccf_add(neg, l0y, p1y); qaccf_add(pos, l1x, p0x); qaccf_add(pos, l1y, p0y);
      break;
    case BG_Z:  // l0x p0y - l0y p0x - l1x p1y + l1y p1x
      qaccf_add(pos, l0x, p0y); qaccf_add(neg, l0y, p0x); qaccf_add(neg, l1x, p1y); qaccf_add(pos, l1y, p1x);
      break;
    case BG_P:  // -2 (l1x p1y - l1y p1x)
      qaccf_add(neg, l1x, p1y); qaccf_add(pos, l1y, p1x);
      return 2 * (qaccf_result(pos) - qaccf_result(neg));
    default:
      return 0;
  }
  return qaccf_result(pos) - qaccf_result(neg);
}

// The pair's two complex products on basis values u, v (see q60_pair_gauss), back to
// the quad at x[0], x[o01], x[o10], x[o11].
__device__ __forceinline__ void bt_pair_products(const QP* g, int64_t ur, int64_t ui, int64_t vr, int64_t vi,
                                                 int64_t* x, uint32_t o01, uint32_t o10, uint32_t o11) {
  qp_cmul(g[0], ur, ui);
  qp_cmul(g[1], vr, vi);
  x[0] = ur + vr;
  x[o01] = ui + vi;
  x[o10] = ui - vi;
  x[o11] = vr - ur;
}

// Real pair forward on one component a thread (18 wide multiply-adds a quad and
// component for both rotations; as the real 4x4 matrix it took 48, as two single
// rotations 48 and two sweeps).
static __device__ __noinline__ void bt_rpair(longlong2* tile, uint32_t TS, uint32_t ta, uint32_t tbb,
                                             const QP* __restrict__ cg) {
  const uint32_t lo = min(ta, tbb), hi = max(ta, tbb);
  const QP c[2] = {cg[0], cg[1]};
  int64_t* comp = reinterpret_cast<int64_t*>(tile) + (threadIdx.x & 1);
  for (uint32_t i = threadIdx.x >> 1; i < (TS >> 2); i += BT_THREADS / 2) {
    uint32_t j = i + (i & ~(lo - 1));
    j = j + (j & ~(hi - 1));
    int64_t* x = comp + 2 * j;
    const int64_t p0 = x[0], p1 = x[2 * ta], p2 = x[2 * tbb], p3 = x[2 * (ta | tbb)];
    bt_pair_products(c, p0 - p3, p1 + p2, p0 + p3, p1 - p2, x, 2 * ta, 2 * tbb, 2 * (ta | tbb));
  }
}

// Real pair backward: the products on psi and lambda, and with gens the generator
// terms of both members.  On one component, with z_b = p_b0 + i p_b1, u = z_0 + i z_1,
// v = z_0 - i z_1 on psi and U, V the same on lambda, the members' terms
//   a: sum_b l_b1 p_b0 - l_b0 p_b1,   b: sum_a l_1a p_0a - l_0a p_1a
// are (Im conj(u) U +- Im conj(v) V) / 2: four products instead of eight.  *out_u and
// *out_v receive the two sums over the tile (kept to all four limb products: they are
// summed over the state; |sum| <= 2 ||psi|| ||lambda|| <= 3.2, below 2^62).
static __device__ __noinline__ void bt_rpair_back(longlong2* P, longlong2* Lt, uint32_t TS, uint32_t ta,
                                                  uint32_t tbb, bool gens, const QP* __restrict__ cg, int64_t* out_u,
                                                  int64_t* out_v) {
  int64_t su = 0, sv = 0;
  const uint32_t lo = min(ta, tbb), hi = max(ta, tbb);
  const QP c[2] = {cg[0], cg[1]};
  const uint32_t o01 = 2 * ta, o10 = 2 * tbb, o11 = 2 * (ta | tbb);
  int64_t* cp = reinterpret_cast<int64_t*>(P) + (threadIdx.x & 1);
  int64_t* cl = reinterpret_cast<int64_t*>(Lt) + (threadIdx.x & 1);
  auto im = [](int64_t ar, int64_t ai, int64_t br, int64_t bi) {  // Im conj(a) b
    QAccF acc{0, 0, 0};
    qaccf_add(acc, q60_split(ar), q60_split(bi));
    qaccf_add(acc, q60_split(-ai), q60_split(br));
    return qaccf_result(acc);
  };
  for (uint32_t i = threadIdx.x >> 1; i < (TS >> 2); i += BT_THREADS / 2) {
    uint32_t j = i + (i & ~(lo - 1));
    j = j + (j & ~(hi - 1));
    int64_t *x = cp + 2 * j, *y = cl + 2 * j;
    const int64_t p0 = x[0], p1 = x[o01], p2 = x[o10], p3 = x[o11];
    const int64_t l0 = y[0], l1 = y[o01], l2 = y[o10], l3 = y[o11];
    const int64_t ur = p0 - p3, ui = p1 + p2, vr = p0 + p3, vi = p1 - p2;
    const int64_t Ur = l0 - l3, Ui = l1 + l2, Vr = l0 + l3, Vi = l1 - l2;
    if (gens) {
      su += im(ur, ui, Ur, Ui);
      sv += im(vr, vi, Vr, Vi);
    }
    bt_pair_products(c, ur, ui, vr, vi, x, o01, o10, o11);
    bt_pair_products(c, Ur, Ui, Vr, Vi, y, o01, o10, o11);
  }
  *out_u = su;
  *out_v = sv;
}

// A run of X and CNOT gates (members in program order, or reversed) as one
// permutation of the tile P, and of Lt if given: amplitude j moves to the index that
// the gates take j to.  That map is affine over bits, so a thread follows its first
// index and the strides of its loop through the gates once.  (A sweep and a barrier
// per gate otherwise, 11 of them for the ring of an ansatz layer.)
static __device__ __noinline__ void bt_perm(longlong2* P, longlong2* Lt, uint32_t TS, const BOp* mem, int nm,
                                            bool reverse, uint64_t base) {
  constexpr int E = (1 << BT_M) / BT_THREADS;  // amplitudes per thread
  uint32_t d = threadIdx.x, s0 = BT_THREADS, s1 = 2 * BT_THREADS, s2 = 4 * BT_THREADS;
  static_assert(E == 8, "three stride bits");
  for (int k = 0; k < nm; ++k) {
    const BOp& op = mem[reverse ? nm - 1 - k : k];
    if ((base & op.ext) != op.ext) continue;
    const uint32_t c = op.lcm, t = 1u << op.tb;
    if ((d & c) == c) d ^= t;
    if (c) {  // the linear part: no control, no change
      if (s0 & c) s0 ^= t;
      if (s1 & c) s1 ^= t;
      if (s2 & c) s2 ^= t;
    }
  }
  for (int a = 0; a < 2; ++a) {
    longlong2* tile = a ? Lt : P;
    if (!tile) break;
    longlong2 v[E];
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (threadIdx.x + e * BT_THREADS < TS) v[e] = tile[threadIdx.x + e * BT_THREADS];
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (threadIdx.x + e * BT_THREADS < TS)
        tile[d ^ ((e & 1) ? s0 : 0u) ^ ((e & 2) ? s1 : 0u) ^ ((e & 4) ? s2 : 0u)] = v[e];
  }
}

// Backward step of a diagonal group in one sweep: per amplitude the members'
// generator terms and then E on psi and on lambda.  With w = Im(conj(l_j) p_j), once per
// amplitude, a Z member's term is (-1)^bit w and a P member's -2 [bit] w; the members
// commute with each other and with each other's generators, so every term may be taken
// before the group runs.
static __device__ void bt_back_dgroup(longlong2* P, longlong2* Lt, uint32_t TS, const BOp* mem, int nm,
                                      const QC* __restrict__ E, int64_t* out) {
  int tbs[BT_DG_MAX], gens[BT_DG_MAX];
#pragma unroll
  for (int m = 0; m < BT_DG_MAX; ++m) {
    out[m] = 0;
    tbs[m] = m < nm ? mem[m].tb : 0;
    gens[m] = m < nm ? mem[m].gen : BG_NONE;
  }
  for (uint32_t j = threadIdx.x; j < TS; j += BT_THREADS) {
    const longlong2 p = P[j], l = Lt[j];
    const QL px = q60_split(p.x), py = q60_split(p.y), lx = q60_split(l.x), ly = q60_split(l.y);
    QAccF pos{0, 0, 0}, neg{0, 0, 0};
    qaccf_add(pos, lx, py);
    qaccf_add(neg, ly, px);
    const int64_t w = qaccf_result(pos) - qaccf_result(neg);
    uint32_t idx = 0;
#pragma unroll
    for (int m = 0; m < BT_DG_MAX; ++m) {
      const bool one = (j >> tbs[m]) & 1u;
      if (m < nm) idx |= (uint32_t)one << m;
      if (gens[m] == BG_Z) out[m] += one ? -w : w;
      else if (gens[m] == BG_P && one) out[m] -= 2 * w;
    }
    const QC u = E[idx];
    int64_t re, im;
    q60_gauss_mul(u, px, py, q60_split(p.x + p.y), &re, &im);
    P[j] = make_longlong2(re, im);
    q60_gauss_mul(u, lx, ly, q60_split(l.x + l.y), &re, &im);
    Lt[j] = make_longlong2(re, im);
  }
}

__device__ __forceinline__ longlong2 bt_unit(longlong2 a, int code) {
  switch (code) {
    case U_ONE: return a;
    case U_I: return make_longlong2(-a.y, a.x);
    case U_MINUS_ONE: return make_longlong2(-a.x, -a.y);
    default: return make_longlong2(a.y, -a.x);
  }
}

// Matrices of these passes are in Gauss form (qc_make_gauss): u * a with three
// limb products; a real entry keeps its value in u.re.
__device__ __forceinline__ longlong2 bt_mul(longlong2 a, int code, const QC& u) {
  if (code != U_GENERAL) return bt_unit(a, code);
  int64_t re, im;
  q60_gauss_mul(u, q60_split(a.x), q60_split(a.y), q60_split(a.x + a.y), &re, &im);
  return make_longlong2(re, im);
}

__device__ __forceinline__ uint32_t bt_expand(uint32_t i, uint32_t fixed, uint32_t set) {
  while (fixed) {
    int f = __ffs(fixed) - 1;
    fixed &= fixed - 1;
    i = ((i >> f) << (f + 1)) | (i & ((1u << f) - 1));
  }
  return i | set;
}

static __device__ void bt_apply(longlong2* tile, uint32_t TS, const BOp& op, int kind, int c0, int c1, const QC* U,
                         uint64_t base) {
  const uint32_t lcm = op.lcm;
  if (kind == BK_SCALAR) {
    const bool one = (base >> op.tb) & 1ull;
    const int code = one ? c1 : c0;
    if (code == U_ONE) return;
    const QC& u = U[one ? 3 : 0];
    const uint32_t cnt = TS >> __popc(lcm);
    for (uint32_t i = threadIdx.x; i < cnt; i += BT_THREADS) {
      uint32_t j = bt_expand(i, lcm, lcm);
      tile[j] = bt_mul(tile[j], code, u);
    }
    return;
  }
  const uint32_t tb = 1u << op.tb;
  const uint32_t fixed = lcm | tb;
  const uint32_t cnt = TS >> __popc(fixed);
  for (uint32_t i = threadIdx.x; i < cnt; i += BT_THREADS) {
    // without in-tile controls the insertion of one zero bit is a mask and an add
    const uint32_t j0 = lcm ? bt_expand(i, fixed, lcm) : i + (i & ~(tb - 1)), j1 = j0 | tb;
    if (kind == OP_PHASE1) {
      tile[j1] = bt_mul(tile[j1], c1, U[3]);
      continue;
    }
    longlong2 a0 = tile[j0], a1 = tile[j1], b0, b1;
    if (kind == OP_DIAG) {
      b0 = bt_mul(a0, c0, U[0]);
      b1 = bt_mul(a1, c1, U[3]);
    } else if (kind == OP_ANTI) {
      b0 = bt_mul(a1, c0, U[1]);
      b1 = bt_mul(a0, c1, U[2]);
    } else if (kind == OP_GENERAL) {
      const QL r0 = q60_split(a0.x), i0 = q60_split(a0.y), r1 = q60_split(a1.x), i1 = q60_split(a1.y);
      const QL s0 = q60_split(a0.x + a0.y), s1 = q60_split(a1.x + a1.y);
      int64_t re, im;
      q60_gauss_row(U[0], U[1], r0, i0, s0, r1, i1, s1, &re, &im);
      b0 = make_longlong2(re, im);
      q60_gauss_row(U[2], U[3], r0, i0, s0, r1, i1, s1, &re, &im);
      b1 = make_longlong2(re, im);
    } else {  // real entries: u.re of the Gauss form
      const QL r0 = q60_split(a0.x), i0 = q60_split(a0.y), r1 = q60_split(a1.x), i1 = q60_split(a1.y);
      int64_t out[4];
#pragma unroll
      for (int row = 0; row < 2; ++row) {
        const QC& u0 = U[2 * row];
        const QC& u1 = U[2 * row + 1];
        QAcc re = qacc_new(), im = qacc_new();
        qacc_add(re, u0.re, r0);
        qacc_add(re, u1.re, r1);
        qacc_add(im, u0.re, i0);
        qacc_add(im, u1.re, i1);
        out[2 * row] = qacc_round(re);
        out[2 * row + 1] = qacc_round(im);
      }
      b0 = make_longlong2(out[0], out[1]);
      b1 = make_longlong2(out[2], out[3]);
    }
    tile[j0] = b0;
    tile[j1] = b1;
  }
}

// sum_k s_k * l_k * p_k for four signed products of Q60 values, in Q60 units
// (all four limb products kept, one rounding: these terms are summed over the
// whole state).
__device__ __forceinline__ int64_t bt_dot4(const int64_t* l, const int64_t* p, const int* sg) {
  QAccF acc{0, 0, 0};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (sg[k] == 0) continue;
    qaccf_add(acc, q60_split(sg[k] > 0 ? l[k] : -l[k]), q60_split(p[k]));
  }
  return qaccf_result(acc);
}

// This thread's share of Im <lambda| G |psi> over the op's pairs in the tile, in
// Q60 units, summed exactly in an int64: every partial sum is bounded by
// sum |l_x| |p_y| over distinct pairs (x, y) times the generator's largest
// weight (2), i.e. by 2 ||lambda|| ||psi|| <= 2 * 1.25^2 < 4 (Cauchy-Schwarz),
// so it stays below 2^62.  No FP64 arithmetic per pair (GB300 issues FP64 at
// 1/74 of its FP32 rate).
static __device__ int64_t bt_gen_partial(const longlong2* P, const longlong2* Lt, uint32_t TS, const BOp& op,
                                         uint64_t base) {
  if (op.kf == BK_SCALAR) {
    // diagonal generator on a qubit outside the tile: per amplitude,
    // Z -> (-1)^bit Im(conj(l) p), P -> -2 [bit] Im(conj(l) p)
    const bool one = (base >> op.tb) & 1ull;
    if (op.gen == BG_P && !one) return 0;
    const int64_t w = op.gen == BG_P ? -2 : (one ? -1 : 1);
    const uint32_t cnt = TS >> __popc(op.lcm);
    int64_t acc = 0;
    for (uint32_t i = threadIdx.x; i < cnt; i += BT_THREADS) {
      const uint32_t j = bt_expand(i, op.lcm, op.lcm);
      const int64_t l[4] = {Lt[j].x, Lt[j].y, 0, 0}, p[4] = {P[j].y, P[j].x, 0, 0};
      const int sg[4] = {1, -1, 0, 0};
      acc += w * bt_dot4(l, p, sg);
    }
    return acc;
  }
  const uint32_t tb = 1u << op.tb;
  const uint32_t fixed = op.lcm | tb;
  const uint32_t cnt = TS >> __popc(fixed);
  int64_t acc = 0;
  for (uint32_t i = threadIdx.x; i < cnt; i += BT_THREADS) {
    const uint32_t j0 = op.lcm ? bt_expand(i, fixed, op.lcm) : i + (i & ~(tb - 1)), j1 = j0 | tb;
    const longlong2 p0 = P[j0], p1 = P[j1], l0 = Lt[j0], l1 = Lt[j1];
    int64_t l[4], p[4];
    int sg[4];
    switch (op.gen) {
      case BG_X:  // l0x p1y - l0y p1x + l1x p0y - l1y p0x
        l[0] = l0.x; p[0] = p1.y; sg[0] = 1; l[1] = l0.y; p[1] = p1.x; sg[1] = -1;
        l[2] = l1.x; p[2] = p0.y; sg[2] = 1; l[3] = l1.y; p[3] = p0.x; sg[3] = -1;
        break;
      case BG_Y:  // -l0x p1x - l0y p1y + l1x p0x + l1y p0y
        l[0] = l0.x; p[0] = p1.x; sg[0] = -1; l[1] = l0.y; p[1] = p1.y; sg[1] = -1;
        l[2] = l1.x; p[2] = p0.x; sg[2] = 1; l[3] = l1.y; p[3] = p0.y; sg[3] = 1;
        break;
      case BG_Z:  // l0x p0y - l0y p0x - l1x p1y + l1y p1x
        l[0] = l0.x; p[0] = p0.y; sg[0] = 1; l[1] = l0.y; p[1] = p0.x; sg[1] = -1;
        l[2] = l1.x; p[2] = p1.y; sg[2] = -1; l[3] = l1.y; p[3] = p1.x; sg[3] = 1;
        break;
      default:    // P: -2 (l1x p1y - l1y p1x)
        l[0] = l1.x; p[0] = p1.y; sg[0] = -1; l[1] = l1.y; p[1] = p1.x; sg[1] = 1;
        l[2] = 0; p[2] = 0; sg[2] = 0; l[3] = 0; p[3] = 0; sg[3] = 0;
        break;
    }
    const int64_t v = bt_dot4(l, p, sg);
    acc += op.gen == BG_P ? 2 * v : v;
  }
  return acc;
}

// Backward step of a pair op of class REAL with a generator (RY, H-type rows):
// for each of this thread's pairs, the generator term and then U on the psi pair
// and on the lambda pair, from one load and one limb split of each (real entries
// in u.re of the Gauss form).  Returns the thread's partial.
static __device__ int64_t bt_back_real(longlong2* P, longlong2* Lt, uint32_t TS, const BOp& op,
                                       const QC* __restrict__ U) {
  const uint32_t tb = 1u << op.tb;
  const uint32_t fixed = op.lcm | tb;
  const uint32_t cnt = TS >> __popc(fixed);
  int64_t acc = 0;
  for (uint32_t i = threadIdx.x; i < cnt; i += BT_THREADS) {
    const uint32_t j0 = op.lcm ? bt_expand(i, fixed, op.lcm) : i + (i & ~(tb - 1)), j1 = j0 | tb;
    const longlong2 p0 = P[j0], p1 = P[j1], l0 = Lt[j0], l1 = Lt[j1];
    const QL p0x = q60_split(p0.x), p0y = q60_split(p0.y), p1x = q60_split(p1.x), p1y = q60_split(p1.y);
    const QL l0x = q60_split(l0.x), l0y = q60_split(l0.y), l1x = q60_split(l1.x), l1y = q60_split(l1.y);
    acc += bt_pair_gen(op.gen, l0x, l0y, l1x, l1y, p0x, p0y, p1x, p1y);
#pragma unroll
    for (int row = 0; row < 2; ++row) {
      const QL u0 = U[2 * row].re, u1 = U[2 * row + 1].re;
      QAcc pr = qacc_new(), pi = qacc_new(), lr = qacc_new(), li = qacc_new();
      qacc_add(pr, u0, p0x);
      qacc_add(pr, u1, p1x);
      qacc_add(pi, u0, p0y);
      qacc_add(pi, u1, p1y);
      qacc_add(lr, u0, l0x);
      qacc_add(lr, u1, l1x);
      qacc_add(li, u0, l0y);
      qacc_add(li, u1, l1y);
      const uint32_t jr = row ? j1 : j0;
      P[jr] = make_longlong2(qacc_round(pr), qacc_round(pi));
      Lt[jr] = make_longlong2(qacc_round(lr), qacc_round(li));
    }
  }
  return acc;
}

// An antidiagonal op with unit factors (X, CNOT, Y, Toffoli) on psi and lambda in
// one sweep over the pairs: swaps with sign or i factors, no arithmetic.
static __device__ void bt_anti_both(longlong2* P, longlong2* Lt, uint32_t TS, const BOp& op, int c0, int c1) {
  const uint32_t tb = 1u << op.tb;
  const uint32_t fixed = op.lcm | tb;
  const uint32_t cnt = TS >> __popc(fixed);
  for (uint32_t i = threadIdx.x; i < cnt; i += BT_THREADS) {
    const uint32_t j0 = op.lcm ? bt_expand(i, fixed, op.lcm) : i + (i & ~(tb - 1)), j1 = j0 | tb;
    const longlong2 p0 = P[j0], p1 = P[j1], l0 = Lt[j0], l1 = Lt[j1];
    P[j0] = bt_unit(p1, c0);
    P[j1] = bt_unit(p0, c1);
    Lt[j0] = bt_unit(l1, c0);
    Lt[j1] = bt_unit(l0, c1);
  }
}

// Sum over the warp, exactly: three integer reductions of 24, 24 and 16 bits.
__device__ __forceinline__ int64_t bt_warp_sum(int64_t v) {
  const uint32_t a = __reduce_add_sync(0xffffffffu, (uint32_t)v & 0xffffffu);
  const uint32_t b = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 24) & 0xffffffu);
  const int32_t c = __reduce_add_sync(0xffffffffu, (int32_t)(v >> 48));
  return (int64_t)a + ((int64_t)b << 24) + (int64_t)c * (1ll << 48);
}

// Adds this thread's partial to its warp's accumulator of `slot` without a CTA
// barrier.  Accumulators hold twice the Q60 value (v2 = 2 x the partial) and stay
// exact: a slot's sum over the whole state is below 4 in magnitude (bt_gen_partial),
// twice that below 8 = 2^63.  wacc holds (BT_THREADS / 32) rows of nslots.  (As doubles
// they took two FP64 instructions a slot, warp and op, 37 cycles of the SM's FP64 pipe
// each, and a conversion.)
__device__ __forceinline__ void bt_warp_accumulate(int64_t v2, int64_t* wacc, int nslots, int slot) {
  v2 = bt_warp_sum(v2);
  if ((threadIdx.x & 31) == 0) wacc[(threadIdx.x >> 5) * nslots + slot] += v2;
}

// After a barrier: the CTA's total of `slot`.
__device__ __forceinline__ double bt_warp_total(const int64_t* wacc, int nslots, int slot) {
  int64_t t = 0;
#pragma unroll
  for (int w = 0; w < BT_THREADS / 32; ++w) t += wacc[w * nslots + slot];
  return 0.5 * q60_to_double(t);
}

// The records a pass works from (ops, group diagonals, pair coefficients), copied to
// shared memory where they fit: with the tiles there, the SM's L1 is too small to hold
// them, and every op began with a chain of loads from L2.
constexpr int BT_ST_OPS = 192, BT_ST_DG = 20, BT_ST_RP = 48;
struct BStage {
  BOp ops[BT_ST_OPS];
  QC dg[16 * BT_ST_DG];
  QP rp[2 * BT_ST_RP];
};
struct BRecords {  // indexed as the global arrays
  const BOp* ops;
  const QC* dg;
  const QP* rp;
};
template <class T>
__device__ __forceinline__ const T* bt_stage(T* dst, const T* src, int begin, int end, int per, int cap) {
  if (end - begin > cap) return src;
  static_assert(sizeof(T) % 8 == 0, "copied in 8-byte words");
  const int words = (int)((end - begin) * per * (sizeof(T) / 8));
  const uint64_t* s8 = reinterpret_cast<const uint64_t*>(src + (size_t)begin * per);
  uint64_t* d8 = reinterpret_cast<uint64_t*>(dst);
  for (int i = threadIdx.x; i < words; i += BT_THREADS) d8[i] = s8[i];
  return dst - (ptrdiff_t)begin * per;
}
// (A barrier must follow before the records are read, and one must precede when the
// stage holds another pass's.)
__device__ __forceinline__ BRecords bt_records(BStage* st, const BPass& ps, const BOp* ops, const QC* dg,
                                               const QP* rp) {
  BRecords r;
  r.ops = bt_stage(st->ops, ops, ps.op_begin, ps.op_end, 1, BT_ST_OPS);
  r.dg = bt_stage(st->dg, dg, ps.dg_begin, ps.dg_end, 16, BT_ST_DG);
  r.rp = bt_stage(st->rp, rp, ps.rp_begin, ps.rp_end, 2, BT_ST_RP);
  return r;
}

// Tile loads and stores.  Loads are asynchronous copies (the tiles hold the same Q60
// integers as memory): all of a thread's are in flight at once and take no registers;
// bt_load_wait comes before the barrier.
__device__ __forceinline__ void bt_load(longlong2* tile, const longlong2* src, uint64_t base, const uint64_t* offs,
                                        int L, uint32_t TS) {
  const uint32_t lowmask = (1u << L) - 1;
  for (uint32_t j = threadIdx.x; j < TS; j += BT_THREADS) cp_async16(tile + j, src + base + offs[j >> L] + (j & lowmask));
}
__device__ __forceinline__ void bt_load_wait() { cp_async_wait_all(); }
__device__ __forceinline__ void bt_store(const longlong2* tile, longlong2* dst, uint64_t base, const uint64_t* offs,
                                         int L, uint32_t TS) {
  constexpr int E = (1 << BT_M) / BT_THREADS;
  const uint32_t lowmask = (1u << L) - 1;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const uint32_t j = threadIdx.x + e * BT_THREADS;
    if (j < TS) dst[base + offs[j >> L] + (j & lowmask)] = tile[j];
  }
}

static __device__ double bt_block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double r = 0.0;
#pragma unroll
  for (int i = 0; i < BT_THREADS / 32; ++i) r += red[i];
  return r;
}

// ---- lambda = (H / S) psi -------------------------------------------------------------
// The terms of H / S as
//   runs    X masks whose only term has no Z and the same real coefficient: their
//           amplitudes are added first and multiplied once;
//   groups  every other X mask, with its terms: the signed coefficient sums
//           d = sum_t (-1)^popc(x & zm_t) c_t are exact in int64 (sum |c_t| <= 1).
// |lambda_y| <= |psi|_inf <= 1.25 and every product is rounded once.
constexpr int HRUN_MAX = 32;  // a run's amplitude sum stays below sqrt(32) * 1.25 < 8
struct HRun {
  int64_t c;  // coef / S, Q60
  int begin, end;
};
struct HGroup {
  uint64_t xm;
  int begin, end, imag;  // imag: some term has an imaginary factor
};
struct HTerm {
  int64_t c;  // coef / S with the real sign of i^ny, Q60
  uint64_t zm;
  int imag;   // i^ny is imaginary
};

// The runs, groups and terms of a Pauli sum; xms: the X masks of the runs in order.
static inline void h_plan(const qs_pauli* terms, size_t nt, double S, std::vector<HRun>* runs,
                          std::vector<uint64_t>* xms, std::vector<HGroup>* groups, std::vector<HTerm>* hterms) {
  std::vector<uint64_t> order;
  std::vector<std::vector<size_t>> of;
  for (size_t k = 0; k < nt; ++k) {  // by X mask, in order of first appearance
    size_t g = 0;
    while (g < order.size() && order[g] != terms[k].xmask) ++g;
    if (g == order.size()) {
      order.push_back(terms[k].xmask);
      of.emplace_back();
    }
    of[g].push_back(k);
  }
  std::vector<std::pair<int64_t, uint64_t>> plain;
  for (size_t g = 0; g < order.size(); ++g) {
    if (of[g].size() == 1 && terms[of[g][0]].zmask == 0) {
      plain.push_back({q60_from_double(terms[of[g][0]].coef / S), order[g]});
      continue;
    }
    HGroup gr{order[g], (int)hterms->size(), 0, 0};
    for (size_t k : of[g]) {
      const int ny = __builtin_popcountll(terms[k].xmask & terms[k].zmask) & 3;
      const double c = terms[k].coef / S;
      hterms->push_back(HTerm{q60_from_double(ny >= 2 ? -c : c), terms[k].zmask, ny & 1});
      gr.imag |= ny & 1;
    }
    gr.end = (int)hterms->size();
    groups->push_back(gr);
  }
  std::stable_sort(plain.begin(), plain.end(),
                   [](const auto& a, const auto& b) { return a.first < b.first; });
  for (size_t k = 0; k < plain.size(); ++k) {
    if (k == 0 || runs->back().c != plain[k].first || runs->back().end - runs->back().begin == HRUN_MAX)
      runs->push_back(HRun{plain[k].first, (int)xms->size(), (int)xms->size()});
    xms->push_back(plain[k].second);
    ++runs->back().end;
  }
}

#ifdef __CUDACC__
// c * s for a Q60 coefficient |c| <= 1 and a sum |s| < 8, rounded once: limbs of 32
// bits with signed low limbs, c in units of 2^-62.
__device__ __forceinline__ int64_t h_mul_sum(int64_t c, int64_t s) {
  const int64_t C = c << 2;
  const int32_t cl = (int32_t)C, sl = (int32_t)s;
  const int32_t ch = (int32_t)(C >> 32) + (int32_t)((uint32_t)cl >> 31);
  const int32_t sh = (int32_t)(s >> 32) + (int32_t)((uint32_t)sl >> 31);
  const int64_t hi = madw(ch, sh, 0), mid = madw(cl, sh, madw(ch, sl, 1ll << 29));
  return (hi << 2) + (mid >> 30);
}

__device__ __forceinline__ bool h_parity(uint64_t x, uint64_t zm) {
  const uint32_t hi = (uint32_t)(x >> 32) & (uint32_t)(zm >> 32);
  return __popc(((uint32_t)x & (uint32_t)zm) ^ hi) & 1;
}

// Row y of (H / S) psi; load(x) gives psi_x in Q60.
template <class F>
__device__ __forceinline__ longlong2 h_row(const HRun* runs, int nruns, const uint64_t* xms, const HGroup* groups,
                                           int ngroups, const HTerm* terms, uint64_t y, F&& load) {
  int64_t ore = 0, oim = 0;
  for (int r = 0; r < nruns; ++r) {
    const HRun run = runs[r];
    int64_t sr = 0, si = 0;
    int k = run.begin;
    for (; k + 4 <= run.end; k += 4) {  // four gathers in flight
      const longlong2 a = load(y ^ xms[k]), b = load(y ^ xms[k + 1]), c = load(y ^ xms[k + 2]),
                      d = load(y ^ xms[k + 3]);
      sr += (a.x + b.x) + (c.x + d.x);
      si += (a.y + b.y) + (c.y + d.y);
    }
    for (; k < run.end; ++k) {
      const longlong2 a = load(y ^ xms[k]);
      sr += a.x;
      si += a.y;
    }
    ore += h_mul_sum(run.c, sr);
    oim += h_mul_sum(run.c, si);
  }
  for (int g = 0; g < ngroups; ++g) {
    const HGroup gr = groups[g];
    const uint64_t x = y ^ gr.xm;
    const longlong2 p = load(x);
    int64_t dre = 0, dim = 0;
    if (!gr.imag) {
      for (int k = gr.begin; k < gr.end; ++k) {
        const int64_t c = terms[k].c;
        dre += h_parity(x, terms[k].zm) ? -c : c;
      }
    } else {
      for (int k = gr.begin; k < gr.end; ++k) {
        const int64_t v = h_parity(x, terms[k].zm) ? -terms[k].c : terms[k].c;
        if (terms[k].imag) dim += v;
        else dre += v;
      }
    }
    const QL px = q60_split(p.x), py = q60_split(p.y), qr = q60_split_coef(dre);
    QAcc re = qacc_new(), im = qacc_new();
    qacc_add(re, qr, px);  // re: dre px - dim py
    qacc_add(im, qr, py);  // im: dre py + dim px
    if (gr.imag) {
      qacc_add(re, q60_split_coef(-dim), py);
      qacc_add(im, q60_split_coef(dim), px);
    }
    ore += qacc_round(re);
    oim += qacc_round(im);
  }
  return make_longlong2(ore, oim);
}
#endif

// Runs of up to BT_DG_MAX consecutive uncontrolled diagonal ops (forward and
// adjoint class) on distinct tile qubits, with a Z, P or no generator, of the
// ops [begin, end) become diagonal groups: a BK_DGROUP head (gate = group index,
// nmem members) is inserted before the members, which turn into BK_MEMBER
// records.  Heads are appended to `heads` (their index in the new op list);
// src[i - begin] receives the old index of new op i (-1 for a head).
// Consecutive uncontrolled real rotations on distinct tile qubits become real pairs
// the same way (a BK_RPAIR head, gate = index into `pairs`, two BK_MEMBER records),
// and runs of X and CNOT gates without a gradient permutations (a BK_PERM head).
static inline void group_diagonals(std::vector<BOp>& ops, size_t begin, std::vector<int>* heads,
                                   std::vector<int>* src, std::vector<int>* pairs) {
  auto eligible = [](const BOp& o) {
    const bool df = o.kf == OP_DIAG || o.kf == OP_PHASE1, db = o.kb == OP_DIAG || o.kb == OP_PHASE1;
    return df && db && o.lcm == 0 && o.ext == 0 && (o.gen == BG_NONE || o.gen == BG_Z || o.gen == BG_P);
  };
  auto real = [](const BOp& o) {
    return o.kf == OP_REAL && o.kb == OP_REAL && o.rot && o.lcm == 0 && o.ext == 0 &&
           (o.gen == BG_NONE || o.gen == BG_Y);
  };
  auto swaps = [](const BOp& o) {
    return o.kf == OP_ANTI && o.kb == OP_ANTI && o.c0f == U_ONE && o.c1f == U_ONE && o.c0b == U_ONE &&
           o.c1b == U_ONE && __builtin_popcount(o.lcm) <= 1 && o.gen == BG_NONE;
  };
  // Only the pass's own ops are copied: the list of a whole batch copied once a pass was
  // most of its creation (128 sets of 10..18 qubits, host time 210 -> 5 ms on one x86 core).
  const std::vector<BOp> in(ops.begin() + begin, ops.end());
  std::vector<BOp>& out = ops;
  out.resize(begin);
  src->clear();
  size_t i = 0;
  while (i < in.size()) {
    size_t run = i;
    while (run < in.size() && run - i < 127 && swaps(in[run])) ++run;
    if (run - i >= 2) {
      BOp h;
      memset(&h, 0, sizeof h);
      h.kf = h.kb = BK_PERM;
      h.nmem = (int8_t)(run - i);
      h.slot = -1;
      h.param = -1;
      h.gen = BG_NONE;
      out.push_back(h);
      src->push_back(-1);
      for (size_t k = i; k < run; ++k) {
        BOp mo = in[k];
        mo.kf = mo.kb = BK_MEMBER;
        out.push_back(mo);
        src->push_back((int)(begin + k));
      }
      i = run;
      continue;
    }
    if (i + 1 < in.size() && real(in[i]) && real(in[i + 1]) && in[i].tb != in[i + 1].tb) {
      BOp h;
      memset(&h, 0, sizeof h);
      h.kf = h.kb = BK_RPAIR;
      h.nmem = 2;
      h.gate = (int)pairs->size();
      h.slot = -1;
      h.param = -1;
      h.gen = BG_NONE;
      pairs->push_back((int)out.size());
      out.push_back(h);
      src->push_back(-1);
      for (size_t k = i; k < i + 2; ++k) {
        BOp mo = in[k];
        mo.kf = mo.kb = BK_MEMBER;
        out.push_back(mo);
        src->push_back((int)(begin + k));
      }
      i += 2;
      continue;
    }
    size_t j = i;
    uint32_t bits = 0;
    while (j < in.size() && j - i < (size_t)BT_DG_MAX && eligible(in[j]) && !((bits >> in[j].tb) & 1)) {
      bits |= 1u << in[j].tb;
      ++j;
    }
    if (j - i >= 2) {
      BOp h;
      memset(&h, 0, sizeof h);
      h.kf = h.kb = BK_DGROUP;
      h.nmem = (int8_t)(j - i);
      h.gate = (int)heads->size();
      h.slot = -1;
      h.param = -1;
      h.gen = BG_NONE;
      heads->push_back((int)out.size());
      out.push_back(h);
      src->push_back(-1);
      for (size_t k = i; k < j; ++k) {
        BOp mo = in[k];
        mo.kf = mo.kb = BK_MEMBER;
        out.push_back(mo);
        src->push_back((int)(begin + k));
      }
      i = j;
    } else {
      out.push_back(in[i]);
      src->push_back((int)(begin + i));
      ++i;
    }
  }
}

}  // namespace qs
