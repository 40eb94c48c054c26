// Adjoint differentiation of <psi(theta)| H |psi(theta)> for parametrised
// circuits (the paper's variational circuits, Section "Variational quantum
// circuit", with qop expectations; it does not say how gradients are taken --
// this is the adjoint recursion of Jones & Gacon, arXiv:2009.02823):
//   psi = U_G ... U_1 |0>,  lambda = H psi,  E = Re <psi|lambda>,
//   for k = G..1:  dE/dtheta_k += Im <lambda| G_k |psi>   (if U_k = exp(-i theta G_k / 2))
//                  psi <- U_k^dag psi,  lambda <- U_k^dag lambda.
// One fused kernel per backward gate reads both vectors once, forms the
// generator inner product (FP64, deterministic per-CTA partials) and applies
// U_k^dag to both.  lambda is kept scaled by 1/S, S a power of two >= sum|coef|,
// so that its components stay inside the Q60 range of the gate engine.
#include <math.h>

#include <algorithm>
#include <memory>
#include <new>
#include <vector>

#include "fixed.h"
#include "internal.h"
#include "q60tile.cuh"

namespace qs {

enum GenKind : int { GEN_NONE = 0, GEN_X = 1, GEN_Y = 2, GEN_Z = 3, GEN_P = 4 };

struct AdjArgs {
  double2 m[4];     // U^dag (FP64 engine)
  QC q[4];          // U^dag (Q60 engine)
  uint64_t cmask;
  int64_t items;
  int t, nfix;
  int fix[QS_MAX_QUBITS];
  int cls, code0, code1;
  int gen;          // GenKind
  double gsign;     // -1 for a dagger record
  int slot;         // partial-sum slot of this gate
};

__device__ __forceinline__ double adj_neg(double x) {
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
}

__device__ __forceinline__ double2 adj_unit(double2 a, int code) {
  switch (code) {
    case U_ONE: return a;
    case U_I: return make_double2(adj_neg(a.y), a.x);
    case U_MINUS_ONE: return make_double2(adj_neg(a.x), adj_neg(a.y));
    default: return make_double2(a.y, adj_neg(a.x));
  }
}

// Apply the op to the pair (a0, a1) in place.
template <bool FX>
__device__ __forceinline__ void adj_pair(const AdjArgs& g, double2& a0, double2& a1) {
  const int cls = g.cls;
  if (!FX) {
    auto mulc = [](double2 a, int code, double2 u) {
      if (code != U_GENERAL) return adj_unit(a, code);
      return make_double2(fma(u.x, a.x, -u.y * a.y), fma(u.x, a.y, u.y * a.x));
    };
    if (cls == OP_PHASE1) {
      a1 = mulc(a1, g.code1, g.m[3]);
    } else if (cls == OP_DIAG) {
      a0 = mulc(a0, g.code0, g.m[0]);
      a1 = mulc(a1, g.code1, g.m[3]);
    } else if (cls == OP_ANTI) {
      double2 b0 = mulc(a1, g.code0, g.m[1]), b1 = mulc(a0, g.code1, g.m[2]);
      a0 = b0;
      a1 = b1;
    } else if (cls == OP_REAL) {
      double2 b0 = make_double2(fma(g.m[0].x, a0.x, g.m[1].x * a1.x), fma(g.m[0].x, a0.y, g.m[1].x * a1.y));
      double2 b1 = make_double2(fma(g.m[2].x, a0.x, g.m[3].x * a1.x), fma(g.m[2].x, a0.y, g.m[3].x * a1.y));
      a0 = b0;
      a1 = b1;
    } else if (cls == OP_GENERAL) {
      const double2 u0 = g.m[0], u1 = g.m[1], u2 = g.m[2], u3 = g.m[3];
      double2 b0, b1;
      b0.x = fma(u0.x, a0.x, fma(-u0.y, a0.y, fma(u1.x, a1.x, -u1.y * a1.y)));
      b0.y = fma(u0.x, a0.y, fma(u0.y, a0.x, fma(u1.x, a1.y, u1.y * a1.x)));
      b1.x = fma(u2.x, a0.x, fma(-u2.y, a0.y, fma(u3.x, a1.x, -u3.y * a1.y)));
      b1.y = fma(u2.x, a0.y, fma(u2.y, a0.x, fma(u3.x, a1.y, u3.y * a1.x)));
      a0 = b0;
      a1 = b1;
    }
    return;
  }
  auto qmul = [](double2 a, int code, const QC& u) {
    if (code != U_GENERAL) return adj_unit(a, code);
    const QL ar = q60_split(q60_from_double(a.x)), ai = q60_split(q60_from_double(a.y));
    QAcc re = qacc_new(), im = qacc_new();
    qacc_add(re, u.re, ar);
    qacc_add(re, u.nim, ai);
    qacc_add(im, u.re, ai);
    qacc_add(im, u.im, ar);
    return make_double2(q60_to_double(qacc_round(re)), q60_to_double(qacc_round(im)));
  };
  if (cls == OP_PHASE1) {
    a1 = qmul(a1, g.code1, g.q[3]);
  } else if (cls == OP_DIAG) {
    a0 = qmul(a0, g.code0, g.q[0]);
    a1 = qmul(a1, g.code1, g.q[3]);
  } else if (cls == OP_ANTI) {
    double2 b0 = qmul(a1, g.code0, g.q[1]), b1 = qmul(a0, g.code1, g.q[2]);
    a0 = b0;
    a1 = b1;
  } else if (cls == OP_REAL || cls == OP_GENERAL) {
    const QL r0 = q60_split(q60_from_double(a0.x)), i0 = q60_split(q60_from_double(a0.y));
    const QL r1 = q60_split(q60_from_double(a1.x)), i1 = q60_split(q60_from_double(a1.y));
    int64_t out[4];
#pragma unroll
    for (int row = 0; row < 2; ++row) {
      const QC& u0 = g.q[2 * row];
      const QC& u1 = g.q[2 * row + 1];
      QAcc re = qacc_new(), im = qacc_new();
      qacc_add(re, u0.re, r0);
      qacc_add(re, u1.re, r1);
      qacc_add(im, u0.re, i0);
      qacc_add(im, u1.re, i1);
      if (cls == OP_GENERAL) {
        qacc_add(re, u0.nim, i0);
        qacc_add(re, u1.nim, i1);
        qacc_add(im, u0.im, r0);
        qacc_add(im, u1.im, r1);
      }
      out[2 * row] = qacc_round(re);
      out[2 * row + 1] = qacc_round(im);
    }
    a0 = make_double2(q60_to_double(out[0]), q60_to_double(out[1]));
    a1 = make_double2(q60_to_double(out[2]), q60_to_double(out[3]));
  }
}

// Im <lambda| G |psi> over one pair.
__device__ __forceinline__ double gen_im(int gen, double2 l0, double2 l1, double2 p0, double2 p1) {
  switch (gen) {
    case GEN_X: return fma(l0.x, p1.y, -l0.y * p1.x) + fma(l1.x, p0.y, -l1.y * p0.x);
    case GEN_Y: return -fma(l0.x, p1.x, l0.y * p1.y) + fma(l1.x, p0.x, l1.y * p0.y);
    case GEN_Z: return fma(l0.x, p0.y, -l0.y * p0.x) - fma(l1.x, p1.y, -l1.y * p1.x);
    case GEN_P: return -2.0 * fma(l1.x, p1.y, -l1.y * p1.x);
    default: return 0.0;
  }
}

__device__ __forceinline__ double adj_block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
  return r;
}

template <bool FX>
__global__ void __launch_bounds__(256) k_adj_step(double2* __restrict__ psi, double2* __restrict__ lam,
                                                  const AdjArgs g, double* __restrict__ part) {
  __shared__ double sh[8];
  const uint64_t tb = 1ull << g.t;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  double acc = 0.0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < (uint64_t)g.items; i += stride) {
    uint64_t x0 = i;
    for (int k = 0; k < g.nfix; ++k) {
      int f = g.fix[k];
      x0 = ((x0 >> f) << (f + 1)) | (x0 & ((1ull << f) - 1));
    }
    x0 |= g.cmask;
    const uint64_t x1 = x0 | tb;
    double2 p0 = psi[x0], p1 = psi[x1], l0 = lam[x0], l1 = lam[x1];
    if (g.gen != GEN_NONE) acc += gen_im(g.gen, l0, l1, p0, p1);
    adj_pair<FX>(g, p0, p1);
    adj_pair<FX>(g, l0, l1);
    psi[x0] = p0;
    psi[x1] = p1;
    lam[x0] = l0;
    lam[x1] = l1;
  }
  if (g.gen != GEN_NONE) {
    double s = adj_block_sum(acc, sh);
    if (threadIdx.x == 0) part[(size_t)g.slot * gridDim.x + blockIdx.x] = s * g.gsign;
  }
}

// lambda = (H / S) psi (h_row in q60tile.cuh) as a gather.  FX: psi and lambda hold
// Q60 integers, else complex128.
constexpr int HMAX = 48;
struct HArgs {
  uint64_t N;
  int nruns, ngroups, accumulate;
  HRun runs[HMAX];
  uint64_t xms[HMAX];
  HGroup groups[HMAX];
  HTerm terms[HMAX];
};

template <bool FX>
__global__ void __launch_bounds__(256) k_apply_h(const double2* __restrict__ psi, double2* __restrict__ lam,
                                                 const __grid_constant__ HArgs h) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  auto load = [](const double2* a, uint64_t x) {
    if (FX) return reinterpret_cast<const longlong2*>(a)[x];
    const double2 p = a[x];
    return make_longlong2(q60_from_double_nb(p.x), q60_from_double_nb(p.y));
  };
  for (uint64_t y = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; y < h.N; y += stride) {
    longlong2 out = h_row(h.runs, h.nruns, h.xms, h.groups, h.ngroups, h.terms, y,
                          [&](uint64_t x) { return load(psi, x); });
    if (FX) {
      longlong2* l = reinterpret_cast<longlong2*>(lam) + y;
      if (h.accumulate) out = make_longlong2(out.x + l->x, out.y + l->y);
      *l = out;
    } else {
      double2 v = make_double2(q60_to_double_nb(out.x), q60_to_double_nb(out.y));
      if (h.accumulate) v = make_double2(v.x + lam[y].x, v.y + lam[y].y);
      lam[y] = v;
    }
  }
}

// per-CTA partials of Re <psi|lambda>
template <bool FX>
__global__ void __launch_bounds__(256) k_dot_re(const double2* __restrict__ a, const double2* __restrict__ b, uint64_t N,
                                                double* __restrict__ part) {
  __shared__ double sh[8];
  double acc = 0.0;
  __int128 eq = 0;  // FX: exact products (units 2^-120)
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < N; i += (uint64_t)gridDim.x * blockDim.x) {
    if (FX) {
      const longlong2 u = reinterpret_cast<const longlong2*>(a)[i], v = reinterpret_cast<const longlong2*>(b)[i];
      eq += (__int128)dot2_exact(split31(u.x), split31(v.x), split31(u.y), split31(v.y));
    } else {
      const double2 u = a[i], v = b[i];
      acc += fma(u.x, v.x, u.y * v.y);
    }
  }
  if (FX) acc = q120_to_double(eq);
  double s = adj_block_sum(acc, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// out[j] = sum over the CTA partials of slot j: one CTA a slot, its threads' partials in
// CTA order, then a fixed tree (one thread a slot waited for memory 608 times).
__global__ void __launch_bounds__(256) k_slot_sums(const double* __restrict__ part, int nblocks,
                                                   double* __restrict__ out) {
  __shared__ double sh[8];
  double s = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += 256) s += part[(size_t)blockIdx.x * nblocks + b];
  s = adj_block_sum(s, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// ---- fused backward sweep (Q60): tile passes over psi and lambda at once --------------
// The backward sweep applies U_G^dag .. U_1^dag, so it is the forward sweep of the
// reversed, daggered program; greedy tile passes over that list only reorder ops
// that commute, and an op that commutes with U_k also commutes with U_k's
// generator (same qubits, same diagonal structure), so every generator inner
// product is taken on the same (psi, lambda) as in the gate-by-gate sweep.
constexpr int ADJ_GRID_STRIDE = 608;  // partial-sum slots per gradient (>= CTAs of any pass)

struct AdjPassArgs {
  BPass ps;
  const BOp* ops;   // ops of this pass (device), in execution order
  const QC* mats;   // 4 entries per op (device)
  const QC* dgm;    // 16 entries per diagonal group (device)
  const QP* rpm;    // 2 entries per real pair (device)
  double* part;     // [slot][ADJ_GRID_STRIDE]
  int slot_base;
};

// psi and lambda hold Q60 integers from the last forward pass on: no conversion and no
// rounding to double between passes.
__global__ void __launch_bounds__(BT_THREADS, 3) k_adj_pass(longlong2* __restrict__ psi, longlong2* __restrict__ lam,
                                                         const __grid_constant__ AdjPassArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const BPass& ps = a.ps;
  const int m = ps.m;
  const int L = m - ps.nhigh;
  const uint32_t TS = 1u << m;
  const uint32_t H = 1u << ps.nhigh;
  longlong2* tP = reinterpret_cast<longlong2*>(smem);
  longlong2* tL = tP + TS;
  uint64_t* offs = reinterpret_cast<uint64_t*>(tL + TS);
  int64_t* wacc = reinterpret_cast<int64_t*>(offs + H);  // [warps][nslots]
  for (uint32_t h = threadIdx.x; h < H; h += BT_THREADS) {
    uint64_t o = 0;
    for (int b = 0; b < ps.nhigh; ++b) o |= (uint64_t)((h >> b) & 1u) << ps.qhigh[b];
    offs[h] = o;
  }
  for (int s = threadIdx.x; s < ps.nslots * (BT_THREADS / 32); s += BT_THREADS) wacc[s] = 0;
  const uint64_t ntiles = 1ull << ps.nout;
  for (uint64_t r = blockIdx.x; r < ntiles; r += gridDim.x) {
    uint64_t base = 0;
    for (int b = 0; b < ps.nout; ++b) base |= ((r >> b) & 1ull) << ps.outpos[b];
    __syncthreads();
    bt_load(tP, psi, base, offs, L, TS);
    bt_load(tL, lam, base, offs, L, TS);
    bt_load_wait();
    __syncthreads();
    for (int k = ps.op_begin; k < ps.op_end; ++k) {
      const BOp& op = a.ops[k];
      if (op.kb == BK_MEMBER || (base & op.ext) != op.ext) continue;
      // each thread reads and then rewrites only its own pairs (amplitudes) of this
      // op, so the generator partial and the update need no barrier between them
      if (op.kb == BK_DGROUP) {
        int64_t gp[BT_DG_MAX];
        const BOp* mem = a.ops + k + 1;
        bt_back_dgroup(tP, tL, TS, mem, op.nmem, a.dgm + 16 * op.gate, gp);
        for (int mm = 0; mm < op.nmem; ++mm)
          if (mem[mm].slot >= 0) bt_warp_accumulate(2 * gp[mm], wacc, ps.nslots, mem[mm].slot);
        __syncthreads();
        continue;
      }
      if (op.kb == BK_RPAIR) {
        const BOp* mem = a.ops + k + 1;
        int64_t gu, gv;
        bt_rpair_back(tP, tL, TS, 1u << mem[0].tb, 1u << mem[1].tb, mem[0].slot >= 0 || mem[1].slot >= 0,
                      a.rpm + 2 * op.gate, &gu, &gv);
        if (mem[0].slot >= 0) bt_warp_accumulate(gu + gv, wacc, ps.nslots, mem[0].slot);
        if (mem[1].slot >= 0) bt_warp_accumulate(gu - gv, wacc, ps.nslots, mem[1].slot);
        __syncthreads();
        continue;
      }
      if (op.kb == BK_PERM) {
        bt_perm(tP, tL, TS, a.ops + k + 1, op.nmem, false, base);
        __syncthreads();
        continue;
      }
      if (op.slot < 0 && op.kb == OP_ANTI && op.c0b != U_GENERAL && op.c1b != U_GENERAL) {
        bt_anti_both(tP, tL, TS, op, op.c0b, op.c1b);  // psi and lambda in one sweep
        __syncthreads();
        continue;
      }
      if (op.slot >= 0 && op.kb == OP_REAL) {  // one pass over the pairs
        bt_warp_accumulate(2 * bt_back_real(tP, tL, TS, op, a.mats + 4 * k), wacc, ps.nslots, op.slot);
        __syncthreads();
        continue;
      }
      if (op.slot >= 0) bt_warp_accumulate(2 * bt_gen_partial(tP, tL, TS, op, base), wacc, ps.nslots, op.slot);
      bt_apply(tP, TS, op, op.kb, op.c0b, op.c1b, a.mats + 4 * k, base);
      bt_apply(tL, TS, op, op.kb, op.c0b, op.c1b, a.mats + 4 * k, base);
      __syncthreads();
    }
    bt_store(tP, psi, base, offs, L, TS);
    bt_store(tL, lam, base, offs, L, TS);
  }
  __syncthreads();
  for (int k = ps.op_begin + threadIdx.x; k < ps.op_end; k += BT_THREADS) {
    const BOp& op = a.ops[k];
    if (op.slot >= 0)
      a.part[(size_t)(a.slot_base + op.slot) * ADJ_GRID_STRIDE + blockIdx.x] =
          bt_warp_total(wacc, ps.nslots, op.slot) * op.gsign;
  }
}

static int gen_of(const qs_gate& g);

// Backward sweep as tile passes; slot_param receives, per gradient slot in
// execution order, the parameter it belongs to.
static int backward_fused(qs_state* s, double2* lam, const qs_gate* gates, size_t ng, const double* params,
                          double* part, std::vector<int>& slot_param) {
  const int n = s->n;
  std::vector<qs_gate> R(ng);
  std::vector<int> tgt(ng);
  std::vector<uint64_t> cms(ng);
  for (size_t i = 0; i < ng; ++i) {
    R[i] = gates[ng - 1 - i];
    R[i].dagger = !R[i].dagger;
    QS_TRY(gate_qubits(R[i], n, &tgt[i], &cms[i]));
  }
  const int m = std::min(n, BT_M);
  const uint64_t low = (1ull << std::min(n, 3)) - 1;
  GateQueue remaining = gate_queue(tgt, cms), rest;
  std::vector<uint32_t> pass;
  std::vector<BOp> ops;
  std::vector<Mat2> opm;  // each op's matrix (double), parallel to ops
  std::vector<QC> mats;
  std::vector<QC> dgm;    // 16 Gauss-form entries per diagonal group
  std::vector<int> dgheads, dgsrc, rpheads;
  std::vector<QP> rpm;    // 2 coefficients per real pair
  std::vector<BPass> passes;
  int slot_base = 0;
  std::vector<int> slot_bases;
  while (!remaining.empty()) {
    const uint64_t Q = greedy_pass(R.data(), tgt, cms, remaining, m, low, BT_MAX_OPS, pass, rest);
    BPass bp;
    memset(&bp, 0, sizeof bp);
    int local[64];
    int mm = 0;
    for (int b = 0; b < n; ++b) local[b] = ((Q >> b) & 1) ? mm++ : -1;
    int L = 0;
    while (L < n && ((Q >> L) & 1)) ++L;
    bp.m = mm;
    for (int b = L; b < n; ++b)
      if ((Q >> b) & 1) bp.qhigh[bp.nhigh++] = b;
    for (int b = 0; b < n; ++b)
      if (!((Q >> b) & 1)) bp.outpos[bp.nout++] = b;
    bp.op_begin = (int)ops.size();
    int slot = 0;
    for (uint32_t i : pass) {
      const qs_gate& orig = gates[ng - 1 - i];
      Mat2 mt;
      QS_TRY(gate_matrix(R[i], params, &mt));
      Op1 o1 = classify(tgt[i], cms[i], mt);
      BOp op;
      memset(&op, 0, sizeof op);
      op.gen = orig.param_idx >= 0 ? (int8_t)gen_of(orig) : (int8_t)BG_NONE;
      if (o1.cls == OP_IDENTITY && op.gen == BG_NONE) continue;
      op.kb = op.kf = (int8_t)o1.cls;
      op.c0b = (int8_t)o1.code0;
      op.c1b = (int8_t)o1.code1;
      op.c0f = op.c0b;
      op.c1f = op.c1b;
      op.rot = o1.cls == OP_REAL && mt.m[0].re * mt.m[3].re - mt.m[1].re * mt.m[2].re > 0.0;
      uint32_t lcm = 0;
      uint64_t ext = 0;
      for (int b = 0; b < n; ++b)
        if ((cms[i] >> b) & 1) {
          if (local[b] >= 0) lcm |= 1u << local[b];
          else ext |= 1ull << b;
        }
      op.lcm = lcm;
      op.ext = ext;
      if (local[tgt[i]] >= 0) {
        op.tb = (int8_t)local[tgt[i]];
        if (o1.cls == OP_IDENTITY) op.kb = op.kf = OP_PHASE1;  // identity matrix, kept for its gradient slot
      } else {
        op.tb = (int8_t)tgt[i];
        op.kb = op.kf = BK_SCALAR;
      }
      op.gsign = orig.dagger ? -1.0 : 1.0;
      op.slot = -1;
      op.param = orig.param_idx;
      if (op.gen != BG_NONE) {
        op.slot = (int16_t)slot++;
        slot_param.push_back(orig.param_idx);
      }
      ops.push_back(op);
      opm.push_back(mt);
    }
    // runs of diagonal ops -> diagonal groups; then the matrix tables in op order
    const size_t ng0 = dgheads.size(), np0 = rpheads.size();
    group_diagonals(ops, bp.op_begin, &dgheads, &dgsrc, &rpheads);
    std::vector<Mat2> pm(dgsrc.size());
    for (size_t k = 0; k < dgsrc.size(); ++k) {
      if (dgsrc[k] >= 0) pm[k] = opm[dgsrc[k]];
      else pm[k] = Mat2{};
    }
    opm.resize(bp.op_begin);
    opm.insert(opm.end(), pm.begin(), pm.end());
    for (size_t k = bp.op_begin; k < ops.size(); ++k)
      for (int e = 0; e < 4; ++e) mats.push_back(qc_make_gauss(opm[k].m[e].re, opm[k].m[e].im));  // bt_apply's form
    for (size_t gi = ng0; gi < dgheads.size(); ++gi) {
      const int head = dgheads[gi];
      const int nm = ops[head].nmem;
      for (int idx = 0; idx < 16; ++idx) {
        double re = 1.0, im = 0.0;
        for (int mm = 0; mm < nm && idx < (1 << nm); ++mm) {
          const C2 u = opm[head + 1 + mm].m[((idx >> mm) & 1) ? 3 : 0];
          const double r2 = re * u.re - im * u.im, i2 = re * u.im + im * u.re;
          re = r2;
          im = i2;
        }
        dgm.push_back(qc_make_gauss(re, im));
      }
    }
    for (size_t pi = np0; pi < rpheads.size(); ++pi) {
      double ra[4], rb[4];
      for (int e = 0; e < 4; ++e) {
        ra[e] = opm[rpheads[pi] + 1].m[e].re;
        rb[e] = opm[rpheads[pi] + 2].m[e].re;
      }
      QP c[2];
      int flags;  // rotations: 0
      q60_pair_gauss_coef(ra, rb, c, &flags);
      rpm.insert(rpm.end(), c, c + 2);
    }
    bp.op_end = (int)ops.size();
    bp.nslots = slot;
    passes.push_back(bp);
    slot_bases.push_back(slot_base);
    slot_base += slot;
    std::swap(remaining, rest);
  }
  // one upload from pinned memory into the workspace (or, if that is too small, into
  // memory of this call)
  auto up16 = [](size_t b) { return (b + 15) & ~(size_t)15; };
  const size_t ob = up16(sizeof(BOp) * ops.size()), mb = up16(sizeof(QC) * mats.size()),
               db = up16(sizeof(QC) * dgm.size()), rb = up16(sizeof(QP) * rpm.size()), total = ob + mb + db + rb;
  ScratchBuf big;
  char* dev = (char*)s->ws;
  if (total > s->ws_bytes) {
    QS_TRY(take_scratch(s, total, &big));
    dev = (char*)big.p;
  }
  QS_TRY(ensure_pinned(s, total + 16));
  char* host = (char*)s->pinned;
  if (!ops.empty()) memcpy(host, ops.data(), sizeof(BOp) * ops.size());
  if (!mats.empty()) memcpy(host + ob, mats.data(), sizeof(QC) * mats.size());
  if (!dgm.empty()) memcpy(host + ob + mb, dgm.data(), sizeof(QC) * dgm.size());
  if (!rpm.empty()) memcpy(host + ob + mb + db, rpm.data(), sizeof(QP) * rpm.size());
  cudaError_t e = total ? cudaMemcpyAsync(dev, host, total, cudaMemcpyHostToDevice, s->stream) : cudaSuccess;
  const BOp* d_ops = (const BOp*)dev;
  const QC* d_mats = (const QC*)(dev + ob);
  const QC* d_dgm = (const QC*)(dev + ob + mb);
  const QP* d_rpm = (const QP*)(dev + ob + mb + db);
  int rc = e == cudaSuccess ? QS_OK : cuda_fail(e, "adjoint op tables");
  static bool attr = false;
  if (rc == QS_OK && !attr) {
    e = cudaFuncSetAttribute(k_adj_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    if (e != cudaSuccess) rc = cuda_fail(e, "adjoint pass attribute");
    attr = true;
  }
  for (size_t p = 0; rc == QS_OK && p < passes.size(); ++p) {
    AdjPassArgs a;
    a.ps = passes[p];
    a.ops = d_ops;
    a.mats = d_mats;
    a.dgm = d_dgm;
    a.rpm = d_rpm;
    a.part = part;
    a.slot_base = slot_bases[p];
    const uint32_t TS = 1u << a.ps.m;
    const size_t smem = 2 * sizeof(longlong2) * TS + sizeof(uint64_t) * ((size_t)1 << a.ps.nhigh) +
                        sizeof(double) * ((size_t)a.ps.nslots * (BT_THREADS / 32) + 8);
    const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(3, (220 * 1024) / (smem + 1024)));
    const uint64_t grid = std::min<uint64_t>(1ull << a.ps.nout, (uint64_t)std::min(ADJ_GRID_STRIDE, 152 * per_sm));
    {
      KTimer kt(s, QS_K_ADJOINT, a.ps.m, a.ps.op_end - a.ps.op_begin, 0, 0, 2.0 * (double)(1ull << n), 0.0);
      k_adj_pass<<<(unsigned)grid, BT_THREADS, smem, s->stream>>>(reinterpret_cast<longlong2*>(s->amps),
                                                                  reinterpret_cast<longlong2*>(lam), a);
    }
    rc = launch_check("adjoint pass");
  }
  return rc;
}

static bool g_adj_fused = true;

extern "C" int qs_set_adjoint_fused(int on) {
  g_adj_fused = on != 0;
  return QS_OK;
}

static int gen_of(const qs_gate& g) {
  switch (g.type) {
    case QS_RX: return GEN_X;
    case QS_RY: return GEN_Y;
    case QS_RZ: return GEN_Z;
    case QS_P: case QS_CR: return GEN_P;
    default: return GEN_NONE;
  }
}

// Launch lambda = (H/S) psi for the whole Pauli sum (several launches if it is long).
static int apply_hamiltonian(qs_state* s, const double2* psi, double2* lam, const qs_pauli* terms, size_t nterms,
                             double S, bool fx) {
  std::vector<HRun> runs;
  std::vector<uint64_t> xms;
  std::vector<HGroup> groups;
  std::vector<HTerm> hterms;
  h_plan(terms, nterms, S, &runs, &xms, &groups, &hterms);
  std::unique_ptr<HArgs> h(new (std::nothrow) HArgs);
  if (!h) return fail(QS_ERR_OOM, "host allocation failed");
  h->N = 1ull << s->n;
  const int grid = (int)std::min<uint64_t>((h->N + 255) / 256, 152 * 16);
  size_t ri = 0, gi = 0;
  h->accumulate = 0;
  do {
    h->nruns = h->ngroups = 0;
    int nx = 0, nt = 0;
    while (ri < runs.size() && nx + runs[ri].end - runs[ri].begin <= HMAX) {
      HRun& r = h->runs[h->nruns++] = runs[ri];
      r.begin = nx;
      for (int k = runs[ri].begin; k < runs[ri].end; ++k) h->xms[nx++] = xms[k];
      r.end = nx;
      ++ri;
    }
    while (gi < groups.size() && nt + groups[gi].end - groups[gi].begin <= HMAX && h->ngroups < HMAX) {
      HGroup& g = h->groups[h->ngroups++] = groups[gi];
      g.begin = nt;
      for (int k = groups[gi].begin; k < groups[gi].end; ++k) h->terms[nt++] = hterms[k];
      g.end = nt;
      ++gi;
    }
    if (gi < groups.size() && nt == 0) return fail(QS_ERR_UNSUPPORTED, "more than %d terms share one X mask", HMAX);
    {
      KTimer kt(s, QS_K_ADJOINT, 0, nx + nt, 0, 0, (double)h->N * (1 + nx + h->ngroups), 0.0);
      if (fx) k_apply_h<true><<<grid, 256, 0, s->stream>>>(psi, lam, *h);
      else k_apply_h<false><<<grid, 256, 0, s->stream>>>(psi, lam, *h);
    }
    QS_TRY(launch_check("apply_h"));
    h->accumulate = 1;
  } while (ri < runs.size() || gi < groups.size());
  return QS_OK;
}

}  // namespace qs

using namespace qs;

extern "C" int qs_adjoint_grad(qs_state* s, const qs_gate* gates, size_t ng, const double* params, size_t np,
                               const qs_pauli* terms, size_t nterms, double* energy, double* grad) {
  clear_error();
  QS_TRY(check_state(s));
  if (s->prec == 64) return fail(QS_ERR_UNSUPPORTED, "adjoint gradients need a complex128 state");
  if (!energy || (np && !grad) || (nterms && !terms)) return fail(QS_ERR_INVALID_ARG, "NULL argument");
  QS_TRY(validate_gates(gates, ng, s->n, params));
  const uint64_t full = s->n >= 64 ? ~0ull : ((1ull << s->n) - 1);
  double csum = 0.0;
  for (size_t k = 0; k < nterms; ++k) {
    if ((terms[k].xmask | terms[k].zmask) & ~full) return fail(QS_ERR_INVALID_ARG, "term %zu exceeds n", k);
    csum += fabs(terms[k].coef);
  }
  size_t nslots = 0;
  for (size_t k = 0; k < ng; ++k) {
    if (gates[k].param_idx < 0) continue;
    if ((size_t)gates[k].param_idx >= np) return fail(QS_ERR_INVALID_ARG, "gate %zu reads params[%d] >= np", k,
                                                      gates[k].param_idx);
    if (gen_of(gates[k]) == GEN_NONE)
      return fail(QS_ERR_UNSUPPORTED, "gate %zu: gradients are defined for RX, RY, RZ, P and CR parameters", k);
    ++nslots;
  }
  const int n = s->n;
  const uint64_t N = 1ull << n;
  const size_t bytes = N * sizeof(double2);
  // lambda lives next to the state for the duration of the call
  const int nblocks = 608;
  ScratchBuf buf;
  QS_TRY(take_scratch(s, bytes + sizeof(double) * (nslots + 1) * (nblocks + 1), &buf));
  double2* lam = (double2*)buf.p;
  double* part = (double*)(lam + N);
  double* sums = part + (size_t)nblocks * (nslots + 1);
  int rc = QS_OK;
  cudaError_t e = cudaSuccess;
  // forward: psi = U_G ... U_1 |0>, fused
  const double S = csum > 0 ? exp2(ceil(log2(csum))) : 1.0;
  qs_plan* plan = nullptr;
  bool fixed = false, held = false;  // held: the amplitudes are Q60 integers
  if ((rc = qs_set_zero(s)) == QS_OK && (rc = qs_plan_create(n, gates, ng, QS_PLAN_GREEDY, 5, &plan)) == QS_OK &&
      (rc = choose_fixed(s, &fixed)) == QS_OK) {
    const bool keep = fixed && g_adj_fused;
    rc = qs_apply_plan(s, gates, ng, params, plan, fixed, keep ? &held : nullptr);
    if (rc == QS_OK && keep && !held) rc = launch_q60_hold(s, &held);
  }
  if (plan) qs_plan_free(plan);
  if (rc == QS_OK) rc = apply_hamiltonian(s, s->amps, lam, terms, nterms, S, held);
  if (rc == QS_OK) {
    KTimer kt(s, QS_K_ADJOINT, 0, 0, 0, 0, 2.0 * N, 2.0 * N);
    double* dot = part + (size_t)nslots * nblocks;
    if (held) k_dot_re<true><<<nblocks, 256, 0, s->stream>>>(s->amps, lam, N, dot);
    else k_dot_re<false><<<nblocks, 256, 0, s->stream>>>(s->amps, lam, N, dot);
    rc = launch_check("dot");
  }
  // backward
  std::vector<int> slot_param;
  size_t slot = 0;
  const bool fused = held;
  if (rc == QS_OK && fused) {
    e = cudaMemsetAsync(part, 0, sizeof(double) * nblocks * nslots, s->stream);
    rc = e == cudaSuccess ? backward_fused(s, lam, gates, ng, params, part, slot_param) : cuda_fail(e, "memset");
  }
  for (size_t kk = fused ? 0 : ng; rc == QS_OK && kk-- > 0;) {
    const qs_gate& g = gates[kk];
    qs_gate inv = g;
    inv.dagger = !g.dagger;
    int t;
    uint64_t cm;
    Mat2 m;
    if ((rc = gate_qubits(inv, n, &t, &cm)) != QS_OK) break;
    if ((rc = gate_matrix(inv, params, &m)) != QS_OK) break;
    Op1 op = classify(t, cm, m);
    AdjArgs a;
    for (int i = 0; i < 4; ++i) {
      a.m[i] = make_double2(m.m[i].re, m.m[i].im);
      a.q[i] = qc_make(m.m[i].re, m.m[i].im);
    }
    a.cmask = cm;
    a.t = t;
    a.cls = op.cls;
    a.code0 = op.code0;
    a.code1 = op.code1;
    a.gen = g.param_idx >= 0 ? gen_of(g) : GEN_NONE;
    a.gsign = g.dagger ? -1.0 : 1.0;
    a.slot = (int)slot;
    if (a.gen == GEN_NONE && op.cls == OP_IDENTITY) continue;
    uint64_t fx = cm | (1ull << t);
    a.nfix = 0;
    for (int b = 0; b < 64; ++b)
      if ((fx >> b) & 1) a.fix[a.nfix++] = b;
    a.items = (int64_t)1 << (n - a.nfix);
    {
      KTimer kt(s, QS_K_ADJOINT, 1, 1, 1ull << t, cm, 4.0 * a.items, a.gen != GEN_NONE ? 8.0 * a.items : 0.0);
      if (fixed) k_adj_step<true><<<nblocks, 256, 0, s->stream>>>(s->amps, lam, a, part);
      else k_adj_step<false><<<nblocks, 256, 0, s->stream>>>(s->amps, lam, a, part);
    }
    rc = launch_check("adjoint step");
    if (a.gen != GEN_NONE) {
      slot_param.push_back(g.param_idx);
      ++slot;
    }
  }
  std::vector<double> host(nslots + 1);
  if (rc == QS_OK) {
    KTimer kt(s, QS_K_ADJOINT, 0, (int)nslots + 1, 0, 0, 0.0, 0.0);
    k_slot_sums<<<(unsigned)(nslots + 1), 256, 0, s->stream>>>(part, nblocks, sums);
    rc = launch_check("slot sums");
  }
  if (rc == QS_OK) {
    e = cudaMemcpyAsync(host.data(), sums, sizeof(double) * (nslots + 1), cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) rc = cuda_fail(e, "adjoint readback");
  }
  if (held) {  // the state is complex128 again, also after an error
    const int rc2 = launch_q60_release(s, &held);
    if (rc == QS_OK) rc = rc2;
  }
  if (rc != QS_OK) {
    s->bound = 0;
    return rc;
  }
  *energy = host[nslots] * S;
  for (size_t j = 0; j < np; ++j) grad[j] = 0.0;
  for (size_t j = 0; j < nslots; ++j) grad[slot_param[j]] += host[j] * S;
  // the state now holds U_1^dag ... U_G^dag psi_G = |0> up to rounding
  return QS_OK;
}
