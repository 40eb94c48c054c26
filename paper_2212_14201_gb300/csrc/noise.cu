// Noisy simulation by Monte-Carlo trajectories (the paper's NoiseQVM, Section
// "Multi-simulation methods", noise simulation method): one-qubit Kraus channels
// attached to gate types, a rotation error on rotation angles, and a readout
// confusion matrix on sampled bits.
//
// Kraus sets as the paper prints them (row-major 2x2):
//   DAMPING       [[1,0],[0,sqrt(1-p)]], [[0,sqrt(p)],[0,0]]
//   DEPHASING     sqrt(1-p) I, sqrt(p) Z           (PHASEFLIP: the same set)
//   DECOHERENCE   Kdamp_i Kdeph_j, i, j = 1, 2 (order 11, 12, 21, 22), with
//                 p_damp = 1 - exp(-tg/T1), p_deph = (1 - exp(-(tg/T2 - tg/(2 T1)))) / 2
//   DEPOLARIZING  sqrt(1 - 3p/4) I, sqrt(p)/2 X, sqrt(p)/2 Y, sqrt(p)/2 Z
//   BITFLIP       sqrt(1-p) I, sqrt(p) X
//   BITPHASEFLIP  sqrt(1-p) I, sqrt(p) Y
//   PHASE_DAMPING [[1,0],[0,sqrt(1-p)]], [[0,0],[0,sqrt(p)]]
// A trajectory, gate by gate: a rotation's theta gets e (2u - 1) (one draw);
// the gate; then for each matching rule and each qubit the gate touches
// (ascending) one draw u picks the smallest j with u W < w_1 + ... + w_j, and
// psi <- K_j psi / sqrt(w_j).  Weights w_j = ||K_j psi||^2;
// for a set of scaled unitaries w_j is the squared scale (no pass), and the
// chosen Pauli joins the gate stream, so such stretches stay fusable.
// Every K_j above is real with a diagonal K_j^dag K_j: the weights need only the
// populations of the qubit, and a diagonal K_j (the usual no-decay operator) scales
// them.  So the joint populations of up to JOINT_MAX qubits that channels touch next
// are read in one pass, the draws of a whole gate layer are decided from that table
// on the host, and the chosen diagonal operators are applied together.
#include <math.h>

#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "fixed.h"
#include "internal.h"

namespace qs {

// ---- product of real diagonal factors on a few qubits ----------------------------------
// a_x *= f[key], key = the listed qubits' bits of x.  Moves the state once for all of
// them.  complex128: two FP64 products per amplitude (2^22 amplitudes: 17 us at GB300's
// FP64 rate, about what their bytes take from L2).  complex64: the factor as a pair of
// floats, two FP32 operations a component and one rounding of the exact product, as a
// double product rounded to float gives it but for ties (the FP64 pipe, conversions
// included, made a trajectory with one operator a time 1.25 times as long as FP32
// kernels do: n = 22, decoherence on every U3, 5.7 ms).
constexpr int JOINT_MAX = 11;
struct FloatPair {
  float hi, lo;
};
__host__ __device__ inline double scale_factor(double f, double2*) { return f; }
__host__ __device__ inline FloatPair scale_factor(double f, float2*) {
  const float hi = (float)f;
  return FloatPair{hi, (float)(f - (double)hi)};
}
template <class A>
using ScaleFactor = decltype(scale_factor(0.0, (A*)nullptr));
// CAP: most qubits of a launch.  One operator at a time has a small variant: the
// arguments of the large one are 16 KB to copy and launch with.
template <class A, int CAP>
struct ScaleArgs {
  uint64_t N;
  int nq;
  int q[CAP];
  ScaleFactor<A> f[1 << CAP];
};

__device__ __forceinline__ double2 scale_amp(double2 v, double f) { return make_double2(v.x * f, v.y * f); }
__device__ __forceinline__ float2 scale_amp(float2 v, FloatPair f) {
  return make_float2(fmaf(v.x, f.hi, v.x * f.lo), fmaf(v.y, f.hi, v.y * f.lo));
}

template <class A, int CAP>
__global__ void __launch_bounds__(256) k_scale(A* __restrict__ a, const __grid_constant__ ScaleArgs<A, CAP> g) {
  __shared__ ScaleFactor<A> f[1 << CAP];
  for (int i = threadIdx.x; i < (1 << g.nq); i += 256) f[i] = g.f[i];
  __syncthreads();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  auto factor = [&](uint64_t x) {
    uint32_t key = 0;
#pragma unroll
    for (int j = 0; j < CAP; ++j)
      if (j < g.nq) key |= (uint32_t)((x >> g.q[j]) & 1) << j;
    return f[key];
  };
  uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  for (; x + 3 * stride < g.N; x += 4 * stride) {  // four loads in flight
    A v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = a[x + k * stride];
#pragma unroll
    for (int k = 0; k < 4; ++k) a[x + k * stride] = scale_amp(v[k], factor(x + k * stride));
  }
  for (; x < g.N; x += stride) a[x] = scale_amp(a[x], factor(x));
}

// ---- readout error on sampled indices ----------------------------------------------
__global__ void k_readout(uint64_t* __restrict__ samples, uint64_t shots, int n, double f0, double f1,
                          uint64_t seed) {
  for (uint64_t s = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; s < shots; s += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t x = samples[s];
    for (int i = 0; i < n; ++i) {
      const int bit = (int)((x >> i) & 1);
      const double u = u01_of(splitmix64(seed, s * (uint64_t)n + (uint64_t)i));
      if (u >= (bit ? f1 : f0)) x ^= 1ull << i;
    }
    samples[s] = x;
  }
}

// ---- Kraus sets ---------------------------------------------------------------------
struct KrausSet {
  int m = 0;
  bool unital = true;  // every operator c_j U_j with U_j in {I, X, Y, Z}
  Mat2 K[4];
  int pauli[4];        // unital sets: 0 = I, 1 = X, 2 = Y, 3 = Z
  double w[4];         // unital sets: c_j^2
};

static Mat2 m2(double a, double b, double c, double d) {
  Mat2 r;
  r.m[0] = {a, 0};
  r.m[1] = {b, 0};
  r.m[2] = {c, 0};
  r.m[3] = {d, 0};
  return r;
}

static Mat2 m2mul(const Mat2& A, const Mat2& B) {
  Mat2 r;
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const C2 x = A.m[2 * i], y = B.m[j], u = A.m[2 * i + 1], v = B.m[2 + j];
      r.m[2 * i + j] = {x.re * y.re - x.im * y.im + u.re * v.re - u.im * v.im,
                        x.re * y.im + x.im * y.re + u.re * v.im + u.im * v.re};
    }
  return r;
}

static int kraus_set(const qs_noise_rule& r, KrausSet* ks) {
  const double p = r.p;
  if (r.model != QS_NOISE_DECOHERENCE && !(p >= 0.0 && p <= 1.0))
    return fail(QS_ERR_INVALID_ARG, "noise probability %g outside [0, 1]", p);
  const double s = sqrt(p), c = sqrt(1.0 - p);
  auto pauli_set = [&](int P, double scale) {
    ks->m = 2;
    ks->unital = true;
    ks->pauli[0] = 0;
    ks->w[0] = c * c;
    ks->pauli[1] = P;
    ks->w[1] = scale * scale;
    ks->K[0] = m2(c, 0, 0, c);
  };
  switch (r.model) {
    case QS_NOISE_DAMPING:
      ks->m = 2;
      ks->unital = false;
      ks->K[0] = m2(1, 0, 0, c);
      ks->K[1] = m2(0, s, 0, 0);
      return QS_OK;
    case QS_NOISE_PHASE_DAMPING:
      ks->m = 2;
      ks->unital = false;
      ks->K[0] = m2(1, 0, 0, c);
      ks->K[1] = m2(0, 0, 0, s);
      return QS_OK;
    case QS_NOISE_DEPHASING:
    case QS_NOISE_PHASEFLIP: pauli_set(3, s); return QS_OK;
    case QS_NOISE_BITFLIP: pauli_set(1, s); return QS_OK;
    case QS_NOISE_BITPHASEFLIP: pauli_set(2, s); return QS_OK;
    case QS_NOISE_DEPOLARIZING: {
      ks->m = 4;
      ks->unital = true;
      const double a = sqrt(1.0 - 0.75 * p), h = 0.5 * s;
      ks->w[0] = a * a;
      for (int j = 1; j < 4; ++j) ks->w[j] = h * h;
      for (int j = 0; j < 4; ++j) ks->pauli[j] = j;
      return QS_OK;
    }
    case QS_NOISE_DECOHERENCE: {
      if (!(r.t1 > 0.0) || !(r.t2 > 0.0) || !(r.tgate >= 0.0))
        return fail(QS_ERR_INVALID_ARG, "decoherence needs T1 > 0, T2 > 0, tgate >= 0");
      const double pa = 1.0 - exp(-r.tgate / r.t1);
      const double pd = 0.5 * (1.0 - exp(-(r.tgate / r.t2 - r.tgate / (2.0 * r.t1))));
      if (!(pd >= 0.0 && pd <= 1.0)) return fail(QS_ERR_INVALID_ARG, "decoherence: T2 > 2 T1 gives no valid dephasing");
      const Mat2 D[2] = {m2(1, 0, 0, sqrt(1.0 - pa)), m2(0, sqrt(pa), 0, 0)};
      const Mat2 P[2] = {m2(sqrt(1.0 - pd), 0, 0, sqrt(1.0 - pd)), m2(sqrt(pd), 0, 0, -sqrt(pd))};
      ks->m = 4;
      ks->unital = false;
      for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) ks->K[2 * i + j] = m2mul(D[i], P[j]);
      return QS_OK;
    }
    default: return fail(QS_ERR_INVALID_ARG, "unknown noise model %d", r.model);
  }
}

static bool is_rotation(int type) {
  return type == QS_RX || type == QS_RY || type == QS_RZ || type == QS_U3 || type == QS_P || type == QS_CR;
}

static bool two_qubit(int type) { return type == QS_CNOT || type == QS_CZ || type == QS_CR; }

// ---- the trajectory driver -----------------------------------------------------------
struct Trajectory {
  qs_state* s;
  bool fuse;
  uint64_t seed, k = 0;
  std::vector<qs_gate> pending;  // parameter-free records (angles resolved)

  double draw() { return u01_of(splitmix64(seed, k++)); }

  // Diagonal operators chosen but not yet applied (real factors, at most one entry a
  // qubit).  Every pending gate commutes with them: it is diagonal or its target is
  // another qubit, so they may be applied before it.
  struct Scale {
    int q;
    double f0, f1;
  };
  std::vector<Scale> scales;
  // Joint populations of `jq` in the state with every pending gate and factor
  // applied (entry bit i: qubit jq[i]); no pending non-diagonal gate has its target
  // among them, so gates on other qubits leave them as they are.
  std::vector<int> jq;
  std::vector<double> joint;

  int joint_bit(int q) const {
    for (size_t i = 0; i < jq.size(); ++i)
      if (jq[i] == q) return (int)i;
    return -1;
  }

  // Appends a gate; target: its target qubit, diagonal: whether it is diagonal.
  int push(const qs_gate& g, int target, bool diagonal) {
    if (!diagonal) {
      for (const Scale& c : scales)
        if (c.q == target) {
          QS_TRY(apply_scales());
          break;
        }
      if (joint_bit(target) >= 0) jq.clear();
    }
    pending.push_back(g);
    return QS_OK;
  }

  template <int CAP, class A>
  void launch_scales(A* a) {
    ScaleArgs<A, CAP> g;
    g.N = 1ull << s->n;
    g.nq = (int)scales.size();
    for (int j = 0; j < g.nq; ++j) g.q[j] = scales[j].q;
    // qubit by qubit, doubling the filled prefix: 2^12 products for eleven qubits (entry by
    // entry it is 11 x 2^11 with a choice in each, 27 us a launch on the host's core)
    double f[1 << CAP];
    f[0] = 1.0;
    for (int j = 0; j < g.nq; ++j)
      for (int k = 0, h = 1 << j; k < h; ++k) {
        f[k + h] = f[k] * scales[j].f1;
        f[k] *= scales[j].f0;
      }
    for (int k = 0; k < (1 << g.nq); ++k) g.f[k] = scale_factor(f[k], a);
    const int nblocks = (int)std::min<uint64_t>(152 * 8, (g.N + 255) / 256);
    k_scale<A, CAP><<<nblocks, 256, 0, s->stream>>>(a, g);
  }

  int apply_scales() {
    if (scales.empty()) return QS_OK;
    const double N = (double)(1ull << s->n);
    KTimer kt(s, QS_K_DIAG, 1, (int)scales.size(), 0, 0, N, 2.0 * N);
    with_amps(s, [&](auto* a) {
      if (scales.size() <= 2) launch_scales<2>(a);
      else launch_scales<JOINT_MAX>(a);
      return QS_OK;
    });
    scales.clear();
    return launch_check("scale");
  }

  // Joint populations of q and the other qubits in `ahead` (distinct, q first).  On large
  // states a read of one to three qubits takes longer than one of seven (k_marginal_tiny
  // and its few sums against k_marginal_rows: n = 22, 48 and 35 us), so it is read with
  // the highest other qubits, which are added up here.
  int read_joint(const std::vector<int>& ahead) {
    QS_TRY(apply_scales());
    QS_TRY(flush());
    jq = ahead;
    std::vector<int> read = ahead;
    uint64_t in = 0;
    for (int b : ahead) in |= 1ull << b;
    for (int b = s->n - 1; s->n >= 20 && read.size() < 7; --b)
      if (!((in >> b) & 1)) read.push_back(b);
    joint.resize((size_t)1 << read.size());
    const int rc = marginal_host(s, read.data(), (int)read.size(), joint.data(), false);
    if (rc != QS_OK) jq.clear();
    const size_t len = (size_t)1 << jq.size();
    for (size_t k = len; k < joint.size(); ++k) joint[k & (len - 1)] += joint[k];
    joint.resize(len);
    return rc;
  }

  int flush() {
    if (pending.empty()) return QS_OK;
    int rc = QS_OK;
    if (fuse && pending.size() > 1) {
      qs_plan* p = nullptr;
      rc = qs_plan_create(s->n, pending.data(), pending.size(), QS_PLAN_GREEDY, 5, &p);
      if (rc == QS_OK) rc = qs_apply(s, pending.data(), pending.size(), nullptr, p);
      if (p) qs_plan_free(p);
    } else {
      rc = apply_per_gate(s, pending.data(), pending.size(), nullptr);
    }
    pending.clear();
    return rc;
  }

  // ahead(): q and the qubits of the channels that follow, as far as one table serves them.
  template <class F>
  int channel(const KrausSet& ks, int q, F&& ahead) {
    double w[4] = {0, 0, 0, 0};
    if (ks.unital) {
      for (int j = 0; j < ks.m; ++j) w[j] = ks.w[j];
    } else {
      if (joint_bit(q) < 0) QS_TRY(read_joint(ahead()));
      const int b = joint_bit(q);
      // four sums per outcome: one would wait for every addition before the next
      double s0[4] = {0, 0, 0, 0}, s1[4] = {0, 0, 0, 0};
      const size_t h = (size_t)1 << b, half = joint.size() / 2;
      for (size_t k = 0; k < half; ++k) {
        const size_t j = k + (k & ~(h - 1));  // bit b clear
        s0[k & 3] += joint[j];
        s1[k & 3] += joint[j + h];
      }
      const double p[2] = {(s0[0] + s0[1]) + (s0[2] + s0[3]), (s1[0] + s1[1]) + (s1[2] + s1[3])};
      for (int j = 0; j < ks.m; ++j) {
        const Mat2& K = ks.K[j];
        w[j] = (K.m[0].re * K.m[0].re + K.m[2].re * K.m[2].re) * p[0] +
               (K.m[1].re * K.m[1].re + K.m[3].re * K.m[3].re) * p[1];
      }
    }
    double W = 0.0;
    for (int j = 0; j < ks.m; ++j) W += w[j];
    const double u = draw();
    int pick = ks.m - 1;
    double c = 0.0;
    for (int j = 0; j < ks.m; ++j) {
      c += w[j];
      if (u * W < c) {
        pick = j;
        break;
      }
    }
    if (!(w[pick] > 0.0)) return fail(QS_ERR_INVALID_ARG, "noise channel picked an operator of zero weight");
    if (ks.unital) {
      static const int codes[4] = {QS_I, QS_X, QS_Y, QS_Z};
      if (ks.pauli[pick] != 0) {
        qs_gate g{};
        g.type = codes[ks.pauli[pick]];
        g.q0 = q;
        g.q1 = -1;
        g.param_idx = -1;
        return push(g, q, ks.pauli[pick] == 3);
      }
      return QS_OK;
    }
    Mat2 M = ks.K[pick];
    const double sc = 1.0 / sqrt(w[pick]);
    for (int e = 0; e < 4; ++e) M.m[e] = {M.m[e].re * sc, M.m[e].im * sc};
    if (M.m[1].re == 0.0 && M.m[2].re == 0.0) {
      const double f0 = M.m[0].re, f1 = M.m[3].re;
      const int b = joint_bit(q);
      for (size_t k = 0; k < joint.size(); ++k) joint[k] *= (k >> b) & 1 ? f1 * f1 : f0 * f0;
      for (Scale& c : scales)
        if (c.q == q) {
          c.f0 *= f0;
          c.f1 *= f1;
          return QS_OK;
        }
      scales.push_back({q, f0, f1});
      return scales.size() == JOINT_MAX ? apply_scales() : QS_OK;
    }
    QS_TRY(apply_scales());
    QS_TRY(flush());
    jq.clear();
    // A renormalised Kraus operator is not unitary, but the state it produces is
    // normalised: the Q60 kernel applies it when every entry has |re| + |im| < 1.9
    // (its Gauss-form sums then stay below 2, the limb range), e.g. the usual
    // no-decay operator of amplitude damping; otherwise (the rare jump operators,
    // scaled by 1 / sqrt(p)) the FP64 kernel.
    bool fixed = false;
    QS_TRY(choose_fixed(s, &fixed));
    for (int e = 0; e < 4 && fixed; ++e)
      if (fabs(M.m[e].re) + fabs(M.m[e].im) >= 1.9) fixed = false;
    return launch_op1(s, classify(q, 0, M), fixed);
  }
};

}  // namespace qs

using namespace qs;

extern "C" int qs_run_noisy(qs_state* s, const qs_gate* gates, size_t ng, const double* params,
                            const qs_noise_rule* rules, size_t nrules, double rotation_error, uint64_t seed, int fuse,
                            uint64_t* ndraws) {
  clear_error();
  QS_TRY(check_state(s));
  QS_TRY(validate_gates(gates, ng, s->n, params));
  if (nrules && !rules) return fail(QS_ERR_INVALID_ARG, "rules is NULL");
  if (!(rotation_error >= 0.0)) return fail(QS_ERR_INVALID_ARG, "rotation_error must be >= 0");
  std::vector<KrausSet> sets(nrules);
  for (size_t r = 0; r < nrules; ++r) {
    QS_TRY(kraus_set(rules[r], &sets[r]));
    if (rules[r].gate_type < -1 || rules[r].gate_type > QS_CR)
      return fail(QS_ERR_INVALID_ARG, "rule %zu: gate type %d", r, rules[r].gate_type);
  }
  Trajectory tr;
  tr.s = s;
  tr.fuse = fuse != 0;
  tr.seed = seed;
  auto matches = [&](const qs_noise_rule& R, const qs_gate& g) {
    return (R.gate_type < 0 || R.gate_type == g.type) && (R.q0 < 0 || R.q0 == g.q0) &&
           (R.q1 < 0 || R.q1 == (two_qubit(g.type) ? g.q1 : -1));
  };
  // q, then the qubits that channels with weights touch in the next gates, until the
  // table is full or a gate changes the populations of one of them.  A qubit whose
  // populations change before its channel is left out: its entry would be of no use, and
  // that gate would end the table (a rotation with a channel on every qubit of a layer
  // then reads one qubit, not eleven, for each).
  constexpr size_t kAheadGates = 256;  // (looked at again at every table)
  const uint64_t all = (1ull << s->n) - 1;
  auto ahead = [&](size_t k, int q) {
    std::vector<int> list{q};
    uint64_t in = 1ull << q, moved = 0;
    for (size_t j = k; j < ng && j < k + kAheadGates && (in | moved) != all; ++j) {
      int t;
      uint64_t cm;
      if (gate_qubits(gates[j], s->n, &t, &cm) != QS_OK) break;
      if (j > k && !structurally_diagonal(gates[j].type)) {
        if ((in >> t) & 1) break;
        moved |= 1ull << t;
      }
      for (size_t r = 0; r < nrules; ++r) {
        if (sets[r].unital || !matches(rules[r], gates[j])) continue;
        for (uint64_t b = (cm | (1ull << t)) & ~(in | moved); b; b &= b - 1) {
          if (list.size() == JOINT_MAX) return list;
          list.push_back(__builtin_ctzll(b));
          in |= b & (0 - b);
        }
      }
    }
    return list;
  };
  int rc = QS_OK;
  for (size_t k = 0; k < ng && rc == QS_OK; ++k) {
    qs_gate g = gates[k];
    if (g.param_idx >= 0) {  // resolve the angle into the record
      g.p[0] = params[g.param_idx];
      g.param_idx = -1;
    }
    if (rotation_error > 0.0 && is_rotation(g.type)) g.p[0] += rotation_error * (2.0 * tr.draw() - 1.0);
    int t;
    uint64_t cm;
    if ((rc = gate_qubits(g, s->n, &t, &cm)) != QS_OK) break;
    if ((rc = tr.push(g, t, structurally_diagonal(g.type))) != QS_OK) break;
    for (size_t r = 0; r < nrules && rc == QS_OK; ++r) {
      if (!matches(rules[r], g)) continue;
      for (uint64_t b = cm | (1ull << t); b && rc == QS_OK; b &= b - 1) {
        const int q = __builtin_ctzll(b);
        rc = tr.channel(sets[r], q, [&] { return ahead(k, q); });
      }
    }
  }
  if (rc == QS_OK) rc = tr.apply_scales();
  if (rc == QS_OK) rc = tr.flush();
  if (ndraws) *ndraws = tr.k;
  if (rc == QS_OK) QS_CUDA(cudaStreamSynchronize(s->stream));
  return rc;
}

extern "C" int qs_readout_error(uint64_t* samples, size_t shots, int n, double f0, double f1, uint64_t seed,
                                int on_device, void* stream) {
  clear_error();
  if (shots && !samples) return fail(QS_ERR_INVALID_ARG, "samples is NULL");
  if (n < 1 || n > 64) return fail(QS_ERR_INVALID_ARG, "n=%d outside 1..64", n);
  if (!(f0 >= 0.0 && f0 <= 1.0 && f1 >= 0.0 && f1 <= 1.0)) return fail(QS_ERR_INVALID_ARG, "fidelities outside [0, 1]");
  if (!shots) return QS_OK;
  cudaStream_t st = (cudaStream_t)stream;
  uint64_t* d = samples;
  if (!on_device) QS_CUDA(dmalloc_async(&d, shots * sizeof(uint64_t), st));
  int rc = QS_OK;
  cudaError_t e = cudaSuccess;
  if (!on_device) e = cudaMemcpyAsync(d, samples, shots * sizeof(uint64_t), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
    const uint64_t grid = std::min<uint64_t>((shots + 255) / 256, (uint64_t)std::max(1, sms) * 8);
    note_launch(1);
    k_readout<<<(unsigned)grid, 256, 0, st>>>(d, shots, n, f0, f1, seed);
    rc = launch_check("readout kernel");
    if (rc == QS_OK && !on_device) e = cudaMemcpyAsync(samples, d, shots * sizeof(uint64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && rc == QS_OK) e = cudaStreamSynchronize(st);
  }
  if (!on_device) cudaFreeAsync(d, st);
  if (rc != QS_OK) return rc;
  if (e != cudaSuccess) return cuda_fail(e, "readout error");
  return QS_OK;
}
