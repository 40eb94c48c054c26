// Tile-pass kernel.  A pass has a qubit set Q (m qubits, always containing the
// contiguous low run 0..L-1).  For each assignment r of the n-m qubits outside Q
// (a "tile"), the 2^m amplitudes x = deposit(r, ~Q) | deposit(j, Q) are loaded
// into shared memory (runs of 2^L contiguous amplitudes), every op of the pass is
// applied there in program order, and the tile is written back once.
//   - one-qubit ops on a tile qubit: pairs (j, j | 2^b) with the in-tile controls set;
//   - controls outside the tile are constant within a tile: the op is skipped for
//     tiles where one of them is 0;
//   - a diagonal op whose target lies outside the tile is a scalar for the tile.
// Gate matrices travel in the kernel parameters (constant bank).
// Two arithmetic engines share the structure: FP64 (tile of double2) and Q60
// fixed point (tile of int64 pairs, converted once on load and once on store).
#include <algorithm>
#include <type_traits>

#include "q60pair.cuh"
#include "tile.h"

namespace qs {

// Shared-memory swizzle of the tile: element j (16 or 8 bytes) lives at
// j ^ sw(j), where sw folds tile bits 3, 4, 5 into bits 0..2 with the vectors 7,
// 3, 5 (a linear map, so the physical index of a sum of disjoint bit sets is the
// XOR of theirs).  An op on tile bits B enumerates its pairs, quads or octets with
// consecutive threads on the lowest tile bits outside B; without the swizzle a
// quarter-warp hits one bank group as soon as B contains bits 0..2 (up to 8-way
// conflicts).  With these vectors every op on at most three tile bits has its
// lanes on at least four distinct bank groups (the best a 3-bit swizzle of bits
// 3..5 allows; 18 of the 299 such bit sets keep a 2-way conflict).
__device__ __forceinline__ uint32_t tsw_bits(uint32_t j) { return (0x3958f8u >> (3u * ((j >> 3) & 7u))) & 7u; }
__device__ __forceinline__ uint32_t tsw(uint32_t j) { return j ^ tsw_bits(j); }
// In a loop over i = threadIdx.x + k * THREADS (THREADS >= 256) whose element index
// j inserts zero bits into i, bits 3..7 of j come from the low bits of i, i.e. from
// threadIdx.x alone: the swizzle is one XOR with a per-thread constant.
// Elements of 8 bytes (complex64) have 16 to a row of banks: their swizzle folds bits
// 4..7 into bits 0..3 with the vectors 5, 10, 3, 8, so that the groups of four bits
// that runs of rotations are cut into ({0,3,6,9}, {1,4,7,10}, {2,5,8,11}), any three
// or all of the low bits and most pairs keep the 16 lanes of a half-warp apart (with
// the map above every one of those groups had a two-way conflict).
template <int BYTES>
__device__ __forceinline__ uint32_t tsw_bits_of(uint32_t j) {
  if (BYTES == 8) return (uint32_t)(0x41EB72D8C963FA50ull >> (4u * ((j >> 4) & 15u))) & 15u;
  return tsw_bits(j);
}
template <int BYTES>
__device__ __forceinline__ uint32_t tsw_of(uint32_t j) {
  return j ^ tsw_bits_of<BYTES>(j);
}

// Insert zero bits at the set positions of `fixed` (ascending), then OR `set`.
__device__ __forceinline__ uint32_t tile_expand(uint32_t i, uint32_t fixed, uint32_t set) {
  while (fixed) {
    int f = __ffs(fixed) - 1;
    fixed &= fixed - 1;
    i = ((i >> f) << (f + 1)) | (i & ((1u << f) - 1));
  }
  return i | set;
}

// The sign mask of table t in the tile at `base`: amplitude j takes the sign
// (-1)^popc(j & S), S = XOR over the terms (q, t) with x_q = 1 of bit t (two terms
// on the same tile bit cancel when both of their outside qubits are set).
__device__ __forceinline__ uint32_t table_sign_mask(const TileArgs& g, int t, uint64_t base) {
  if (t >= TILE_MAX_SIGNED_TABLES) return 0;
  const TileSigns& sg = g.signs[t];
  uint32_t S = 0;
  for (int i = 0; i < sg.n; ++i)
    if ((base >> sg.q[i]) & 1ull) S ^= 1u << sg.t[i];
  return S;
}

// ---- FP64 engine -------------------------------------------------------------------
// a * T (Q60), T = c + i d from a phase table entry {c.h, c.l, d.h, d.l} (16 bytes),
// negated when neg: three products (nine wide multiply-adds; the multiply-add pipe
// bounds the pass), the limbs of d - c, -(c + d) and of the amplitude's sum as limb
// sums (|low limb| < 2^31; middle accumulator at most 5.5 in units of 2^60).
__device__ __forceinline__ longlong2 table_mul(const int4 e, longlong2 a, bool neg) {
  const int32_t m = neg ? -1 : 0;
  const QL c{(e.x ^ m) - m, (e.y ^ m) - m}, d{(e.z ^ m) - m, (e.w ^ m) - m};
  const QL ar = q60_split(a.x), ai = q60_split(a.y);
  QAcc re = qacc_new();
  qacc_add(re, c, ql_add(ar, ai));
  QAcc im = re;
  qacc_add(re, QL{-c.h - d.h, -c.l - d.l}, ai);
  qacc_add(im, ql_sub(d, c), ar);
  return make_longlong2(qacc_round(re), qacc_round(im));
}

struct EngF64 {
  using T = double2;  // shared-memory element
  using G = double2;  // global element
  static constexpr int kMinBlocks = 3;  // CTAs per SM the register budget must allow (256 threads; 64 KiB tiles)
  static __device__ __forceinline__ double neg(double x) {
    return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
  }
  static __device__ __forceinline__ T load(const double2& a) { return a; }
  static __device__ __forceinline__ double2 store(const T& a) { return a; }
  static __device__ __forceinline__ T unit(T a, int code) {
    switch (code) {
      case U_ONE: return a;
      case U_I: return make_double2(neg(a.y), a.x);
      case U_MINUS_ONE: return make_double2(neg(a.x), neg(a.y));
      default: return make_double2(a.y, neg(a.x));
    }
  }
  static __device__ __forceinline__ T mul(T a, int code, const TileOp& op, int e) {
    if (code != U_GENERAL) return unit(a, code);
    const double2 u = op.m[e];
    return make_double2(fma(u.x, a.x, -u.y * a.y), fma(u.x, a.y, u.y * a.x));
  }
  static __device__ __forceinline__ void real2(const TileOp& op, T a0, T a1, T& b0, T& b1) {
    b0 = make_double2(fma(op.m[0].x, a0.x, op.m[1].x * a1.x), fma(op.m[0].x, a0.y, op.m[1].x * a1.y));
    b1 = make_double2(fma(op.m[2].x, a0.x, op.m[3].x * a1.x), fma(op.m[2].x, a0.y, op.m[3].x * a1.y));
  }
  static __device__ __forceinline__ void general2(const TileOp& op, T a0, T a1, T& b0, T& b1) {
    const double2 u0 = op.m[0], u1 = op.m[1], u2 = op.m[2], u3 = op.m[3];
    b0.x = fma(u0.x, a0.x, fma(-u0.y, a0.y, fma(u1.x, a1.x, -u1.y * a1.y)));
    b0.y = fma(u0.x, a0.y, fma(u0.y, a0.x, fma(u1.x, a1.y, u1.y * a1.x)));
    b1.x = fma(u2.x, a0.x, fma(-u2.y, a0.y, fma(u3.x, a1.x, -u3.y * a1.y)));
    b1.y = fma(u2.x, a0.y, fma(u2.y, a0.x, fma(u3.x, a1.y, u3.y * a1.x)));
  }
};

// ---- Q60 fixed-point engine ----------------------------------------------------------
struct EngQ60 {
  using T = longlong2;
  using G = double2;
  static constexpr int kMinBlocks = 3;  // 64 KiB tiles: three per SM; registers must not cut that
  static __device__ __forceinline__ T load(const double2& a) {
    return make_longlong2(q60_from_double_nb(a.x), q60_from_double_nb(a.y));
  }
  static __device__ __forceinline__ double2 store(const T& a) {
    return make_double2(q60_to_double_nb(a.x), q60_to_double_nb(a.y));
  }
  static __device__ __forceinline__ T unit(T a, int code) {
    switch (code) {
      case U_ONE: return a;
      case U_I: return make_longlong2(-a.y, a.x);
      case U_MINUS_ONE: return make_longlong2(-a.x, -a.y);
      default: return make_longlong2(a.y, -a.x);
    }
  }
  static __device__ __forceinline__ T mul(T a, int code, const TileOp& op, int e) {
    if (code != U_GENERAL) return unit(a, code);
    const QC& u = op.q[e];
    int64_t re, im;
    q60_gauss_mul(u, q60_split(a.x), q60_split(a.y), q60_split(a.x + a.y), &re, &im);
    return make_longlong2(re, im);
  }
  // x0 + i x1 of each component times c + i s (a reflection flips x1 first)
  static __device__ __forceinline__ void real2(const TileOp& op, T a0, T a1, T& b0, T& b1) {
    if (op.code1) a1 = make_longlong2(-a1.x, -a1.y);
    const QC& u = op.q[0];
    int64_t x0, x1, y0, y1;
    q60_gauss_mul(u, q60_split(a0.x), q60_split(a1.x), q60_split(a0.x + a1.x), &x0, &x1);
    q60_gauss_mul(u, q60_split(a0.y), q60_split(a1.y), q60_split(a0.y + a1.y), &y0, &y1);
    b0 = make_longlong2(x0, y0);
    b1 = make_longlong2(x1, y1);
  }
  static __device__ __forceinline__ void general2(const TileOp& op, T a0, T a1, T& b0, T& b1) {
    const QL r0 = q60_split(a0.x), i0 = q60_split(a0.y), r1 = q60_split(a1.x), i1 = q60_split(a1.y);
    // Gauss form: three limb products per complex product
    const QL s0 = q60_split(a0.x + a0.y), s1 = q60_split(a1.x + a1.y);
    int64_t re, im;
    q60_gauss_row(op.q[0], op.q[1], r0, i0, s0, r1, i1, s1, &re, &im);
    b0 = make_longlong2(re, im);
    q60_gauss_row(op.q[2], op.q[3], r0, i0, s0, r1, i1, s1, &re, &im);
    b1 = make_longlong2(re, im);
  }
};

// Two FP32 operations in one instruction (Blackwell's packed FP32): a complex64
// amplitude is the pair.  The same roundings as fmaf and a product on each half.
using F2 = unsigned long long;
__device__ __forceinline__ F2 f2_pack(float x, float y) {
  F2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ float2 f2_unpack(F2 a) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(a));
  return v;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  F2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// u * v for complex u, v: fma(u.x, v, (-u.y, u.y) (v.y, v.x)) in both halves
__device__ __forceinline__ F2 f2_cmul(float2 u, F2 v) {
  const float2 w = f2_unpack(v);
  return f2_fma(f2_pack(u.x, u.x), v, f2_mul(f2_pack(-u.y, u.y), f2_pack(w.y, w.x)));
}

// A table entry negated where `odd` is: sign terms make an entry's sign the parity of
// j & S.  Callers take that parity once per group of amplitudes and skip the signs of
// a tile without any (n = 26 brickwork of 16 layers 15.81 -> 15.34 ms).
__device__ __forceinline__ float2 entry_sign(float2 e, uint32_t odd) {
  const uint32_t m = odd << 31;
  return make_float2(__uint_as_float(__float_as_uint(e.x) ^ m), __uint_as_float(__float_as_uint(e.y) ^ m));
}

// ---- FP32 engine (complex64 states) -------------------------------------------------
// The op's matrix arrives rounded to float by the host (no conversion on the FP64 pipe).
struct EngF32 {
  using T = float2;
  using G = float2;
  // 32 KiB tiles, four per SM: 64 registers, of which the groups of 16 amplitudes with
  // eight table entries in flight spill 88 bytes.
  static constexpr int kMinBlocks = 4;
  static __device__ __forceinline__ T load(const float2& a) { return a; }
  static __device__ __forceinline__ float2 store(const T& a) { return a; }
  static __device__ __forceinline__ float2 u(const TileOp& op, int e) { return op.f[e]; }
  static __device__ __forceinline__ T unit(T a, int code) {
    switch (code) {
      case U_ONE: return a;
      case U_I: return make_float2(-a.y, a.x);
      case U_MINUS_ONE: return make_float2(-a.x, -a.y);
      default: return make_float2(a.y, -a.x);
    }
  }
  static __device__ __forceinline__ T mul(T a, int code, const TileOp& op, int e) {
    if (code != U_GENERAL) return unit(a, code);
    const float2 w = u(op, e);
    return make_float2(fmaf(w.x, a.x, -w.y * a.y), fmaf(w.x, a.y, w.y * a.x));
  }
  static __device__ __forceinline__ void real2(const TileOp& op, T a0, T a1, T& b0, T& b1) {
    const float m0 = op.f[0].x, m1 = op.f[1].x, m2 = op.f[2].x, m3 = op.f[3].x;
    b0 = make_float2(fmaf(m0, a0.x, m1 * a1.x), fmaf(m0, a0.y, m1 * a1.y));
    b1 = make_float2(fmaf(m2, a0.x, m3 * a1.x), fmaf(m2, a0.y, m3 * a1.y));
  }
  static __device__ __forceinline__ void general2(const TileOp& op, T a0, T a1, T& b0, T& b1) {
    const float2 u0 = u(op, 0), u1 = u(op, 1), u2 = u(op, 2), u3 = u(op, 3);
    b0.x = fmaf(u0.x, a0.x, fmaf(-u0.y, a0.y, fmaf(u1.x, a1.x, -u1.y * a1.y)));
    b0.y = fmaf(u0.x, a0.y, fmaf(u0.y, a0.x, fmaf(u1.x, a1.y, u1.y * a1.x)));
    b1.x = fmaf(u2.x, a0.x, fmaf(-u2.y, a0.y, fmaf(u3.x, a1.x, -u3.y * a1.y)));
    b1.y = fmaf(u2.x, a0.y, fmaf(u2.y, a0.x, fmaf(u3.x, a1.y, u3.y * a1.x)));
  }
};

// All pairs (j, j | tb) of one op in the tile, the op class fixed at compile time;
// unrolled twice so that a thread has independent pairs in flight (four times: the
// kernel outgrows the instruction cache, n = 26 random circuit 26.4 -> 26.7 ms).
template <class E, int KIND, int THREADS>
__device__ __forceinline__ void pair_loop(typename E::T* tile, uint32_t cnt, uint32_t fixed, uint32_t lcm, uint32_t tb,
                                          const TileOp& op) {
  using T = typename E::T;
  constexpr int B = sizeof(T);
  const uint32_t tbp = tsw_of<B>(tb);
  const uint32_t csw = tsw_bits_of<B>(lcm ? tile_expand(threadIdx.x, fixed, lcm) : threadIdx.x + (threadIdx.x & ~(tb - 1)));
#pragma unroll 2
  for (uint32_t i = threadIdx.x; i < cnt; i += THREADS) {
    // without in-tile controls the insertion of one zero bit is a mask and an add
    const uint32_t j0 = (lcm ? tile_expand(i, fixed, lcm) : i + (i & ~(tb - 1))) ^ csw, j1 = j0 ^ tbp;
    const T a0 = tile[j0], a1 = tile[j1];
    T b0, b1;
    if (KIND == TOP_DIAG) {
      b0 = E::mul(a0, op.code0, op, 0);
      b1 = E::mul(a1, op.code1, op, 3);
    } else if (KIND == TOP_ANTI) {
      b0 = E::mul(a1, op.code0, op, 1);
      b1 = E::mul(a0, op.code1, op, 2);
    } else if (KIND == TOP_REAL) {
      E::real2(op, a0, a1, b0, b1);
    } else {
      E::general2(op, a0, a1, b0, b1);
    }
    tile[j0] = b0;
    tile[j1] = b1;
  }
}

// Two real rotations on tile bits a and b on the quads (j, j|a, j|b, j|a|b), as
// two complex products per quad and component (q60pair.cuh): 36 wide
// multiply-adds per quad where the 4x4 matrix takes 96.  With a phase table
// (tab != nullptr, the table op just before the pair): every amplitude of the
// quad is first multiplied by its table entry, which saves the table op's own
// shared-memory round trip, index arithmetic and barrier.
template <int THREADS>
__device__ __forceinline__ void quad_real(longlong2* tile, uint32_t TS, uint32_t ta, uint32_t tbb, const QP* m0,
                                          int flags, const int4* tab, uint32_t S) {
  const uint32_t lo = min(ta, tbb), hi = max(ta, tbb);
  const uint32_t pa = tsw(ta), pb = tsw(tbb);
  uint32_t csw;
  {
    uint32_t j = threadIdx.x + (threadIdx.x & ~(lo - 1));
    csw = tsw_bits(j + (j & ~(hi - 1)));
  }
  const uint32_t cnt = TS >> 2;
#pragma unroll 2
  for (uint32_t i = threadIdx.x; i < cnt; i += THREADS) {
    uint32_t j = i + (i & ~(lo - 1));  // insert a zero bit at lo, then at hi
    j = j + (j & ~(hi - 1));
    const uint32_t jj[4] = {j, j | ta, j | tbb, j | ta | tbb};
    const uint32_t pj = j ^ csw;
    const uint32_t pp[4] = {pj, pj ^ pa, pj ^ pb, pj ^ pa ^ pb};
    longlong2 v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      v[c] = tile[pp[c]];
      if (tab) v[c] = table_mul(__ldg(tab + jj[c]), v[c], __popc(jj[c] & S) & 1);
    }
    if (flags) {  // reflections: the sign flip of their bit-1 half first
#pragma unroll
      for (int c = 1; c < 4; ++c)
        if (__popc(c & flags) & 1) v[c] = make_longlong2(-v[c].x, -v[c].y);
    }
    int64_t r[4], im[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      r[c] = v[c].x;
      im[c] = v[c].y;
    }
    q60_pair_gauss(r[0], r[1], r[2], r[3], m0);
    q60_pair_gauss(im[0], im[1], im[2], im[3], m0);
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = make_longlong2(r[c], im[c]);
#pragma unroll
    for (int c = 0; c < 4; ++c) tile[pp[c]] = v[c];
  }
}

// Three real rotations on tile bits ta, tb, tc on the octets (index bit(ta) +
// 2 bit(tb) + 4 bit(tc)) as four complex products per octet and component
// (q60pair.cuh): 16 real products per octet and component where a pair and a
// single rotation take 24.  With a phase table, as in quad_real.
template <int THREADS>
__device__ __forceinline__ void octet_real(longlong2* tile, uint32_t TS, uint32_t ta, uint32_t tb, uint32_t tc,
                                           const QW* G, int flags, const int4* tab, uint32_t S) {
  const uint32_t p0 = min(ta, min(tb, tc)), p2 = max(ta, max(tb, tc));
  const uint32_t p1 = (ta | tb | tc) & ~(p0 | p2);
  const uint32_t pa = tsw(ta), pb = tsw(tb), pc = tsw(tc);
  uint32_t csw;
  {
    uint32_t j = threadIdx.x + (threadIdx.x & ~(p0 - 1));
    j = j + (j & ~(p1 - 1));
    csw = tsw_bits(j + (j & ~(p2 - 1)));
  }
  const uint32_t cnt = TS >> 3;
  for (uint32_t i = threadIdx.x; i < cnt; i += THREADS) {
    uint32_t j = i + (i & ~(p0 - 1));  // insert zero bits at p0 < p1 < p2
    j = j + (j & ~(p1 - 1));
    j = j + (j & ~(p2 - 1));
    uint32_t jj[8], pp[8];
    const uint32_t pj = j ^ csw;
    longlong2 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      jj[k] = j | ((k & 1) ? ta : 0u) | ((k & 2) ? tb : 0u) | ((k & 4) ? tc : 0u);
      pp[k] = pj ^ ((k & 1) ? pa : 0u) ^ ((k & 2) ? pb : 0u) ^ ((k & 4) ? pc : 0u);
      v[k] = tile[pp[k]];
      if (tab) v[k] = table_mul(__ldg(tab + jj[k]), v[k], __popc(jj[k] & S) & 1);
    }
    if (flags) {  // reflections: the sign flip of their bit-1 half first
#pragma unroll
      for (int k = 1; k < 8; ++k)
        if (__popc(k & flags) & 1) v[k] = make_longlong2(-v[k].x, -v[k].y);
    }
    int64_t r[8], im[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      r[k] = v[k].x;
      im[k] = v[k].y;
    }
    q60_triple_gauss(r, G);
    q60_triple_gauss(im, G);
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = make_longlong2(r[k], im[k]);
#pragma unroll
    for (int k = 0; k < 8; ++k) tile[pp[k]] = v[k];
  }
}

// Four real rotations on tile bits ta < ... (any order) on one component of 16
// amplitudes per work item: item t takes group t >> 1 and component t & 1, so the
// two lanes of a pair read the two halves of the same 16-byte amplitudes.
template <int THREADS>
__device__ __forceinline__ void quad4_real(longlong2* tile, uint32_t TS, uint32_t ta, uint32_t tb, uint32_t tc,
                                           uint32_t td, const QW* G0, const QW* G1, int flags) {
  const uint32_t all = ta | tb | tc | td;
  uint32_t p[4], rest = all;
#pragma unroll
  for (int e = 0; e < 4; ++e) {  // the four bits in ascending order
    p[e] = rest & (0u - rest);
    rest ^= p[e];
  }
  const uint32_t pa = tsw(ta), pb = tsw(tb), pc = tsw(tc), pd = tsw(td);
  const uint32_t grp0 = threadIdx.x >> 1;
  uint32_t csw;
  {
    uint32_t j = grp0;
#pragma unroll
    for (int e = 0; e < 4; ++e) j = j + (j & ~(p[e] - 1));
    csw = tsw_bits(j);
  }
  int64_t* comp = reinterpret_cast<int64_t*>(tile) + (threadIdx.x & 1);
  const uint32_t cnt = TS >> 4;
  for (uint32_t g = grp0; g < cnt; g += THREADS / 2) {
    uint32_t j = g;
#pragma unroll
    for (int e = 0; e < 4; ++e) j = j + (j & ~(p[e] - 1));  // insert zero bits at p[0] < ... < p[3]
    const uint32_t pj = j ^ csw;
    uint32_t pp[16];
    int64_t x[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      pp[k] = pj ^ ((k & 1) ? pa : 0u) ^ ((k & 2) ? pb : 0u) ^ ((k & 4) ? pc : 0u) ^ ((k & 8) ? pd : 0u);
      x[k] = comp[2 * pp[k]];
    }
    if (flags) {
#pragma unroll
      for (int k = 1; k < 16; ++k)
        if (__popc(k & flags) & 1) x[k] = -x[k];
    }
    q60_quad4_gauss(x, G0, G1);
#pragma unroll
    for (int k = 0; k < 16; ++k) comp[2 * pp[k]] = x[k];
  }
}

// The same two ops for the FP32 engine (complex64 states): a real 4x4 on quads with
// its 16 entries as floats in f[] of the op's two slots, optionally after a phase
// table of float2 entries (one per amplitude of the tile).
template <int THREADS>
__device__ __forceinline__ void quad_real_f32(float2* tile, uint32_t TS, uint32_t ta, uint32_t tbb, const float* m0,
                                              const float* m1, const float2* tab, uint32_t S) {
  const uint32_t lo = min(ta, tbb), hi = max(ta, tbb);
  const uint32_t pa = tsw_of<8>(ta), pb = tsw_of<8>(tbb);
  uint32_t csw;
  {
    uint32_t j = threadIdx.x + (threadIdx.x & ~(lo - 1));
    csw = tsw_bits_of<8>(j + (j & ~(hi - 1)));
  }
  const uint32_t cnt = TS >> 2;
#pragma unroll 2
  for (uint32_t i = threadIdx.x; i < cnt; i += THREADS) {
    uint32_t j = i + (i & ~(lo - 1));
    j = j + (j & ~(hi - 1));
    const uint32_t jj[4] = {j, j | ta, j | tbb, j | ta | tbb};
    const uint32_t pj = j ^ csw;
    const uint32_t pp[4] = {pj, pj ^ pa, pj ^ pb, pj ^ pa ^ pb};
    F2 v[4];
    F2* t2 = reinterpret_cast<F2*>(tile);
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = t2[pp[c]];
    if (tab) {
      float2 e[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) e[c] = __ldg(tab + jj[c]);
      if (S) {
        const uint32_t odd = __popc(j & S), oa = (S & ta) != 0, ob = (S & tbb) != 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) e[c] = entry_sign(e[c], odd ^ ((c & 1) ? oa : 0u) ^ ((c & 2) ? ob : 0u));
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = f2_cmul(e[c], v[c]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      F2 x = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int e = 4 * k + c;
        const float u = e < 8 ? m0[e] : m1[e - 8];
        x = f2_fma(f2_pack(u, u), v[c], x);
      }
      t2[pp[k]] = x;
    }
  }
}

// FP32 engine: four real rotations (row-major 2x2 each, r[4q..4q+3] for bits a, b,
// c, d) on groups of 16 amplitudes held in registers, one after another, after an
// optional phase table: one shared-memory round trip for up to five ops.
template <int THREADS>
__device__ __forceinline__ void quad4_f32(float2* tile, uint32_t TS, uint32_t ta, uint32_t tb, uint32_t tc,
                                          uint32_t td, const float* r, const float2* tab, uint32_t S) {
  const uint32_t all = ta | tb | tc | td;
  uint32_t p[4], rest = all;
#pragma unroll
  for (int e = 0; e < 4; ++e) {  // the four bits in ascending order
    p[e] = rest & (0u - rest);
    rest ^= p[e];
  }
  const uint32_t pa = tsw_of<8>(ta), pb = tsw_of<8>(tb), pc = tsw_of<8>(tc), pd = tsw_of<8>(td);
  uint32_t csw;
  {
    uint32_t j = threadIdx.x;
#pragma unroll
    for (int e = 0; e < 4; ++e) j = j + (j & ~(p[e] - 1));
    csw = tsw_bits_of<8>(j);
  }
  const uint32_t cnt = TS >> 4;
  for (uint32_t g = threadIdx.x; g < cnt; g += THREADS) {
    uint32_t j = g;
#pragma unroll
    for (int e = 0; e < 4; ++e) j = j + (j & ~(p[e] - 1));  // insert zero bits at p[0] < ... < p[3]
    const uint32_t pj = j ^ csw;
    auto slot = [&](int k) {
      return pj ^ ((k & 1) ? pa : 0u) ^ ((k & 2) ? pb : 0u) ^ ((k & 4) ? pc : 0u) ^ ((k & 8) ? pd : 0u);
    };
    F2 v[16];
    F2* t2 = reinterpret_cast<F2*>(tile);
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = t2[slot(k)];
    if (tab) {
      const uint32_t odd = __popc(j & S), oa = (S & ta) != 0, ob = (S & tb) != 0, oc = (S & tc) != 0,
                     od = (S & td) != 0;
#pragma unroll
      for (int h = 0; h < 16; h += 8) {  // eight entries in flight
        float2 e[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          e[k] = __ldg(tab + (j | ((k & 1) ? ta : 0u) | ((k & 2) ? tb : 0u) | ((k & 4) ? tc : 0u) | (h ? td : 0u)));
        if (S) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            e[k] = entry_sign(e[k], odd ^ ((k & 1) ? oa : 0u) ^ ((k & 2) ? ob : 0u) ^ ((k & 4) ? oc : 0u) ^ (h ? od : 0u));
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) v[h + k] = f2_cmul(e[k], v[h + k]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const F2 m00 = f2_pack(r[4 * q], r[4 * q]), m01 = f2_pack(r[4 * q + 1], r[4 * q + 1]),
               m10 = f2_pack(r[4 * q + 2], r[4 * q + 2]), m11 = f2_pack(r[4 * q + 3], r[4 * q + 3]);
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (!(k & (1 << q))) {
          const F2 x0 = v[k], x1 = v[k | (1 << q)];
          v[k] = f2_fma(m01, x1, f2_mul(m00, x0));
          v[k | (1 << q)] = f2_fma(m11, x1, f2_mul(m10, x0));
        }
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) t2[slot(k)] = v[k];
  }
}

// Loads a tile into shared memory with eight global loads in flight per thread
// before their shared-memory stores (thread t takes j = t, t + THREADS, ...; the
// swizzle tsq depends only on bits the stride keeps).
template <int THREADS, class T, class S, class F>
__device__ __forceinline__ void load_tile(T* tile, const S* src, uint64_t base, const uint64_t* offs, int L,
                                          uint32_t lowmask, uint32_t TS, uint32_t tsq, F conv) {
  constexpr uint32_t U = 8;
  uint32_t j = threadIdx.x;
  for (; j + (U - 1) * THREADS < TS; j += U * THREADS) {
    S v[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const uint32_t jj = j + u * THREADS;
      v[u] = src[base + offs[jj >> L] + (jj & lowmask)];
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) tile[(j + u * THREADS) ^ tsq] = conv(v[u]);
  }
  for (; j < TS; j += THREADS) tile[j ^ tsq] = conv(src[base + offs[j >> L] + (j & lowmask)]);
}

// The same load with a phase table applied on the way in (the pass's first op):
// element j is multiplied by tab[j], negated where popc(j & S) is odd; four loads
// in flight (the table entries take the other registers).
template <int THREADS, class S, class F>
__device__ __forceinline__ void load_tile_table(longlong2* tile, const S* src, uint64_t base, const uint64_t* offs,
                                                int L, uint32_t lowmask, uint32_t TS, uint32_t tsq, F conv,
                                                const int4* tab, uint32_t Sg) {
  constexpr uint32_t U = 4;
  uint32_t j = threadIdx.x;
  for (; j + (U - 1) * THREADS < TS; j += U * THREADS) {
    S v[U];
    int4 e[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const uint32_t jj = j + u * THREADS;
      v[u] = src[base + offs[jj >> L] + (jj & lowmask)];
      e[u] = __ldg(tab + jj);
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const uint32_t jj = j + u * THREADS;
      tile[jj ^ tsq] = table_mul(e[u], conv(v[u]), __popc(jj & Sg) & 1);
    }
  }
  for (; j < TS; j += THREADS)
    tile[j ^ tsq] = table_mul(__ldg(tab + j), conv(src[base + offs[j >> L] + (j & lowmask)]), __popc(j & Sg) & 1);
}

// Stores a tile the same way, eight shared-memory reads before their global stores.
template <int THREADS, class T, class D, class F>
__device__ __forceinline__ void store_tile(const T* tile, D* dst, uint64_t base, const uint64_t* offs, int L,
                                           uint32_t lowmask, uint32_t TS, uint32_t tsq, F conv) {
  constexpr uint32_t U = 8;
  uint32_t j = threadIdx.x;
  for (; j + (U - 1) * THREADS < TS; j += U * THREADS) {
    T v[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) v[u] = tile[(j + u * THREADS) ^ tsq];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const uint32_t jj = j + u * THREADS;
      dst[base + offs[jj >> L] + (jj & lowmask)] = conv(v[u]);
    }
  }
  for (; j < TS; j += THREADS) dst[base + offs[j >> L] + (j & lowmask)] = conv(tile[j ^ tsq]);
}

// The same store with a phase table applied on the way out (the pass's last op).
template <int THREADS, class D, class F>
__device__ __forceinline__ void store_tile_table(const longlong2* tile, D* dst, uint64_t base, const uint64_t* offs,
                                                 int L, uint32_t lowmask, uint32_t TS, uint32_t tsq, F conv,
                                                 const int4* tab, uint32_t Sg) {
  constexpr uint32_t U = 4;
  uint32_t j = threadIdx.x;
  for (; j + (U - 1) * THREADS < TS; j += U * THREADS) {
    longlong2 v[U];
    int4 e[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      v[u] = tile[(j + u * THREADS) ^ tsq];
      e[u] = __ldg(tab + j + u * THREADS);
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const uint32_t jj = j + u * THREADS;
      dst[base + offs[jj >> L] + (jj & lowmask)] = conv(table_mul(e[u], v[u], __popc(jj & Sg) & 1));
    }
  }
  for (; j < TS; j += THREADS)
    dst[base + offs[j >> L] + (j & lowmask)] = conv(table_mul(__ldg(tab + j), tile[j ^ tsq], __popc(j & Sg) & 1));
}

template <class E, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? E::kMinBlocks : 1) k_tile(typename E::G* __restrict__ a, const __grid_constant__ TileArgs g) {
  using T = typename E::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int m = g.m;
  const int L = m - g.nhigh;
  const uint32_t TS = 1u << m;
  const uint32_t H = 1u << g.nhigh;
  uint64_t* offs = reinterpret_cast<uint64_t*>(smem_raw);  // [H] offsets of the high tile bits
  T* tile = reinterpret_cast<T*>(smem_raw + ((H * sizeof(uint64_t) + 15) & ~(size_t)15));
  for (uint32_t h = threadIdx.x; h < H; h += THREADS) {
    uint64_t o = 0;
    for (int b = 0; b < g.nhigh; ++b) o |= (uint64_t)((h >> b) & 1u) << g.qhigh[b];
    offs[h] = o;
  }
  const uint32_t lowmask = (1u << L) - 1;
  const uint32_t tsq = tsw_bits_of<sizeof(T)>(threadIdx.x);  // swizzle of the sequential loops over j
  for (uint64_t r = blockIdx.x; r < g.ntiles; r += gridDim.x) {
    uint64_t base = 0;
    for (int b = 0; b < g.nout; ++b) base |= ((r >> b) & 1ull) << g.outpos[b];
    __syncthreads();  // offs ready / previous tile stored
    auto conv = [](const typename E::G& v) { return E::load(v); };
    if constexpr (std::is_same<E, EngQ60>::value) {
      const int lt = ((g.io >> 8) & 255) - 1;  // a phase table applied on load
      if (lt >= 0) {
        const int4* tab = reinterpret_cast<const int4*>(g.tables) + (size_t)lt * TS;
        const uint32_t Sg = table_sign_mask(g, lt, base);
        if (g.io & 1)
          load_tile_table<THREADS>(tile, reinterpret_cast<const longlong2*>(a), base, offs, L, lowmask, TS, tsq,
                                   [](const longlong2& v) { return v; }, tab, Sg);
        else
          load_tile_table<THREADS>(tile, a, base, offs, L, lowmask, TS, tsq, conv, tab, Sg);
      } else if (g.io & 1) {  // Q60 in memory as in the tile: asynchronous copies
        const longlong2* src = reinterpret_cast<const longlong2*>(a);
        for (uint32_t j = threadIdx.x; j < TS; j += THREADS)
          cp_async16(tile + (j ^ tsq), src + base + offs[j >> L] + (j & lowmask));
        cp_async_wait_all();
      } else {
        load_tile<THREADS>(tile, a, base, offs, L, lowmask, TS, tsq, conv);
      }
    } else {
      load_tile<THREADS>(tile, a, base, offs, L, lowmask, TS, tsq, conv);
    }
    __syncthreads();
    for (int k = 0; k < g.nops; ++k) {
      const TileOp& op = g.ops[k];
      if ((base & op.ext_cmask) != op.ext_cmask) continue;  // uniform across the CTA
      const uint32_t lcm = op.lcmask;
      if constexpr (std::is_same<E, EngF32>::value) {
        if (op.kind == TOP_DTABLE) {
          const float2* tf = reinterpret_cast<const float2*>(g.tables) + (size_t)lcm * TS;
          const uint32_t S = table_sign_mask(g, (int)lcm, base);
          const uint32_t odd = __popc(threadIdx.x & S);
#pragma unroll 8
          for (uint32_t j = threadIdx.x; j < TS; j += THREADS) {
            float2 u = __ldg(tf + j);
            if (S) u = entry_sign(u, odd ^ __popc((j - threadIdx.x) & S));
            F2* t2 = reinterpret_cast<F2*>(tile);
            t2[j ^ tsq] = f2_cmul(u, t2[j ^ tsq]);
          }
          __syncthreads();
          continue;
        }
        if (op.kind == TOP_REAL4) {
          const float2* tab =
              op.code1 >= 0 ? reinterpret_cast<const float2*>(g.tables) + (size_t)op.code1 * TS : nullptr;
          quad4_f32<THREADS>(tile, TS, 1u << op.tb, 1u << op.code0, 1u << ((op.lcmask >> 8) & 31),
                             1u << ((op.lcmask >> 16) & 31), reinterpret_cast<const float*>(op.q), tab,
                             op.code1 >= 0 ? table_sign_mask(g, op.code1, base) : 0u);
          __syncthreads();
          continue;
        }
        if (op.kind == TOP_REAL2) {
          const float2* tab =
              op.code1 >= 0 ? reinterpret_cast<const float2*>(g.tables) + (size_t)op.code1 * TS : nullptr;
          quad_real_f32<THREADS>(tile, TS, 1u << op.tb, 1u << op.code0, reinterpret_cast<const float*>(op.f),
                                 reinterpret_cast<const float*>(g.ops[k + 1].f), tab,
                                 op.code1 >= 0 ? table_sign_mask(g, op.code1, base) : 0u);
          ++k;  // the continuation slot
          __syncthreads();
          continue;
        }
      }
      if constexpr (std::is_same<E, EngQ60>::value) {
        if (op.kind == TOP_DTABLE) {
          // one table entry per amplitude, read through the read-only path (every
          // tile reads the same table: it stays in L2)
          const int4* tab = reinterpret_cast<const int4*>(g.tables) + (size_t)lcm * TS;
          const uint32_t S = table_sign_mask(g, (int)lcm, base);
#pragma unroll 8
          for (uint32_t j = threadIdx.x; j < TS; j += THREADS)
            tile[j ^ tsq] = table_mul(__ldg(tab + j), tile[j ^ tsq], __popc(j & S) & 1);
          __syncthreads();
          continue;
        }
        if (op.kind == TOP_REAL4) {
          // 24 coefficients: 12 in q[] of this slot and 12 in the next slot's
          quad4_real<THREADS>(tile, TS, 1u << op.tb, 1u << op.code0, 1u << ((op.lcmask >> 8) & 31),
                              1u << ((op.lcmask >> 16) & 31), reinterpret_cast<const QW*>(op.q),
                              reinterpret_cast<const QW*>(g.ops[k + 1].q), (int)(op.lcmask & 15));
          ++k;  // the continuation slot
          __syncthreads();
          continue;
        }
        if (op.kind == TOP_REAL3) {
          const int4* tab = op.code1 >= 0 ? reinterpret_cast<const int4*>(g.tables) + (size_t)op.code1 * TS : nullptr;
          const QW* G = reinterpret_cast<const QW*>(op.q);  // 12 coefficients
          if (tab)
            octet_real<THREADS>(tile, TS, 1u << op.tb, 1u << op.code0, 1u << (op.lcmask >> 8), G,
                                (int)(op.lcmask & 7), tab, table_sign_mask(g, op.code1, base));
          else
            octet_real<THREADS>(tile, TS, 1u << op.tb, 1u << op.code0, 1u << (op.lcmask >> 8), G,
                                (int)(op.lcmask & 7), nullptr, 0u);
          __syncthreads();
          continue;
        }
        if (op.kind == TOP_REAL2) {
          const int4* tab = op.code1 >= 0 ? reinterpret_cast<const int4*>(g.tables) + (size_t)op.code1 * TS : nullptr;
          if (tab)
            quad_real<THREADS>(tile, TS, 1u << op.tb, 1u << op.code0, reinterpret_cast<const QP*>(op.q),
                               (int)op.lcmask, tab, table_sign_mask(g, op.code1, base));
          else
            quad_real<THREADS>(tile, TS, 1u << op.tb, 1u << op.code0, reinterpret_cast<const QP*>(op.q),
                               (int)op.lcmask, nullptr, 0u);
          ++k;  // the continuation slot
          __syncthreads();
          continue;
        }
      }
      if (op.kind == TOP_SCALAR) {
        const bool one = (base >> op.tb) & 1ull;
        const int code = one ? op.code1 : op.code0;
        if (code == U_ONE) continue;
        const int e = one ? 3 : 0;
        const uint32_t cnt = TS >> __popc(lcm);
        for (uint32_t i = threadIdx.x; i < cnt; i += THREADS) {
          const uint32_t j = tsw_of<sizeof(T)>(tile_expand(i, lcm, lcm));
          tile[j] = E::mul(tile[j], code, op, e);
        }
      } else {
        const uint32_t tb = 1u << op.tb;
        const uint32_t fixed = lcm | tb;
        const uint32_t cnt = TS >> __popc(fixed);
        if (op.kind == TOP_PHASE1) {
          for (uint32_t i = threadIdx.x; i < cnt; i += THREADS) {
            const uint32_t j = tsw_of<sizeof(T)>(tile_expand(i, fixed, lcm) | tb);
            tile[j] = E::mul(tile[j], op.code1, op, 3);
          }
        } else if (op.kind == TOP_GENERAL) {
          pair_loop<E, TOP_GENERAL, THREADS>(tile, cnt, fixed, lcm, tb, op);
        } else if (op.kind == TOP_REAL) {
          pair_loop<E, TOP_REAL, THREADS>(tile, cnt, fixed, lcm, tb, op);
        } else if (op.kind == TOP_ANTI) {
          pair_loop<E, TOP_ANTI, THREADS>(tile, cnt, fixed, lcm, tb, op);
        } else {
          pair_loop<E, TOP_DIAG, THREADS>(tile, cnt, fixed, lcm, tb, op);
        }
      }
      __syncthreads();
    }
    if constexpr (std::is_same<E, EngQ60>::value) {
      const int st = ((g.io >> 16) & 255) - 1;  // a phase table applied on store
      if (st >= 0) {
        const int4* tab = reinterpret_cast<const int4*>(g.tables) + (size_t)st * TS;
        const uint32_t Sg = table_sign_mask(g, st, base);
        if (g.io & 2)
          store_tile_table<THREADS>(tile, reinterpret_cast<longlong2*>(a), base, offs, L, lowmask, TS, tsq,
                                    [](const longlong2& v) { return v; }, tab, Sg);
        else
          store_tile_table<THREADS>(tile, a, base, offs, L, lowmask, TS, tsq,
                                    [](const longlong2& v) { return E::store(v); }, tab, Sg);
        continue;
      }
      if (g.io & 2) {
        store_tile<THREADS>(tile, reinterpret_cast<longlong2*>(a), base, offs, L, lowmask, TS, tsq,
                            [](const longlong2& v) { return v; });
        continue;
      }
    }
    store_tile<THREADS>(tile, a, base, offs, L, lowmask, TS, tsq, [](const T& v) { return E::store(v); });
  }
}

// Phase tables from their factors: a CTA takes a run of entries of one table, forms
// the products over the tile's low six bits and over the rest once (at most 64 + 128
// products), and an entry is their product times its terms.  Bound by FP64 issue
// (six FP64 instructions a complex product): 25 tables of 4096 entries a few
// microseconds.
constexpr uint32_t TABLE_RUN = 1024;
__global__ void __launch_bounds__(256) k_phase_tables(const __grid_constant__ TableArgs g, void* out) {
  __shared__ double2 lo[64], hi[1 << (TILE_MAX_M - 6)];
  const uint32_t TS = 1u << g.m, run = min(TS, TABLE_RUN), per = TS / run;
  const int t = blockIdx.x / per;
  const uint32_t j0 = (blockIdx.x % per) * run;
  const double* d = g.w + g.off[t];
  const int lb = min(g.m, 6), hb = g.m - lb;
  auto mul = [](double2 x, double2 y) {
    return make_double2(fma(x.x, y.x, -x.y * y.y), fma(x.x, y.y, x.y * y.x));
  };
  auto prod = [&](uint32_t bits, int b0, int nb) {
    double2 v = make_double2(1.0, 0.0);
    for (int b = 0; b < nb; ++b) {
      const double* e = d + 4 * (b0 + b);
      const bool one = (bits >> b) & 1;
      v = mul(v, make_double2(one ? e[2] : e[0], one ? e[3] : e[1]));
    }
    return v;
  };
  if (threadIdx.x < (1u << lb)) lo[threadIdx.x] = prod(threadIdx.x, 0, lb);
  const uint32_t h = threadIdx.x - 64;  // the next threads: the high products
  if (threadIdx.x >= 64 && h < (1u << hb)) hi[h] = prod(h, lb, hb);
  __syncthreads();
  const double* sg = d + 4 * g.m;
  const double* tm = sg + g.ns[t];
  for (uint32_t j = j0 + threadIdx.x; j < j0 + run; j += 256) {
    double2 v = mul(lo[j & ((1u << lb) - 1)], hi[j >> lb]);
    uint32_t neg = 0;
    for (int k = 0; k < g.ns[t]; ++k) {
      const uint32_t mask = (uint32_t)sg[k];
      neg ^= (j & mask) == mask;
    }
    for (int k = 0; k < g.nt[t]; ++k) {
      const uint32_t code = (uint32_t)tm[5 * k], mask = code >> 5;
      const int e = (j >> (code & 31)) & 1 ? 3 : 1;
      if ((j & mask) == mask) v = mul(v, make_double2(tm[5 * k + e], tm[5 * k + e + 1]));
    }
    if (neg) v = make_double2(-v.x, -v.y);
    if (g.f32) {
      reinterpret_cast<float2*>(out)[(size_t)t * TS + j] = make_float2((float)v.x, (float)v.y);
    } else {
      const QL c = q60_split_coef(q60_from_double(v.x)), s = q60_split_coef(q60_from_double(v.y));
      reinterpret_cast<int4*>(out)[(size_t)t * TS + j] = make_int4(c.h, c.l, s.h, s.l);
    }
  }
}

int launch_tables(qs_state* s, const TableArgs& g, void* out) {
  const uint32_t TS = 1u << g.m;
  note_launch(1);
  k_phase_tables<<<g.ntab * (TS / std::min(TS, TABLE_RUN)), 256, 0, s->stream>>>(g, out);
  return launch_check("phase tables");
}

// In-place Q60 integer pairs -> complex128 (the same rounding as a tile pass's store).
__global__ void k_q60_release(double2* __restrict__ a, size_t N) {
  longlong2* v = reinterpret_cast<longlong2*>(a);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    const longlong2 x = v[i];
    a[i] = make_double2(q60_to_double_nb(x.x), q60_to_double_nb(x.y));
  }
}

// The other way, as a tile pass's load.
__global__ void k_q60_hold(double2* __restrict__ a, size_t N) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    const double2 v = a[i];
    reinterpret_cast<longlong2*>(a)[i] = make_longlong2(q60_from_double_nb(v.x), q60_from_double_nb(v.y));
  }
}

template <class E, int THREADS>
static int launch_engine_t(qs_state* s, const TileArgs& g, size_t smem, bool* queued) {
  static bool attr_set = false;
  static int sms = 0;
  if (!attr_set) {
    QS_CUDA(cudaFuncSetAttribute(k_tile<E, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    QS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s->device));
    attr_set = true;
  }
  int per_sm = 0;
  QS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tile<E, THREADS>, THREADS, smem));
  const uint64_t grid = std::min<uint64_t>(g.ntiles, (uint64_t)std::max(1, sms) * std::max(1, per_sm));
  k_tile<E, THREADS><<<(unsigned)grid, THREADS, smem, s->stream>>>(reinterpret_cast<typename E::G*>(s->amps), g);
  return launch_check("tile kernel", queued);
}

// 256 threads per CTA (measured at n=30, 12-qubit tiles: 512 threads with 2 CTAs
// per SM and 1024 with one are 2-6 % slower); a 13-qubit tile (one CTA per SM)
// runs 512 threads, and so does a pass of at most one tile of 11 qubits or more per
// SM, where a CTA has the SM to itself.
template <class E>
static int launch_engine(qs_state* s, const TileArgs& g, bool* queued) {
  const size_t H = (size_t)1 << g.nhigh;
  const size_t smem = ((H * sizeof(uint64_t) + 15) & ~(size_t)15) + (sizeof(typename E::T) << g.m);
  if (g.m >= 13 || (g.m >= 11 && g.ntiles <= 152)) return launch_engine_t<E, 512>(s, g, smem, queued);
  return launch_engine_t<E, 256>(s, g, smem, queued);
}

int launch_q60_release(qs_state* s, bool* held) {
  const size_t N = (size_t)1 << s->n;
  const int blocks = (int)std::min<size_t>((N + 255) / 256, 152 * 16);
  KTimer kt(s, QS_K_OTHER, 0, 0, 0, 0, (double)N, 0.0);
  k_q60_release<<<blocks, 256, 0, s->stream>>>(s->amps, N);
  bool queued = false;
  const int rc = launch_check("q60 release", &queued);
  if (queued) *held = false;
  return rc;
}

int launch_q60_hold(qs_state* s, bool* held) {
  const size_t N = (size_t)1 << s->n;
  KTimer kt(s, QS_K_OTHER, 0, 0, 0, 0, (double)N, 0.0);
  k_q60_hold<<<(int)std::min<size_t>((N + 255) / 256, 152 * 16), 256, 0, s->stream>>>(s->amps, N);
  bool queued = false;
  const int rc = launch_check("q60 hold", &queued);
  if (queued) *held = true;
  return rc;
}

int launch_tile(qs_state* s, const TileArgs& g, bool fixed, bool* queued) {
  if (s->prec == 64) return launch_engine<EngF32>(s, g, queued);
  return fixed ? launch_engine<EngQ60>(s, g, queued) : launch_engine<EngF64>(s, g, queued);
}

}  // namespace qs
