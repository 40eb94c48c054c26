// Host-side harness for the rotation groups with three real products a complex
// product (compiled by the test suite with g++; the same inline functions the kernels
// use).  Each call applies the group to one component and writes the complex
// coefficients it used (c, d as exact integers) and the reflection flags.
#include "q60pair.cuh"

extern "C" {
static void wide(const qs::QW* g, long long* out) {  // c, d in units of 2^-64
  const long long c = ((long long)g[0].h << 32) + g[0].l, dc = ((long long)g[1].h << 32) + g[1].l;
  out[0] = c;
  out[1] = c + dc;
}
int gc_triple(const double* ra, const double* rb, const double* rc, long long* x, long long* c) {
  qs::QW G[12];
  int flags = 0;
  qs::q60_triple_gauss_coef(ra, rb, rc, G, &flags);
  for (int k = 0; k < 4; ++k) wide(G + 3 * k, c + 2 * k);
  int64_t v[8];
  for (int k = 0; k < 8; ++k) v[k] = (__builtin_popcount(k & flags) & 1) ? -x[k] : x[k];
  qs::q60_triple_gauss(v, G);
  for (int k = 0; k < 8; ++k) x[k] = v[k];
  return flags;
}
int gc_quad(const double* ra, const double* rb, const double* rc, const double* rd, long long* x, long long* c) {
  qs::QW G[24];
  int flags = 0;
  qs::q60_quad4_gauss_coef(ra, rb, rc, rd, G, &flags);
  for (int k = 0; k < 8; ++k) wide(G + 3 * k, c + 2 * k);
  int64_t v[16];
  for (int k = 0; k < 16; ++k) v[k] = (__builtin_popcount(k & flags) & 1) ? -x[k] : x[k];
  qs::q60_quad4_gauss(v, G, G + 12);
  for (int k = 0; k < 16; ++k) x[k] = v[k];
  return flags;
}
int gc_pair(const double* ra, const double* rb, long long* x, long long* c) {
  qs::QP g[2];
  int flags = 0;
  qs::q60_pair_gauss_coef(ra, rb, g, &flags);
  for (int k = 0; k < 2; ++k) {  // units of 2^-60
    const long long cc = (long long)g[k].c.h * (1ll << 30) + g[k].c.l2 / 2;
    c[2 * k] = cc;
    c[2 * k + 1] = cc + (long long)g[k].d.h * (1ll << 30) + g[k].d.l;
  }
  int64_t v[4];
  for (int k = 0; k < 4; ++k) v[k] = (__builtin_popcount(k & flags) & 1) ? -x[k] : x[k];
  qs::q60_pair_gauss(v[0], v[1], v[2], v[3], g);
  for (int k = 0; k < 4; ++k) x[k] = v[k];
  return flags;
}
}
