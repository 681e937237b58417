// Excitations of one sample from tables in shared memory: the lists of
// occupied and virtual orbitals, the single excitations of each spin with
// their signs, and the index pairs of the double excitations.  Shared by the
// kernels that enumerate connected determinants, one CTA per sample or part
// of one, so that an excitation costs a few shared-memory loads instead of
// its own unranking from the occupation bits.
#pragma once

#include "common.cuh"

namespace anqs {

constexpr int MAXS = 256;  // singles of one spin: at most 16 x 16
constexpr int MAXP = 512;  // pairs of a list: at most C(32, 2) = 496 (a spin without electrons)

// Per-sample tables in shared memory.  A single (i, a) of spin s has index
// r_i * n_virt + r_a in the order of the occupied and virtual lists.
struct Exc {
  uint64_t x;
  uint32_t str[2];
  int ok;
  uint8_t occ[2][32], vir[2][32];
  uint8_t sgn[2][MAXS];   // parity of the electrons strictly between the two spin-orbitals
  uint8_t si[2][MAXS], sa[2][MAXS];
  uint32_t rank[2][MAXS]; // alpha: rank of the new string times nb_p[n]; beta: rank of the new string
  uint32_t g[2][MAXS];    // alpha: (a n + i) n^2, beta: a n + i
  uint16_t po[2][MAXP], pv[2][MAXP];  // pairs r1 | r2 << 8, lexicographic
  uint32_t own[2];        // rank(alpha) * nb_p[n], rank(beta)
};

// q = v / d for v d <= 2^32 by multiplication with ceil(2^32 / d): the product's
// excess over v / d is v e / (2^32 d) with e < d, below 1 / d.  The largest here:
// pairs of pairs, v < 120^2, d <= 496; singles of both spins, v < 2^16, d <= 256;
// excitations and row variants, v < 2^17, d <= 32.
struct FastDiv {
  uint32_t d, m;
};
__host__ __device__ inline FastDiv fast_div(uint32_t d) {
  return FastDiv{d, d > 1 ? uint32_t((0xffffffffull + d) / d) : 0u};
}
__device__ __forceinline__ uint32_t fdiv(const FastDiv& f, uint32_t v) { return f.d > 1 ? __umulhi(v, f.m) : v; }

// pair lists of both spins (they depend on the electron counts only)
__device__ __forceinline__ void build_pairs(const HamView& hv, Exc& E) {
  for (int s = 0; s < 2; ++s) {
    const int ne = s ? hv.nb : hv.na, nv = hv.n - ne;
    for (int t = 0; t < 2; ++t) {
      const int m = t ? nv : ne;
      uint16_t* o = t ? E.pv[s] : E.po[s];
      for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = e / m, j = e % m;
        if (i < j) o[i * (2 * m - i - 1) / 2 + j - i - 1] = uint16_t(i | j << 8);
      }
    }
  }
}

// tables of sample x; begins and ends with the CTA synchronised
template <bool RANK>
__device__ __forceinline__ void build_exc(const HamView& hv, const SectorView& sv, uint64_t x, Exc& E) {
  const int n = hv.n;
  const uint32_t oa = even_bits(x), ob = even_bits(x >> 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    E.x = x;
    E.str[0] = oa;
    E.str[1] = ob;
    E.ok = __popc(oa) == hv.na && __popc(ob) == hv.nb && (n == 32 || (x >> (2 * n)) == 0);
  }
  if (threadIdx.x < 64) {
    const int s = threadIdx.x >> 5, p = threadIdx.x & 31;
    if (p < n) {
      const uint32_t o = s ? ob : oa, below = o & ((1u << p) - 1u);
      const int k = __popc(below);
      if ((o >> p) & 1u) E.occ[s][k] = uint8_t(p);
      else E.vir[s][p - k] = uint8_t(p);
    }
  }
  __syncthreads();
  if (!E.ok) return;
  for (int s = 0; s < 2; ++s) {
    const int ne = s ? hv.nb : hv.na, nv = n - ne;
    for (int e = threadIdx.x; e < ne * nv; e += blockDim.x) {
      const int i = E.occ[s][e / nv], a = E.vir[s][e % nv];
      const int lo = 2 * min(i, a) + s, hi = 2 * max(i, a) + s;
      E.sgn[s][e] = uint8_t(__popcll(x & ((1ull << hi) - 1ull) & ~((2ull << lo) - 1ull)) & 1);
      E.si[s][e] = uint8_t(i);
      E.sa[s][e] = uint8_t(a);
      E.g[s][e] = uint32_t(a * n + i) * (s ? 1u : uint32_t(n * n));
      if constexpr (RANK) {
        const uint32_t t = E.str[s] ^ (1u << i) ^ (1u << a);
        E.rank[s][e] = s ? __ldg(sv.rkb + (1u << n) + t) : __ldg(sv.rka + (1u << n) + t) * sv.nb_p[n];
      }
    }
  }
  if constexpr (RANK) {
    if (threadIdx.x == 0) E.own[0] = __ldg(sv.rka + (1u << n) + oa) * sv.nb_p[n];
    if (threadIdx.x == 32) E.own[1] = __ldg(sv.rkb + (1u << n) + ob);
  }
  __syncthreads();
}

// parity of an opposite-spin double I -> A (alpha), J -> B (beta) as the
// product of the two singles: the beta move changes the occupation of J and
// B, which lie between I and A when lo <= orbital < hi
__device__ __forceinline__ int sign_ab(const Exc& E, uint32_t ea, uint32_t eb, int i, int a, int j, int b) {
  const int lo = min(i, a), hi = max(i, a);
  return E.sgn[0][ea] ^ E.sgn[1][eb] ^ int(j >= lo && j < hi) ^ int(b >= lo && b < hi);
}

// parity of a same-spin double I<J -> A<B as I -> A, then J -> B
__device__ __forceinline__ int sign_ss(const Exc& E, int s, uint32_t po, uint32_t pv, uint32_t nvirt, int i, int j, int a,
                                       int b) {
  const int lo = min(j, b), hi = max(j, b);
  return E.sgn[s][(po & 255u) * nvirt + (pv & 255u)] ^ E.sgn[s][(po >> 8) * nvirt + (pv >> 8)] ^
         int(i > lo && i < hi) ^ int(a > lo && a < hi);
}

// v with its sign flipped if odd: on the integer pipe (the FP64 pipe takes two
// lanes per clock and SM on this GPU, and a conditional negation is an FP64
// instruction)
__device__ __forceinline__ double flip_sign(double v, int odd) {
  return __hiloint2double(__double2hiint(v) ^ (odd << 31), __double2loint(v));
}

// two-electron integral (pq|rs)
__device__ __forceinline__ double Gint(const HamView& hv, int p, int q, int r, int s) {
  const int n = hv.n;
  return __ldg(hv.g + ((size_t(p) * n + q) * n + r) * n + s);
}

// h_ai + sum_{J occ} ([AI|JJ] - [AJ|JI]) of the single I -> A of spin s
__device__ __forceinline__ double single_value(const HamView& hv, const Exc& E, int s, int i, int a) {
  double v = __ldg(hv.h + a * hv.n + i);
  for (int t = 0; t < 2; ++t) {
    const int ne = t ? hv.nb : hv.na;
    for (int m = 0; m < ne; ++m) {
      const int jj = E.occ[t][m];
      v += Gint(hv, a, i, jj, jj);
      if (t == s) v -= Gint(hv, a, jj, jj, i);
    }
  }
  return v;
}

}  // namespace anqs
