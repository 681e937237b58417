// Prefix trees of the samples' connected determinants, for sectors without a
// prefix index (eloc_unique.cu covers the others).
//
// A connected determinant x' differs from its sample x in at most four slots,
// so the 33,508 determinants of a sample of the 52-qubit workload (26
// orbitals, 9 + 9 electrons) have 201,800 distinct prefixes, where evaluating
// every position after the first difference takes 731,500.  The tree is built
// level by level: whether a prefix can still be completed to at most a double
// excitation follows from how many electrons it has removed and added per spin
// and what the sample has beyond it, so each node yields its children without
// looking at any list, and the children of all nodes come out in node order:
// the determinants of a sample are contiguous and neighbours share prefixes
// (their keys and values come from the same cache lines).
//
// Levels 0..n-1 are evaluated by the network one level per launch (a node
// attends to the stored keys and values of its own prefixes); level n are the
// determinants.  Their amplitude is the sum of the terms up to the first
// differing slot plus the sum of the later ones, and E_loc comes straight from
// the pairs (x, x').
#include <algorithm>

#include "common.cuh"

namespace anqs {
namespace {

constexpr int BT = 256;       // threads of the level kernels
constexpr uint32_t NPB = 1024;  // nodes per CTA

// node counts sit next to each other and are read and written by successive
// kernels: always through L2
__device__ __forceinline__ uint64_t count_at(const uint64_t* cnt, int t) {
  return __ldcg(reinterpret_cast<const unsigned long long*>(cnt) + t);
}

__device__ __forceinline__ bool good_sample(const HamView& hv, uint64_t x) {
  return __popcll(x & 0x5555555555555555ull) == hv.na && __popcll(x & 0xAAAAAAAAAAAAAAAAull) == hv.nb &&
         (hv.n == 32 || (x >> (2 * hv.n)) == 0);
}

// outcomes (bits) of slot t after prefix q of sample x that lead to a
// determinant at most a double excitation away: per spin, r electrons removed
// and a added so far take max(r, a) moves, whose missing removals and
// additions must still find occupied and empty orbitals in the later slots
__device__ __forceinline__ unsigned child_mask(const HamView& hv, uint64_t x, uint64_t q, int t) {
  const uint64_t upto = t + 1 >= 32 ? ~0ull : (1ull << (2 * (t + 1))) - 1ull;
  const uint64_t E = 0x5555555555555555ull, xp = x & upto, rest = x & ~upto;
  const int left = hv.n - 1 - t;
  unsigned m = 0;
#pragma unroll
  for (unsigned v = 0; v < 4; ++v) {
    const uint64_t d = (q | (uint64_t(v) << (2 * t))) ^ xp;
    int moves = 0;
    bool ok = true;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const uint64_t S = E << s;
      const int r = __popcll(d & xp & S), a = __popcll(d & ~xp & S), k = r > a ? r : a;
      const int occ = __popcll(rest & S);
      ok = ok && k - r <= occ && k - a <= left - occ;
      moves += k;
    }
    if (ok && moves <= 2) m |= 1u << v;
  }
  return m;
}

// level 0: one root per sample of the group that lies in the sector (electron
// counts), in order
__global__ void __launch_bounds__(BT) root_kernel(HamView hv, const uint64_t* __restrict__ xs, Count n_x_,
                                                  uint64_t first, uint64_t group, uint64_t* __restrict__ x,
                                                  uint32_t* __restrict__ src, uint64_t* __restrict__ cnt) {
  ANQS_PDL_ENTRY();
  __shared__ uint32_t s_w[BT / 32], s_base;
  const uint64_t n_x = n_x_.get(), hi = first + group < n_x ? first + group : n_x;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_base = 0;
  __syncthreads();
  for (uint64_t l0 = first; l0 < hi; l0 += BT) {
    const uint64_t l = l0 + threadIdx.x;
    const bool ok = l < hi && good_sample(hv, xs[l]);
    const unsigned b = __ballot_sync(0xffffffffu, ok);
    if (lane == 0) s_w[wp] = __popc(b);
    __syncthreads();
    uint32_t at = s_base + __popc(b & ((1u << lane) - 1u)), total = 0;
    for (int q = 0; q < BT / 32; ++q) {
      if (q < wp) at += s_w[q];
      total += s_w[q];
    }
    if (ok) {
      x[at] = 0;
      src[at] = uint32_t(l);
    }
    __syncthreads();
    if (threadIdx.x == 0) s_base += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) cnt[0] = s_base;
}

// children of level t's nodes per CTA
__global__ void __launch_bounds__(BT) child_count_kernel(HamView hv, const uint64_t* __restrict__ xs, int t,
                                                         const uint64_t* __restrict__ x,
                                                         const uint32_t* __restrict__ src,
                                                         const uint64_t* __restrict__ cnt, uint32_t* __restrict__ bsum) {
  ANQS_PDL_ENTRY();
  __shared__ uint32_t s_sum;
  const uint64_t rows = count_at(cnt, t);
  if (uint64_t(blockIdx.x) * NPB >= rows) return;
  if (threadIdx.x == 0) s_sum = 0;
  __syncthreads();
  uint32_t c = 0;
  for (uint32_t i = threadIdx.x; i < NPB; i += BT) {
    const uint64_t r = uint64_t(blockIdx.x) * NPB + i;
    if (r < rows) c += __popc(child_mask(hv, xs[src[r]], x[r], t));
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum, c);
  __syncthreads();
  if (threadIdx.x == 0) bsum[blockIdx.x] = s_sum;
}

// the children in order: prefix, sample and parent of each; cnt[t + 1]
__global__ void __launch_bounds__(BT) child_emit_kernel(HamView hv, const uint64_t* __restrict__ xs, int t,
                                                        const uint64_t* __restrict__ x,
                                                        const uint32_t* __restrict__ src, uint64_t* __restrict__ cnt,
                                                        const uint32_t* __restrict__ bsum, uint64_t* __restrict__ xn,
                                                        uint32_t* __restrict__ srcn, uint32_t* __restrict__ parn) {
  ANQS_PDL_ENTRY();
  __shared__ uint32_t s_base, s_w[BT / 32];
  const uint64_t rows = count_at(cnt, t);
  const uint32_t blocks = uint32_t((rows + NPB - 1) / NPB);
  if (blockIdx.x == 0 && blocks == 0 && threadIdx.x == 0) cnt[t + 1] = 0;
  if (blockIdx.x >= blocks) return;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_base = 0;
  __syncthreads();
  uint32_t c = 0;
  for (uint32_t i = threadIdx.x; i < blockIdx.x; i += BT) c += __ldcg(bsum + i);
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) atomicAdd(&s_base, c);
  __syncthreads();
  uint32_t base = s_base;
  for (uint32_t i0 = 0; i0 < NPB; i0 += BT) {
    const uint64_t r = uint64_t(blockIdx.x) * NPB + i0 + threadIdx.x;
    uint64_t q = 0;
    uint32_t l = 0;
    unsigned m = 0;
    if (r < rows) {
      q = x[r];
      l = src[r];
      m = child_mask(hv, xs[l], q, t);
    }
    const uint32_t k = __popc(m);
    uint32_t inc = k;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) s_w[wp] = inc;
    __syncthreads();
    uint32_t at = base + inc - k, total = 0;
#pragma unroll
    for (int g = 0; g < BT / 32; ++g) {
      if (g < wp) at += s_w[g];
      total += s_w[g];
    }
    while (m) {
      const uint64_t v = uint64_t(__ffs(m)) - 1ull;
      m &= m - 1u;
      xn[at] = q | v << (2 * t);
      srcn[at] = l;
      parn[at++] = uint32_t(r);
    }
    base += total;
    __syncthreads();
  }
  if (blockIdx.x == blocks - 1 && threadIdx.x == 0) cnt[t + 1] = base;
}

// anc[i][u] of level p's nodes: the parent's table, then the parent (id node0 + par)
__global__ void anc_kernel(int p, const uint64_t* __restrict__ cnt, const uint32_t* __restrict__ par,
                           const uint32_t* __restrict__ from, uint64_t node0, uint32_t* __restrict__ anc) {
  ANQS_PDL_ENTRY();
  const uint64_t total = count_at(cnt, p) * TRIE_ANC;
  for (uint64_t k = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; k < total; k += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t i = k / TRIE_ANC;
    const int u = int(k % TRIE_ANC);
    if (u >= p) continue;
    const uint32_t r = par[i];
    anc[k] = u + 1 < p ? from[uint64_t(r) * TRIE_ANC + u] : uint32_t(node0 + r);
  }
}

// Amplitude of every determinant: the terms of its path up to its first slot
// that differs from the sample, plus the sum of the later ones; a sample's
// own (all terms in order) goes to own[l].
__global__ void amp_kernel(int n, const uint64_t* __restrict__ xs, const uint64_t* __restrict__ cnt,
                           const uint64_t* __restrict__ x, const uint32_t* __restrict__ src,
                           const uint32_t* __restrict__ par, const uint32_t* __restrict__ anc, uint64_t node0,
                           const float2* __restrict__ terms, float2* __restrict__ amp, float2* __restrict__ own) {
  ANQS_PDL_ENTRY();
  const uint64_t rows = count_at(cnt, n);
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < rows; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t xp = x[i], d = xp ^ xs[src[i]];
    const int j = d ? (__ffsll(static_cast<long long>(d)) - 1) >> 1 : n - 1;
    const uint32_t r = par[i];
    const uint32_t* a = anc + uint64_t(r) * TRIE_ANC;
    float la = 0.f, ph = 0.f, sl = 0.f, sp = 0.f;
    for (int p = 0; p < n; p += 8) {  // eight loads in flight
      float2 t[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        t[e] = make_float2(0.f, 0.f);
        if (p + e < n) {
          const uint64_t id = p + e + 1 < n ? uint64_t(a[p + e]) : node0 + r;
          t[e] = __ldcg(terms + id * 4 + ((xp >> (2 * (p + e))) & 3ull));
        }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (p + e <= j) {
          la += t[e].x;
          ph += t[e].y;
        } else if (p + e < n) {
          sl += t[e].x;
          sp += t[e].y;
        }
      }
    }
    const float2 v = j + 1 < n ? make_float2(la + sl, ph + sp) : make_float2(la, ph);
    amp[i] = v;
    if (!d) own[src[i]] = v;
  }
}

__device__ __forceinline__ int par_below(uint64_t x, int q) { return __popcll(x & ((1ull << q) - 1ull)) & 1; }

__device__ __forceinline__ double G(const HamView& hv, int p, int q, int r, int s) {
  const int n = hv.n;
  return __ldg(hv.g + ((size_t(p) * n + q) * n + r) * n + s);
}

// H_xx' of a connected pair (Slater-Condon, Jordan-Wigner sign)
__device__ double element(const HamView& hv, uint64_t x, uint64_t xp) {
  const uint64_t E = 0x5555555555555555ull;
  uint64_t hole = x & ~xp, part = xp & ~x;
  if (__popcll(hole) == 1) {  // single I -> A: h_ai + sum_{J occ} ([AI|JJ] - [AJ|JI])
    const int I = __ffsll(static_cast<long long>(hole)) - 1, A = __ffsll(static_cast<long long>(part)) - 1;
    const int s = I & 1, i = I >> 1, a = A >> 1, lo = min(I, A), hi = max(I, A);
    double v = __ldg(hv.h + a * hv.n + i);
    for (int t = 0; t < 2; ++t)
      for (uint64_t m = x & (E << t); m; m &= m - 1) {
        const int jj = (__ffsll(static_cast<long long>(m)) - 1) >> 1;
        v += G(hv, a, i, jj, jj);
        if (t == s) v -= G(hv, a, jj, jj, i);
      }
    return (__popcll(x & ((1ull << hi) - 1ull) & ~((2ull << lo) - 1ull)) & 1) ? -v : v;
  }
  // double: same spin I<J -> A<B, or the alpha move first
  int I, J, A, B;
  const bool mixed = __popcll(hole & E) == 1;
  if (mixed) {
    I = __ffsll(static_cast<long long>(hole & E)) - 1, J = __ffsll(static_cast<long long>(hole & ~E)) - 1;
    A = __ffsll(static_cast<long long>(part & E)) - 1, B = __ffsll(static_cast<long long>(part & ~E)) - 1;
  } else {
    I = __ffsll(static_cast<long long>(hole)) - 1, J = 63 - __clzll(static_cast<long long>(hole));
    A = __ffsll(static_cast<long long>(part)) - 1, B = 63 - __clzll(static_cast<long long>(part));
  }
  const int i = I >> 1, j = J >> 1, a = A >> 1, b = B >> 1;
  double v = G(hv, a, i, b, j);
  if (!mixed) v -= G(hv, a, j, b, i);
  // sign of <x'| a+_A a+_B a_J a_I |x>, operators applied right to left
  uint64_t y = x;
  int sg = par_below(y, I);
  y ^= 1ull << I;
  sg ^= par_below(y, J);
  y ^= 1ull << J;
  sg ^= par_below(y, B);
  y ^= 1ull << B;
  sg ^= par_below(y, A);
  return sg ? -v : v;
}

// part[l][q] = part q of sum_x' H_xx' psi(x') / psi(x) over sample l's
// determinants (and H_xx in part 0); NaN for samples outside the sector
constexpr int ET = 128;
__global__ void __launch_bounds__(ET) trie_eloc_kernel(HamView hv, const uint64_t* __restrict__ xs, Count n_x_,
                                                       uint64_t first, uint64_t group, int parts,
                                                       const uint64_t* __restrict__ x, const float2* __restrict__ amp,
                                                       const float2* __restrict__ own, double* __restrict__ part) {
  ANQS_PDL_ENTRY();
  __shared__ double red[2][ET / 32];
  __shared__ uint32_t s_before;
  const uint64_t n_x = n_x_.get(), hi = first + group < n_x ? first + group : n_x;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, n = hv.n;
  for (uint64_t it = blockIdx.x; first + it / parts < hi; it += gridDim.x) {
    const uint64_t l = first + it / parts;
    const int pt = int(it % parts);
    const uint64_t xl = xs[l];
    __syncthreads();
    if (threadIdx.x == 0) s_before = 0;
    __syncthreads();
    // samples of the group before l that have a tree: K + 1 determinants each
    uint32_t c = 0;
    for (uint64_t q = first + threadIdx.x; q < l; q += ET) c += good_sample(hv, xs[q]);
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0 && c) atomicAdd(&s_before, c);
    __syncthreads();
    double re = 0.0, im = 0.0;
    if (good_sample(hv, xl)) {
      const uint64_t m = uint64_t(hv.K) + 1, r0 = uint64_t(s_before) * m;
      const float2 o = __ldcg(own + l);
      for (uint64_t i = r0 + m * pt / parts + threadIdx.x; i < r0 + m * (pt + 1) / parts; i += ET) {
        const uint64_t xp = __ldcg(reinterpret_cast<const unsigned long long*>(x) + i);
        if (xp == xl) continue;
        const double h = element(hv, xl, xp);
        const float2 t = __ldcg(amp + i);
        const float r = expf(t.x - o.x);
        float s, co;
        sincosf(t.y - o.y, &s, &co);
        const double hr = h * double(r);
        re = fma(hr, double(co), re);
        im = fma(hr, double(s), im);
      }
      if (pt == 0) {  // <x|H|x> = E_nuc + sum_I h_ii + 1/2 sum_{I,J occ} ([II|JJ] - [IJ|JI])
        for (int t = threadIdx.x; t < 4 * n * n; t += ET) {
          const int I = t / (2 * n), J = t - I * 2 * n;
          if (!((xl >> I) & (xl >> J) & 1ull)) continue;
          const int i = I >> 1, j = J >> 1;
          re += 0.5 * G(hv, i, i, j, j);
          if ((I & 1) == (J & 1)) re -= 0.5 * G(hv, i, j, j, i);
          if (I == J) re += __ldg(hv.h + i * n + i);
        }
        if (threadIdx.x == 0) re += hv.e_nuc;
      }
    } else {
      re = __longlong_as_double(0x7ff8000000000000ll);
      im = hv.K ? re : 0.0;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
      red[0][wp] = re;
      red[1][wp] = im;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double sr = 0.0, si = 0.0;
#pragma unroll
      for (int q = 0; q < ET / 32; ++q) {
        sr += red[0][q];
        si += red[1][q];
      }
      part[(l * parts + pt) * 2] = sr;
      part[(l * parts + pt) * 2 + 1] = si;
    }
  }
}

constexpr int FT = 256;
__global__ void __launch_bounds__(FT) trie_finish_kernel(Count n_x_, int parts, const double* __restrict__ part,
                                                         double* ere, double* eim, const uint64_t* __restrict__ counts,
                                                         double* stats) {
  ANQS_PDL_ENTRY();
  const uint64_t n_x = n_x_.get();
  for (uint64_t l = threadIdx.x; l < n_x; l += FT) {
    double sr = 0.0, si = 0.0;
    for (int q = 0; q < parts; ++q) {
      sr += part[(l * parts + q) * 2];
      si += part[(l * parts + q) * 2 + 1];
    }
    ere[l] = sr;
    eim[l] = si;
  }
  if (!counts) return;
  __threadfence();
  __syncthreads();
  cta_energy_stats<FT>(ere, eim, counts, n_x, stats);
}

}  // namespace

// Most distinct prefixes of t = 0..n slots that one sample's connected
// determinants (and the sample) can have, over how many electrons the sample
// has there.  Once per Hamiltonian: a call asks for them several times.
void trie_level_nodes(const HamView& hv, uint64_t* nodes) {
  const int n = hv.n;
  for (int t = 0; t <= n; ++t) {
    // prefixes of one spin that take k moves, for a of ne electrons in the t slots: r removed and s added, k the
    // larger, and the missing k - r and k - s still possible in the later slots
    auto spin = [&](int a, int ne, uint64_t (&c)[3]) {
      const int occ = ne - a, vir = n - t - occ, e = t - a;
      const uint64_t A[3] = {1, uint64_t(a), uint64_t(a) * uint64_t(a > 0 ? a - 1 : 0) / 2};
      const uint64_t B[3] = {1, uint64_t(e), uint64_t(e) * uint64_t(e > 0 ? e - 1 : 0) / 2};
      for (int k = 0; k <= 2; ++k) {
        c[k] = 0;
        for (int r = 0; r <= k; ++r)
          for (int s = 0; s <= k; ++s)
            if (std::max(r, s) == k && k - r <= occ && k - s <= vir) c[k] += A[r] * B[s];
      }
    };
    uint64_t cb[ANQS_MAX_ORB + 1][3], best = 0;
    const int b0 = std::max(0, hv.nb - (n - t)), b1 = std::min(t, hv.nb);
    for (int b = b0; b <= b1; ++b) spin(b, hv.nb, cb[b]);
    for (int a = std::max(0, hv.na - (n - t)); a <= std::min(t, hv.na); ++a) {
      uint64_t ca[3];
      spin(a, hv.na, ca);
      for (int b = b0; b <= b1; ++b)
        best = std::max(best, ca[0] * (cb[b][0] + cb[b][1] + cb[b][2]) + ca[1] * (cb[b][0] + cb[b][1]) + ca[2] * cb[b][0]);
    }
    nodes[t] = best;
  }
}

void plan_trie(const anqs_ham* H, uint64_t n_x, uint64_t max_nodes, Arena& A, TrieWs& w) {
  const int n = H->v.n;
  w = TrieWs{};
  const uint64_t* per = H->tree_nodes;
  uint64_t inner = 0;
  for (int p = 0; p + 1 < n; ++p) inner += per[p];
  w.group = std::max<uint64_t>(1, inner ? max_nodes / inner : n_x);
  w.group = std::min(w.group, std::max<uint64_t>(1, (1ull << 31) / (uint64_t(H->v.K) + 1)));
  w.group = std::min(w.group, n_x);
  uint64_t most = 0;
  for (int p = 0; p <= n; ++p) {
    w.cap[p] = per[p] * w.group;
    w.node0[p] = p ? w.node0[p - 1] + w.cap[p - 1] : 0;
    most = std::max(most, w.cap[p]);
  }
  w.parts = int(std::max<uint64_t>(1, std::min<uint64_t>(32, H->v.K / 512)));
  w.cnt = A.take<uint64_t>(ANQS_MAX_ORB + 2);
  for (int b = 0; b < 2; ++b) {
    w.x[b] = A.take<uint64_t>(most);
    w.src[b] = A.take<uint32_t>(most);
    w.par[b] = A.take<uint32_t>(most);
    w.anc[b] = A.take<uint32_t>((n > 1 ? std::max(w.cap[n - 1], w.cap[n - 2]) : w.cap[n - 1]) * TRIE_ANC);
  }
  w.bsum = A.take<uint32_t>((most + NPB - 1) / NPB);
  w.amp = A.take<float2>(w.cap[n]);
  w.own = A.take<float2>(n_x);
  w.part = A.take<double>(n_x * uint64_t(w.parts) * 2);
}

int launch_trie_level(const anqs_ham* H, const uint64_t* x, Count n_x, uint64_t c, int p, const TrieWs& w,
                      TrieLevel& lv, cudaStream_t s) {
  const int b = p & 1, a = 1 - b;
  ProfScope ps(PROF_TC_SORT, s);
  if (p == 0) {
    ANQS_CUDA_LAUNCH("root_kernel", launch_k(root_kernel, dim3(1), dim3(BT), 0, s, H->v, x, n_x, c * w.group, w.group, w.x[0], w.src[0], w.cnt));
  } else {
    const unsigned blocks = unsigned((w.cap[p - 1] + NPB - 1) / NPB);
    ANQS_CUDA_LAUNCH("child_count_kernel", launch_k(child_count_kernel, dim3(blocks), dim3(BT), 0, s, H->v, x, p - 1, w.x[a], w.src[a], w.cnt, w.bsum));
    ANQS_CUDA_LAUNCH("child_emit_kernel", launch_k(child_emit_kernel, dim3(blocks), dim3(BT), 0, s, H->v, x, p - 1, w.x[a], w.src[a], w.cnt, w.bsum, w.x[b], w.src[b], w.par[b]));
    if (p < H->v.n) {
      const unsigned grid = unsigned(std::min<uint64_t>((w.cap[p] * TRIE_ANC + 255) / 256, 152 * 8));
      ANQS_CUDA_LAUNCH("anc_kernel", launch_k(anc_kernel, dim3(grid), dim3(256), 0, s, p, w.cnt, w.par[b], w.anc[a], w.node0[p - 1], w.anc[b]));
    }
  }
  lv.p = p;
  lv.x = w.x[b];
  lv.rows = Count{w.cap[p], w.cnt + p, 1};
  lv.anc = w.anc[b];
  lv.node0 = w.node0[p];
  return ANQS_OK;
}

int launch_trie_eloc(const anqs_ham* H, const uint64_t* x, Count n_x, uint64_t c, const TrieWs& w, const float2* terms,
                     cudaStream_t s) {
  const int n = H->v.n, b = n & 1, a = 1 - b;
  TrieLevel lv;
  ANQS_TRY(launch_trie_level(H, x, n_x, c, n, w, lv, s));  // the determinants
  {
    ProfScope ps(PROF_TC_FINALIZE, s);
    const unsigned grid = unsigned(std::min<uint64_t>((w.cap[n] + 127) / 128, 152 * 16));
    ANQS_CUDA_LAUNCH("amp_kernel", launch_k(amp_kernel, dim3(grid), dim3(128), 0, s, n, x, w.cnt, w.x[b], w.src[b], w.par[b], w.anc[a], w.node0[n - 1], terms, w.amp, w.own));
  }
  ProfScope ps(PROF_TC_ELOC, s);
  const unsigned grid = unsigned(std::min<uint64_t>(w.group * w.parts, 152 * 16));
  ANQS_CUDA_LAUNCH("trie_eloc_kernel", launch_k(trie_eloc_kernel, dim3(grid), dim3(ET), 0, s, H->v, x, n_x, c * w.group, w.group, w.parts, w.x[b], w.amp, w.own, w.part));
  return ANQS_OK;
}

int launch_trie_finish(const anqs_ham* H, Count n_x, const TrieWs& w, double* ere, double* eim, const uint64_t* counts,
                       double* stats, cudaStream_t s) {
  (void)H;
  ProfScope ps(PROF_STATS, s);
  ANQS_CUDA_LAUNCH("trie_finish_kernel", launch_k(trie_finish_kernel, dim3(1), dim3(FT), 0, s, n_x, w.parts, w.part, ere, eim, counts, stats));
  return ANQS_OK;
}

}  // namespace anqs
