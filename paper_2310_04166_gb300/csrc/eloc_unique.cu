// Local energies over the distinct connected determinants of a sample set.
//
// The connected sets of different samples overlap: 10,816 samples of the
// 20-qubit workload have 6.6e6 connected determinants, but the sector holds
// 14,400.  So the amplitudes are evaluated once per distinct determinant (for
// the slot networks once per distinct prefix) and the local energies look
// them up.  The steps of a call:
//   mark    one thread per (sample, excitation) sets the bit of x' in a bitmap
//           over the sector; who sets it also sets the bits of its prefixes
//   count, emit
//           popcounts of the bitmap, their prefix sums, and the list of the
//           marked prefixes level by level (a rank structure: the id of any
//           prefix is one 8-byte load and a popcount)
//   (network: one row per node, or per distinct determinant; other files)
//   sums    the slot terms of each determinant's path, in slot order
//   eloc    one CTA per sample (or a part of it): the excitations are
//           enumerated again, with H_xx' and its sign, and the amplitudes
//           looked up; nothing of the connected set is written to memory.
//           Statistics in the last CTA.
// Sectors of few prefixes skip mark, count and emit: every prefix is a node.
// Where the connected determinants outnumber a larger sector's, all bits are
// set without looking at them (covers_sector).
//
// All float32 sums run in the order of an evaluation of each connected
// determinant by itself, so the amplitudes have its bits.
#include <algorithm>
#include <cmath>

#include "excite.cuh"

namespace anqs {
namespace {

// whether a determinant of the right electron counts lies in the sector (its
// last slot is allowed after its prefix): always, without Z2 symmetries
__device__ __forceinline__ bool in_sector(const HamView& hv, uint32_t a, uint32_t b) {
  if (hv.nz == 0) return true;
  const int p = hv.n - 1;
  const uint32_t m = (1u << p) - 1u;
  const uint64_t x = spread_bits(a) | spread_bits(b) << 1;
  return (slot_mask(hv, p, __popc(a & m), __popc(b & m), x) >> ((x >> (2 * p)) & 3ull)) & 1u;
}

// ---- mark, count, emit --------------------------------------------------------
__device__ __forceinline__ bool set_bit(uint32_t* w, uint32_t bit) {  // true if it was clear
  if (__ldcg(w) & bit) return false;
  return !(atomicOr(w, bit) & bit);
}

__device__ __forceinline__ void mark_det(const HamView& hv, const SectorView& sv, uint32_t* bits, uint32_t idx,
                                         uint32_t a, uint32_t b, int levels) {
  uint32_t* w = bits + sv.woff[sv.n] + (idx >> 5);
  const uint32_t bit = 1u << (idx & 31u);
  if (__ldcg(w) & bit) return;
  if (!in_sector(hv, a, b)) return;
  if ((atomicOr(w, bit) & bit) || !levels) return;
  // the first to set a prefix's bit goes on to its own prefixes
  for (int p = sv.n - 1; p >= 0; --p) {
    const uint32_t i = prefix_index(sv, p, a, b);
    if (!set_bit(bits + sv.woff[p] + (i >> 5), 1u << (i & 31u))) return;
  }
}

// Whether a call's connected determinants outnumber the sector's so far that
// all its prefixes are taken as marked: hardly any is left out then, and one
// word is written per 32 determinants instead of an atomic or a load per
// connected one (6.6e6 of a 14,400-determinant sector: 126 us).  From the
// device's count: a buffer may hold fewer samples than it has room for.
// Not with Z2 symmetries, where the index also holds other sectors' prefixes.
// How often (cover) depends on what a determinant costs the network: the sets
// of samples that follow its distribution leave a third of the sector out at
// four connected determinants per one, a tenth at twelve.  16-bit MLP, 12
// orbitals, 5 + 5 electrons (us, all and marked): 274 and 202 at 1.5 per one,
// 284 and 304 at 4, 337 and 439 at 12; FP32 MLP 5,990 and 3,870 at 4, 6,050
// and 5,330 at 12, where marking takes 100.
constexpr uint32_t kCover = 32;  // 16-bit MLP: kCoverMlpTc
__device__ __forceinline__ bool covers_sector(const HamView& hv, const SectorView& sv, uint32_t cover, uint64_t n_x) {
  return hv.nz == 0 && n_x * uint64_t(hv.K) >= uint64_t(cover) * sv.na_p[sv.n] * sv.nb_p[sv.n];
}

constexpr int MT_ = 128;

__global__ void __launch_bounds__(MT_) mark_kernel(HamView hv, SectorView sv, const uint64_t* __restrict__ xs,
                                                   Count n_x_, int splits, uint32_t* __restrict__ bits, int levels,
                                                   uint32_t cover) {
  ANQS_PDL_ENTRY();
  __shared__ Exc E;
  const uint64_t items = n_x_.get() * uint64_t(splits);
  const uint32_t K = hv.K;
  if (covers_sector(hv, sv, cover, n_x_.get())) {
    for (int p = levels ? 0 : sv.n; p <= sv.n; ++p) {
      const uint32_t all = sv.na_p[p] * sv.nb_p[p], words = (all + 31u) / 32u;
      for (uint32_t w = blockIdx.x * MT_ + threadIdx.x; w < words; w += gridDim.x * MT_)
        bits[sv.woff[p] + w] = w + 1 < words || !(all & 31u) ? ~0u : (1u << (all & 31u)) - 1u;
    }
    return;
  }
  build_pairs(hv, E);
  const uint32_t nvb = hv.n - hv.nb, nsb = hv.nb * nvb;
  const FastDiv dsb = fast_div(nsb);
  FastDiv dp[2];
  for (int s = 0; s < 2; ++s) {
    const uint32_t nv = hv.n - (s ? hv.nb : hv.na);
    dp[s] = fast_div(nv * (nv - 1) / 2);
  }
  for (uint64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const uint64_t l = it / uint32_t(splits);
    const uint32_t part = uint32_t(it - l * uint32_t(splits));
    build_exc<true>(hv, sv, __ldcg(reinterpret_cast<const unsigned long long*>(xs) + l), E);
    if (!E.ok) continue;
    const uint32_t k0 = uint32_t(uint64_t(K) * part / uint32_t(splits)),
                   k1 = uint32_t(uint64_t(K) * (part + 1) / uint32_t(splits));
    if (part == 0 && threadIdx.x == 0) mark_det(hv, sv, bits, E.own[0] + E.own[1], E.str[0], E.str[1], levels);
    for (uint32_t k = k0 + threadIdx.x; k < k1; k += MT_) {
      uint32_t idx, a = E.str[0], b = E.str[1];
      if (k < hv.nsa) {
        a ^= (1u << E.si[0][k]) ^ (1u << E.sa[0][k]);
        idx = E.rank[0][k] + E.own[1];
      } else if (k < hv.nsa + hv.nsb) {
        const uint32_t e = k - hv.nsa;
        b ^= (1u << E.si[1][e]) ^ (1u << E.sa[1][e]);
        idx = E.own[0] + E.rank[1][e];
      } else {
        uint32_t r = k - hv.nsa - hv.nsb;
        if (r < hv.ndaa + hv.ndbb) {
          const int s = r < hv.ndaa ? 0 : 1;
          if (s) r -= hv.ndaa;
          const uint32_t q = fdiv(dp[s], r), po = E.po[s][q], pv = E.pv[s][r - q * dp[s].d];
          const uint32_t flip = (1u << E.occ[s][po & 255u]) ^ (1u << E.occ[s][po >> 8]) ^
                                (1u << E.vir[s][pv & 255u]) ^ (1u << E.vir[s][pv >> 8]);
          if (s) {
            b ^= flip;
            idx = E.own[0] + __ldg(sv.rkb + (1u << sv.n) + b);
          } else {
            a ^= flip;
            idx = __ldg(sv.rka + (1u << sv.n) + a) * sv.nb_p[sv.n] + E.own[1];
          }
        } else {
          r -= hv.ndaa + hv.ndbb;
          const uint32_t ea = fdiv(dsb, r), eb = r - ea * nsb;
          a ^= (1u << E.si[0][ea]) ^ (1u << E.sa[0][ea]);
          b ^= (1u << E.si[1][eb]) ^ (1u << E.sa[1][eb]);
          idx = E.rank[0][ea] + E.rank[1][eb];
        }
      }
      mark_det(hv, sv, bits, idx, a, b, levels);
    }
  }
}

// the prefixes of the samples alone (one thread per sample)
__global__ void mark_samples_kernel(HamView hv, SectorView sv, const uint64_t* __restrict__ xs, Count n_x_,
                                    uint32_t* __restrict__ bits) {
  ANQS_PDL_ENTRY();
  const uint64_t n_x = n_x_.get();
  const int n = sv.n;
  for (uint64_t l = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; l < n_x; l += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t x = xs[l];
    const uint32_t a = even_bits(x), b = even_bits(x >> 1);
    if (__popc(a) != hv.na || __popc(b) != hv.nb || (x >> (2 * n)) != 0 || !in_sector(hv, a, b)) continue;
    for (int p = n - 1; p >= 0; --p) {
      const uint32_t i = prefix_index(sv, p, a, b);
      if (!set_bit(bits + sv.woff[p] + (i >> 5), 1u << (i & 31u))) break;
    }
  }
}

constexpr int CT = 256;  // threads of the count and emit kernels

// Bitmap words per CTA: one per thread, so that the 450 words of a 20-qubit
// sector occupy two SMs for a microsecond (with 4,096 words per CTA one CTA
// expanded them all, 27 us), and more where the CTAs, each of which sums the
// counts of all CTAs before it, would number above 4,096.
constexpr uint32_t CW_MAX = 4096;
uint32_t words_per_cta(uint32_t words) { return std::min(CW_MAX, std::max<uint32_t>(1, (words + 4096 * CT - 1) / (4096 * CT)) * CT); }

// nodes of each CTA's CW words, and the total of the determinants' level (words from leaf_w on)
__global__ void __launch_bounds__(CT) count_kernel(const uint32_t* __restrict__ bits, uint32_t words, uint32_t CW,
                                                   uint32_t leaf_w, uint32_t* __restrict__ bsum,
                                                   unsigned long long* __restrict__ n_leaves) {
  ANQS_PDL_ENTRY();
  __shared__ uint32_t s_sum, s_leaf;
  if (threadIdx.x == 0) s_sum = s_leaf = 0;
  __syncthreads();
  const uint32_t w0 = blockIdx.x * CW;
  uint32_t c = 0, f = 0;
#pragma unroll 4
  for (uint32_t i = threadIdx.x; i < CW; i += CT)
    if (w0 + i < words) {
      const uint32_t k = __popc(__ldcg(bits + w0 + i));
      c += k;
      f += w0 + i >= leaf_w ? k : 0u;
    }
  c = __reduce_add_sync(0xffffffffu, c);
  f = __reduce_add_sync(0xffffffffu, f);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s_sum, c);
    atomicAdd(&s_leaf, f);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    bsum[blockIdx.x] = s_sum;
    if (s_leaf) atomicAdd(n_leaves, static_cast<unsigned long long>(s_leaf));
  }
}

// words: those of the levels below `levels`; writes off[0 .. levels]
__global__ void __launch_bounds__(CT) emit_kernel(SectorView sv, int levels, const uint32_t* __restrict__ bits, uint32_t words,
                                                  uint32_t CW, const uint32_t* __restrict__ bsum, uint2* __restrict__ packed,
                                                  uint64_t* __restrict__ node_x, uint32_t* __restrict__ off) {
  ANQS_PDL_ENTRY();
  __shared__ uint32_t s_base, s_warp[CT / 32];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_base = 0;
  __syncthreads();
  {  // nodes before this CTA's words
    uint32_t c = 0;
    for (uint32_t i = threadIdx.x; i < blockIdx.x; i += CT) c += __ldcg(bsum + i);
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) atomicAdd(&s_base, c);
  }
  __syncthreads();
  uint32_t base = s_base;
  const uint32_t w_end = min(words, (blockIdx.x + 1) * CW);
  for (uint32_t w0 = blockIdx.x * CW; w0 < w_end; w0 += CT) {
    const uint32_t w = w0 + threadIdx.x;
    uint32_t v = w < w_end ? __ldcg(bits + w) : 0u;
    const uint32_t c = __popc(v);
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) s_warp[wp] = inc;
    __syncthreads();
    uint32_t before = 0, total = 0;
#pragma unroll
    for (int q = 0; q < CT / 32; ++q) {
      if (q < wp) before += s_warp[q];
      total += s_warp[q];
    }
    const uint32_t id = base + before + inc - c;
    int p = 0;
    uint32_t i0 = 0;
    if (w < w_end) {
      packed[w] = make_uint2(v, id);
      while (w >= sv.woff[p + 1]) ++p;
      if (w == sv.woff[p]) off[p] = id;
      if (w + 1 == words) off[levels] = id + c;
      i0 = (w - sv.woff[p]) * 32u;
    }
    // the warp's words, a lane per bit, four words' lookups in flight (one word
    // at a time waited for its two loads 32 times: 14 us for any sector); a
    // word's nodes are written side by side
    const uint32_t some = __ballot_sync(0xffffffffu, v != 0u);
#pragma unroll 1
    for (int q0 = 0; q0 < 32; q0 += 4) {
      if (!((some >> q0) & 15u)) continue;
      uint32_t sa[4], sb[4], at[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t vq = __shfl_sync(0xffffffffu, v, q0 + e), idq = __shfl_sync(0xffffffffu, id, q0 + e),
                       idx = __shfl_sync(0xffffffffu, i0, q0 + e) + uint32_t(lane);
        const int pq = __shfl_sync(0xffffffffu, p, q0 + e);
        const bool on = (vq >> lane) & 1u;
        const uint32_t nb = sv.nb_p[pq], ra = idx / nb, rb = idx - ra * nb;
        sa[e] = on ? __ldg(sv.sta + sv.soa[pq] + ra) : 0u;
        sb[e] = on ? __ldg(sv.stb + sv.sob[pq] + rb) : 0u;
        at[e] = on ? idq + __popc(vq & ((1u << lane) - 1u)) : 0xffffffffu;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (at[e] != 0xffffffffu) node_x[at[e]] = spread_bits(sa[e]) | spread_bits(sb[e]) << 1;
    }
    base += total;
    __syncthreads();
  }
}

// ---- path sums ------------------------------------------------------------------
// sums[node of level hi] = from[its level-lo prefix] + the terms of slots lo .. hi - 1
// (of each variant: consecutive threads take the variants of a node)
__global__ void path_sum_kernel(SectorView sv, NodeView nv, const float2* __restrict__ terms, int lo, int hi,
                                const float2* __restrict__ from, float2* __restrict__ sums, uint32_t var) {
  ANQS_PDL_ENTRY();
  const uint32_t i0 = __ldcg(nv.off + hi), i1 = __ldcg(nv.off + hi + 1), lo0 = __ldcg(nv.off + lo);
  const uint64_t total = uint64_t(i1 - i0) * var;
  for (uint64_t k = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; k < total; k += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t r = var == 1 ? uint32_t(k) : uint32_t(k / var), vr = var == 1 ? 0u : uint32_t(k - uint64_t(r) * var);
    const uint32_t id = i0 + r;
    const uint64_t x = __ldcg(reinterpret_cast<const unsigned long long*>(nv.x) + id);
    const uint32_t a = even_bits(x), b = even_bits(x >> 1);
    float la = 0.f, ph = 0.f;
    if (lo) {
      const float2 t = __ldcg(from + size_t(node_id(sv, nv, lo, prefix_index(sv, lo, a, b)) - lo0) * var + vr);
      la = t.x;
      ph = t.y;
    }
    for (int p = lo; p < hi; p += 4) {  // four slots' loads in flight
      float2 t[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        t[e] = make_float2(0.f, 0.f);
        if (p + e < hi)
          t[e] = __ldcg(terms + (size_t(node_id(sv, nv, p + e, prefix_index(sv, p + e, a, b))) * var + vr) * 4 +
                        ((x >> (2 * (p + e))) & 3ull));
      }
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (p + e < hi) {
          la += t[e].x;
          ph += t[e].y;
        }
    }
    sums[k] = make_float2(la, ph);
  }
}

// out[leaf][p] = per[id] + per[stride + id], id the node of the leaf's level p + 1 prefix
__global__ void path_terms_kernel(SectorView sv, NodeView nv, const float2* __restrict__ per, uint64_t stride,
                                  float2* __restrict__ out) {
  ANQS_PDL_ENTRY();
  const int n = sv.n;
  const uint32_t i0 = __ldcg(nv.off + n);
  const uint64_t total = uint64_t(__ldcg(nv.off + n + 1) - i0) * n;
  for (uint64_t t = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; t < total; t += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t r = uint32_t(t / uint32_t(n));
    const int p = int(t - uint64_t(r) * uint32_t(n)) + 1;
    const uint64_t x = __ldcg(reinterpret_cast<const unsigned long long*>(nv.x) + i0 + r);
    const float2* at = per + node_id(sv, nv, p, prefix_index(sv, p, even_bits(x), even_bits(x >> 1)));
    const float2 u = __ldcg(at), v = __ldcg(at + stride);
    out[t] = make_float2(u.x + v.x, u.y + v.y);
  }
}

// Rows r < leaves of raw network outputs [r][n][8] (determinants x[r]) to
// tab[r][n + 1]: entry j < n is the amplitude of the determinant as the
// connected determinant of a sample that first differs in slot j (the sum of
// the terms up to j, plus the sum of the later ones), entry n its own (all
// terms in order).  One thread per determinant.
__global__ void byj_kernel(HamView hv, const uint64_t* __restrict__ xs, Count rows_, const float* __restrict__ raw,
                           float2* __restrict__ tab) {
  ANQS_PDL_ENTRY();
  const int n = hv.n;
  const uint64_t rows = rows_.get();
  for (uint64_t r = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; r < rows; r += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t x = __ldcg(reinterpret_cast<const unsigned long long*>(xs) + r);
    float2 t[IDX_MAX_ORB];
    bool dead = false;
    int ca = 0, cb = 0;
    for (int p = 0; p < n; ++p) {
      const float4* o4 = reinterpret_cast<const float4*>(raw + (r * n + p) * 8);
      const float4 q0 = __ldcg(o4), q1 = __ldcg(o4 + 1);
      const float o[4] = {q0.x, q0.y, q0.z, q0.w};
      const unsigned pmk = slot_mask(hv, p, ca, cb, x), mk = norm_mask(hv, p, pmk);
      float mx = -INFINITY;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if ((mk >> u) & 1u) mx = fmaxf(mx, o[u]);
      float sum = 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if ((mk >> u) & 1u) sum += __expf(o[u] - mx);
      const float lse = mx + __logf(sum);
      const int v = int((x >> (2 * p)) & 3ull);
      const float ov = v == 0 ? o[0] : v == 1 ? o[1] : v == 2 ? o[2] : o[3];
      t[p].x = ((pmk >> v) & 1u) ? 0.5f * (ov - lse) : -INFINITY;
      t[p].y = v == 0 ? q1.x : v == 1 ? q1.y : v == 2 ? q1.z : q1.w;
      dead = dead || !((pmk >> v) & 1u);
      ca += v & 1;
      cb += v >> 1;
    }
    float2* d = tab + r * (n + 1);
    float la = 0.f, ph = 0.f;
    for (int j = 0; j < n; ++j) {
      la += t[j].x;
      ph += t[j].y;
      float sl = 0.f, sp = 0.f;
      for (int p = j + 1; p < n; ++p) {
        sl += t[p].x;
        sp += t[p].y;
      }
      d[j] = j + 1 < n ? make_float2(la + sl, ph + sp) : make_float2(la, ph);
      if (dead) d[j].x = -INFINITY;
    }
    d[n] = make_float2(dead ? -INFINITY : la, ph);
  }
}

// rows of each chunk of `chunk` determinants
__global__ void chunk_counts_kernel(const uint64_t* __restrict__ total, uint64_t chunk, int n, uint64_t* __restrict__ out) {
  ANQS_PDL_ENTRY();
  const uint64_t t = *total;
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    const uint64_t lo = uint64_t(c) * chunk;
    out[c] = t <= lo ? 0 : (t - lo < chunk ? t - lo : chunk);
  }
}

// ---- E_loc ------------------------------------------------------------------------
constexpr int ET = 128;
constexpr uint64_t kTailStats = 1024;  // samples up to which eloc_direct_kernel's last CTA reduces the statistics

// a * b with the sign flipped if odd, exactly: the 48-bit product of two float
// significands fits into a double, and multiplying and packing them as
// integers keeps three conversions and a multiplication off the FP64 pipe.
__device__ __forceinline__ double exact_product(float a, float b, int odd) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  const uint32_t ea = (ua >> 23) & 255u, eb = (ub >> 23) & 255u;
  if (ea - 1u < 254u && eb - 1u < 254u) {  // both normal
    // significands scaled by 2^3 each: the product has bit 52 or 53 set
    const uint64_t m = uint64_t((ua << 3 & 0x03fffff8u) | 0x04000000u) * ((ub << 3 & 0x03fffff8u) | 0x04000000u);
    const uint32_t top = uint32_t(m >> 53);
    const uint64_t r = m >> top;  // bit 52 set; a bit shifted out is zero
    const uint32_t hi = uint32_t(r >> 32) + ((ea + eb + 768u + top) << 20);
    return __hiloint2double(int(hi | (((ua ^ ub) & 0x80000000u) ^ (uint32_t(odd) << 31))), int(uint32_t(r)));
  }
  return flip_sign(double(a) * double(b), odd);
}

// h_ai + sum_{J occ} ([AI|JJ] - [AJ|JI]) of the single I -> A of spin s, one
// table entry per occupied orbital
__device__ __forceinline__ double single_sum(const HamView& hv, const Exc& E, int s, int i, int a) {
  const int n = hv.n, row = (a * n + i) * n * n;
  double v = __ldg(hv.h + a * n + i);
  for (int t = 0; t < 2; ++t) {
    const double* src = (t == s ? hv.ga : hv.g) + row;
    const int ne = t ? hv.nb : hv.na;
    for (int m = 0; m < ne; ++m) v += __ldg(src + E.occ[t][m] * (n + 1));
  }
  return v;
}

// One CTA per (sample, part).  The FP64 pipe bounds it: it takes two lanes per
// clock and SM, so a term costs two FP64 operations, the accumulations of its
// real and imaginary part (7 when the amplitude ratio was converted and
// multiplied there: the pipe was 80% busy), the diagonal comes from pair
// energies and one warp adds up the CTA's 128 partial sums.
template <AmpMode MODE>
__global__ void __launch_bounds__(ET) eloc_direct_kernel(HamView hv, SectorView sv, NodeView nv,
                                                         const uint64_t* __restrict__ xs, Count n_x_, int splits,
                                                         AmpSrc A, double* ere, double* eim, double* part,
                                                         StatsOut so) {
  ANQS_PDL_ENTRY();
  constexpr bool RANK = MODE != AMP_ARRAY;
  __shared__ Exc E;
  __shared__ double red[2][ET];
  __shared__ int s_last;
  const uint64_t n_x = n_x_.get();
  const int n = hv.n, lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const uint32_t K = hv.K;
  const uint64_t items = n_x * uint64_t(splits);
  build_pairs(hv, E);
  const uint32_t nvb = n - hv.nb, nsb = hv.nb * nvb, nva = n - hv.na;
  const FastDiv dsb = fast_div(nsb);
  FastDiv dp[2];
  for (int s = 0; s < 2; ++s) {
    const uint32_t nv_ = s ? nvb : nva;
    dp[s] = fast_div(nv_ * (nv_ - 1) / 2);
  }
  const uint32_t var = A.variants;
  const FastDiv dvar = fast_div(var);
  uint32_t leaf0 = 0;
  if constexpr (RANK) leaf0 = __ldcg(nv.off + n);
  const bool all = !nv.packed || covers_sector(hv, sv, nv.cover, n_x);  // every determinant of the sector has a row
  // row of determinant index idx in the amplitude tables; false if it is not there
  auto leaf = [&](uint32_t idx, uint32_t& r) -> bool {
    if (all) {
      r = idx;
      return true;
    }
    const uint2 w = __ldcg(nv.packed + sv.woff[n] + (idx >> 5));
    r = w.y - leaf0 + uint32_t(__popc(w.x & ((1u << (idx & 31u)) - 1u)));
    return (w.x >> (idx & 31u)) & 1u;
  };
  for (uint64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const uint64_t l = it / uint32_t(splits);
    const uint32_t pt = uint32_t(it - l * uint32_t(splits));
    build_exc<RANK>(hv, sv, __ldcg(reinterpret_cast<const unsigned long long*>(xs) + l), E);
    double re = 0.0, im = 0.0, dg = 0.0;
    const uint32_t vbase = uint32_t(l * K % var);
    if (E.ok) {
      float lx, px;
      if constexpr (MODE == AMP_SUM || MODE == AMP_BYJ) {
        uint32_t r;
        lx = -INFINITY;
        px = 0.f;
        if (leaf(E.own[0] + E.own[1], r)) {
          if (MODE == AMP_SUM && !A.tab) {
            lx = __ldcg(A.la + r);
            px = __ldcg(A.ph + r);
          } else {
            const float2 t = __ldcg(A.tab + (MODE == AMP_SUM ? size_t(r) * var + uint32_t(l % var) : size_t(r) * (n + 1) + n));
            lx = t.x;
            px = t.y;
          }
        }
      } else {
        lx = __ldcg(A.la_x + l);
        px = __ldcg(A.ph_x + l);
      }
      // log|psi(x')| and phase of excitation k (determinant index idx, strings a and b, first differing slot j)
      auto add = [&](uint32_t k, uint32_t idx, uint32_t a, uint32_t b, int j, double h, int odd) {
        float la, ph;
        if constexpr (MODE == AMP_ARRAY) {
          la = __ldcg(A.la + l * K + k);
          ph = __ldcg(A.ph + l * K + k);
        } else {
          uint32_t r;
          const bool there = leaf(idx, r);
          la = -INFINITY;
          ph = 0.f;
          if constexpr (MODE == AMP_TERMS) {
            const float* cc = A.cache + (l * n + j) * TC_CACHE_F;
            const int vj = int((a >> j) & 1u) + 2 * int((b >> j) & 1u);
            la = __ldcg(cc) + __ldcg(cc + 2 + vj);
            ph = __ldcg(cc + 1) + __ldcg(cc + 6 + vj);
            if (!there) la = -INFINITY;
            else
              for (int p = j + 1; p < n; ++p) {
                const float2 t = __ldcg(A.tab + size_t(r) * n + p);
                la += t.x;
                ph += t.y;
              }
          } else if (there) {
            if (MODE == AMP_SUM && !A.tab) {
              la = __ldcg(A.la + r);
              ph = __ldcg(A.ph + r);
            } else {
              uint32_t vr = 0;
              if (MODE == AMP_SUM && var > 1) {
                vr = vbase + k;
                vr -= fdiv(dvar, vr) * var;
              }
              const float2 t = __ldcg(A.tab + (MODE == AMP_SUM ? size_t(r) * var + vr : size_t(r) * (n + 1) + j));
              la = t.x;
              ph = t.y;
            }
          }
        }
        const float r = expf(la - lx);
        float s, co;
        sincosf(ph - px, &s, &co);
        re = fma(h, exact_product(r, co, odd), re);
        im = fma(h, exact_product(r, s, odd), im);
      };
      const uint32_t k0 = uint32_t(uint64_t(K) * pt / uint32_t(splits)),
                     k1 = uint32_t(uint64_t(K) * (pt + 1) / uint32_t(splits));
      const uint32_t ks = hv.nsa + hv.nsb, kd = ks + hv.ndaa + hv.ndbb;
      // opposite-spin doubles (I_a, A_a, I_b, A_b): [AI|BJ], as the product of the two singles
      for (uint32_t k = max(k0, kd) + threadIdx.x; k < k1; k += ET) {
        const uint32_t r = k - kd, ea = fdiv(dsb, r), eb = r - ea * nsb;
        const int i = E.si[0][ea], a = E.sa[0][ea], j = E.si[1][eb], b = E.sa[1][eb];
        const int sg = sign_ab(E, ea, eb, i, a, j, b);
        const double v = __ldg(hv.g + E.g[0][ea] + E.g[1][eb]);
        uint32_t idx = 0;
        if constexpr (RANK) idx = E.rank[0][ea] + E.rank[1][eb];
        add(k, idx, E.str[0] ^ (1u << i) ^ (1u << a), E.str[1] ^ (1u << j) ^ (1u << b), min(min(i, a), min(j, b)), v, sg);
      }
      // same-spin doubles I<J -> A<B: [AI|BJ] - [AJ|BI], as I -> A then J -> B
      for (uint32_t k = max(k0, ks) + threadIdx.x; k < min(k1, kd); k += ET) {
        uint32_t r = k - ks;
        const int s = r < hv.ndaa ? 0 : 1;
        if (s) r -= hv.ndaa;
        const uint32_t q = fdiv(dp[s], r), po = E.po[s][q], pv = E.pv[s][r - q * dp[s].d];
        const uint32_t nv_ = s ? nvb : nva;
        const int i = E.occ[s][po & 255u], j = E.occ[s][po >> 8], a = E.vir[s][pv & 255u], b = E.vir[s][pv >> 8];
        const int sg = sign_ss(E, s, po, pv, nv_, i, j, a, b);
        const double v = __ldg(hv.ga + ((a * n + i) * n + b) * n + j);
        const uint32_t flip = (1u << i) ^ (1u << j) ^ (1u << a) ^ (1u << b);
        const uint32_t sa = E.str[0] ^ (s ? 0u : flip), sb = E.str[1] ^ (s ? flip : 0u);
        uint32_t idx = 0;
        if constexpr (RANK)
          idx = s ? E.own[0] + __ldg(sv.rkb + (1u << n) + sb) : __ldg(sv.rka + (1u << n) + sa) * sv.nb_p[n] + E.own[1];
        add(k, idx, sa, sb, min(min(i, j), min(a, b)), v, sg);
      }
      // singles I -> A of spin s: h_ai + sum_{J occ} ([AI|JJ] - [AJ|JI])
      for (uint32_t k = k0 + threadIdx.x; k < min(k1, ks); k += ET) {
        const int s = k < hv.nsa ? 0 : 1;
        const uint32_t e = s ? k - hv.nsa : k;
        const int i = E.si[s][e], a = E.sa[s][e];
        const double v = single_sum(hv, E, s, i, a);
        uint32_t idx = 0;
        if constexpr (RANK) idx = s ? E.own[0] + E.rank[1][e] : E.rank[0][e] + E.own[1];
        const uint32_t flip = (1u << i) ^ (1u << a);
        add(k, idx, E.str[0] ^ (s ? 0u : flip), E.str[1] ^ (s ? flip : 0u), min(i, a), v, E.sgn[s][e]);
      }
      if (pt == 0) {  // <x|H|x> = E_nuc + sum_I h_ii + sum_{I<J occ} ([II|JJ] - [IJ|JI])
        const int ca = hv.na * (hv.na - 1) / 2, cs = ca + hv.nb * (hv.nb - 1) / 2, cd = cs + hv.na * hv.nb;
        for (int t = threadIdx.x; t < cd + hv.na + hv.nb; t += ET) {
          const double* src;
          if (t < cs) {
            const int s = t >= ca ? 1 : 0;
            const uint32_t po = E.po[s][s ? t - ca : t];
            src = hv.pair + E.occ[s][po & 255u] * n + E.occ[s][po >> 8];
          } else if (t < cd) {
            const int q = (t - cs) / hv.nb;
            src = hv.pair + n * n + E.occ[0][q] * n + E.occ[1][t - cs - q * hv.nb];
          } else {
            const int I = t - cd;
            src = hv.h + (I < hv.na ? E.occ[0][I] : E.occ[1][I - hv.na]) * (n + 1);
          }
          dg += __ldg(src);
        }
        if (threadIdx.x == 0) dg += hv.e_nuc;
      }
    } else {  // a determinant outside the sector
      const double nan = __longlong_as_double(0x7ff8000000000000ll);
      re = nan;
      im = K ? nan : 0.0;
    }
    red[0][threadIdx.x] = re + dg;
    red[1][threadIdx.x] = im;
    __syncthreads();
    if (wp == 0) {  // lanes 0..15 the real parts, 16..31 the imaginary ones
      const double* r = red[lane >> 4] + (lane & 15);
      double v = 0.0;
#pragma unroll
      for (int q = 0; q < ET; q += 16) v += r[q];
#pragma unroll
      for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      const double vi = __shfl_sync(0xffffffffu, v, 16);
      if (lane == 0) {
        if (splits == 1) {
          ere[l] = v;
          eim[l] = vi;
        } else {
          part[2 * it] = v;
          part[2 * it + 1] = vi;
        }
      }
    }
  }
  if (splits == 1 && !so.counts) return;
  if (threadIdx.x == 0) {
    __threadfence();  // this CTA's rows (written by thread 0) before its ticket
    s_last = atomicAdd(so.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (splits > 1) {  // the parts of each sample, in order
    for (uint64_t l = threadIdx.x; l < n_x; l += ET) {
      double sr = 0.0, si = 0.0;
      for (int q = 0; q < splits; ++q) {
        sr += __ldcg(part + 2 * (l * uint32_t(splits) + q));
        si += __ldcg(part + 2 * (l * uint32_t(splits) + q) + 1);
      }
      ere[l] = sr;
      eim[l] = si;
    }
    __threadfence();
    __syncthreads();
  }
  if (so.counts) cta_energy_stats<ET>(ere, eim, so.counts, n_x, so.stats);
}

// Statistics of more than kTailStats samples: a CTA per 512 of them, the last
// one adds up the partial sums in order.  One CTA alone, bound by its SM's FP64
// pipe, takes 2 ns per sample.
constexpr int SB = 152;  // CTAs at most
__global__ void __launch_bounds__(ET) stats_kernel(const double* ere, const double* eim,
                                                   const uint64_t* __restrict__ counts, Count n_x_, double* part,
                                                   uint32_t* ticket, double* stats) {
  ANQS_PDL_ENTRY();
  __shared__ double red[4][ET / 32];
  __shared__ int s_last;
  const uint64_t n_x = n_x_.get();
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const double kr = n_x ? __ldcg(ere) : 0.0, ki = n_x ? __ldcg(eim) : 0.0;
  double t[4] = {0.0, 0.0, 0.0, 0.0};  // sums of n, n d, n |d|^2 with d the distance from the first sample's energy
  for (uint64_t l = blockIdx.x * uint64_t(ET) + threadIdx.x; l < n_x; l += uint64_t(gridDim.x) * ET) {
    const double c = double(__ldcg(reinterpret_cast<const unsigned long long*>(counts) + l));
    const double dr = __ldcg(ere + l) - kr, di = __ldcg(eim + l) - ki;
    t[0] += c;
    t[1] = fma(c, dr, t[1]);
    t[2] = fma(c, di, t[2]);
    t[3] = fma(c, fma(dr, dr, di * di), t[3]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int o = 16; o; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
    if (lane == 0) red[k][wp] = t[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k) {
      double v = 0.0;
      for (int q = 0; q < ET / 32; ++q) v += red[k][q];
      part[4 * blockIdx.x + k] = v;
    }
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || wp) return;
  __threadfence();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    t[k] = 0.0;
    for (uint32_t b = lane; b < gridDim.x; b += 32) t[k] += __ldcg(part + 4 * b + k);
#pragma unroll
    for (int o = 16; o; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
  }
  if (lane) return;
  const double mr = t[1] / t[0], mi = t[2] / t[0];
  stats[0] = kr + mr;
  stats[1] = ki + mi;
  stats[2] = fmax(0.0, t[3] / t[0] - fma(mr, mr, mi * mi));
  stats[3] = t[0];
}

// CTAs per sample: a whole sample each when there are enough to fill the GPU
// (16 CTAs of 128 threads per SM are resident at most), else parts of at
// least one excitation per thread.  (With parts of 512 one sample of 10 orbitals,
// 875 excitations, was one CTA: 70 us of marking, seven chains of dependent
// loads and atomics one after the other, and 33 us of assembly.)
constexpr uint64_t kFillCtas = 152 * 8, kPart = 128;

int split_of(uint64_t n_x, uint32_t K) {
  if (n_x == 0) return 1;
  const uint64_t want = (kFillCtas + n_x - 1) / n_x, most = std::max<uint64_t>(1, K / kPart);
  return int(std::max<uint64_t>(1, std::min<uint64_t>(std::min(want, most), 128)));
}

uint64_t index_words(const anqs_ham* H) { return H->sv.woff[H->sv.n + 1]; }

// every prefix of a small sector is evaluated when the call's connected
// determinants outnumber the sector's at least fourfold.  Below that it is the
// better form too where it was measured (7 orbitals, 5 + 5 electrons, half a
// connected determinant per determinant: 16-bit MLP 39 us against 69 marked,
// FP32 MLP 57 against 91, NADE 52 against 77, transformer 66 against 81); the
// line keeps a call of few samples from a sector's whole network work.
bool use_full(const anqs_ham* H, uint64_t n_x) {
  return H->has_full && n_x * uint64_t(H->v.K) >= 4ull * H->sv.na_p[H->v.n] * H->sv.nb_p[H->v.n];
}

// The last slots of a determinant's path are summed from its level n - 3 prefix
// where the extra launch pays.  Two steps against one, 16-bit MLP: 4,900
// determinants 41 us against 38 (hence the 16,384), 63,504 94 against 90, 213,444
// 140 against 142, 853,776 379 against 402; FP32 MLP (32 places): 63,504 645
// against 696.
constexpr int kMidSlots = 3;

int mid_level(const anqs_ham* H, uint64_t leaves) {
  return H->v.n > 2 * kMidSlots && leaves > 16384 ? H->v.n - kMidSlots : 0;
}

uint64_t level_bound(const anqs_ham* H, uint64_t n_x, int p) {
  const uint64_t all = uint64_t(H->sv.na_p[p]) * H->sv.nb_p[p];
  return use_full(H, n_x) ? all : std::min<uint64_t>(all, n_x * (uint64_t(H->v.K) + 1));
}

}  // namespace

// The bitmap's fixed cost (zeroing, scanning: 20 bytes per word) against the
// connected set's own (at least 29 bytes per determinant without it).  A line on
// scratch before time.  Index against list, 16-bit MLP 3 x 128: 14 orbitals 7 + 7
// (1.05 M words), 4 samples 99 us against 101, 64 samples 217 against 431; 16
// orbitals 6 + 6 (5.93 M words), 4 samples (words = 292 m) 185 against 148, 16
// samples (73 m) 255 against 274, 256 samples (4.6 m) 761 against 2,633.
bool unique_applies(const anqs_ham* H, uint64_t n_x) {
  if (!H->has_index) return false;
  if (use_full(H, n_x)) return true;
  const uint64_t m = n_x * (uint64_t(H->v.K) + 1);
  return index_words(H) <= (1ull << 20) || index_words(H) <= 8 * m;
}

bool unique_full(const anqs_ham* H, uint64_t n_x) { return use_full(H, n_x); }

// As if the connected sets fell into the sector at random, times 0.7: sets of
// samples that follow a network's distribution overlap more (16 to 95 samples
// of 11 to 18 orbitals: 0.3 to 0.7 of a random set's determinants).
double unique_expected(const anqs_ham* H, uint64_t n_x) {
  const double all = double(H->sv.na_p[H->v.n]) * double(H->sv.nb_p[H->v.n]);
  if (use_full(H, n_x)) return all;
  return std::max(0.7 * all * -std::expm1(-double(n_x) * (double(H->v.K) + 1.0) / all), std::min(all, double(H->v.K) + 1.0));
}

void plan_unique(const anqs_ham* H, uint64_t n_x, bool levels, Arena& A, UniqueWs& w) {
  const int n = H->v.n;
  w = UniqueWs{};
  w.full = use_full(H, n_x);
  w.levels = levels;
  for (int p = levels ? 0 : n; p <= n; ++p) w.max_nodes += level_bound(H, n_x, p);
  w.max_leaves = level_bound(H, n_x, n);
  const uint64_t words = index_words(H);  // reserved in the full form too: a smaller call may run without it
  w.bits_bytes = 256 + words * sizeof(uint32_t);
  char* z = A.take<char>(w.bits_bytes);
  w.ticket = reinterpret_cast<uint32_t*>(z);
  w.part = A.take<double>(eloc_partials(H, n_x));
  w.bits = z ? reinterpret_cast<uint32_t*>(z + 256) : nullptr;
  w.packed = A.take<uint2>(words);
  w.bsum = A.take<uint32_t>((words + words_per_cta(uint32_t(words)) - 1) / words_per_cta(uint32_t(words)));
  w.n_leaves = z ? reinterpret_cast<uint64_t*>(z + 8) : nullptr;
  w.node_x = A.take<uint64_t>(w.max_nodes);
  w.leaf_x = w.node_x;  // without levels, the determinants are the only nodes
  w.off = A.take<uint32_t>(n + 2);
  w.nodes = w.full ? NodeView{H->d_full_x, H->d_full_off, nullptr, kCover} : NodeView{w.node_x, w.off, w.packed, kCover};
}

int launch_unique(const anqs_ham* H, const uint64_t* x, Count n_x, const UniqueWs& w, cudaStream_t s) {
  ANQS_CUDA(cudaMemsetAsync(w.ticket, 0, w.full ? sizeof(uint32_t) : w.bits_bytes, s));
  if (w.full) return ANQS_OK;
  const int splits = split_of(n_x.n, H->v.K);
  {
    ProfScope ps(PROF_CONNECT, s);
    const unsigned grid = unsigned(std::min<uint64_t>(n_x.n * splits, 152 * 12));
    ANQS_CUDA_LAUNCH("mark_kernel", launch_k(mark_kernel, dim3(grid), dim3(MT_), 0, s, H->v, H->sv, x, n_x, splits, w.bits, w.levels ? 1 : 0, w.nodes.cover));
  }
  ProfScope ps(PROF_TC_SORT, s);
  const uint32_t words = uint32_t(index_words(H)), cw = words_per_cta(words);
  const unsigned blocks = (words + cw - 1) / cw;
  ANQS_CUDA_LAUNCH("count_kernel", launch_k(count_kernel, dim3(blocks), dim3(CT), 0, s, w.bits, words, cw, H->sv.woff[H->v.n], w.bsum, reinterpret_cast<unsigned long long*>(w.n_leaves)));
  ANQS_CUDA_LAUNCH("emit_kernel", launch_k(emit_kernel, dim3(blocks), dim3(CT), 0, s, H->sv, H->v.n + 1, w.bits, words, cw, w.bsum, w.packed, w.node_x, w.off));
  return ANQS_OK;
}

int launch_path_terms(const anqs_ham* H, const UniqueWs& w, const float2* per, float2* out, cudaStream_t s) {
  ProfScope ps(PROF_TC_FINALIZE, s);
  const unsigned grid = unsigned(std::min<uint64_t>((w.max_leaves * H->v.n + 255) / 256, 152 * 8));
  ANQS_CUDA_LAUNCH("path_terms_kernel", launch_k(path_terms_kernel, dim3(grid ? grid : 1), dim3(256), 0, s, H->sv, w.nodes, per, w.max_nodes, out));
  return ANQS_OK;
}

int launch_byj(const HamView& hv, const uint64_t* x, Count rows, const float* raw, float2* tab, cudaStream_t s) {
  ProfScope ps(PROF_TC_FINALIZE, s);
  const unsigned grid = unsigned(std::min<uint64_t>((rows.n + 63) / 64, 152 * 16));
  ANQS_CUDA_LAUNCH("byj_kernel", launch_k(byj_kernel, dim3(grid ? grid : 1), dim3(64), 0, s, hv, x, rows, raw, tab));
  return ANQS_OK;
}

int launch_chunk_counts(const uint64_t* total, uint64_t chunk, int n, uint64_t* out, cudaStream_t s) {
  ANQS_CUDA_LAUNCH("chunk_counts_kernel", launch_k(chunk_counts_kernel, dim3(1), dim3(256), 0, s, total, chunk, n, out));
  return ANQS_OK;
}

const uint64_t* unique_leaf_x(const anqs_ham* H, const UniqueWs& w) {
  return w.full ? H->d_full_x + H->full_off[H->v.n] : w.leaf_x;
}

bool use_unique(const anqs_ham* H, bool preferred, size_t plain, size_t unique, size_t ws_bytes) {
  if (!H->has_index) return false;
  return preferred ? unique <= ws_bytes || plain > ws_bytes : plain > ws_bytes && unique <= ws_bytes;
}

// The samples' prefixes: what marking and listing them costs is repaid where
// many samples share them.  Prefixes against rows, transformer d 64, 2 blocks, 14
// orbitals 7 + 7: 1 sample 367 us against 295, 256 samples 508 against 451, 4,000
// samples 1,163 against 1,816; 18 orbitals 6 + 6, far beyond the line: 681
// against 301, 777 against 487, 1,828 against 2,383.  2^21 bitmap words cost
// about 20 us to clear and scan.
bool tree_applies(const anqs_ham* H) { return H->has_index && H->sv.woff[H->v.n] <= (1u << 21); }

void plan_tree(const anqs_ham* H, uint64_t n_x, Arena& A, TreeWs& w) {
  const int n = H->v.n;
  const uint32_t words = H->sv.woff[n];
  w = TreeWs{};
  for (int p = 0; p < n; ++p) w.max_rows += std::min<uint64_t>(uint64_t(H->sv.na_p[p]) * H->sv.nb_p[p], n_x);
  w.zero_bytes = 256 + words * sizeof(uint32_t);
  char* z = A.take<char>(w.zero_bytes);
  w.n_rows = reinterpret_cast<uint64_t*>(z);
  w.bits = z ? reinterpret_cast<uint32_t*>(z + 256) : nullptr;
  w.packed = A.take<uint2>(words);
  w.bsum = A.take<uint32_t>((words + words_per_cta(uint32_t(words)) - 1) / words_per_cta(uint32_t(words)));
  w.node_x = A.take<uint64_t>(w.max_rows);
  w.off = A.take<uint32_t>(n + 1);
  w.nodes = NodeView{w.node_x, w.off, w.packed, kCover};
}

int launch_tree(const anqs_ham* H, const uint64_t* x, Count n_x, const TreeWs& w, cudaStream_t s) {
  const uint32_t words = H->sv.woff[H->v.n];
  const uint32_t cw = words_per_cta(words);
  const unsigned blocks = (words + cw - 1) / cw;
  ANQS_CUDA(cudaMemsetAsync(w.n_rows, 0, w.zero_bytes, s));
  ANQS_CUDA_LAUNCH("mark_samples_kernel", launch_k(mark_samples_kernel, dim3(unsigned(std::min<uint64_t>((n_x.n + 63) / 64, 152 * 16))), dim3(64), 0, s, H->v, H->sv, x, n_x, w.bits));
  ANQS_CUDA_LAUNCH("count_kernel", launch_k(count_kernel, dim3(blocks), dim3(CT), 0, s, w.bits, words, cw, 0u, w.bsum, reinterpret_cast<unsigned long long*>(w.n_rows)));
  ANQS_CUDA_LAUNCH("emit_kernel", launch_k(emit_kernel, dim3(blocks), dim3(CT), 0, s, H->sv, H->v.n, w.bits, words, cw, w.bsum, w.packed, w.node_x, w.off));
  return ANQS_OK;
}

Count unique_leaves(const UniqueWs& w) {
  return w.full ? host_count(w.max_leaves) : Count{w.max_leaves, w.n_leaves, 1};
}

uint64_t path_sums_mid(const anqs_ham* H, uint64_t n_x) {
  const int mid = mid_level(H, level_bound(H, n_x, H->v.n));
  return mid ? level_bound(H, n_x, mid) : 0;
}

int launch_path_sums(const anqs_ham* H, const UniqueWs& w, const float2* terms, float2* mid, float2* sums,
                     cudaStream_t s, uint32_t variants) {
  const int n = H->v.n, m = mid_level(H, w.max_leaves);
  ProfScope ps(PROF_TC_FINALIZE, s);
  if (m)
    ANQS_CUDA_LAUNCH("path_sum_kernel", launch_k(path_sum_kernel, dim3(152 * 4), dim3(256), 0, s, H->sv, w.nodes, terms, 0, m, static_cast<const float2*>(nullptr), mid, variants));
  const unsigned grid = unsigned(std::min<uint64_t>((w.max_leaves * variants + 127) / 128, 152 * 16));
  ANQS_CUDA_LAUNCH("path_sum_kernel", launch_k(path_sum_kernel, dim3(grid ? grid : 1), dim3(128), 0, s, H->sv, w.nodes, terms, m, n, static_cast<const float2*>(mid), sums, variants));
  return ANQS_OK;
}

// n_x * split_of(n_x) stays below 1216 + n_x; never less for more samples.
// A call of more samples that is not split keeps its statistics' sums there.
uint64_t eloc_partials(const anqs_ham* H, uint64_t n_x) {
  return std::max<uint64_t>(H->v.K >= 2 * kPart ? 2 * (kFillCtas + std::min<uint64_t>(n_x, kFillCtas)) : 0,
                            n_x > kTailStats ? 4 * SB : 0);
}

int launch_eloc_direct(const anqs_ham* H, const uint64_t* x, Count n_x, const NodeView& nodes, const AmpSrc& amp,
                       double* ere, double* eim, double* part, const StatsOut& so, cudaStream_t s) {
  const int splits = split_of(n_x.n, H->v.K);
  const unsigned grid = unsigned(std::min<uint64_t>(n_x.n * splits, 152 * 16));
  const bool tail = splits > 1 || n_x.n <= kTailStats;  // else the statistics are a launch of their own
  const StatsOut in_kernel = tail ? so : StatsOut{};
  ProfScope ps(PROF_TC_ELOC, s);
  auto go = [&](auto kern) {
    return launch_k(kern, dim3(grid), dim3(ET), 0, s, H->v, H->sv, nodes, x, n_x, splits, amp, ere, eim, part, in_kernel);
  };
  switch (amp.mode) {
    case AMP_SUM: ANQS_CUDA_LAUNCH("eloc_direct_kernel", go(eloc_direct_kernel<AMP_SUM>)); break;
    case AMP_BYJ: ANQS_CUDA_LAUNCH("eloc_direct_kernel", go(eloc_direct_kernel<AMP_BYJ>)); break;
    case AMP_TERMS: ANQS_CUDA_LAUNCH("eloc_direct_kernel", go(eloc_direct_kernel<AMP_TERMS>)); break;
    case AMP_ARRAY: ANQS_CUDA_LAUNCH("eloc_direct_kernel", go(eloc_direct_kernel<AMP_ARRAY>)); break;
  }
  if (!tail && so.counts) {
    const unsigned blocks = unsigned(std::min<uint64_t>((n_x.n + 511) / 512, SB));
    ANQS_CUDA_LAUNCH("stats_kernel", launch_k(stats_kernel, dim3(blocks), dim3(ET), 0, s, ere, eim, so.counts, n_x, part, so.ticket, so.stats));
  }
  return ANQS_OK;
}

}  // namespace anqs
