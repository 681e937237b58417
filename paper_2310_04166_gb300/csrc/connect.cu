// Connected set of a determinant: single and double excitations that keep
// N_alpha and N_beta, with Jordan-Wigner signs and Slater-Condon elements
// (Eq. local_energy_def, Eq. sq_hamiltonian, Sec. IV.A).
//
// One CTA per determinant l, or part of its list.  The excitations come in a
// fixed order (alpha singles, beta singles, alpha-alpha doubles, beta-beta
// doubles, alpha-beta doubles), so that the output needs no sort and every row
// has the same length K.  Integer work
// (x', sign, first slot) is exact; matrix elements are FP64.
#include <algorithm>

#include "excite.cuh"

namespace anqs {
namespace {

__device__ __forceinline__ uint32_t spin_occ(uint64_t x, int s, int n) {
  uint32_t m = 0;
  for (int p = 0; p < n; ++p) m |= uint32_t((x >> (2 * p + s)) & 1ull) << p;
  return m;
}

// position of the r-th (0-based) set bit of m
__device__ __forceinline__ int nth_bit(uint32_t m, int r) {
  for (int i = 0; i < r; ++i) m &= m - 1;
  return __ffs(m) - 1;
}

// Items bid, bid + nb, ... of the (sample, part) list, one per turn of the
// CTA: the sample's tables, then the part's excitations in the fixed order,
// consecutive threads on consecutive rows.  Bound by the 17 bytes written per
// row.  A thread that unranked its own row from the occupation bits spent
// about ten times the instructions of one that reads the tables: 8.6e6 rows
// (256 samples, 26 orbitals, 9 + 9 electrons) took 233 us.
__device__ __forceinline__ void connected_body(const HamView& hv, const uint64_t* __restrict__ xs, Count n_x,
                                               uint64_t* __restrict__ xp_out, double* __restrict__ h_out,
                                               uint8_t* __restrict__ j_out, int parts, uint64_t bid, uint64_t nb) {
  __shared__ Exc E;
  const uint32_t K = hv.K;
  const int n = hv.n;
  const uint64_t items = n_x.get() * uint64_t(parts);
  build_pairs(hv, E);
  const uint32_t nvirt[2] = {uint32_t(n - hv.na), uint32_t(n - hv.nb)}, nsb = hv.nsb;
  const FastDiv dsb = fast_div(nsb);
  const FastDiv dp[2] = {fast_div(nvirt[0] * (nvirt[0] - 1) / 2), fast_div(nvirt[1] * (nvirt[1] - 1) / 2)};
  const uint32_t ks = hv.nsa + hv.nsb, kd = ks + hv.ndaa + hv.ndbb;
  for (uint64_t it = bid; it < items; it += nb) {
    const uint64_t l = it / uint32_t(parts);
    const uint32_t part = uint32_t(it - l * uint32_t(parts));
    const uint32_t k0 = uint32_t(uint64_t(K) * part / uint32_t(parts)),
                   k1 = uint32_t(uint64_t(K) * (part + 1) / uint32_t(parts));
    build_exc<false>(hv, SectorView{}, __ldg(xs + l), E);
    const uint64_t x = E.x, row = l * K;
    auto put = [&](uint32_t k, uint64_t xn, double v, int j) {
      __stcs(reinterpret_cast<unsigned long long*>(xp_out) + row + k, xn);
      __stcs(h_out + row + k, v);
      if (j_out) j_out[row + k] = uint8_t(j);
    };
    if (!E.ok) {
      for (uint32_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) put(k, x, __longlong_as_double(0x7ff8000000000000ll), 255);
      continue;
    }
    for (uint32_t k = k0 + threadIdx.x; k < min(k1, ks); k += blockDim.x) {
      const int s = k < hv.nsa ? 0 : 1;
      const uint32_t e = s ? k - hv.nsa : k;
      const int i = E.si[s][e], a = E.sa[s][e];
      const double v = single_value(hv, E, s, i, a);
      put(k, x ^ (1ull << (2 * i + s)) ^ (1ull << (2 * a + s)), flip_sign(v, E.sgn[s][e]), min(i, a));
    }
    // same-spin doubles I<J -> A<B: [AI|BJ] - [AJ|BI]
    for (uint32_t k = max(k0, ks) + threadIdx.x; k < min(k1, kd); k += blockDim.x) {
      uint32_t r = k - ks;
      const int s = r < hv.ndaa ? 0 : 1;
      if (s) r -= hv.ndaa;
      const FastDiv d = s ? dp[1] : dp[0];
      const uint32_t q = fdiv(d, r), po = E.po[s][q], pv = E.pv[s][r - q * d.d];
      const int i = E.occ[s][po & 255u], j = E.occ[s][po >> 8], a = E.vir[s][pv & 255u], b = E.vir[s][pv >> 8];
      const double v = __ldg(hv.ga + ((a * n + i) * n + b) * n + j);
      put(k, x ^ (1ull << (2 * i + s)) ^ (1ull << (2 * j + s)) ^ (1ull << (2 * a + s)) ^ (1ull << (2 * b + s)),
          flip_sign(v, sign_ss(E, s, po, pv, s ? nvirt[1] : nvirt[0], i, j, a, b)), min(min(i, j), min(a, b)));
    }
    // opposite-spin doubles (I_a, A_a, I_b, A_b): [AI|BJ] (exchange term vanishes by spin)
    for (uint32_t k = max(k0, kd) + threadIdx.x; k < k1; k += blockDim.x) {
      const uint32_t r = k - kd, ea = fdiv(dsb, r), eb = r - ea * nsb;
      const int i = E.si[0][ea], a = E.sa[0][ea], j = E.si[1][eb], b = E.sa[1][eb];
      const double v = __ldg(hv.g + E.g[0][ea] + E.g[1][eb]);
      put(k, x ^ (1ull << (2 * i)) ^ (1ull << (2 * a)) ^ (2ull << (2 * j)) ^ (2ull << (2 * b)),
          flip_sign(v, sign_ab(E, ea, eb, i, a, j, b)), min(min(i, a), min(j, b)));
    }
  }
}

// The tensor-core local energy's control words (TC_CTL_WORDS, optional) are
// zeroed by block 0 of the call's first kernel, on the stream of the kernels
// that use them (sort histogram, statistics ticket).
__device__ __forceinline__ void zero_ctl(uint32_t* ctl) {
  if (ctl && blockIdx.x == 0 && threadIdx.x < TC_CTL_WORDS) ctl[threadIdx.x] = 0u;
}

__global__ void connected_kernel(HamView hv, const uint64_t* __restrict__ xs, Count n_x,
                                 uint64_t* __restrict__ xp_out, double* __restrict__ h_out,
                                 uint8_t* __restrict__ j_out, int parts, uint32_t* __restrict__ ctl) {
  ANQS_PDL_ENTRY();
  zero_ctl(ctl);
  connected_body(hv, xs, n_x, xp_out, h_out, j_out, parts, blockIdx.x, gridDim.x);
}

// <x|H|x> = E_nuc + sum_I h_ii + 1/2 sum_{I,J occ} ([II|JJ] - [IJ|JI]).
// One warp per determinant: lane i takes the occupied spin-orbital pairs
// (I, J) with I*N_occ + J = i mod 32, then the FP64 partial sums are reduced.
// one warp per sample, blocks bid = 0..nb-1
__device__ __forceinline__ void diagonal_body(const HamView& hv, const uint64_t* __restrict__ xs, Count n_x_,
                                              double* __restrict__ hdiag, uint64_t bid, uint64_t nb) {
  const int n = hv.n;
  const uint64_t n_x = n_x_.get();
  const int lane = threadIdx.x & 31;
  const uint64_t warps = nb * (blockDim.x >> 5);
  for (uint64_t l = bid * (blockDim.x >> 5) + (threadIdx.x >> 5); l < n_x; l += warps) {
    const uint64_t x = __ldg(xs + l);
    const uint32_t oa = spin_occ(x, 0, n), ob = spin_occ(x, 1, n);
    const bool ok = (__popc(oa) == hv.na) && (__popc(ob) == hv.nb) && (n == 32 || (x >> (2 * n)) == 0);
    // occupied spin-orbitals as (spatial index, spin)
    const int ne = hv.na + hv.nb;
    double e = 0.0;
    if (ok) {
      for (int t = lane; t < ne * ne + ne; t += 32) {
        if (t < ne * ne) {
          const int I = t / ne, J = t % ne;
          const int si = I < hv.na ? 0 : 1, sj = J < hv.na ? 0 : 1;
          const int i = nth_bit(si ? ob : oa, si ? I - hv.na : I);
          const int j = nth_bit(sj ? ob : oa, sj ? J - hv.na : J);
          e += 0.5 * Gint(hv, i, i, j, j);
          if (si == sj) e -= 0.5 * Gint(hv, i, j, j, i);
        } else {
          const int I = t - ne * ne;
          const int si = I < hv.na ? 0 : 1;
          const int i = nth_bit(si ? ob : oa, si ? I - hv.na : I);
          e += __ldg(hv.h + i * n + i);
        }
      }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane == 0) hdiag[l] = ok ? hv.e_nuc + e : __longlong_as_double(0x7ff8000000000000ll);
  }
}

__global__ void diagonal_kernel(HamView hv, const uint64_t* __restrict__ xs, Count n_x, double* __restrict__ hdiag,
                                uint32_t* __restrict__ ctl) {
  ANQS_PDL_ENTRY();
  zero_ctl(ctl);
  diagonal_body(hv, xs, n_x, hdiag, blockIdx.x, gridDim.x);
}

// [pq|rs] - [ps|rq] for the same-spin doubles and the pair energies of the
// diagonal, once per Hamiltonian
__global__ void integral_tables_kernel(int n, const double* __restrict__ g, double* __restrict__ ga,
                                       double* __restrict__ pair) {
  const uint32_t n1 = uint32_t(n), n2 = n1 * n1, all = n2 * n2;
  auto G = [&](uint32_t p, uint32_t q, uint32_t r, uint32_t s) { return g[(p * n1 + q) * n2 + r * n1 + s]; };
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < all; t += gridDim.x * blockDim.x) {
    const uint32_t p = t / (n2 * n1), q = t / n2 % n1, r = t / n1 % n1, s = t % n1;
    ga[t] = g[t] - G(p, s, r, q);
    if (t < n2) {
      const double J = 0.5 * G(r, r, s, s) + 0.5 * G(s, s, r, r);
      pair[t] = J - (0.5 * G(r, s, s, r) + 0.5 * G(s, r, r, s));
      pair[n2 + t] = J;
    }
  }
}

// the connected set on blocks [0, nb_c) and the diagonal on the rest, in one
// launch
__global__ void connected_diag_kernel(HamView hv, const uint64_t* __restrict__ xs, Count n_x,
                                      uint64_t* __restrict__ xp_out, double* __restrict__ h_out,
                                      uint8_t* __restrict__ j_out, double* __restrict__ hdiag, unsigned nb_c,
                                      int parts, uint32_t* __restrict__ ctl) {
  ANQS_PDL_ENTRY();
  zero_ctl(ctl);
  if (blockIdx.x < nb_c) connected_body(hv, xs, n_x, xp_out, h_out, j_out, parts, blockIdx.x, nb_c);
  else diagonal_body(hv, xs, n_x, hdiag, blockIdx.x - nb_c, gridDim.x - nb_c);
}

}  // namespace

int launch_integral_tables(int n, const double* g, double* ga, double* pair, cudaStream_t s) {
  const unsigned all = unsigned(n) * unsigned(n) * unsigned(n) * unsigned(n);
  const unsigned grid = std::min(152u * 8u, (all + 255u) / 256u);
  ANQS_CUDA_LAUNCH("integral_tables_kernel", launch_k(integral_tables_kernel, dim3(grid), dim3(256), 0, s, n, g, ga, pair));
  return ANQS_OK;
}

int launch_connected(const HamView& hv, const uint64_t* x, Count n_x, uint64_t* xp, double* hval,
                     uint8_t* first_slot, double* hdiag, cudaStream_t s, uint32_t* ctl) {
  const int threads = 256;
  // parts of a sample: enough items for 8 CTAs per SM, of at least 1,024 rows
  const uint64_t want = n_x.n ? (152 * 8 + n_x.n - 1) / n_x.n : 1;
  const int parts = int(std::max<uint64_t>(1, std::min<uint64_t>(want, hv.K / 1024)));
  uint64_t total = n_x.n * hv.K, bc = std::min<uint64_t>(n_x.n * parts, 152 * 16);
  if (total && hdiag) {
    uint64_t bd = (n_x.n + 7) / 8;
    if (bd > 152ull * 16) bd = 152ull * 16;
    ProfScope ps(PROF_CONNECT, s);
    ANQS_CUDA_LAUNCH("connected_diag_kernel", launch_k(connected_diag_kernel, dim3(unsigned(bc + bd)), dim3(threads), 0, s, hv, x, n_x, xp, hval, first_slot, hdiag, unsigned(bc), parts, ctl));
    return ANQS_OK;
  }
  if (total) {
    ProfScope ps(PROF_CONNECT, s);
    ANQS_CUDA_LAUNCH("connected_kernel", launch_k(connected_kernel, dim3(unsigned(bc)), dim3(threads), 0, s, hv, x, n_x, xp, hval, first_slot, parts, ctl));
    ctl = nullptr;
  }
  if (hdiag) {
    uint64_t blocks = (n_x.n + 7) / 8;  // 8 warps per CTA
    if (blocks > 152ull * 16) blocks = 152ull * 16;
    if (blocks == 0) blocks = 1;
    ProfScope ps(PROF_DIAGONAL, s);
    ANQS_CUDA_LAUNCH("diagonal_kernel", launch_k(diagonal_kernel, dim3(unsigned(blocks)), dim3(threads), 0, s, hv, x, n_x, hdiag, ctl));
  }
  return ANQS_OK;
}

}  // namespace anqs
