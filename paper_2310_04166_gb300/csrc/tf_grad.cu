// Hand-written adjoint of the masked log psi for the causal-transformer
// ansatz (FP32): the VMC gradient of Eq. grad_def is the vector-Jacobian
// product of sum_l [cot_la_l log|psi(x_l)| + cot_ph_l arg psi(x_l)] with the
// cotangents 2 w_l Re(E_loc,l - E) and 2 w_l Im(E_loc,l - E).
//
// The adjoint runs as batched passes over all rows (struct Rows: distinct
// prefixes of the samples, or (sample, position) pairs) with every activation
// of the forward stored in the workspace
// (or, when the workspace is too small for that, only the block inputs, each
// block's activations being recomputed from its input before its backward):
// embedding; per block LN1, q|k|v, causal attention (probabilities kept),
// output projection + residual, LN2, FFN (pre-activation kept) + residual;
// final LN and head.  The backward walks the same steps in reverse.  Matrix
// products go through one SGEMM tile (operands normal or transposed, optional
// bias, residual input, ReLU on an operand, ReLU'-mask of the result); weight
// gradients are products over the R rows, split along R across CTAs and
// accumulated with atomics into the flat gradient.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace anqs {
namespace {

// The rows of a pass, one per distinct prefix of the samples ("node", tree
// form) or one per (sample, position) (flat form).  Positions see only the
// tokens before them, so samples that share a prefix share its activations,
// and the cotangents of its outputs add up: 10,816 samples x 10 positions of
// the 20-qubit workload are 27,000 distinct prefixes.
struct Rows {
  const uint64_t* x;    // prefix bits (higher bits may be set)
  const uint8_t* lv;    // position
  const uint32_t* anc;  // [row][n]: rows of positions 0..lv of the same sequence (anc[lv] = row)
  Count rows;
  int n;
};

__global__ void flat_rows_kernel(const uint64_t* __restrict__ xs, Count rows_, int n, uint64_t* __restrict__ x,
                                 uint8_t* __restrict__ lv, uint32_t* __restrict__ anc) {
  ANQS_PDL_ENTRY();
  const uint64_t rows = rows_.get();
  for (uint64_t r = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; r < rows; r += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t s = r / n;
    const int t = int(r - s * n);
    x[r] = xs[s];
    lv[r] = uint8_t(t);
    for (int u = 0; u <= t; ++u) anc[r * n + u] = uint32_t(s * n + u);
  }
}

__global__ void tree_rows_kernel(SectorView sv, NodeView nv, uint8_t* __restrict__ lv, uint32_t* __restrict__ anc) {
  ANQS_PDL_ENTRY();
  const int n = sv.n;
  const uint32_t rows = __ldcg(nv.off + n);
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += gridDim.x * blockDim.x) {
    const uint64_t x = __ldcg(reinterpret_cast<const unsigned long long*>(nv.x) + r);
    const uint32_t a = even_bits(x), b = even_bits(x >> 1);
    int p = 0;
    while (r >= __ldcg(nv.off + p + 1)) ++p;
    lv[r] = uint8_t(p);
    for (int u = 0; u < p; ++u) anc[size_t(r) * n + u] = node_id(sv, nv, u, prefix_index(sv, u, a, b));
    anc[size_t(r) * n + p] = r;
  }
}

constexpr int BM = 64, BN = 64, BK = 32, GT = 128;
constexpr int LV = BM * BK / 4 / GT;  // 4-vectors of A, and of B, that a thread loads per K step
static_assert(BM == BN, "one index for both operands");

// A matrix whose rows come in segments (the q, k and v weights lie one
// behind the other with their biases between): row i starts at
// (i / seg) * stride + (i % seg) * ld.
struct Seg {
  int seg;
  size_t stride;
};

struct Gm {
  const float* A;
  int lda;
  const float* B;
  int ldb;
  Seg sb;            // segments of B's rows
  float* C;
  int ldc;
  Seg sc;            // segments of C's rows (weight products)
  const float* Cin;  // residual input (may alias C), or null
  int ldcin;
  const float* bias;  // per column (segments as B's), or null
  const float* mask;  // result zeroed where mask <= 0, or null
  int ldmask;
  float* colsum;      // += the sums of A's columns (weight products: the bias gradient; segments as C's), or null
  Count M, K;         // M (rows) and K may be device counts
  int N;
  int relu_a, relu_b, atomic;
  int b_vec;          // B and bias are 16-byte aligned (parameters may be any float tensor, say a slice)
  int c_vec;          // C is
  uint64_t k_chunk;   // split-K: K range per blockIdx.z
};

__device__ __forceinline__ float4 ld4(const float* p, int vec) {
  if (vec) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[1], p[2], p[3]);
}

__device__ __forceinline__ size_t seg_row(const Seg& s, int i, int ld) {
  return s.seg ? size_t(i / s.seg) * s.stride + size_t(i % s.seg) * ld : size_t(i) * ld;
}

// c += a b of two floats each (one instruction, the rounding of two fmaf)
__device__ __forceinline__ void fma2(uint64_t a, uint64_t b, uint64_t& c) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t both(float v) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
  return r;
}

struct GmSmem {
  float A[2][BK][BM + 4], B[2][BK][BN + 4];
};

// C[m][n] = sum_k opA(m, k) opB(k, n), opA(m, k) = A[m][k] (TA: A[k][m]),
// opB(k, n) = B[k][n] (TB: B[n][k]); tile (bx, by), K part bz.  64 x 64 tile
// per CTA of 128 threads, 8 x 4 per thread (3 16-byte shared loads for 32
// FMAs, paired along the rows; a 4 x 4 tile is bound by its shared loads), the
// next K step's operands loaded to registers while this one runs.  A CTA waits
// for those loads in every step (so the steps are 32 deep), and what counts is
// how many share an SM: with
// 128 x 64 tiles the 26,000 rows of the 20-qubit workload were 205 CTAs of a
// 64-column product, and half of every tile of a 64-row weight product empty.
// All leading dimensions, segments and widths are multiples of 4 floats.
template <bool TA, bool TB>
__device__ __forceinline__ void gemm_tile(const Gm& g, unsigned bx, unsigned by, unsigned bz, GmSmem& sm) {
  const uint64_t M = g.M.get(), K = g.K.get();
  const uint64_t m0 = uint64_t(by) * BM;
  const int n0 = bx * BN, tid = threadIdx.x;
  if (m0 >= M) return;
  const uint64_t k_lo = uint64_t(bz) * g.k_chunk;
  if (k_lo >= K && !(k_lo == 0)) return;
  const uint64_t k_hi = k_lo + g.k_chunk < K ? k_lo + g.k_chunk : K;
  const int tx = tid % 16, ty = tid / 16;
  float4 ra[LV], rb[LV];
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  auto load = [&](uint64_t k0) {
#pragma unroll
    for (int i = 0; i < LV; ++i) {
      const int e = tid + GT * i;
      ra[i] = rb[i] = zero;
      if (TA) {  // [k][m]: vectors along m
        const uint64_t m = m0 + uint64_t(e % 16) * 4, k = k0 + e / 16;
        if (k < k_hi) {
          const float* p = g.A + k * g.lda + m;
          if (m + 4 <= M) ra[i] = *reinterpret_cast<const float4*>(p);
          else {
            if (m < M) ra[i].x = p[0];
            if (m + 1 < M) ra[i].y = p[1];
            if (m + 2 < M) ra[i].z = p[2];
          }
        }
      } else {  // [m][k]: vectors along k
        const uint64_t m = m0 + e / (BK / 4), k = k0 + uint64_t(e % (BK / 4)) * 4;
        if (m < M && k + 4 <= k_hi) ra[i] = *reinterpret_cast<const float4*>(g.A + m * g.lda + k);
      }
      if (g.relu_a) {
        ra[i].x = fmaxf(ra[i].x, 0.f), ra[i].y = fmaxf(ra[i].y, 0.f);
        ra[i].z = fmaxf(ra[i].z, 0.f), ra[i].w = fmaxf(ra[i].w, 0.f);
      }
      if (TB) {  // [n][k]: vectors along k
        const int n = n0 + e / (BK / 4);
        const uint64_t k = k0 + uint64_t(e % (BK / 4)) * 4;
        if (n < g.N && k + 4 <= k_hi) rb[i] = ld4(g.B + seg_row(g.sb, n, g.ldb) + k, g.b_vec);
      } else {  // [k][n]: vectors along n
        const int n = n0 + (e % 16) * 4;
        const uint64_t k = k0 + e / 16;
        if (k < k_hi && n < g.N) rb[i] = ld4(g.B + (g.sb.seg ? seg_row(g.sb, int(k), g.ldb) : k * g.ldb) + n, g.b_vec);
      }
      if (g.relu_b) {
        rb[i].x = fmaxf(rb[i].x, 0.f), rb[i].y = fmaxf(rb[i].y, 0.f);
        rb[i].z = fmaxf(rb[i].z, 0.f), rb[i].w = fmaxf(rb[i].w, 0.f);
      }
    }
  };
  auto store = [&](int b) {
#pragma unroll
    for (int i = 0; i < LV; ++i) {
      const int e = tid + GT * i, r = e / (BK / 4), k = (e % (BK / 4)) * 4;
      if (TA) *reinterpret_cast<float4*>(&sm.A[b][e / 16][(e % 16) * 4]) = ra[i];
      else sm.A[b][k][r] = ra[i].x, sm.A[b][k + 1][r] = ra[i].y, sm.A[b][k + 2][r] = ra[i].z, sm.A[b][k + 3][r] = ra[i].w;
      if (TB) sm.B[b][k][r] = rb[i].x, sm.B[b][k + 1][r] = rb[i].y, sm.B[b][k + 2][r] = rb[i].z, sm.B[b][k + 3][r] = rb[i].w;
      else *reinterpret_cast<float4*>(&sm.B[b][e / 16][(e % 16) * 4]) = rb[i];
    }
  };
  uint64_t acc2[4][4] = {};  // rows 2 i and 2 i + 1 of the thread's eight
  float cs = 0.f;
  const bool sums = g.colsum && bx == 0;
  load(k_lo);
  store(0);
  __syncthreads();
  int b = 0;
  for (uint64_t k0 = k_lo; k0 < k_hi; k0 += BK) {
    const bool more = k0 + BK < k_hi;
    if (more) load(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(&sm.A[b][kk][ty * 8]);
      const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(&sm.A[b][kk][ty * 8 + 4]);
      const float4 bb = *reinterpret_cast<const float4*>(&sm.B[b][kk][tx * 4]);
      const uint64_t av[4] = {a0.x, a0.y, a1.x, a1.y}, bv[4] = {both(bb.x), both(bb.y), both(bb.z), both(bb.w)};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) fma2(av[i], bv[j], acc2[i][j]);
    }
    if (sums && tid < BM)
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) cs += sm.A[b][kk][tid];
    if (more) store(b ^ 1);
    __syncthreads();
    b ^= 1;
  }
  if (sums && tid < BM && m0 + tid < M) atomicAdd(g.colsum + seg_row(g.sc, int(m0 + tid), 1), cs);
  const int n = n0 + tx * 4;
  if (n >= g.N) return;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint64_t m = m0 + ty * 8 + i;
    if (m >= M) break;
    float a[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) a[j] = __uint_as_float(uint32_t(acc2[i / 2][j] >> (32 * (i & 1))));
    float4 v = make_float4(a[0], a[1], a[2], a[3]);
    float* c = g.C + (g.sc.seg ? seg_row(g.sc, int(m), g.ldc) : m * g.ldc) + n;
    if (g.atomic) {
      if (g.c_vec) {
        atomicAdd(reinterpret_cast<float4*>(c), v);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) atomicAdd(c + j, a[j]);
      }
      continue;
    }
    if (g.bias) {
      const float4 t = ld4(g.bias + seg_row(g.sb, n, 1), g.b_vec);
      v.x += t.x, v.y += t.y, v.z += t.z, v.w += t.w;
    }
    if (g.Cin) {
      const float4 t = *reinterpret_cast<const float4*>(g.Cin + m * g.ldcin + n);
      v.x += t.x, v.y += t.y, v.z += t.z, v.w += t.w;
    }
    if (g.mask) {
      const float4 t = *reinterpret_cast<const float4*>(g.mask + m * g.ldmask + n);
      v.x = t.x > 0.f ? v.x : 0.f, v.y = t.y > 0.f ? v.y : 0.f;
      v.z = t.z > 0.f ? v.z : 0.f, v.w = t.w > 0.f ? v.w : 0.f;
    }
    *reinterpret_cast<float4*>(c) = v;
  }
}

// one product with a transposed B (the forward pass)
__global__ void __launch_bounds__(GT, 4) sgemm_kernel(Gm g) {
  ANQS_PDL_ENTRY();
  __shared__ __align__(16) GmSmem sm;
  gemm_tile<false, true>(g, blockIdx.x, blockIdx.y, 0, sm);
}

// A layer's two products of the backward pass, both from the cotangents of its
// outputs: the input's cotangents d = dY W (CTAs from nw on, dx tiles wide) and
// the weight gradient w += dY^T X (CTAs below nw: wx tiles wide, wy high, parts
// of the rows).  In one launch, because neither fills the GPU by itself; the
// weight product's CTAs run longest and come first.
__global__ void __launch_bounds__(GT, 4) sgemm_bwd_kernel(Gm w, Gm d, unsigned nw, unsigned wx, unsigned wy, unsigned dx) {
  ANQS_PDL_ENTRY();
  __shared__ __align__(16) GmSmem sm;
  if (blockIdx.x < nw) {
    const unsigned t = blockIdx.x % (wx * wy);
    gemm_tile<true, false>(w, t % wx, t / wx, blockIdx.x / (wx * wy), sm);
  } else {
    const unsigned t = blockIdx.x - nw;
    gemm_tile<false, false>(d, t % dx, t / dx, 0, sm);
  }
}

// h0[r] = tok[token(r)] + pos[position of r]
__global__ void embed_kernel(TfView m, Rows R, float* __restrict__ h0) {
  ANQS_PDL_ENTRY();
  const uint64_t rows = R.rows.get();
  const int D = m.d;
  const float* tok = m.params;
  const float* pos = m.params + 5 * size_t(D);
  for (uint64_t idx = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; idx < rows * D;
       idx += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t r = idx / D;
    const int c = int(idx % D), t = R.lv[r];
    const int token = t == 0 ? 4 : int((R.x[r] >> (2 * (t - 1))) & 3ull);
    h0[idx] = tok[token * D + c] + pos[t * D + c];
  }
}

// y = xhat * g + b, xhat = (x - mean) rs, one warp per row; keeps xhat and rs
template <int D>
__global__ void ln_fwd_kernel(const float* __restrict__ X, const float* __restrict__ gam,
                              const float* __restrict__ bet, float* __restrict__ Xh, float* __restrict__ Y,
                              float* __restrict__ RS, Count rows_) {
  ANQS_PDL_ENTRY();
  constexpr int E = D / 32;
  const uint64_t rows = rows_.get();
  const int lane = threadIdx.x & 31;
  for (uint64_t r = (blockIdx.x * uint64_t(blockDim.x) + threadIdx.x) >> 5; r < rows;
       r += (uint64_t(gridDim.x) * blockDim.x) >> 5) {
    float v[E], s = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      v[e] = X[r * D + lane + 32 * e];
      s += v[e];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float mean = s / float(D);
    float q = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      v[e] -= mean;
      q = fmaf(v[e], v[e], q);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    const float rs = 1.0f / sqrtf(q / float(D) + 1e-5f);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int c = lane + 32 * e;
      const float xh = v[e] * rs;
      Xh[r * D + c] = xh;
      Y[r * D + c] = fmaf(xh, gam[c], bet[c]);
    }
    if (lane == 0) RS[r] = rs;
  }
}

// dX = dRes + rs (gy - mean(gy) - xhat mean(gy xhat)), gy = dY * g (dRes may
// alias dX or be null); dg += sum_r dY xhat, db += sum_r dY
template <int D>
__global__ void __launch_bounds__(256) ln_bwd_kernel(const float* __restrict__ dY, const float* __restrict__ Xh,
                                                     const float* __restrict__ gam, const float* __restrict__ RS,
                                                     const float* dRes, float* dX, float* __restrict__ dg,
                                                     float* __restrict__ db, Count rows_) {
  ANQS_PDL_ENTRY();
  constexpr int E = D / 32;
  __shared__ float s_dg[D], s_db[D];
  for (int c = threadIdx.x; c < D; c += blockDim.x) s_dg[c] = s_db[c] = 0.f;
  __syncthreads();
  const uint64_t rows = rows_.get();
  const int lane = threadIdx.x & 31;
  float pg[E] = {}, pb[E] = {};
  for (uint64_t r = (blockIdx.x * uint64_t(blockDim.x) + threadIdx.x) >> 5; r < rows;
       r += (uint64_t(gridDim.x) * blockDim.x) >> 5) {
    float dy[E], xh[E], gy[E], s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int c = lane + 32 * e;
      dy[e] = dY[r * D + c];
      xh[e] = Xh[r * D + c];
      gy[e] = dy[e] * gam[c];
      s1 += gy[e];
      s2 = fmaf(gy[e], xh[e], s2);
      pg[e] = fmaf(dy[e], xh[e], pg[e]);
      pb[e] += dy[e];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    const float m1 = s1 / float(D), m2 = s2 / float(D), rs = RS[r];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int c = lane + 32 * e;
      float v = rs * (gy[e] - m1 - xh[e] * m2);
      if (dRes) v += dRes[r * D + c];
      dX[r * D + c] = v;
    }
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {
    atomicAdd(&s_dg[lane + 32 * e], pg[e]);
    atomicAdd(&s_db[lane + 32 * e], pb[e]);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < D; c += blockDim.x) {
    atomicAdd(dg + c, s_dg[c]);
    atomicAdd(db + c, s_db[c]);
  }
}

// Causal attention of one (row, head) per thread over the row's ancestors;
// keeps the probabilities P[r][h][u].  qkv [row][3 D].  The heads of a row are
// neighbouring threads, so a warp reads whole key and value rows.  E4: the
// head width in 4-vectors, held in registers (0: any width, one element or
// 4-vector at a time).  Scores wait in shared memory: through global memory
// (P itself) every one was written and read back three times, and the kernel
// waited for that (26,000 rows x 4 heads: 30 us).
constexpr int AT = 128;  // threads of the attention kernels
template <int E4>
__global__ void __launch_bounds__(AT) attn_fwd_kernel(const float* __restrict__ qkv, float* __restrict__ P,
                                                      float* __restrict__ O, int D, int H, Rows R) {
  ANQS_PDL_ENTRY();
  __shared__ float sp[32][AT];
  const uint64_t rows = R.rows.get();
  const int dh = D / H, n = R.n, tid = threadIdx.x;
  const float scale = 1.0f / sqrtf(float(dh));
  for (uint64_t task = blockIdx.x * uint64_t(blockDim.x) + tid; task < rows * H; task += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t r = task / H;
    const int hd = int(task - r * H), t = R.lv[r];
    const float* q = qkv + r * 3 * D + hd * dh;
    const uint32_t* anc = R.anc + r * n;
    float* prow = P + task * n;
    float mx = -INFINITY;
    float4 qv[E4 ? E4 : 1];
#pragma unroll
    for (int e = 0; e < E4; ++e) qv[e] = *reinterpret_cast<const float4*>(q + 4 * e);
#pragma unroll 2
    for (int u = 0; u <= t; ++u) {
      const float* k = qkv + size_t(anc[u]) * 3 * D + D + hd * dh;
      float dot = 0.f;
      if constexpr (E4 > 0) {
#pragma unroll
        for (int e = 0; e < E4; ++e) {
          const float4 a = qv[e], b = *reinterpret_cast<const float4*>(k + 4 * e);
          dot = fmaf(a.x, b.x, dot), dot = fmaf(a.y, b.y, dot), dot = fmaf(a.z, b.z, dot), dot = fmaf(a.w, b.w, dot);
        }
      } else if (dh % 4 == 0) {
        for (int e = 0; e < dh; e += 4) {
          const float4 a = *reinterpret_cast<const float4*>(q + e), b = *reinterpret_cast<const float4*>(k + e);
          dot = fmaf(a.x, b.x, dot), dot = fmaf(a.y, b.y, dot), dot = fmaf(a.z, b.z, dot), dot = fmaf(a.w, b.w, dot);
        }
      } else {
        for (int e = 0; e < dh; ++e) dot = fmaf(q[e], k[e], dot);
      }
      sp[u][tid] = dot * scale;
      mx = fmaxf(mx, dot * scale);
    }
    float sum = 0.f;
    for (int u = 0; u <= t; ++u) {
      const float p = expf(sp[u][tid] - mx);
      sp[u][tid] = p;
      sum += p;
    }
    const float inv = 1.0f / sum;
    float* o = O + r * D + hd * dh;
    if constexpr (E4 > 0) {
      float4 acc[E4] = {};
#pragma unroll 2
      for (int u = 0; u <= t; ++u) {
        const float p = sp[u][tid] * inv;
        prow[u] = p;
        const float* v = qkv + size_t(anc[u]) * 3 * D + 2 * D + hd * dh;
#pragma unroll
        for (int e = 0; e < E4; ++e) {
          const float4 w = *reinterpret_cast<const float4*>(v + 4 * e);
          acc[e].x = fmaf(p, w.x, acc[e].x), acc[e].y = fmaf(p, w.y, acc[e].y);
          acc[e].z = fmaf(p, w.z, acc[e].z), acc[e].w = fmaf(p, w.w, acc[e].w);
        }
      }
#pragma unroll
      for (int e = 0; e < E4; ++e) *reinterpret_cast<float4*>(o + 4 * e) = acc[e];
    } else {
      for (int u = 0; u <= t; ++u) prow[u] = sp[u][tid] = sp[u][tid] * inv;
      if (dh % 4 == 0) {
        for (int e = 0; e < dh; e += 4) {
          float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int u = 0; u <= t; ++u) {
            const float p = sp[u][tid];
            const float4 w = *reinterpret_cast<const float4*>(qkv + size_t(anc[u]) * 3 * D + 2 * D + hd * dh + e);
            a.x = fmaf(p, w.x, a.x), a.y = fmaf(p, w.y, a.y), a.z = fmaf(p, w.z, a.z), a.w = fmaf(p, w.w, a.w);
          }
          *reinterpret_cast<float4*>(o + e) = a;
        }
        continue;
      }
      for (int e = 0; e < dh; ++e) {
        float a = 0.f;
        for (int u = 0; u <= t; ++u) a = fmaf(sp[u][tid], qkv[size_t(anc[u]) * 3 * D + 2 * D + hd * dh + e], a);
        o[e] = a;
      }
    }
  }
}

// Backward of the attention of one (row, head): dS[r][h][u] (with the score
// scale) and dQ.  dP_u = dO . V_u; dS_u = P_u (dP_u - sum_u' P_u' dP_u') scale.
// The row's dQ | dK | dV slots hold dQ after it; dK and dV are zeroed here for
// attn_bwd_kv_kernel.
template <int E4>
__global__ void __launch_bounds__(AT) attn_bwd_q_kernel(const float* __restrict__ qkv, const float* __restrict__ P,
                                                        const float* __restrict__ dO, float* __restrict__ dS,
                                                        float* __restrict__ dqkv, int D, int H, Rows R) {
  ANQS_PDL_ENTRY();
  __shared__ float sp[32][AT];
  const uint64_t rows = R.rows.get();
  const int dh = D / H, n = R.n, tid = threadIdx.x;
  const float scale = 1.0f / sqrtf(float(dh));
  for (uint64_t task = blockIdx.x * uint64_t(blockDim.x) + tid; task < rows * H; task += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t r = task / H;
    const int hd = int(task - r * H), t = R.lv[r];
    const uint32_t* anc = R.anc + r * n;
    const float* prow = P + task * n;
    float* srow = dS + task * n;
    const float* go = dO + r * D + hd * dh;
    float dot = 0.f;
    float4 gv[E4 ? E4 : 1];
#pragma unroll
    for (int e = 0; e < E4; ++e) gv[e] = *reinterpret_cast<const float4*>(go + 4 * e);
#pragma unroll 2
    for (int u = 0; u <= t; ++u) {
      const float* v = qkv + size_t(anc[u]) * 3 * D + 2 * D + hd * dh;
      float a = 0.f;
      if constexpr (E4 > 0) {
#pragma unroll
        for (int e = 0; e < E4; ++e) {
          const float4 x = gv[e], y = *reinterpret_cast<const float4*>(v + 4 * e);
          a = fmaf(x.x, y.x, a), a = fmaf(x.y, y.y, a), a = fmaf(x.z, y.z, a), a = fmaf(x.w, y.w, a);
        }
      } else if (dh % 4 == 0) {
        for (int e = 0; e < dh; e += 4) {
          const float4 x = *reinterpret_cast<const float4*>(go + e), y = *reinterpret_cast<const float4*>(v + e);
          a = fmaf(x.x, y.x, a), a = fmaf(x.y, y.y, a), a = fmaf(x.z, y.z, a), a = fmaf(x.w, y.w, a);
        }
      } else {
        for (int e = 0; e < dh; ++e) a = fmaf(go[e], v[e], a);
      }
      sp[u][tid] = a;
      dot = fmaf(prow[u], a, dot);
    }
    float* gq = dqkv + r * 3 * D + hd * dh;
    if constexpr (E4 > 0) {
      float4 acc[E4] = {};
#pragma unroll 2
      for (int u = 0; u <= t; ++u) {
        const float ds = prow[u] * (sp[u][tid] - dot) * scale;
        srow[u] = ds;
        const float* k = qkv + size_t(anc[u]) * 3 * D + D + hd * dh;
#pragma unroll
        for (int e = 0; e < E4; ++e) {
          const float4 w = *reinterpret_cast<const float4*>(k + 4 * e);
          acc[e].x = fmaf(ds, w.x, acc[e].x), acc[e].y = fmaf(ds, w.y, acc[e].y);
          acc[e].z = fmaf(ds, w.z, acc[e].z), acc[e].w = fmaf(ds, w.w, acc[e].w);
        }
      }
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int e = 0; e < E4; ++e) {
        *reinterpret_cast<float4*>(gq + 4 * e) = acc[e];
        *reinterpret_cast<float4*>(gq + D + 4 * e) = zero;
        *reinterpret_cast<float4*>(gq + 2 * D + 4 * e) = zero;
      }
    } else {
      for (int u = 0; u <= t; ++u) srow[u] = sp[u][tid] = prow[u] * (sp[u][tid] - dot) * scale;
      if (dh % 4 == 0) {
        for (int e = 0; e < dh; e += 4) {
          float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int u = 0; u <= t; ++u) {
            const float p = sp[u][tid];
            const float4 w = *reinterpret_cast<const float4*>(qkv + size_t(anc[u]) * 3 * D + D + hd * dh + e);
            a.x = fmaf(p, w.x, a.x), a.y = fmaf(p, w.y, a.y), a.z = fmaf(p, w.z, a.z), a.w = fmaf(p, w.w, a.w);
          }
          *reinterpret_cast<float4*>(gq + e) = a;
          *reinterpret_cast<float4*>(gq + D + e) = make_float4(0.f, 0.f, 0.f, 0.f);
          *reinterpret_cast<float4*>(gq + 2 * D + e) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        continue;
      }
      for (int e = 0; e < dh; ++e) {
        float a = 0.f;
        for (int u = 0; u <= t; ++u) a = fmaf(sp[u][tid], qkv[size_t(anc[u]) * 3 * D + D + hd * dh + e], a);
        gq[e] = a;
        gq[D + e] = 0.f;
        gq[2 * D + e] = 0.f;
      }
    }
  }
}

// dK_u = sum over the rows r below key u of dS[r][u] q_r, dV_u = the same of
// P[r][u] dO_r.  A CTA takes KVR consecutive rows and one ancestor level;
// thread = column (dK's, then dV's).  Rows of one level are ordered so that
// neighbours mostly share their ancestors: the sums stay in a register while
// the ancestor is the same and are added to its row when it changes (one add
// per run instead of one per (row, key)).
constexpr int KVR = 64;
__global__ void attn_bwd_kv_kernel(const float* __restrict__ qkv, const float* __restrict__ P,
                                   const float* __restrict__ dO, const float* __restrict__ dS,
                                   float* __restrict__ dqkv, int D, int H, Rows R) {
  ANQS_PDL_ENTRY();
  const uint64_t rows = R.rows.get(), r0 = uint64_t(blockIdx.x) * KVR;
  if (r0 >= rows) return;
  const uint64_t r1 = r0 + KVR < rows ? r0 + KVR : rows;
  const int n = R.n, u = blockIdx.y, dh = D / H;
  __shared__ uint32_t key[KVR];
  for (int i = threadIdx.x; i < KVR; i += blockDim.x) {
    const uint64_t r = r0 + i;
    key[i] = r < r1 && R.lv[r] >= u ? R.anc[r * n + u] : 0xffffffffu;
  }
  __syncthreads();
  for (int col = threadIdx.x; col < 2 * D; col += blockDim.x) {
    const int kv = col / D, c = col - kv * D, hd = c / dh;
    const int ldw = H * n, ldv = kv ? D : 3 * D;
    const float* w = (kv ? P : dS) + hd * n + u + r0 * ldw;
    const float* v = (kv ? dO + c : qkv + c) + r0 * ldv;
    uint32_t cur = 0xffffffffu;
    float acc = 0.f;
    for (int i0 = 0; i0 < int(r1 - r0); i0 += 8) {  // eight rows' loads in flight (rows beyond have no key)
      float wr[8], vr[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const bool on = key[i0 + e] != 0xffffffffu;
        wr[e] = on ? w[e * ldw] : 0.f;
        vr[e] = on ? v[e * ldv] : 0.f;
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint32_t k = key[i0 + e];
        if (k != cur) {
          if (cur != 0xffffffffu) atomicAdd(dqkv + size_t(cur) * 3 * D + (1 + kv) * D + c, acc);
          cur = k;
          acc = 0.f;
        }
        if (k != 0xffffffffu) acc = fmaf(wr[e], vr[e], acc);
      }
      w += 8 * ldw;
      v += 8 * ldv;
    }
    if (cur != 0xffffffffu) atomicAdd(dqkv + size_t(cur) * 3 * D + (1 + kv) * D + c, acc);
  }
}

// Cotangents of every row's slot terms: cot[r][v] += cl, cot[r][4 + v] += cp
// over the samples whose path takes outcome v at row r (FP64: a root row adds
// up all samples).  Samples outside the sector add nothing.  nv.packed null:
// flat rows.
__global__ void cot_rows_kernel(HamView hv, SectorView sv, NodeView nv, const uint64_t* __restrict__ x, Count nx_,
                                const float* __restrict__ cl, const float* __restrict__ cp, double* __restrict__ cot) {
  ANQS_PDL_ENTRY();
  const uint64_t nx = nx_.get();
  const int n = hv.n, lane = threadIdx.x & 31;
  for (uint64_t s0 = (blockIdx.x * uint64_t(blockDim.x) + threadIdx.x) - lane; s0 < nx;
       s0 += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t s = s0 + lane;
    const uint64_t xs = s < nx ? x[s] : 0ull;
    bool dead = s >= nx || (n < 32 && (xs >> (2 * n)) != 0);
    for (int p = 0; p < n; ++p) {
      const uint64_t below = xs & ((1ull << (2 * p)) - 1ull);
      const unsigned pm = slot_mask(hv, p, __popcll(below & 0x5555555555555555ull),
                                    __popcll(below & 0xAAAAAAAAAAAAAAAAull), xs);
      if (!((pm >> ((xs >> (2 * p)) & 3ull)) & 1u)) dead = true;
    }
    const double l = dead ? 0.0 : double(cl[s]), c = dead ? 0.0 : double(cp[s]);
    const uint32_t a = even_bits(xs), b = even_bits(xs >> 1);
    for (int p = 0; p < n; ++p) {
      const int v = int((xs >> (2 * p)) & 3ull);
      uint32_t row = 0xffffffffu;
      if (!dead) row = nv.packed ? node_id(sv, nv, p, prefix_index(sv, p, a, b)) : uint32_t(s * n + p);
      if (p < 4 && nv.packed) {  // few rows take all samples: one add per warp and row
        const unsigned peers = __match_any_sync(0xffffffffu, dead ? 0xffffffffu : row * 4 + v);
        double tl = 0.0, tc = 0.0;
        const int lead = __ffs(peers) - 1;
        for (int o = 0; o < 32; ++o) {
          const double ol = __shfl_sync(0xffffffffu, l, o), oc = __shfl_sync(0xffffffffu, c, o);
          if ((peers >> o) & 1u) tl += ol, tc += oc;
        }
        if (lane == lead && !dead) {
          atomicAdd(cot + size_t(row) * 8 + v, tl);
          atomicAdd(cot + size_t(row) * 8 + 4 + v, tc);
        }
      } else if (!dead) {
        atomicAdd(cot + size_t(row) * 8 + v, l);
        atomicAdd(cot + size_t(row) * 8 + 4 + v, c);
      }
    }
  }
}

// head cotangents d out8[r] from the masked log-softmax of the row's slot:
// d l_u = (sum of cl with outcome u - p_u sum of cl) / 2, d phi_u = sum of cp with outcome u
__global__ void head_dout_kernel(HamView hv, Rows R, const float* __restrict__ out8, const double* __restrict__ cot,
                                 float* __restrict__ dout8) {
  ANQS_PDL_ENTRY();
  const uint64_t rows = R.rows.get();
  for (uint64_t r = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; r < rows; r += uint64_t(gridDim.x) * blockDim.x) {
    const int p = R.lv[r];
    const uint64_t x = R.x[r], below = x & ((1ull << (2 * p)) - 1ull);
    const unsigned mk = norm_mask(hv, p, slot_mask(hv, p, __popcll(below & 0x5555555555555555ull),
                                                   __popcll(below & 0xAAAAAAAAAAAAAAAAull), x));
    const float* o = out8 + r * 8;
    const double* c = cot + r * 8;
    float* d = dout8 + r * 8;
    float mx = -INFINITY;
    for (int u = 0; u < 4; ++u)
      if ((mk >> u) & 1u) mx = fmaxf(mx, o[u]);
    float e[4], sum = 0.f;
    double tot = 0.0;
    for (int u = 0; u < 4; ++u) {
      e[u] = ((mk >> u) & 1u) ? expf(o[u] - mx) : 0.f;
      sum += e[u];
      tot += c[u];
    }
    for (int u = 0; u < 4; ++u) {
      // a row without an allowed outcome takes no samples (outputs that are not finite give NaN)
      d[u] = mk ? float(0.5 * (c[u] - double(e[u] / sum) * tot)) : 0.f;
      d[4 + u] = float(c[4 + u]);
    }
  }
}

// gtok[token(r)] += dH0[r], gpos[position of r] += dH0[r]: thread = column,
// a CTA's rows in order, one add per token and per run of equal positions.
// The rows' positions and tokens come first, so that eight rows' loads are in
// flight (a row at a time, waiting for its position, its token and its value
// in turn, took 60 us for 26,000 rows).
constexpr int EBR = 64;
__global__ void embed_bwd_kernel(TfView m, Rows R, const float* __restrict__ dh0, float* __restrict__ gtok,
                                 float* __restrict__ gpos) {
  ANQS_PDL_ENTRY();
  __shared__ uint8_t s_pos[EBR], s_tok[EBR];
  const uint64_t rows = R.rows.get(), r0 = uint64_t(blockIdx.x) * EBR;
  if (r0 >= rows) return;
  const int D = m.d, cnt = int(r0 + EBR < rows ? EBR : rows - r0);
  for (int i = threadIdx.x; i < EBR; i += blockDim.x) {
    const int t = i < cnt ? R.lv[r0 + i] : 255;
    s_pos[i] = uint8_t(t);
    s_tok[i] = uint8_t(i >= cnt ? 5 : t == 0 ? 4 : int((R.x[r0 + i] >> (2 * (t - 1))) & 3ull));
  }
  __syncthreads();
  for (int c = threadIdx.x; c < D; c += blockDim.x) {
    float tk[5] = {}, ps = 0.f;
    int cur = s_pos[0];
    for (int i0 = 0; i0 < cnt; i0 += 8) {
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = i0 + e < cnt ? dh0[(r0 + i0 + e) * D + c] : 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (i0 + e >= cnt) break;
        const int t = s_pos[i0 + e], token = s_tok[i0 + e];
        if (t != cur) {
          atomicAdd(gpos + cur * D + c, ps);
          cur = t;
          ps = 0.f;
        }
        ps += v[e];
#pragma unroll
        for (int k = 0; k < 5; ++k) tk[k] += k == token ? v[e] : 0.f;
      }
    }
    atomicAdd(gpos + cur * D + c, ps);
#pragma unroll
    for (int k = 0; k < 5; ++k)
      if (tk[k] != 0.f) atomicAdd(gtok + k * D + c, tk[k]);
  }
}

// out[c] += sum_r X[r][c] for c < 8
__global__ void __launch_bounds__(256) colsum8_kernel(const float* __restrict__ X, Count rows_, float* __restrict__ out) {
  ANQS_PDL_ENTRY();
  const uint64_t rows = rows_.get();
  const int c = threadIdx.x & 7;
  float s = 0.f;
  for (uint64_t r = (blockIdx.x * uint64_t(blockDim.x) + threadIdx.x) >> 3; r < rows; r += (uint64_t(gridDim.x) * blockDim.x) >> 3)
    s += X[r * 8 + c];
  s += __shfl_xor_sync(0xffffffffu, s, 8);
  s += __shfl_xor_sync(0xffffffffu, s, 16);
  if ((threadIdx.x & 31) < 8) atomicAdd(out + c, s);
}

// ---- host side ----------------------------------------------------------------

struct LayerOff {  // float offsets of one block's parameters within the flat layout
  size_t ln1_g, ln1_b, wq, bq, wk, bk, wv, bv, wo, bo, ln2_g, ln2_b, w1, b1, w2, b2;
};

LayerOff layer_off(const TfView& m, int l) {
  const size_t D = m.d, per = 12 * D * D + 13 * D;
  LayerOff o;
  o.ln1_g = 5 * D + size_t(m.n) * D + size_t(l) * per;
  o.ln1_b = o.ln1_g + D;
  o.wq = o.ln1_b + D;
  o.bq = o.wq + D * D;
  o.wk = o.bq + D;
  o.bk = o.wk + D * D;
  o.wv = o.bk + D;
  o.bv = o.wv + D * D;
  o.wo = o.bv + D;
  o.bo = o.wo + D * D;
  o.ln2_g = o.bo + D;
  o.ln2_b = o.ln2_g + D;
  o.w1 = o.ln2_b + D;
  o.b1 = o.w1 + 4 * D * D;
  o.w2 = o.b1 + 4 * D;
  o.b2 = o.w2 + 4 * D * D;
  return o;
}

struct Acts {
  float *H[17], *Xh1[16], *A1[16], *RS1[16], *QKV[16], *P[16], *O[16], *Hm[16], *Xh2[16], *A2[16], *RS2[16], *F[16];
  float *Xhf, *Af, *RSf, *out8, *dout8, *dH, *dA, *dHm, *dF, *dQKV, *dO, *dS;
  double* cot;
  // rows
  bool tree;
  uint64_t R;  // bound on the rows
  uint64_t* x;
  uint8_t* lv;
  uint32_t* anc;
  TreeWs t;
};

// Full storage keeps every block's activations; with `ckpt` (activation
// recomputation) only the block inputs H[l] are kept and one set of block
// activations is shared by all blocks: the backward recomputes block l's
// forward from H[l] just before its own backward.
size_t plan(const TfView& m, const anqs_ham* Hm, uint64_t nx, Arena& Ar, Acts& a, bool ckpt = false) {
  const uint64_t D = m.d;
  a.tree = tree_applies(Hm);
  a.x = nullptr;
  if (a.tree) {
    plan_tree(Hm, nx, Ar, a.t);
    a.R = a.t.max_rows;
  } else {
    a.R = nx * m.n;
    a.x = Ar.take<uint64_t>(a.R);
  }
  const uint64_t R = a.R;
  a.lv = Ar.take<uint8_t>(R);
  a.anc = Ar.take<uint32_t>(R * m.n);
  a.cot = Ar.take<double>(R * 8);
  for (int l = 0; l <= m.L; ++l) a.H[l] = Ar.take<float>(R * D);
  for (int l = 0; l < (ckpt ? 1 : m.L); ++l) {
    a.Xh1[l] = Ar.take<float>(R * D);
    a.A1[l] = Ar.take<float>(R * D);
    a.RS1[l] = Ar.take<float>(R);
    a.QKV[l] = Ar.take<float>(R * 3 * D);
    a.P[l] = Ar.take<float>(R * m.H * m.n);
    a.O[l] = Ar.take<float>(R * D);
    a.Hm[l] = Ar.take<float>(R * D);
    a.Xh2[l] = Ar.take<float>(R * D);
    a.A2[l] = Ar.take<float>(R * D);
    a.RS2[l] = Ar.take<float>(R);
    a.F[l] = Ar.take<float>(R * 4 * D);
  }
  for (int l = 1; ckpt && l < m.L; ++l) {
    a.Xh1[l] = a.Xh1[0], a.A1[l] = a.A1[0], a.RS1[l] = a.RS1[0], a.QKV[l] = a.QKV[0];
    a.P[l] = a.P[0], a.O[l] = a.O[0], a.Hm[l] = a.Hm[0], a.Xh2[l] = a.Xh2[0];
    a.A2[l] = a.A2[0], a.RS2[l] = a.RS2[0], a.F[l] = a.F[0];
  }
  a.Xhf = Ar.take<float>(R * D);
  a.Af = Ar.take<float>(R * D);
  a.RSf = Ar.take<float>(R);
  a.out8 = Ar.take<float>(R * 8);
  a.dout8 = Ar.take<float>(R * 8);
  a.dH = Ar.take<float>(R * D);
  a.dA = Ar.take<float>(R * D);
  a.dHm = Ar.take<float>(R * D);
  a.dF = Ar.take<float>(R * 4 * D);
  a.dQKV = Ar.take<float>(R * 3 * D);
  a.dO = Ar.take<float>(R * D);
  a.dS = Ar.take<float>(R * m.H * m.n);
  return Ar.off;
}

unsigned grid_for(uint64_t work, int threads, uint64_t cap) {
  uint64_t b = (work + threads - 1) / threads;
  if (b > cap) b = cap;
  return unsigned(b ? b : 1);
}

void set_vec(Gm& g) {
  g.b_vec = reinterpret_cast<uintptr_t>(g.B) % 16 == 0 && reinterpret_cast<uintptr_t>(g.bias) % 16 == 0;
  g.c_vec = reinterpret_cast<uintptr_t>(g.C) % 16 == 0;
}

// C = A B^T with the options of Gm, M rows (device or host count)
int gemm_nt(Gm g, uint64_t M_host, uint64_t K_host, cudaStream_t s) {
  const uint64_t gy = (M_host + BM - 1) / BM;
  if (gy > 65535u) return set_error(ANQS_ERR_UNSUPPORTED, "too many rows for the transformer adjoint");
  g.k_chunk = K_host ? K_host : 1;
  set_vec(g);
  ANQS_CUDA_LAUNCH("tf sgemm_kernel", launch_k(sgemm_kernel, dim3(unsigned((g.N + BN - 1) / BN), unsigned(gy)), dim3(GT), 0, s, g));
  return ANQS_OK;
}

// The weight product w (Mw x N, over R rows, split over CTAs) and the data
// product d (R x N) of one layer
int gemm_bwd(Gm w, uint64_t Mw, Gm d, uint64_t Kd, uint64_t R, cudaStream_t s) {
  const unsigned wx = unsigned((w.N + BN - 1) / BN), wy = unsigned((Mw + BM - 1) / BM), dx = unsigned((d.N + BN - 1) / BN);
  const uint64_t dy = (R + BM - 1) / BM;
  uint64_t parts = (152 * 4 + wx * wy - 1) / (wx * wy);
  parts = std::max<uint64_t>(1, std::min(parts, (R + 127) / 128));  // at least 128 rows each
  w.k_chunk = ((R + parts - 1) / parts + BK - 1) / BK * BK;
  d.k_chunk = Kd ? Kd : 1;
  if (!w.k_chunk) w.k_chunk = BK;
  if (dy * dx > (1ull << 30)) return set_error(ANQS_ERR_UNSUPPORTED, "too many rows for the transformer adjoint");
  set_vec(w);
  set_vec(d);
  const unsigned nw = unsigned(parts) * wx * wy;
  ANQS_CUDA_LAUNCH("tf sgemm_bwd_kernel", launch_k(sgemm_bwd_kernel, dim3(nw + unsigned(dy) * dx), dim3(GT), 0, s, w, d, nw, wx, wy, dx));
  return ANQS_OK;
}

Gm mk(const float* A, int lda, const float* B, int ldb, float* C, int ldc, Count M, Count K, int N) {
  Gm g = {};
  g.A = A;
  g.lda = lda;
  g.B = B;
  g.ldb = ldb;
  g.C = C;
  g.ldc = ldc;
  g.M = M;
  g.K = K;
  g.N = N;
  return g;
}

template <int D>
int run(const TfView& m, const anqs_ham* Hm, const uint64_t* x, Count nx, const float* cl, const float* cp,
        float* grad, void* ws, size_t ws_bytes, cudaStream_t s) {
  const HamView& hv = Hm->v;
  Arena Ar(ws, ws_bytes);
  Acts a{};
  plan(m, Hm, nx.n, Ar, a);
  bool ckpt = false;
  if (!Ar.fits()) {  // too little workspace for every activation: recompute each block's
    Arena Ac(ws, ws_bytes);
    plan(m, Hm, nx.n, Ac, a, true);
    if (!Ac.fits())
      return set_error(ANQS_ERR_CAPACITY, "transformer adjoint workspace needs %zu bytes (%zu with recomputation)",
                       Ar.off, Ac.off);
    ckpt = true;
  }
  const int n = m.n, L = m.L, H = m.H;
  // attention kernels with the head in registers for widths 4 to 32 in powers of two
  const int e4 = D / H == 4 ? 1 : D / H == 8 ? 2 : D / H == 16 ? 4 : D / H == 32 ? 8 : 0;
  const auto attn_fwd = e4 == 1 ? attn_fwd_kernel<1> : e4 == 2 ? attn_fwd_kernel<2> : e4 == 4 ? attn_fwd_kernel<4>
                        : e4 == 8 ? attn_fwd_kernel<8> : attn_fwd_kernel<0>;
  const auto attn_bwd_q = e4 == 1 ? attn_bwd_q_kernel<1> : e4 == 2 ? attn_bwd_q_kernel<2> : e4 == 4 ? attn_bwd_q_kernel<4>
                          : e4 == 8 ? attn_bwd_q_kernel<8> : attn_bwd_q_kernel<0>;
  const uint64_t R = a.R;
  const Count rows = a.tree ? Count{R, a.t.n_rows, 1} : scaled(nx, n);
  const Count kD = host_count(D), k3D = host_count(3 * D), k4D = host_count(4 * D), k8 = host_count(8);
  const float* P = m.params;
  ProfScope ps(PROF_TF_GRAD, s);
  const unsigned eg = grid_for(R * D, 256, 152 * 16), lg = grid_for(R * 32, 256, 152 * 16);
  const unsigned ag = grid_for(R * H, AT, 152 * 16);
  Rows rw{a.x, a.lv, a.anc, rows, n};
  ANQS_CUDA(cudaMemsetAsync(a.cot, 0, R * 8 * sizeof(double), s));
  if (a.tree) {
    ANQS_TRY(launch_tree(Hm, x, nx, a.t, s));
    rw.x = a.t.nodes.x;
    ANQS_CUDA_LAUNCH("tf tree_rows_kernel", launch_k(tree_rows_kernel, dim3(grid_for(R, 64, 152 * 16)), dim3(64), 0, s, Hm->sv, a.t.nodes, a.lv, a.anc));
  } else {
    ANQS_CUDA_LAUNCH("tf flat_rows_kernel", launch_k(flat_rows_kernel, dim3(grid_for(R, 64, 152 * 16)), dim3(64), 0, s, x, rows, n, a.x, a.lv, a.anc));
  }
  ANQS_CUDA_LAUNCH("tf cot_rows_kernel", launch_k(cot_rows_kernel, dim3(grid_for(nx.n, 64, 152 * 16)), dim3(64), 0, s, hv, Hm->sv, a.t.nodes, x, nx, cl, cp, a.cot));
  ANQS_CUDA_LAUNCH("tf embed_kernel", launch_k(embed_kernel, dim3(eg), dim3(256), 0, s, m, rw, a.H[0]));
  const Seg qkv_seg{D, size_t(D) * D + D};  // wq, bq, wk, bk, wv, bv
  // forward of block l from H[l]: its activations and H[l + 1] (deterministic,
  // so a recomputation reproduces them bit for bit)
  auto fwd_block = [&](int l) -> int {
    const LayerOff o = layer_off(m, l);
    ANQS_CUDA_LAUNCH("tf ln_fwd_kernel", launch_k(ln_fwd_kernel<D>, dim3(lg), dim3(256), 0, s, a.H[l], P + o.ln1_g,
                                                  P + o.ln1_b, a.Xh1[l], a.A1[l], a.RS1[l], rows));
    {
      Gm g = mk(a.A1[l], D, P + o.wq, D, a.QKV[l], 3 * D, rows, kD, 3 * D);
      g.sb = qkv_seg;
      g.bias = P + o.bq;
      ANQS_TRY(gemm_nt(g, R, D, s));
    }
    ANQS_CUDA_LAUNCH("tf attn_fwd_kernel", launch_k(attn_fwd, dim3(ag), dim3(AT), 0, s, a.QKV[l], a.P[l], a.O[l], D, H, rw));
    {
      Gm g = mk(a.O[l], D, P + o.wo, D, a.Hm[l], D, rows, kD, D);
      g.bias = P + o.bo;
      g.Cin = a.H[l];
      g.ldcin = D;
      ANQS_TRY(gemm_nt(g, R, D, s));
    }
    ANQS_CUDA_LAUNCH("tf ln_fwd_kernel", launch_k(ln_fwd_kernel<D>, dim3(lg), dim3(256), 0, s, a.Hm[l], P + o.ln2_g,
                                                  P + o.ln2_b, a.Xh2[l], a.A2[l], a.RS2[l], rows));
    {
      Gm g = mk(a.A2[l], D, P + o.w1, D, a.F[l], 4 * D, rows, kD, 4 * D);
      g.bias = P + o.b1;
      ANQS_TRY(gemm_nt(g, R, D, s));
    }
    {
      Gm g = mk(a.F[l], 4 * D, P + o.w2, 4 * D, a.H[l + 1], D, rows, k4D, D);
      g.relu_a = 1;
      g.bias = P + o.b2;
      g.Cin = a.Hm[l];
      g.ldcin = D;
      ANQS_TRY(gemm_nt(g, R, 4 * D, s));
    }
    return ANQS_OK;
  };
  for (int l = 0; l < L; ++l) ANQS_TRY(fwd_block(l));
  const size_t tail = 5 * size_t(D) + size_t(n) * D + size_t(L) * (12 * size_t(D) * D + 13 * size_t(D));
  const size_t lnf_g = tail, lnf_b = tail + D, head_w = tail + 2 * D, head_b = tail + 10 * D;
  ANQS_CUDA_LAUNCH("tf ln_fwd_kernel", launch_k(ln_fwd_kernel<D>, dim3(lg), dim3(256), 0, s, a.H[L], P + lnf_g,
                                                P + lnf_b, a.Xhf, a.Af, a.RSf, rows));
  {
    Gm g = mk(a.Af, D, P + head_w, D, a.out8, 8, rows, kD, 8);
    g.bias = P + head_b;
    ANQS_TRY(gemm_nt(g, R, D, s));
  }
  ANQS_CUDA_LAUNCH("tf head_dout_kernel", launch_k(head_dout_kernel, dim3(grid_for(R, 128, 152 * 8)), dim3(128), 0, s,
                                                   hv, rw, a.out8, a.cot, a.dout8));
  // ---- backward ----
  // weight gradient gW += dY^T X and bias gradient gb += the column sums of dY
  auto wgrad = [&](const float* dY, int ldy, const float* X, int ldx, int Mo, int Ni, float* gW, float* gb, int relu_x,
                   Seg seg = Seg{}) -> Gm {
    Gm g = mk(dY, ldy, X, ldx, gW, Ni, host_count(Mo), rows, Ni);
    g.relu_b = relu_x;
    g.atomic = 1;
    g.sc = seg;
    g.colsum = gb;
    return g;
  };
  ANQS_CUDA_LAUNCH("tf colsum8_kernel", launch_k(colsum8_kernel, dim3(grid_for(R * 8, 256, 152)), dim3(256), 0, s, a.dout8, rows, grad + head_b));
  {
    const Gm g = mk(a.dout8, 8, P + head_w, D, a.dA, D, rows, k8, D);
    ANQS_TRY(gemm_bwd(wgrad(a.dout8, 8, a.Af, D, 8, D, grad + head_w, nullptr, 0), 8, g, 8, R, s));
  }
  ANQS_CUDA_LAUNCH("tf ln_bwd_kernel",
                   launch_k(ln_bwd_kernel<D>, dim3(lg), dim3(256), 0, s, a.dA, a.Xhf, P + lnf_g, a.RSf,
                            (const float*)nullptr, a.dH, grad + lnf_g, grad + lnf_b, rows));
  for (int l = L - 1; l >= 0; --l) {
    const LayerOff o = layer_off(m, l);
    if (ckpt && l + 1 < L) ANQS_TRY(fwd_block(l));  // the shared activations hold block L-1's after the forward
    {
      Gm g = mk(a.dH, D, P + o.w2, 4 * D, a.dF, 4 * D, rows, kD, 4 * D);
      g.mask = a.F[l];
      g.ldmask = 4 * D;
      ANQS_TRY(gemm_bwd(wgrad(a.dH, D, a.F[l], 4 * D, D, 4 * D, grad + o.w2, grad + o.b2, 1), D, g, D, R, s));
    }
    {
      const Gm g = mk(a.dF, 4 * D, P + o.w1, D, a.dA, D, rows, k4D, D);
      ANQS_TRY(gemm_bwd(wgrad(a.dF, 4 * D, a.A2[l], D, 4 * D, D, grad + o.w1, grad + o.b1, 0), 4 * D, g, 4 * D, R, s));
    }
    ANQS_CUDA_LAUNCH("tf ln_bwd_kernel", launch_k(ln_bwd_kernel<D>, dim3(lg), dim3(256), 0, s, a.dA, a.Xh2[l],
                                                  P + o.ln2_g, a.RS2[l], (const float*)a.dH, a.dHm, grad + o.ln2_g,
                                                  grad + o.ln2_b, rows));
    {
      const Gm g = mk(a.dHm, D, P + o.wo, D, a.dO, D, rows, kD, D);
      ANQS_TRY(gemm_bwd(wgrad(a.dHm, D, a.O[l], D, D, D, grad + o.wo, grad + o.bo, 0), D, g, D, R, s));
    }
    ANQS_CUDA_LAUNCH("tf attn_bwd_q_kernel", launch_k(attn_bwd_q, dim3(ag), dim3(AT), 0, s, a.QKV[l], a.P[l], a.dO, a.dS, a.dQKV, D, H, rw));
    ANQS_CUDA_LAUNCH("tf attn_bwd_kv_kernel", launch_k(attn_bwd_kv_kernel, dim3(unsigned((R + KVR - 1) / KVR), unsigned(n)), dim3(2 * D < 256 ? 2 * D : 256), 0, s, a.QKV[l], a.P[l], a.dO, a.dS, a.dQKV, D, H, rw));
    {
      Gm g = mk(a.dQKV, 3 * D, P + o.wq, D, a.dA, D, rows, k3D, D);
      g.sb = qkv_seg;
      ANQS_TRY(gemm_bwd(wgrad(a.dQKV, 3 * D, a.A1[l], D, 3 * D, D, grad + o.wq, grad + o.bq, 0, qkv_seg), 3 * D, g, 3 * D, R, s));
    }
    ANQS_CUDA_LAUNCH("tf ln_bwd_kernel", launch_k(ln_bwd_kernel<D>, dim3(lg), dim3(256), 0, s, a.dA, a.Xh1[l],
                                                  P + o.ln1_g, a.RS1[l], (const float*)a.dHm, a.dH, grad + o.ln1_g,
                                                  grad + o.ln1_b, rows));
  }
  ANQS_CUDA_LAUNCH("tf embed_bwd_kernel", launch_k(embed_bwd_kernel, dim3(unsigned((R + EBR - 1) / EBR)), dim3(D), 0, s, m, rw, a.dH, grad, grad + 5 * size_t(D)));
  return ANQS_OK;
}

}  // namespace

size_t tf_grad_workspace(const TfView& m, const anqs_ham* H, uint64_t n_x, bool recompute) {
  Arena Ar(nullptr, 0);
  Acts a{};
  return plan(m, H, n_x, Ar, a, recompute);
}

int launch_tf_fp32_grad(const TfView& m, const anqs_ham* H, const uint64_t* x, Count n_x, const float* cl,
                        const float* cp, float* grad, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (n_x.n == 0) return ANQS_OK;
  if (m.n > 32) return set_error(ANQS_ERR_UNSUPPORTED, "n_orb %d", m.n);
  switch (m.d) {
    case 32: return run<32>(m, H, x, n_x, cl, cp, grad, ws, ws_bytes, s);
    case 64: return run<64>(m, H, x, n_x, cl, cp, grad, ws, ws_bytes, s);
    case 128: return run<128>(m, H, x, n_x, cl, cp, grad, ws, ws_bytes, s);
    case 256: return run<256>(m, H, x, n_x, cl, cp, grad, ws, ws_bytes, s);
  }
  return set_error(ANQS_ERR_UNSUPPORTED, "d_model %d", m.d);
}

}  // namespace anqs
