// Statistics of the union of sample sets, and the per-sample cotangents of
// the VMC gradient (Eq. grad_def).
#include <cmath>

#include "common.cuh"

namespace anqs {
namespace {

// cot_la = 2 w Re(eloc - E), cot_ph = 2 w Im(eloc - E), w = n / S
__global__ void cotangent_kernel(const double* __restrict__ ere, const double* __restrict__ eim,
                                 const uint64_t* __restrict__ counts, const double* __restrict__ stats,
                                 Count n_x_, float* __restrict__ cl, float* __restrict__ cp) {
  ANQS_PDL_ENTRY();
  const double Er = stats[0], Ei = stats[1], S = stats[3];
  const uint64_t n_x = n_x_.get();
  for (uint64_t l = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; l < n_x; l += uint64_t(gridDim.x) * blockDim.x) {
    double w = double(counts[l]) / S;
    cl[l] = float(2.0 * w * (ere[l] - Er));
    cp[l] = float(2.0 * w * (eim[l] - Ei));
  }
}

// statistics of the union of `world` disjoint sample sets (law of total
// variance); one thread, world is small.  Empty sets (S_r = 0, whose E_r is
// 0/0) are skipped.
__global__ void stats_combine_kernel(const double* __restrict__ in, int world, double* __restrict__ out) {
  ANQS_PDL_ENTRY();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double s = 0.0, sr = 0.0, si = 0.0;
  for (int r = 0; r < world; ++r) {
    const double w = in[4 * r + 3];
    if (!(w > 0.0)) continue;
    s += w;
    sr = fma(w, in[4 * r + 0], sr);
    si = fma(w, in[4 * r + 1], si);
  }
  const double Er = sr / s, Ei = si / s;
  double v = 0.0;
  for (int r = 0; r < world; ++r) {
    if (!(in[4 * r + 3] > 0.0)) continue;
    const double dr = in[4 * r + 0] - Er, di = in[4 * r + 1] - Ei;
    v = fma(in[4 * r + 3], in[4 * r + 2] + dr * dr + di * di, v);
  }
  out[0] = Er;
  out[1] = Ei;
  out[2] = v / s;
  out[3] = s;
}

}  // namespace

int launch_stats_combine(const double* in, int world, double* out, cudaStream_t s) {
  ProfScope ps(PROF_STATS, s);
  ANQS_CUDA_LAUNCH("stats_combine_kernel", launch_k(stats_combine_kernel, dim3(1), dim3(32), 0, s, in, world, out));
  return ANQS_OK;
}

int launch_grad_cotangents(const double* ere, const double* eim, const uint64_t* counts, const double* stats,
                           Count n_x, float* cl, float* cp, cudaStream_t s) {
  uint64_t blocks = (n_x.n + 255) / 256;
  if (blocks == 0) blocks = 1;
  if (blocks > 152 * 8) blocks = 152 * 8;
  ProfScope ps(PROF_COTANGENT, s);
  ANQS_CUDA_LAUNCH("cotangent_kernel", launch_k(cotangent_kernel, dim3(unsigned(blocks)), dim3(256), 0, s, ere, eim, counts, stats, n_x, cl, cp));
  return ANQS_OK;
}

}  // namespace anqs
