// Covariance of xi from sub-samples of the catalogue (HEALPix pixels of the
// first forest of each pair): with per sub-sample sums N^s_A, W^s_A of
// Eq. (2.4) and the full sums N_A = sum_s N^s_A, W_A = sum_s W^s_A,
// xi_A = N_A / W_A,
//     C_AB = sum_s W^s_A W^s_B (xi^s_A - xi_A)(xi^s_B - xi_B) / (W_A W_B)
//          = sum_s a^s_A a^s_B / (W_A W_B),   a^s_A = N^s_A - W^s_A xi_A,
// the weighted sub-sample covariance (zero rows and columns where W_A = 0).
// FP64 throughout; only sub-samples with pairs enter the sum (list built in
// sub-sample order, so the result does not depend on scheduling).
#include <algorithm>

#include "lya_internal.cuh"

namespace lya {
namespace {

constexpr int kTile = 64;     // output tile edge
constexpr int kSt = 16;       // sub-samples per shared-memory stage

// full sums and xi: 32 bins per block, 32 slices of the sub-samples
// (one thread per bin walking all of them in turn took 0.23 ms for 768 x 2,500)
__global__ void __launch_bounds__(1024) cov_totals_kernel(const double* num_s, const double* wsum_s, int n_sub, int nb,
                                                          double* W, double* xi) {
  __shared__ double sw[32][33], sn[32][33];
  const int t = threadIdx.x & 31, q = threadIdx.x >> 5;
  for (int A0 = blockIdx.x * 32; A0 < nb; A0 += gridDim.x * 32) {
    const int A = A0 + t;
    double w = 0.0, n = 0.0;
    if (A < nb)
      for (int s = q; s < n_sub; s += 32) {
        w += wsum_s[static_cast<int64_t>(s) * nb + A];
        n += num_s[static_cast<int64_t>(s) * nb + A];
      }
    sw[q][t] = w;
    sn[q][t] = n;
    __syncthreads();
    // warp q sums bin q's slices
    w = warp_sum_f64(sw[t][q]);
    n = warp_sum_f64(sn[t][q]);
    if (t == 0 && A0 + q < nb) {
      W[A0 + q] = w;
      xi[A0 + q] = (w != 0.0) ? n / w : 0.0;
    }
    __syncthreads();
  }
}

// flag[s] = 1 if any bin of sub-sample s has weight, one block per sub-sample
// (one block for all of them took 4.0 ms)
__global__ void cov_flag_kernel(const double* wsum_s, int n_sub, int nb, int32_t* flag) {
  for (int s = blockIdx.x; s < n_sub; s += gridDim.x) {
    int any = 0;
    for (int A = threadIdx.x; A < nb; A += blockDim.x) any |= wsum_s[static_cast<int64_t>(s) * nb + A] != 0.0;
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) flag[s] = any;
  }
}

// list[0] = number of flagged sub-samples, list[1 ..] = their indices in order; one block
__global__ void __launch_bounds__(1024) cov_list_kernel(const int32_t* flag, int n_sub, int32_t* list) {
  __shared__ int part[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int base = 0;
  for (int s0 = 0; s0 < n_sub; s0 += 1024) {
    const int s = s0 + threadIdx.x;
    const bool on = s < n_sub && flag[s] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (lane == 0) part[wid] = __popc(m);
    __syncthreads();
    int before = base, all = 0;
    for (int k = 0; k < 32; ++k) {
      if (k < wid) before += part[k];
      all += part[k];
    }
    if (on) list[1 + before + __popc(m & ((1u << lane) - 1u))] = s;
    base += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) list[0] = base;
}

// C tile (64 x 64) per block of 16 x 16 threads, 4 x 4 outputs per thread;
// tiles on and above the diagonal, written to both sides.  Bound by the FP64
// pipe: an entry costs one multiply-add per sub-sample, and a division as much
// as the sum over a dozen sub-samples.
__global__ void __launch_bounds__(256) cov_kernel(const double* num_s, const double* wsum_s, int nb,
                                                  const double* W, const double* xi,
                                                  const int32_t* list, double* cov) {
  if (blockIdx.x < blockIdx.y) return;
  __shared__ double ar[kSt][kTile];
  __shared__ double ac[kSt][kTile];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int r0 = blockIdx.y * kTile, c0 = blockIdx.x * kTile;
  const int m = list[0];
  double acc[4][4] = {};
  for (int k0 = 0; k0 < m; k0 += kSt) {
    for (int e = threadIdx.x; e < kSt * kTile; e += blockDim.x) {
      const int kk = e / kTile, t = e - kk * kTile;
      double vr = 0.0, vc = 0.0;
      if (k0 + kk < m) {
        const int64_t base = static_cast<int64_t>(list[1 + k0 + kk]) * nb;
        const int A = r0 + t, B = c0 + t;
        if (A < nb) vr = num_s[base + A] - wsum_s[base + A] * xi[A];
        if (B < nb) vc = num_s[base + B] - wsum_s[base + B] * xi[B];
      }
      ar[kk][t] = vr;
      ac[kk][t] = vc;
    }
    __syncthreads();
    const int kn = min(kSt, m - k0);
#pragma unroll 2
    for (int kk = 0; kk < kn; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = ar[kk][ty * 4 + u];
        b[u] = ac[kk][tx * 4 + u];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int A = r0 + ty * 4 + u;
    if (A >= nb) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int B = c0 + tx * 4 + v;
      if (B >= nb) continue;
      const double den = W[A] * W[B];
      const double c = (den != 0.0) ? acc[u][v] / den : 0.0;   // (symmetric)
      cov[static_cast<int64_t>(A) * nb + B] = c;
      if (blockIdx.x != blockIdx.y) cov[static_cast<int64_t>(B) * nb + A] = c;
    }
  }
}

}  // namespace

size_t covariance_scratch_bytes(int n_sub, int nb) {
  auto al = [](size_t v) { return (v + 255) & ~size_t(255); };
  return 2 * al(static_cast<size_t>(nb) * 8) + al((static_cast<size_t>(n_sub) + 1) * 4) + al(static_cast<size_t>(n_sub) * 4);
}

cudaError_t launch_covariance(const double* num_s, const double* wsum_s, int n_sub, int nb, double* cov,
                              double* xi_out, void* scratch, cudaStream_t s) {
  if (nb == 0) return cudaSuccess;
  auto al = [](size_t v) { return (v + 255) & ~size_t(255); };
  char* sc = static_cast<char*>(scratch);
  double* W = reinterpret_cast<double*>(sc);
  double* xi = reinterpret_cast<double*>(sc + al(static_cast<size_t>(nb) * 8));
  int32_t* list = reinterpret_cast<int32_t*>(sc + 2 * al(static_cast<size_t>(nb) * 8));
  int32_t* flag = reinterpret_cast<int32_t*>(sc + 2 * al(static_cast<size_t>(nb) * 8) + al((static_cast<size_t>(n_sub) + 1) * 4));
  LYA_COUNT(1), cov_totals_kernel<<<std::min((nb + 31) / 32, 2048), 1024, 0, s>>>(num_s, wsum_s, n_sub, nb, W, xi);
  LYA_COUNT(1), cov_flag_kernel<<<std::min(n_sub, 4096), 256, 0, s>>>(wsum_s, n_sub, nb, flag);
  LYA_COUNT(1), cov_list_kernel<<<1, 1024, 0, s>>>(flag, n_sub, list);
  const int nt = (nb + kTile - 1) / kTile;
  LYA_COUNT(1), cov_kernel<<<dim3(nt, nt), 256, 0, s>>>(num_s, wsum_s, nb, W, xi, list, cov);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && xi_out) e = cudaMemcpyAsync(xi_out, xi, static_cast<size_t>(nb) * 8, cudaMemcpyDeviceToDevice, s);
  return e;
}

}  // namespace lya
