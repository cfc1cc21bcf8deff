// Anisotropic three-point estimator, Eq. (2.8) (Section 2.3):
//   xi3_A = sum_A (w d)_i (w d)_j (w d)_k / sum_A w_i w_j w_k
// over pixel triplets of three distinct forests.  A record is a main vertex i
// with r1 = x_j - x_i, r2 = x_k - x_i (x = d n), binned in (|r1|, |r2|,
// cos alpha, theta1, theta2) and flattened as
//   A = (((i_r1 n_r + i_r2) n_alpha + i_alpha) n_theta + i_theta1) n_theta + i_theta2,
// theta the angle to the main vertex's line of sight, alpha the angle between
// r1 and r2.  Every pixel is a main vertex, the other two pixels take
// (r1, r2) in both orders, and a record needs |r1|, |r2| < r_max.
//
// One block per main-vertex pixel (work taken from an atomic counter):
//  1. gather: for every forest in the vertex forest's neighbour list, the chord
//     of pixels within r_max of the vertex (a contiguous range of the sorted
//     distances, one forest per lane), then the chords' pixels, one per thread:
//     tested exactly in FP64, with r in FP32; the |r| and theta bins come from
//     FP32 and, near a bin edge, from the FP64 square root and arc cosine of the
//     definition, so they are the definition's;
//  2. pairs: blocks of 32 x 32 neighbours dealt to the warps, 32 candidates q in
//     registers against candidates p read once for the whole warp; pixels of
//     the same forest are skipped; cos alpha is FP32; the record and its
//     mirror (sides swapped) are added once, to the bin whose (r, theta) key
//     of side 1 is not above side 2's, with weight 2 when both keys are equal;
//     sums are FP32 products added to FP64 bin sums with global atomics;
//  3. a finalize kernel copies each canonical bin to its mirror and forms xi.
// A counting pass first finds the longest chords of any vertex, and the block's
// shared-memory capacity is sized to them; a vertex with more neighbours than
// one block can hold raises a device flag (reported as LYA_ERR_TOO_LARGE)
// instead of being truncated silently.
// What bounds it: the FP64 atomics in L2, which takes one 32-byte sector per
// 2.3 clocks and SM wherever the bins are random; N and W of a bin therefore
// lie side by side and two lanes add a record, so a record costs one sector and
// not two.  Measured (5,000 SDSS-like forests, r_max 40, 200,000 bins): 411 ms
// with separate arrays and FP64 gathers and counts by whole warps, 381 ms with
// the gather and the count per lane, 204 ms with the sums side by side.
#include <algorithm>
#include <math.h>

#include "lya_internal.cuh"

namespace lya {
namespace {

constexpr int kX3Threads = 256;
constexpr int kX3Batch = 64;   // neighbour forests per gather step (with the static words, below 1,024 bytes)

__global__ void x3_degree_kernel(const int2* pairs, int64_t n, int32_t* deg) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int2 p = pairs[k];
    if (p.x < 0) continue;
    atomicAdd(&deg[p.x], 1);
    atomicAdd(&deg[p.y], 1);
  }
}

__global__ void x3_fill_kernel(const int2* pairs, int64_t n, const int64_t* start, int32_t* cursor,
                               int32_t* nbr) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int2 p = pairs[k];
    if (p.x < 0) continue;
    nbr[start[p.x] + atomicAdd(&cursor[p.x], 1)] = p.y;
    nbr[start[p.y] + atomicAdd(&cursor[p.y], 1)] = p.x;
  }
}

__global__ void x3_scan_kernel(const int32_t* in, int64_t n, int64_t* out) {
  __shared__ int64_t part[1024];
  const int t = threadIdx.x;
  const int64_t chunk = (n + blockDim.x - 1) / blockDim.x;
  const int64_t b = t * chunk, e = min(n, b + chunk);
  int64_t s = 0;
  for (int64_t k = b; k < e; ++k) s += in[k];
  part[t] = s;
  __syncthreads();
  if (t == 0) {
    int64_t run = 0;
    for (int k = 0; k < (int)blockDim.x; ++k) {
      const int64_t v = part[k];
      part[k] = run;
      run += v;
    }
    out[n] = run;
  }
  __syncthreads();
  int64_t run = part[t];
  for (int64_t k = b; k < e; ++k) {
    out[k] = run;
    run += in[k];
  }
}

// forest of packed pixel g: the last forest whose first pixel is <= g
__device__ __forceinline__ int forest_of(const Forests& F, int64_t g) {
  int lo = 0, hi = static_cast<int>(F.n) - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (F.off[mid] <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Pixels [lo, hi) of forest o that can lie within r_max of the vertex at
// distance di on forest f's line of sight: the chord of the sphere along o's
// line of sight, 1e-2 Mpc/h wider.
struct Chord {
  int lo, hi;
};
__device__ __forceinline__ Chord chord(const X3Args& A, int f, int o, double di, double rmax2) {
  Chord c{0, 0};
  const int no = A.F.len[o];
  if (no == 0) return c;
  const double ca = A.F.ux[f] * A.F.ux[o] + A.F.uy[f] * A.F.uy[o] + A.F.uz[f] * A.F.uz[o];
  const double disc = rmax2 - di * di * fmax(0.0, 1.0 - ca * ca);
  if (!(disc > 0.0)) return c;
  const double sq = sqrt(disc);
  const Pix* po = A.pix + A.F.off[o];
  const double ref = A.F.dref[o];
  c.lo = count_below(po, no, static_cast<float>(di * ca - sq - ref) - 1e-2f);
  c.hi = max(c.lo, count_below(po, no, static_cast<float>(di * ca + sq - ref) + 1e-2f));
  return c;
}

__global__ void __launch_bounds__(kX3Threads, 5) xi3_kernel(X3Args A, const int32_t* nbr, const int64_t* nstart,
                                                         int cap, double* sums, unsigned long long* counter, unsigned* err) {
  extern __shared__ __align__(16) unsigned char sm[];
  float4* cr = reinterpret_cast<float4*>(sm);                  // r (FP32) and 1 / |r|
  float2* cw = reinterpret_cast<float2*>(cr + cap);            // (w d, w)
  int2* ck = reinterpret_cast<int2*>(cw + cap);                // ((radial bin << 16) | theta bin, forest)
  __shared__ int s_n, s_f;
  __shared__ long long s_item;
  __shared__ int s_o[kX3Batch], s_lo[kX3Batch], s_pre[kX3Batch + 1];   // chords of a batch of neighbours
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarps = blockDim.x >> 5;
  const double rmax = A.r_max, rmax2 = rmax * rmax;
  const double inv_dr = A.n_r / rmax, inv_dt = A.n_theta / M_PI;
  const float inv_dr_f = static_cast<float>(inv_dr), inv_dt_f = static_cast<float>(inv_dt);
  // FP32 errors of |r| and theta in bins, doubled: |r| n_r / r_max <= n_r is good to 4 roundings; theta =
  // acos(c) to 5e-6 rad where |c| <= 0.9999 (the FP32 rounding of c over sin theta, and of acosf)
  const float guard_r = 1e-6f * static_cast<float>(A.n_r) + 1e-6f, guard_t = 1e-5f * inv_dt_f + 1e-6f;
  const float half_na = 0.5f * static_cast<float>(A.n_alpha);
  const int nr = A.n_r, nt = A.n_theta, na = A.n_alpha;
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      const long long it = static_cast<long long>(atomicAdd(counter, 1ull));
      s_item = it;
      s_n = 0;
      s_f = (it < A.n_pix) ? forest_of(A.F, it) : 0;
    }
    __syncthreads();
    const long long g = s_item;
    if (g >= A.n_pix) break;
    const int f = s_f;
    const int64_t i_in = g - A.F.off[f];
    if (i_in >= A.F.len[f]) continue;    // pixel of a forest that failed the input checks
    const double nax = A.F.ux[f], nay = A.F.uy[f], naz = A.F.uz[f];
    const double di = A.dist[g];
    const double xi = di * nax, yi = di * nay, zi = di * naz;
    const Pix pv = A.pix[g];
    const float w_i = pv.y, wd_i = pv.z;
    // 1. gather the vertex's neighbours within r_max: the chords of up to 64
    //    forests, one per lane, then their pixels, one per thread
    for (int64_t e0 = nstart[f]; e0 < nstart[f + 1]; e0 += kX3Batch) {
      const int nb = static_cast<int>(min(static_cast<int64_t>(kX3Batch), nstart[f + 1] - e0));
      if (wid == 0) {
        int carry = 0;
        if (lane == 0) s_pre[0] = 0;
        for (int m0 = 0; m0 < nb; m0 += 32) {
          const int m = m0 + lane;
          int cnt = 0;
          if (m < nb) {
            const int o = nbr[e0 + m];
            const Chord c = chord(A, f, o, di, rmax2);
            s_o[m] = o;
            s_lo[m] = c.lo;
            cnt = c.hi - c.lo;
          }
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, cnt, d);
            if (lane >= d) cnt += up;
          }
          cnt += carry;
          if (m < nb) s_pre[m + 1] = cnt;
          carry = __shfl_sync(0xffffffffu, cnt, 31);
        }
      }
      __syncthreads();
      const int total = s_pre[nb];
      for (int k0 = wid * 32; k0 < total; k0 += kX3Threads) {
        const int k = k0 + lane;
        bool in = false;
        float4 r4 = make_float4(0.f, 0.f, 0.f, 0.f);
        Pix q = r4;
        int key = 0, o = 0;
        if (k < total) {
          int lo = 0, hi = nb - 1;   // neighbour whose pixels hold candidate k: the last with s_pre <= k
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_pre[mid] <= k) lo = mid; else hi = mid - 1;
          }
          o = s_o[lo];
          const int64_t p = A.F.off[o] + s_lo[lo] + (k - s_pre[lo]);
          const double dj = A.dist[p];
          const double dx = dj * A.F.ux[o] - xi, dy = dj * A.F.uy[o] - yi, dz = dj * A.F.uz[o] - zi;
          const double r2 = dx * dx + dy * dy + dz * dz;
          in = r2 < rmax2 && r2 > 0.0;
          if (in) {
            q = A.pix[p];
            // 1 / |r| to 2e-14: one Newton step from FP32 (an FP64 square root and division cost 20 times that)
            const float r2f = static_cast<float>(r2);
            const float y0f = rsqrtf(r2f);
            const double y0 = y0f;
            const double y = fma(0.5 * y0, fma(-(r2 * y0), y0, 1.0), y0);
            const double dot = dx * nax + dy * nay + dz * naz;
            const float ctf = static_cast<float>(dot * y);
            const float fr = r2f * y0f * inv_dr_f, ft = acosf(fminf(1.f, fmaxf(-1.f, ctf))) * inv_dt_f;
            const float gr = fr - floorf(fr), gt = ft - floorf(ft);
            int ir = static_cast<int>(fr), it = static_cast<int>(ft);
            const bool sure = r2f > 1e-30f && fabsf(gr - 0.5f) < 0.5f - guard_r && fabsf(gt - 0.5f) < 0.5f - guard_t &&
                              fabsf(ctf) <= 0.9999f;
            if (!sure) {   // the definition, near a bin edge
              const double r = sqrt(r2);
              const double ct = dot / r;
              ir = static_cast<int>(r * inv_dr);
              it = static_cast<int>(acos(fmin(1.0, fmax(-1.0, ct))) * inv_dt);
              r4.w = static_cast<float>(1.0 / r);
            } else {
              r4.w = static_cast<float>(y);
            }
            r4.x = static_cast<float>(dx);
            r4.y = static_cast<float>(dy);
            r4.z = static_cast<float>(dz);
            key = (min(ir, nr - 1) << 16) | min(it, nt - 1);
          }
        }
        const unsigned msk = __ballot_sync(0xffffffffu, in);
        int slot = 0;
        if (lane == 0 && msk) slot = atomicAdd(&s_n, __popc(msk));
        slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(msk & ((1u << lane) - 1u));
        if (in && slot < cap) {
          cr[slot] = r4;
          cw[slot] = make_float2(q.z, q.y);
          ck[slot] = make_int2(key, o);
        }
      }
      __syncthreads();
    }
    __syncthreads();
    const int P = s_n;
    if (P > cap && tid == 0) atomicOr(err, FLAG_X3_CAP);
    // 2. unordered pairs (p < q) of neighbours from two distinct forests, in
    //    blocks of 32 x 32 dealt to the warps: the block's candidates q sit in
    //    registers (one per lane), its candidates p are read once for the whole warp
    if (P <= cap) {
      const int tiles = (P + 31) >> 5, units = tiles * (tiles + 1) / 2;
      int t = 0, first = 0;   // unit u = first + c: candidates q of tile t, p of tile c <= t
      for (int u = wid; u < units; u += nwarps) {
        while (u > first + t) {
          first += t + 1;
          ++t;
        }
        const int q = 32 * t + lane;
        const bool qv = q < P;
        const float4 rq = qv ? cr[q] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float2 wq = qv ? cw[q] : make_float2(0.f, 0.f);
        const int2 kq = qv ? ck[q] : make_int2(0, -1);
        const float wdq = wq.x * wd_i, wwq = wq.y * w_i;
        const int qr = kq.x >> 16, qt = kq.x & 0xffff;
        const int p0 = 32 * (u - first), pend = min(p0 + 32, P);
        for (int p = p0; p < pend; ++p) {
          const float4 rp = cr[p];
          const int2 kp = ck[p];
          const float2 wp = cw[p];
          const bool on = qv && p < q && kp.y != kq.y;
          const float ca = (rp.x * rq.x + rp.y * rq.y + rp.z * rq.z) * (rp.w * rq.w);
          const int ia = min(max(static_cast<int>(floorf((ca + 1.0f) * half_na)), 0), na - 1);
          const int pr = kp.x >> 16, pt = kp.x & 0xffff;
          int r1, t1, r2, t2;
          if (kp.x <= kq.x) { r1 = pr; t1 = pt; r2 = qr; t2 = qt; } else { r1 = qr; t1 = qt; r2 = pr; t2 = pt; }
          const float mult = (kp.x == kq.x) ? 2.f : 1.f;
          const int bin = on ? (((r1 * nr + r2) * na + ia) * nt + t1) * nt + t2 : -1;   // (at most 2^28 bins)
          const float vn = wp.x * wdq * mult, vw = wp.y * wwq * mult;
          // two lanes per record, N and W of one bin side by side: L2 takes
          // atomics a 32-byte sector at a time
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int src = (lane >> 1) + 16 * h;
            const int b = __shfl_sync(0xffffffffu, bin, src);
            const float n = __shfl_sync(0xffffffffu, vn, src), w = __shfl_sync(0xffffffffu, vw, src);
            if (b >= 0) red_add_f64_global(sums + 2 * static_cast<int64_t>(b) + (lane & 1), static_cast<double>((lane & 1) ? w : n));
          }
        }
      }
    }
  }
}

// largest number of pixels on any main vertex's chords (an upper bound of its
// neighbours within r_max, 1e-2 Mpc/h wider), one warp per vertex pixel
__global__ void xi3_count_kernel(X3Args A, const int32_t* nbr, const int64_t* nstart, int* max_count) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const double rmax2 = A.r_max * A.r_max;
  int best = 0;
  for (int64_t g = warp; g < A.n_pix; g += nw) {
    const int f = forest_of(A.F, g);
    if (g - A.F.off[f] >= A.F.len[f]) continue;
    int cnt = 0;
    for (int64_t e = nstart[f] + lane; e < nstart[f + 1]; e += 32) {
      const Chord c = chord(A, f, nbr[e], A.dist[g], rmax2);
      cnt += c.hi - c.lo;
    }
    best = max(best, __reduce_add_sync(0xffffffffu, cnt));
  }
  if (lane == 0 && best > 0) atomicMax(max_count, best);
}

// num, wsum and xi of every bin: the sums of its canonical bin (side-1 key <=
// side-2 key), interleaved (N, W)
__global__ void xi3_finalize_kernel(const double* sums, double* num, double* wsum, double* xi, int nr, int nt, int na) {
  const int64_t n = static_cast<int64_t>(nr) * nr * na * nt * nt;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    int64_t rest = k;
    const int t2 = static_cast<int>(rest % nt); rest /= nt;
    const int t1 = static_cast<int>(rest % nt); rest /= nt;
    const int ia = static_cast<int>(rest % na); rest /= na;
    const int r2 = static_cast<int>(rest % nr); rest /= nr;
    const int r1 = static_cast<int>(rest);
    const int64_t m = (r1 * nt + t1 > r2 * nt + t2)
                          ? (((static_cast<int64_t>(r2) * nr + r1) * na + ia) * nt + t2) * nt + t1 : k;
    const double2 v = reinterpret_cast<const double2*>(sums)[m];
    num[k] = v.x;
    wsum[k] = v.y;
    if (xi) xi[k] = (v.y != 0.0) ? v.x / v.y : 0.0;
  }
}

int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 1 << 16) b = 1 << 16;
  return static_cast<int>(b);
}

#define LYA_TRY(x)                    \
  do {                                \
    cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

}  // namespace

cudaError_t run_xi3(const X3Args& a, const DevInfo& dev, void** scratch, size_t* scratch_cap, unsigned* err,
                    cudaStream_t s) {
  const int64_t nf = a.F.n, np = a.n_pairs;
  const int64_t nbins = static_cast<int64_t>(a.n_r) * a.n_r * a.n_alpha * a.n_theta * a.n_theta;
  auto al = [](size_t v) { return (v + 255) & ~size_t(255); };
  size_t o = 0;
  const size_t o_deg = o; o += al((nf + 1) * 4);
  const size_t o_cur = o; o += al((nf + 1) * 4);
  const size_t o_start = o; o += al((nf + 1) * 8);
  const size_t o_nbr = o; o += al(std::max<int64_t>(2 * np, 1) * 4);
  const size_t o_sums = o; o += al(static_cast<size_t>(nbins) * 16);   // (N, W) per bin
  const size_t o_misc = o; o += 256;
  LYA_TRY(grow(scratch, scratch_cap, o));
  char* sc = static_cast<char*>(*scratch);
  int32_t* deg = reinterpret_cast<int32_t*>(sc + o_deg);
  int32_t* cur = reinterpret_cast<int32_t*>(sc + o_cur);
  int64_t* start = reinterpret_cast<int64_t*>(sc + o_start);
  int32_t* nbr = reinterpret_cast<int32_t*>(sc + o_nbr);
  double* sums = reinterpret_cast<double*>(sc + o_sums);
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(sc + o_misc);
  LYA_TRY(cudaMemsetAsync(sums, 0, static_cast<size_t>(nbins) * 16, s));
  LYA_TRY(cudaMemsetAsync(deg, 0, (nf + 1) * 4, s));
  LYA_TRY(cudaMemsetAsync(cur, 0, (nf + 1) * 4, s));
  LYA_TRY(cudaMemsetAsync(counter, 0, 8, s));
  if (np > 0) LYA_COUNT(1), x3_degree_kernel<<<grid_for(np, 256), 256, 0, s>>>(a.pairs, np, deg);
  LYA_COUNT(1), x3_scan_kernel<<<1, 1024, 0, s>>>(deg, nf, start);
  if (np > 0) LYA_COUNT(1), x3_fill_kernel<<<grid_for(np, 256), 256, 0, s>>>(a.pairs, np, start, cur, nbr);
  LYA_TRY(cudaGetLastError());
  // neighbour capacity per block: the longest chords of any vertex (counting
  // pass, synchronising); a list beyond one block's shared memory is reported,
  // not truncated
  const int per_cand = 32;
  int* dmax = reinterpret_cast<int*>(sc + o_misc + 64);
  LYA_TRY(cudaMemsetAsync(dmax, 0, 4, s));
  if (a.n_pix > 0 && nf > 0)
    LYA_COUNT(1), xi3_count_kernel<<<dev.sms * 8, 256, 0, s>>>(a, nbr, start, dmax);
  int hmax = 0;
  LYA_TRY(cudaMemcpyAsync(&hmax, dmax, 4, cudaMemcpyDeviceToHost, s));
  LYA_TRY(cudaStreamSynchronize(s));
  const int cap_max = (dev.smem_optin - 1024) / per_cand;
  const int cap = std::max(std::min(hmax, cap_max), 256);
  const int smem = cap * per_cand;
  if (smem > dev.smem_optin) return cudaErrorInvalidValue;
  LYA_TRY(set_max_dynamic_smem(reinterpret_cast<const void*>(xi3_kernel), smem));
  int per_sm = 0;
  LYA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, xi3_kernel, kX3Threads, smem));
  if (per_sm < 1) return cudaErrorInvalidValue;
  if (a.n_pix > 0 && nf > 0)
    LYA_COUNT(1), xi3_kernel<<<per_sm * dev.sms, kX3Threads, smem, s>>>(a, nbr, start, cap, sums, counter, err);
  LYA_TRY(cudaGetLastError());
  LYA_COUNT(1), xi3_finalize_kernel<<<grid_for(nbins, 256), 256, 0, s>>>(sums, a.num, a.wsum, a.xi, a.n_r, a.n_theta,
                                                                        a.n_alpha);
  return cudaGetLastError();
}

}  // namespace lya
