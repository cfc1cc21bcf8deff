// Forest x quasar cross-correlation, its distortion matrix, and the
// same-forest (1D) correlation -- the extensions the paper names as future
// work (Section 4), built on the estimator of Eq. (2.4), the bisector split of
// Section 2.1 and the projection of Eqs. (2.6)-(2.7).
//
// Cross-correlation.  A quasar q (distance d_q, weight w_q) plays the second
// pixel of Eq. (2.4) with delta = 1:
//     N_A = sum_{(i,q) in A} (w delta)_i w_q,   W_A = sum_{(i,q) in A} w_i w_q,
// r_par = (d_i - d_q) cos(theta/2) signed and binned over [-r_par_max, r_par_max),
// r_perp = (d_i + d_q) sin(theta/2).  The (forest, quasar) list is grouped by
// forest: xcf_kernel.  A lane bins one pixel in FP32 as x = fma(x_i, c/D_par, X0),
// y = fma(x_i, s/D_perp, Y0) (X0, Y0 formed in FP64).
//
// Distortion matrix.  With eta = I - 1 u^T - x v^T the pair (a, q) adds
// w_q (diag(alpha) - alpha alpha^T / W_a - beta beta^T / S_a) on the bins its
// window touches, alpha[B] = sum_{k in B} w_k, beta[B] = sum_{k in B} w_k x_k:
// xdm_kernel; D = D~ / W_A row by row.
//
// 1D correlation.  Described at xi1d_kernel.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "dfloat.cuh"
#include "exact.cuh"
#include "fixed.cuh"

namespace lya {
namespace {

constexpr int kXW = 8;    // warps per block (distortion matrix)
constexpr int kXdmCap = 32;   // least entries of a warp's run list: it passes 64 pairs
constexpr int kXCW = 32;  // warps per block of the cross-correlation (one block per SM)
constexpr int kPad1 = 48;   // sentinels past a forest (a block of 8 rows and 32 lags reaches 39 past it)
constexpr unsigned kFull = 0xffffffffu;

// FP32 bin coordinates of a (forest, quasar) pair:
//   x = (r_par + r_par_max) / D_par = fma(x_i, cP, X0),  y = r_perp / D_perp = fma(x_i, sP, Y0)
// for the packed pixel distance x_i = fl32(d_i - dref), and the window [i0, i1)
// of pixels that can fall in the grid (0.5 Mpc/h wider than the FP32 rounding).
struct XGeo {
  float cP, sP, X0, Y0;
  int i0, i1;
};

__device__ __forceinline__ XGeo pair_geo(const XcfArgs& A, int a, int q, const Pix* fp, int n) {
  const double ax = A.F.ux[a], ay = A.F.uy[a], az = A.F.uz[a];
  const double qx = A.Q.ux[q], qy = A.Q.uy[q], qz = A.Q.uz[q];
  const double dx = ax - qx, dy = ay - qy, dz = az - qz;
  const double sx = ax + qx, sy = ay + qy, sz = az + qz;
  const double s = 0.5 * sqrt(dx * dx + dy * dy + dz * dz);
  const double c = 0.5 * sqrt(sx * sx + sy * sy + sz * sz);
  const double inv_dpar = A.n_par / (2.0 * A.r_par_max), inv_dperp = A.n_perp / A.r_perp_max;
  const double dref = static_cast<double>(A.F.dref[a]), dq = A.Q.dmin[q];
  XGeo g;
  g.cP = static_cast<float>(c * inv_dpar);
  g.sP = static_cast<float>(s * inv_dperp);
  g.X0 = static_cast<float>((dref - dq) * c * inv_dpar + 0.5 * A.n_par);
  g.Y0 = static_cast<float>((dref + dq) * s * inv_dperp);
  const double xq = dq - dref;
  const double half = A.r_par_max / c;
  const double lo = xq - half - 0.5;
  double hi = xq + half + 0.5;
  if (s > 0.0) hi = fmin(hi, A.r_perp_max / s - dref - dq + 0.5);
  g.i0 = count_below(fp, n, static_cast<float>(lo));
  g.i1 = (hi > lo) ? count_below(fp, n, static_cast<float>(hi)) : g.i0;
  if (g.i1 < g.i0) g.i1 = g.i0;
  return g;
}

// Bin of one pixel (-1 outside the grid).  Bins never decrease with x_i.
__device__ __forceinline__ int pixel_bin(const XGeo& g, float x, int n_par, int n_perp) {
  const float xv = fmaf(x, g.cP, g.X0);
  const float yv = fmaf(x, g.sP, g.Y0);
  if (!(xv >= 0.0f) || !(xv < static_cast<float>(n_par)) || !(yv < static_cast<float>(n_perp))) return -1;
  return static_cast<int>(xv) * n_perp + static_cast<int>(yv);
}

// Segmented inclusive scan of two compensated sums (hi, lo) over lanes with
// equal bins (runs are contiguous); returns true on the last lane of a run.
__device__ __forceinline__ bool run_scan(int bin, int lane, float& h1, float& l1, float& h2, float& l2) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int ob = __shfl_up_sync(kFull, bin, d);
    const float oh1 = __shfl_up_sync(kFull, h1, d);
    const float ol1 = __shfl_up_sync(kFull, l1, d);
    const float oh2 = __shfl_up_sync(kFull, h2, d);
    const float ol2 = __shfl_up_sync(kFull, l2, d);
    if (lane >= d && ob == bin) {
      float s, e;
      two_sum(h1, oh1, s, e);
      h1 = s;
      l1 += ol1 + e;
      two_sum(h2, oh2, s, e);
      h2 = s;
      l2 += ol2 + e;
    }
  }
  const int nxt = __shfl_down_sync(kFull, bin, 1);
  return bin >= 0 && (lane == 31 || nxt != bin);
}

__global__ void own_hash_kernel(const int64_t* own, int64_t n, unsigned long long* fp) {
  for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < n; f += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(fp, static_cast<unsigned long long>(
                      splitmix64(static_cast<uint64_t>(f) * 0xD1B54A32D192ED03ull ^ static_cast<uint64_t>(own[f]))));
}

__global__ void qso_prep_kernel(lya_quasars q, Forests Q, unsigned* err, unsigned long long* fp) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < q.n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const double ra = q.ra[k], dec = q.dec[k], d = q.dist[k];
    const float w = q.weight[k];
    const bool fin = isfinite(ra) && isfinite(dec) && isfinite(d) && d > 0.0 && isfinite(w);
    if (!fin) atomicOr(err, FLAG_NONFINITE);
    if (fin && w < 0.0f) atomicOr(err, FLAG_NEGATIVE_W);
    double sr = 0, cr = 1, sd = 0, cd = 1;
    if (fin) {
      sincos(ra, &sr, &cr);
      sincos(dec, &sd, &cd);
    }
    Q.ux[k] = cd * cr;
    Q.uy[k] = cd * sr;
    Q.uz[k] = sd;
    Q.dmin[k] = fin ? d : 1.0;
    Q.len[k] = (fin && w >= 0.0f) ? 1 : 0;
    auto bits = [](double v) { return static_cast<uint64_t>(__double_as_longlong(v)); };
    uint64_t x = splitmix64(static_cast<uint64_t>(k) * 0x9E3779B97F4A7C15ull ^ static_cast<uint64_t>(Q.len[k]));
    x = splitmix64(x ^ bits(ra));
    x = splitmix64(x ^ bits(dec));
    x = splitmix64(x ^ bits(d));
    atomicAdd(fp, static_cast<unsigned long long>(x));
  }
}

// Number of entries of the sorted shared array a[0..n) strictly below v.
__device__ __forceinline__ int count_below_s(const float* a, int n, float v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Two sums times w as unevaluated float pairs (h, l), N and W side by side, to 2^-47 of themselves:
// S = 2^24 H + L, |H| <= 2^24 and L in [-2^23, 2^23) exact in FP32, their products with their errors,
// f = 2^24 times the units of the sums.
__device__ __forceinline__ void run_times(const longlong2& S, float w, F2 f, float2& h, float2& l) {
  const int hn = static_cast<int>((S.x + (1ll << 23)) >> 24), hw = static_cast<int>((S.y + (1ll << 23)) >> 24);
  const int ln = static_cast<int>(static_cast<unsigned>(S.x) - (static_cast<unsigned>(hn) << 24));
  const int lw = static_cast<int>(static_cast<unsigned>(S.y) - (static_cast<unsigned>(hw) << 24));
  const F2 one = f2(1.f, 1.f), neg = f2(-1.f, -1.f), w1 = f2(w, w);
  const float wl = w * 5.9604644775390625e-8f;   // w 2^-24, exact (w > 1e-27)
  const F2 w2 = f2(wl, wl);
  const F2 H = f2(static_cast<float>(hn), static_cast<float>(hw)), L = f2(static_cast<float>(ln), static_cast<float>(lw));
  const F2 np = fma2(H, f2(-w, -w), 0ull), nq = fma2(L, f2(-wl, -wl), 0ull);   // minus the rounded products
  const F2 ns = fma2(np, one, nq);                                             // minus their sum; |p| >= |q| or p = 0
  const F2 err = fma2(fma2(np, neg, ns), one, fma2(nq, neg, 0ull));            // q - (s - p), exact
  h = unf2(fma2(ns, fma2(f, neg, 0ull), 0ull));
  l = unf2(fma2(fma2(err, one, fma2(fma2(H, w1, np), one, fma2(L, w2, nq))), f, 0ull));
}

// sqrt(q) to one unit in the last place: 1 / sqrt(q) to 2e-14 by a Newton step from
// FP32, and the root corrected by its remainder, exact in a fused multiply-add
// (a square root costs twice as many FP64 operations)
__device__ __forceinline__ double root(double q) {
  const float qf = static_cast<float>(q);
  if (!(qf > 1e-30f)) return sqrt(q);
  const double y0 = rsqrtf(qf), h0 = 0.5 * y0;
  const double h = fma(0.5 * h0, fma(-(q * y0), y0, 1.0), h0);   // 1 / (2 sqrt(q))
  const double s = 2.0 * q * h;
  return fma(fma(-s, s, q), h, s);
}

// Window geometry of one (forest, quasar) pair against the forest's staged
// packed distances xs[0..n): as pair_geo, searched in shared memory, the
// window's ends in FP32.
__device__ __forceinline__ XGeo pair_geo_s(const XcfArgs& A, int a, int q, const float* xs, int n) {
  const double ax = A.F.ux[a], ay = A.F.uy[a], az = A.F.uz[a];
  const double qx = A.Q.ux[q], qy = A.Q.uy[q], qz = A.Q.uz[q];
  const double dx = ax - qx, dy = ay - qy, dz = az - qz;
  const double sx = ax + qx, sy = ay + qy, sz = az + qz;
  const double s = 0.5 * root(dx * dx + dy * dy + dz * dz);
  const double c = 0.5 * root(sx * sx + sy * sy + sz * sz);
  const double dref = static_cast<double>(A.F.dref[a]), dq = A.Q.dmin[q];
  const double cp = c * A.inv_dpar, sp = s * A.inv_dperp;
  XGeo g;
  g.cP = static_cast<float>(cp);
  g.sP = static_cast<float>(sp);
  g.X0 = static_cast<float>((dref - dq) * cp + 0.5 * A.n_par);
  g.Y0 = static_cast<float>((dref + dq) * sp);
  // 0 <= x cP + X0 < n_par and x sP + Y0 < n_perp, 0.5 Mpc/h wider (and 1e-5 of the terms)
  const float fnpar = static_cast<float>(A.n_par), fnperp = static_cast<float>(A.n_perp);
  const float lo = -g.X0 / g.cP;
  float hi = (fnpar - g.X0) / g.cP;
  if (g.sP > 0.f) hi = fminf(hi, (fnperp - g.Y0) / g.sP);
  g.i0 = count_below_s(xs, n, lo - (0.5f + 1e-5f * fabsf(lo)));
  g.i1 = count_below_s(xs, n, hi + (0.5f + 1e-5f * fabsf(hi)));
  if (g.i1 < g.i0) g.i1 = g.i0;
  return g;
}

// One block per SM: teams of warps, each staging one forest at a time (atomic
// counter) with integer prefix sums of its packed w delta and w on the forest's
// own power-of-two scales (43 bits; the FP32 values are exact on them down to
// 2^-19 of the largest, and so are the sums).  A forest with smaller weights than
// that (or w delta of 32 neighbouring pixels below 2^-12), and scales out of FP32's
// range, are summed pixel by pixel.  Warps take 32 of the forest's quasars at a time, one pair's geometry
// per lane, then walk each pair's window together: bins ascend along the
// window, so a run of equal bins [j0, j] sits in adjacent lanes, and its last
// lane adds w_q (P[j + 1] - P[j0]) as a float pair to the block's double-float
// histogram (bounded compare-and-swap), flushed to FP64 once per block.  The
// teams are as many and as small as shared memory allows (single warps up to
// about 230 pixels at 5,000 bins): a team waits for its slowest warp at every
// forest.
// What bounds it: issue, about 100 warp instructions per 32 pixels.
// Measured (60,000 x 90,000, 100 x 50 bins): 27.5 ms with a compensated
// segmented scan over the lanes per 32 pixels and FP64 square roots, divisions
// and window ends per pair; 18 ms with the prefix sums in teams of eight warps,
// 16 ms in as many teams as fit, 17.5 ms with the run sums' low halves and the
// sums by pixel for forests that the integers do not hold.
__global__ void __launch_bounds__(kXCW * 32, 1) xcf_kernel(XcfArgs A, int cap, int team_warps, unsigned long long* counter) {
  // [nb] (num hi, num lo, w hi, w lo) | per team: inclusive prefix sums (w delta, w) [cap] | per team: distances [cap]
  extern __shared__ float4 xs4[];
  const int nb = A.n_par * A.n_perp;
  float4* hist = xs4;
  for (int k = threadIdx.x; k < nb; k += blockDim.x) hist[k] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int teams = kXCW / team_warps;
  const int team = wi / team_warps, tw = wi % team_warps, tt = threadIdx.x % (team_warps * 32);
  longlong2* pre = reinterpret_cast<longlong2*>(xs4 + nb) + static_cast<size_t>(team) * cap;
  float* xs = reinterpret_cast<float*>(reinterpret_cast<longlong2*>(xs4 + nb) + static_cast<size_t>(teams) * cap) +
              static_cast<size_t>(team) * cap;
  auto sync = [&]() {
    if (team_warps == 1) __syncwarp();
    else team_sync(1 + team, team_warps * 32);   // (at most 8 teams of more than one warp)
  };
  for (;;) {
    sync();   // the team's previous forest's readers are done
    long long f = 0;
    if (tt == 0) f = static_cast<long long>(atomicAdd(counter, 1ull));
    if (team_warps == 1) {
      f = __shfl_sync(kFull, f, 0);
    } else {   // by way of the staging buffer
      if (tt == 0) pre[0].x = f;
      sync();
      f = pre[0].x;
      sync();
    }
    if (f >= A.F.n) break;
    const int64_t q0 = A.qoff[f], q1 = A.qoff[f + 1];
    const int n = A.F.len[f];
    if (q1 <= q0 || n <= 0 || n > cap) continue;   // uniform over the team
    const Pix* fp = A.pix + A.F.off[f];
    const float mn = A.F.wdmax[f], mw = A.F.wmax[f];
    // smallest w that is not 0, and smallest of the 32-pixel segments' largest |w delta| that is not 0 (not of less
    // than 16 pixels at the forest's end), by the bits of the FP32 values
    uint32_t low_w = 0xFFFFFFFFu, low_n = 0xFFFFFFFFu;
    for (int k0 = 0; k0 < n; k0 += 32) {
      const Pix P = (k0 + lane < n) ? fp[k0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
      const uint32_t top = __reduce_max_sync(kFull, __float_as_uint(fabsf(P.z)));
      if (top && (n - k0 >= 16 || k0 == 0)) low_n = min(low_n, top);
      if (P.y > 0.f) low_w = min(low_w, __float_as_uint(P.y));
    }
    low_w = __reduce_min_sync(kFull, low_w);
    // |value| 2^e < 2^43
    const bool plain = !(mn < 1e18f && mw < 1e18f && (mn == 0.f || (mn > 1e-24f && mn <= 4096.f * __uint_as_float(low_n))) &&
                         (mw == 0.f || (mw > 1e-24f && mw <= 524288.f * __uint_as_float(low_w))));
    const int en = (mn > 0.f && !plain) ? 42 - ilogbf(mn) : 0, ew = (mw > 0.f && !plain) ? 42 - ilogbf(mw) : 0;
    for (int k = tt; k < n; k += team_warps * 32) xs[k] = fp[k].x;
    if (tw == 0 && !plain) {
      const double sn = pow2(en), sw = pow2(ew);
      long long cn = 0, cw = 0;
      for (int base = 0; base < n; base += 32) {
        const int k = base + lane;
        long long vn = 0, vw = 0;
        if (k < n) {
          const Pix P = fp[k];
          vn = __double2ll_rn(static_cast<double>(P.z) * sn);
          vw = __double2ll_rn(static_cast<double>(P.y) * sw);
        }
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const long long on = __shfl_up_sync(kFull, vn, d), ow = __shfl_up_sync(kFull, vw, d);
          if (lane >= d) {
            vn += on;
            vw += ow;
          }
        }
        vn += cn;
        vw += cw;
        if (k < n) pre[k] = make_longlong2(vn, vw);
        cn = __shfl_sync(kFull, vn, 31);
        cw = __shfl_sync(kFull, vw, 31);
      }
    }
    sync();
    const F2 unit = f2(ldexpf(1.f, 24 - en), ldexpf(1.f, 24 - ew));   // see run_times
    for (int64_t qb = q0 + static_cast<int64_t>(tw) * 32; qb < q1; qb += team_warps * 32) {
      XGeo g{0.f, 0.f, 0.f, 0.f, 0, 0};
      float wq = 0.f;
      const int64_t k = qb + lane;
      if (k < q1) {
        const int q = A.pairs[k].y;
        if (q >= 0 && A.Q.len[q] > 0) {
          g = pair_geo_s(A, static_cast<int>(f), q, xs, n);
          wq = A.wq[q];
        }
      }
      const int nq = static_cast<int>((q1 - qb < 32) ? (q1 - qb) : 32);
      for (int t = 0; t < nq; ++t) {
        const int i0 = __shfl_sync(kFull, g.i0, t), i1 = __shfl_sync(kFull, g.i1, t);
        if (i1 <= i0) continue;
        XGeo h;
        h.cP = __shfl_sync(kFull, g.cP, t);
        h.sP = __shfl_sync(kFull, g.sP, t);
        h.X0 = __shfl_sync(kFull, g.X0, t);
        h.Y0 = __shfl_sync(kFull, g.Y0, t);
        const float wqt = __shfl_sync(kFull, wq, t);
        const bool by_pixel = plain || !(wqt < 1e27f && (wqt > 1e-27f || wqt == 0.f));
        for (int base = i0; base < i1; base += 32) {
          const int j = base + lane;
          const int bin = (j < i1) ? pixel_bin(h, xs[j], A.n_par, A.n_perp) : -1;
          const int prev = __shfl_up_sync(kFull, bin, 1), nxt = __shfl_down_sync(kFull, bin, 1);
          const unsigned heads = __ballot_sync(kFull, lane == 0 || prev != bin);
          if (bin >= 0 && (lane == 31 || nxt != bin)) {
            const int j0 = base + 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
            float2 hi = make_float2(0.f, 0.f), lo = hi;   // N, W
            if (!by_pixel) {
              longlong2 S = pre[j];
              if (j0 > 0) {
                const longlong2 p = pre[j0 - 1];
                S.x -= p.x;
                S.y -= p.y;
              }
              run_times(S, wqt, unit, hi, lo);
            } else {
              for (int i = j0; i <= j; ++i) {
                const float pn = wqt * fp[i].z, pw = wqt * fp[i].y;
                float s, e;
                two_sum(hi.x, pn, s, e);
                hi.x = s;
                lo.x += e + fmaf(wqt, fp[i].z, -pn);
                two_sum(hi.y, pw, s, e);
                hi.y = s;
                lo.y += e + fmaf(wqt, fp[i].y, -pw);
              }
            }
            df_atomic_add(reinterpret_cast<float2*>(&hist[bin]), hi.x, lo.x, A.err);
            df_atomic_add(reinterpret_cast<float2*>(&hist[bin]) + 1, hi.y, lo.y, A.err);
          }
          __syncwarp();
        }
      }
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nb; k += blockDim.x) {
    const float4 v = hist[k];
    const double sn = static_cast<double>(v.x) + static_cast<double>(v.y);
    const double sw = static_cast<double>(v.z) + static_cast<double>(v.w);
    if (sn != 0.0) red_add_f64_global(A.num + k, sn);
    if (sw != 0.0) red_add_f64_global(A.wsum + k, sw);
  }
}

// Kept (forest, quasar) pairs, one per warp at a time.  A warp draws its pairs
// 32 at a time and collects the kept ones, at most one per lane and the next 31
// by way of its run lists' memory; with 32 of them (or at the end) each lane computes one pair's geometry, window and normalisers in FP64 (with
// all lanes on one pair that cost as much as the pair's updates), and the warp
// takes the pairs in turn: the runs of its window in shared memory, scaled to
// al = alpha sqrt(w_q / W_a) and be = beta sqrt(w_q / S_a), then the upper
// triangle -(al al^T + be be^T), two FP64 operations per entry, rows r and
// L - 1 - r together so that the lanes stay full.
// What bounds it: the FP64 pipe (two operations of 19 clocks per 32 entries)
// and L2's atomics (entries of consecutive runs are consecutive in G).
// Measured (60,000 x 90,000, 2% of the pairs): 31.0 ms with the geometry in all
// lanes, five FP64 operations per entry and G numbered p n_perp + t; with the
// rest of its call 12 ms as it is.
__global__ void __launch_bounds__(kXW * 32) xdm_kernel(XcfArgs A, int cap) {
  extern __shared__ double dsh[];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nwb = blockDim.x >> 5;
  double* lal = dsh + static_cast<size_t>(wi) * 2 * cap;
  double* lbe = lal + cap;
  int* lA = reinterpret_cast<int*>(dsh + static_cast<size_t>(nwb) * 2 * cap) + static_cast<size_t>(wi) * cap;
  int2* pass = reinterpret_cast<int2*>(lal);   // 64 pairs: cap >= kXdmCap
  const int nb = A.n_par * A.n_perp;
  const int all = A.p_subsample >= 1.0;
  const uint64_t thr = all ? 0 : static_cast<uint64_t>(A.p_subsample * 18446744073709551616.0);
  const int64_t nw = static_cast<int64_t>(gridDim.x) * nwb;
  int held = 0;   // pairs kept so far (uniform), one in `own` of each of the first lanes
  int2 own = make_int2(-1, -1);
  for (int64_t k0 = (blockIdx.x * static_cast<int64_t>(nwb) + wi) * 32;; k0 += nw * 32) {
    const bool last = k0 >= A.n_pairs;
    bool keep = false;
    int2 pr = make_int2(-1, -1);
    if (k0 + lane < A.n_pairs) {
      pr = A.pairs[k0 + lane];
      keep = pr.x >= 0 && pr.y >= 0 &&
             (all || splitmix64(A.seed ^ ((static_cast<uint64_t>(pr.x) << 32) | static_cast<uint64_t>(pr.y))) < thr);
      keep = keep && A.F.len[pr.x] > 0 && A.Q.len[pr.y] > 0;
    }
    const unsigned km = __ballot_sync(kFull, keep);
    if (km) {
      // the new ones behind those held
      __syncwarp();
      if (lane < held) pass[lane] = own;
      if (keep) pass[held + __popc(km & ((1u << lane) - 1u))] = pr;
      held += __popc(km);
      __syncwarp();
      if (lane < held) own = pass[lane];
      if (lane + 32 < held) pr = pass[lane + 32];
      __syncwarp();
    }
    if (held < 32 && !last) continue;
    const int nq = min(held, 32);
    const int2 rest = pr;   // of the first held - 32 lanes: kept for the next turn
    // one pair's geometry per lane
    XGeo mine{0.f, 0.f, 0.f, 0.f, 0, 0};
    double cw = 0.0, cs = 0.0;   // sqrt(w_q / W_a), sqrt(w_q / S_a) (0 where eta lacks the term)
    if (lane < nq) {
      pr = own;
      mine = pair_geo(A, pr.x, pr.y, A.pix + A.F.off[pr.x], A.F.len[pr.x]);
      const double wq = static_cast<double>(A.wq[pr.y]);
      const double Wa = A.F.wsum[pr.x], Sa = A.F.ssum[pr.x];
      if (A.eta_mean_slope && Wa > 0.0) {
        cw = sqrt(wq / Wa);
        cs = (Sa > 0.0) ? sqrt(wq / Sa) : 0.0;
      }
    }
    for (int m = 0; m < nq; ++m) {
      const int a = __shfl_sync(kFull, pr.x, m), q = __shfl_sync(kFull, pr.y, m);
      XGeo g;
      g.i0 = __shfl_sync(kFull, mine.i0, m);
      g.i1 = __shfl_sync(kFull, mine.i1, m);
      g.cP = __shfl_sync(kFull, mine.cP, m);
      g.sP = __shfl_sync(kFull, mine.sP, m);
      g.X0 = __shfl_sync(kFull, mine.X0, m);
      g.Y0 = __shfl_sync(kFull, mine.Y0, m);
      const double sw = __shfl_sync(kFull, cw, m), ss = __shfl_sync(kFull, cs, m);
      const Pix* fp = A.pix + A.F.off[a];
      int L = 0, lastA = -1;
      for (int base = g.i0; base < g.i1; base += 32) {
        const int i = base + lane;
        int bin = -1;
        float ha = 0.f, la = 0.f, hb = 0.f, lb = 0.f;
        if (i < g.i1) {
          const Pix P = fp[i];
          bin = pixel_bin(g, P.x, A.n_par, A.n_perp);
          if (bin >= 0) {
            bin = (bin % A.n_perp) * A.n_par + bin / A.n_perp;   // as G numbers it; also ascending along the window
            ha = P.y;
            hb = P.y * P.w;
            lb = fmaf(P.y, P.w, -hb);
          }
        }
        const bool tail = run_scan(bin, lane, ha, la, hb, lb);
        const unsigned tm = __ballot_sync(kFull, tail);
        if (tm) {
          const int fbin = __shfl_sync(kFull, bin, __ffs(tm) - 1);
          const int merged = (fbin == lastA) ? 1 : 0;   // run continued from the previous chunk
          if (tail) {
            const int r = __popc(tm & ((1u << lane) - 1u));
            const double va = static_cast<double>(ha) + static_cast<double>(la);
            const double vb = static_cast<double>(hb) + static_cast<double>(lb);
            if (r == 0 && merged) {
              lal[L - 1] += va;
              lbe[L - 1] += vb;
            } else {
              const int slot = L + r - merged;
              lA[slot] = bin;
              lal[slot] = va;
              lbe[slot] = vb;
            }
          }
          lastA = __shfl_sync(kFull, bin, 31 - __clz(tm));
          L += __popc(tm) - merged;
        }
        __syncwarp();
      }
      if (L == 0) continue;
      const double wq = static_cast<double>(A.wq[q]);
      for (int r = lane; r < L; r += 32) {
        const double v = wq * lal[r];
        const int64_t b = lA[r];
        red_add_f64_global(A.wdm + b, v);
        if (v != 0.0) red_add_f64_global(A.G + b * nb + b, v);
        lal[r] *= sw;
        lbe[r] *= ss;
      }
      __syncwarp();
      if (sw != 0.0) {
        for (int r = 0; 2 * r < L; ++r) {
          // row r from its diagonal on, then row L - 1 - r (L + 1 entries together; once where they are the same row)
          const int r2 = L - 1 - r;
          const int n1 = L - r, n = (r2 > r) ? L + 1 : n1;
          for (int e = lane; e < n; e += 32) {
            const int row = (e < n1) ? r : r2;
            const int c = (e < n1) ? r + e : r2 + (e - n1);
            const double v = fma(lbe[row], lbe[c], lal[row] * lal[c]);
            if (v != 0.0) red_add_f64_global(A.G + static_cast<int64_t>(lA[row]) * nb + lA[c], -v);
          }
        }
      }
      __syncwarp();
    }
    held -= nq;
    if (lane < held) own = rest;
    if (last) break;   // (a turn leaves pairs only where it has drawn some)
  }
}

// One forest per warp at a time (atomic counter).  Lane l takes the pixel pairs
// (i, i + lag + l) of a group of 32 lags, whose separations change slowly with
// i, so a run of pairs in one bin is tens of pairs long; products and sums are
// the exact integers of exact.cuh, added to the warp's 64-bit histogram per run
// and to FP64 sums per forest.  With S = SumF64 they are FP64: a second launch
// for the forests, left by the first, whose values lie so far apart that a run
// would be rounded by more than 2^-36 of its smallest product (survey weights
// reach 12 of the 15 bits).  p = floor((d_j - d_i) / D) is taken from the
// FP32 packed distances when that value lies farther than `guard` from an
// integer (the FP32 error is below guard / 2), else from the FP64 division of
// the definition, so every bin is the definition's.
// What bounds it: issue (71%), about 55 warp instructions per step of 32 pairs.
// Measured (60,000 SDSS-like forests, 8.5e8 pairs): one warp per pixel with
// FP64 prefix sums and two shared FP64 atomics per run of two pixels 25.1 ms,
// this form 2.5 ms, and 0.05 ms for 21 forests of the second launch (0.13 ms with
// a warp on a whole forest).
template <class S>
__global__ void __launch_bounds__(256) xi1d_kernel(X1Args A, const Pix* pix, int acc_bins, int stage, int per_warp,
                                                   unsigned long long* counter, unsigned* n_wide) {
  constexpr bool kExact = std::is_same<S, Sum64>::value;
  // with FP64 sums an item is one group of 32 lags: a few forests have to fill the GPU
  const unsigned groups = kExact ? 1u : static_cast<unsigned>(A.max_len + 30) / 32u;
  const unsigned long long n_items = kExact ? static_cast<unsigned long long>(A.F.n) : static_cast<unsigned long long>(*n_wide) * groups;
  if (n_items == 0ull) return;
  // per warp: histogram (N, W) of n_bins + 1 bins, u64 | FP64 sums of acc_bins bins | H, L [stage] | distances [stage]
  extern __shared__ __align__(16) unsigned char dyn[];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  unsigned char* mine = dyn + static_cast<size_t>(wi) * per_warp;
  unsigned long long* hist = reinterpret_cast<unsigned long long*>(mine);
  double2* acc = reinterpret_cast<double2*>(hist + 2 * (A.n_bins + 1));
  int4* v = reinterpret_cast<int4*>(acc + acc_bins);
  float* xs = reinterpret_cast<float*>(v + stage);
  for (int q = lane; q < 2 * (A.n_bins + 1); q += 32) hist[q] = 0ull;
  for (int q = lane; q < acc_bins; q += 32) acc[q] = make_double2(0.0, 0.0);
  const double dr = A.r_max / A.n_bins;
  const float inv_dr = static_cast<float>(A.n_bins / A.r_max), fbins = static_cast<float>(A.n_bins);
  const uint32_t base = smem_addr(hist) - 16u * kMagicBits;
  const uint32_t off_grid = kMagicBits + static_cast<uint32_t>(A.n_bins);
  for (;;) {
    unsigned long long f = 0;
    if (lane == 0) f = atomicAdd(counter, 1ull);
    f = __shfl_sync(kFull, f, 0);
    if (f >= n_items) break;
    int first = 1;   // first lag
    if (!kExact) {
      first += 32 * static_cast<int>(f % groups);
      f = static_cast<unsigned long long>(A.wide[f / groups]);
    }
    const int n = A.F.len[f];
    if (n < 2 || n > A.max_len) continue;
    const int64_t o = A.F.off[f];
    __syncwarp();
    // by the high words of the FP64 values: largest |w delta| and |w|, smallest w that is not 0, and smallest of
    // the 32-pixel segments' largest |w delta| that is not 0 (not of less than 16 pixels at the forest's end)
    uint32_t mn = 0u, mw = 0u, ln = 0xFFFFFFFFu, lw = 0xFFFFFFFFu;
    float tn = 0.f, tw = 0.f;
    for (int k0 = 0; k0 < n; k0 += 32) {
      const int k = k0 + lane;
      const float wf = (k < n) ? A.weight[o + k] : 0.f;
      const double w = static_cast<double>(wf), wd = (k < n) ? fabs(w * static_cast<double>(A.delta[o + k])) : 0.0;
      const uint32_t hw = static_cast<uint32_t>(__double2hiint(w)) & 0x7FFFFFFFu;
      const uint32_t top = __reduce_max_sync(kFull, static_cast<uint32_t>(__double2hiint(wd)));
      mn = max(mn, top);
      mw = max(mw, hw);
      if (hw) lw = min(lw, hw);
      if (top && (n - k0 >= 16 || k0 == 0)) ln = min(ln, top);
      tn += static_cast<float>(wd);
      tw += wf;
    }
    mw = __reduce_max_sync(kFull, mw);
    lw = __reduce_min_sync(kFull, lw);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      tn += __shfl_xor_sync(kFull, tn, d);
      tw += __shfl_xor_sync(kFull, tw, d);
    }
    // |value| < 2^(exponent + 1) scaled below 2^54
    const int en = (mn >> 20) ? 53 - (static_cast<int>(mn >> 20) - 1023) : 0;
    const int ew = (mw >> 20) ? 53 - (static_cast<int>(mw >> 20) - 1023) : 0;
    const double sn = pow2(en), sw = pow2(ew);
    // a bin holds at most D / gap + 2 partners of a pixel, and no more than half the square of the values' sum
    // (in units of 2^54); its sum stays below 2^62
    const float qn = static_cast<float>(static_cast<double>(tn) * pow2(en - 54)), qw = static_cast<float>(static_cast<double>(tw) * pow2(ew - 54));
    const float terms = fminf(fminf(static_cast<float>(n) * (static_cast<float>(dr) / A.F.hmin[f] + 2.f),
                                    0.5f * static_cast<float>(n) * static_cast<float>(n)),
                              0.501f * fmaxf(qn * qn, qw * qw) + 1.f);
    const int shift = max(1, static_cast<int>((__float_as_uint(fmaxf(terms, 1.f)) >> 23) & 0xFFu) - 126 - 10);
    // log2 of largest over smallest, from exponent and mantissa in one (0.1: their log2 is less than 0.09 off)
    const float rn = mn ? (ln != 0xFFFFFFFFu ? static_cast<float>(mn - ln) * 9.5367431640625e-7f + 0.1f : 128.f) : 0.f;
    const float rw = mw ? static_cast<float>(mw - lw) * 9.5367431640625e-7f + 0.1f : 0.f;
    if (kExact && 2.f * fmaxf(rn, rw) + static_cast<float>(shift) > 15.f) {
      if (lane == 0) A.wide[atomicAdd(n_wide, 1u)] = static_cast<int32_t>(f);
      continue;
    }
    for (int k = lane; k < n + kPad1; k += 32) {
      const bool in = k < n;
      xs[k] = in ? pix[o + k].x : INFINITY;
      const double w = in ? static_cast<double>(A.weight[o + k]) : 0.0;
      const double wd = in ? w * static_cast<double>(A.delta[o + k]) : 0.0;
      if (kExact) {
        const int2 a = split55(wd, sn), b = split55(w, sw);
        v[k] = make_int4(a.x, a.y, b.x, b.y);
      } else {
        v[k] = pack_f64(wd, w);
      }
    }
    __syncwarp();
    // |FP32 value - exact quotient| < 2^-22 (2 xs_max + r_max) / D + 2^-22 n_bins  (half of the guard)
    const float guard = 2.384185791015625e-7f * ((2.0f * xs[n - 1] + static_cast<float>(A.r_max)) * inv_dr + fbins) + 1e-6f;
    const float half = 0.5f - guard;
    bool more = true;
    for (int lag = first; lag < n && more; lag += 32) {
      // separations grow with the lag: a group none of whose rows can be in range ends the walk
      more = false;
      for (int r0 = 0; r0 < n - lag; r0 += 256) {
        // lane m: whether rows r0 + 8 m .. + 7 can hold a pair in range (that of the smallest lag, 1e-2 bins
        // wider than the rounding)
        const int i0 = r0 + 8 * lane, i1 = min(i0 + 7, n - 1);
        const bool work = i0 + lag < n && (xs[i0 + lag] - xs[i1]) * inv_dr < fbins + 1e-2f;
        unsigned todo = __ballot_sync(kFull, work);
        more = more || todo != 0u;
        S run{};
        uint32_t cur = off_grid;
        for (; todo; todo &= todo - 1u) {
          const int ib = r0 + 8 * (__ffs(todo) - 1);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int i = ib + q, j = i + lag + lane;
            const float t = (xs[j] - xs[i]) * inv_dr;
            const float tm = __fadd_rd(t, kMagic);
            const bool near = fabsf((t - (tm - kMagic)) - 0.5f) > half;
            uint32_t key = __float_as_uint(fminf(tm, kMagic + fbins));
            if (__any_sync(kFull, near)) {   // (never of the padding: its coordinates are infinite or NaN)
              const double pe = floor((A.dist[o + min(j, n - 1)] - A.dist[o + min(i, n - 1)]) / dr);
              const uint32_t exact = (pe < static_cast<double>(A.n_bins)) ? kMagicBits + static_cast<uint32_t>(static_cast<int>(pe)) : off_grid;
              key = near ? exact : key;
            }
            const bool chg = key != cur;
            if (__any_sync(kFull, chg)) {
              if (chg) {
                if (cur != off_grid) add_bin64(run, base + (cur << 4), shift);
                run = S{};
                cur = key;
              }
              __syncwarp();
            }
            add_products(run, v[i], v[j]);
          }
        }
        if (cur != off_grid) add_bin64(run, base + (cur << 4), shift);
        __syncwarp();
      }
      if (!kExact) break;
    }
    // the forest's sums -> FP64 sums
    const double un = pow2(56 + shift - 2 * en), uw = pow2(56 + shift - 2 * ew);
    for (int q = lane; q < A.n_bins; q += 32) {
      const long long hn = static_cast<long long>(hist[2 * q]), hw = static_cast<long long>(hist[2 * q + 1]);
      if ((hn | hw) == 0) continue;
      const double dn = kExact ? static_cast<double>(hn) * un : __longlong_as_double(hn);
      const double dw = kExact ? static_cast<double>(hw) * uw : __longlong_as_double(hw);
      if (q < acc_bins) {
        acc[q].x += dn;
        acc[q].y += dw;
      } else {
        red_add_f64_global(A.num + q, dn);
        red_add_f64_global(A.wsum + q, dw);
      }
      hist[2 * q] = 0ull;
      hist[2 * q + 1] = 0ull;
    }
  }
  // the block's warps together, so that the FP64 sums in global memory take few terms
  __syncthreads();
  for (int q = threadIdx.x; q < acc_bins; q += blockDim.x) {
    double n = 0.0, w = 0.0;
    for (int m = 0; m < static_cast<int>(blockDim.x >> 5); ++m) {
      const double2 t = reinterpret_cast<const double2*>(dyn + static_cast<size_t>(m) * per_warp + 16 * (A.n_bins + 1))[q];
      n += t.x;
      w += t.y;
    }
    if (n != 0.0) red_add_f64_global(A.num + q, n);
    if (w != 0.0) red_add_f64_global(A.wsum + q, w);
  }
}

int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 1 << 16) b = 1 << 16;
  return static_cast<int>(b);
}

}  // namespace

// The grids and forest lengths the entry point takes (16 bytes per bin and 40
// per pixel of the longest forest within a block's shared memory).
int xcf_limit_bytes(int nb, int max_len) {
  const int cap = std::max(max_len, 1);
  return 16 * nb + 2 * 20 * cap;
}

int xdm_warps(const DevInfo& dev, int max_len) {
  const int64_t per_warp = 20LL * std::max(max_len, kXdmCap);
  int w = static_cast<int>(std::min<int64_t>(kXW, dev.smem_optin / per_warp));
  return w;   // 0: forests too long for the run lists
}

// The bins and forest lengths the entry point takes (16 bytes per bin and 28
// per pixel of the longest forest within a block's shared memory).
int xi1d_limit_bytes(int n_bins, int max_len) {
  const int cap = std::max(max_len, 1);
  return 16 * n_bins + 16 * (cap + 1) + 12 * cap;
}

cudaError_t launch_qso_prep(const lya_quasars& q, Forests Q, unsigned* err, unsigned long long* fp,
                            cudaStream_t s) {
  if (q.n <= 0) return cudaSuccess;
  LYA_COUNT(1), qso_prep_kernel<<<grid_for(q.n, 256), 256, 0, s>>>(q, Q, err, fp);
  return cudaGetLastError();
}

cudaError_t launch_own_hash(const int64_t* own, int64_t n, unsigned long long* fp, cudaStream_t s) {
  if (!own || n <= 0) return cudaSuccess;
  LYA_COUNT(1), own_hash_kernel<<<grid_for(n, 256), 256, 0, s>>>(own, n, fp);
  return cudaGetLastError();
}

cudaError_t launch_xcf(const XcfArgs& a, unsigned long long* counter, const DevInfo& dev, cudaStream_t s) {
  if (a.n_pairs == 0) return cudaSuccess;
  const int cap = std::max(a.max_len, 1), nb = a.n_par * a.n_perp;
  // the most teams whose staging fits beside the histogram (power of two; named barriers serve up to 8)
  int team_warps = 1;
  while (team_warps < kXCW && (team_warps == 2 || 16 * nb + (kXCW / team_warps) * 20 * cap > dev.smem_optin))
    team_warps *= 2;
  const int smem = 16 * nb + (kXCW / team_warps) * 20 * cap;
  cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(xcf_kernel), smem);
  if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  const int blocks = static_cast<int>(std::min<int64_t>(dev.sms, a.F.n));
  LYA_COUNT(1), xcf_kernel<<<blocks, kXCW * 32, smem, s>>>(a, cap, team_warps, counter);
  return cudaGetLastError();
}

cudaError_t launch_xdm(const XcfArgs& a, const DevInfo& dev, cudaStream_t s) {
  if (a.n_pairs == 0 || a.p_subsample <= 0.0) return cudaSuccess;
  const int warps = xdm_warps(dev, a.max_len);
  if (warps < 1) return cudaErrorInvalidConfiguration;
  const int cap = std::max(a.max_len, kXdmCap);
  const int smem = warps * 20 * cap;
  cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(xdm_kernel), smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, xdm_kernel, warps * 32, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int64_t want = (a.n_pairs + warps - 1) / warps;
  const int blocks = static_cast<int>(std::min<int64_t>(static_cast<int64_t>(dev.sms) * per_sm, want));
  LYA_COUNT(1), xdm_kernel<<<blocks, warps * 32, smem, s>>>(a, cap);
  return cudaGetLastError();
}

cudaError_t launch_xi1d(const X1Args& a, const Pix* pix, unsigned long long* counter, const DevInfo& dev, cudaStream_t s) {
  if (a.F.n == 0) return cudaSuccess;
  // FP64 sums per warp where the grid is small enough not to crowd out warps
  const int acc_bins = a.n_bins <= 512 ? a.n_bins : 0;
  const int stage = std::max(a.max_len, 1) + kPad1;
  const int per_warp = (16 * (a.n_bins + 1 + acc_bins) + 20 * stage + 15) & ~15;
  const int warps = std::max(1, std::min(8, dev.smem_optin / per_warp));
  const int smem = warps * per_warp;
  cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(xi1d_kernel<Sum64>), smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(reinterpret_cast<const void*>(xi1d_kernel<SumF64>), smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, xi1d_kernel<Sum64>, warps * 32, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  unsigned* n_wide = reinterpret_cast<unsigned*>(counter + 1);
  e = cudaMemsetAsync(counter, 0, 2 * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  const int blocks =
      static_cast<int>(std::min<int64_t>(static_cast<int64_t>(dev.sms) * per_sm, (a.F.n + warps - 1) / warps));
  LYA_COUNT(1), xi1d_kernel<Sum64><<<blocks, warps * 32, smem, s>>>(a, pix, acc_bins, stage, per_warp, counter, n_wide);
  e = cudaGetLastError();
  // the forests left by it (the kernel ends at once where there are none)
  if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  LYA_COUNT(1), xi1d_kernel<SumF64><<<blocks, warps * 32, smem, s>>>(a, pix, acc_bins, stage, per_warp, counter, n_wide);
  return cudaGetLastError();
}

}  // namespace lya
