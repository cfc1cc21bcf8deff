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
// Two kernels with the same arithmetic: xi3_group_kernel (several vertices a block,
// sums of a class in shared memory; see there) where it pays, and xi3_kernel: one
// block per main-vertex pixel (work taken from an atomic counter):
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
// What bounds xi3_kernel: the FP64 atomics in L2, which takes one 32-byte sector per
// 2.3 clocks and SM wherever the bins are random; N and W of a bin therefore
// lie side by side and two lanes add a record, so a record costs one sector and
// not two.  Measured (5,000 SDSS-like forests, r_max 40, 200,000 bins): 411 ms
// with separate arrays and FP64 gathers and counts by whole warps, 381 ms with
// the gather and the count per lane, 204 ms with the sums side by side.
#include <algorithm>
#include <math.h>

#include "exact.cuh"
#include "fixed.cuh"

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

// Bins of a neighbour pixel: |r| and the angle to the vertex's line of sight,
// from FP32, and near a bin edge from the definition in FP64.
struct X3Bin {
  double rmax2, inv_dr, inv_dt;
  float inv_dr_f, inv_dt_f, guard_r, guard_t;
  int nr, nt;
  // pixel p of forest o against the vertex at x with line of sight u: false beyond r_max
  __device__ __forceinline__ bool candidate(const X3Args& A, int o, int64_t p, const double* x, const double* u,
                                            float4* r4, int* ir, int* it) const {
    const double dj = A.dist[p];
    const double dx = dj * A.F.ux[o] - x[0], dy = dj * A.F.uy[o] - x[1], dz = dj * A.F.uz[o] - x[2];
    const double r2 = dx * dx + dy * dy + dz * dz;
    if (!(r2 < rmax2 && r2 > 0.0)) return false;
    // 1 / |r| to FP64 by two Newton steps from FP32 (a square root and a division cost five times that)
    const float r2f = static_cast<float>(r2);
    const float y0f = rsqrtf(r2f);
    const double y0 = y0f;
    const double y1 = fma(0.5 * y0, fma(-(r2 * y0), y0, 1.0), y0);
    const double y = fma(0.5 * y1, fma(-(r2 * y1), y1, 1.0), y1);
    const double dot = dx * u[0] + dy * u[1] + dz * u[2];
    const float ctf = static_cast<float>(dot * y);
    const float fr = r2f * y0f * inv_dr_f, ft = acosf(fminf(1.f, fmaxf(-1.f, ctf))) * inv_dt_f;
    const float gr = fr - floorf(fr), gt = ft - floorf(ft);
    int jr = static_cast<int>(fr), jt = static_cast<int>(ft);
    const bool sure = r2f > 1e-30f && fabsf(gr - 0.5f) < 0.5f - guard_r && fabsf(gt - 0.5f) < 0.5f - guard_t &&
                      fabsf(ctf) <= 0.9999f;
    if (!sure) {   // the definition, near a bin edge
      const double r = sqrt(r2);
      const double ct = dot / r;
      jr = static_cast<int>(r * inv_dr);
      jt = static_cast<int>(acos(fmin(1.0, fmax(-1.0, ct))) * inv_dt);
      r4->w = static_cast<float>(1.0 / r);
    } else {
      r4->w = static_cast<float>(y);
    }
    r4->x = static_cast<float>(dx);
    r4->y = static_cast<float>(dy);
    r4->z = static_cast<float>(dz);
    *ir = min(jr, nr - 1);
    *it = min(jt, nt - 1);
    return true;
  }
};
__device__ __forceinline__ X3Bin x3_bin(const X3Args& A) {
  X3Bin b;
  b.rmax2 = A.r_max * A.r_max;
  b.inv_dr = A.n_r / A.r_max;
  b.inv_dt = A.n_theta / M_PI;
  b.inv_dr_f = static_cast<float>(b.inv_dr);
  b.inv_dt_f = static_cast<float>(b.inv_dt);
  // FP32 errors of |r| and theta in bins, doubled: |r| n_r / r_max <= n_r is good to 4 roundings; theta =
  // acos(c) to 5e-6 rad where |c| <= 0.9999 (the FP32 rounding of c over sin theta, and of acosf)
  b.guard_r = 1e-6f * static_cast<float>(A.n_r) + 1e-6f;
  b.guard_t = 1e-5f * b.inv_dt_f + 1e-6f;
  b.nr = A.n_r;
  b.nt = A.n_theta;
  return b;
}

// SPLIT: sums straight in num and wsum, where the device has no room for `sums`.
template <bool SPLIT>
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
  const double rmax2 = A.r_max * A.r_max;
  const X3Bin bin3 = x3_bin(A);
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
    const double xv[3] = {di * nax, di * nay, di * naz}, uv[3] = {nax, nay, naz};
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
          int ir, it;
          in = bin3.candidate(A, o, p, xv, uv, &r4, &ir, &it);
          if (in) {
            q = A.pix[p];
            key = (ir << 16) | it;
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
            double* const at = SPLIT ? ((lane & 1) ? A.wsum : A.num) + b : sums + 2 * static_cast<int64_t>(b) + (lane & 1);
            if (b >= 0) red_add_f64_global(at, static_cast<double>((lane & 1) ? w : n));
          }
        }
      }
    }
  }
}

// ----------------------------------------------------------------------------
// Several main vertices per block: their records of one (r1, r2) class, whose
// n_alpha n_theta^2 bins fit in shared memory, are summed there before they go
// to the FP64 bin sums, so L2 sees one reduction per touched bin, group of
// vertices and sum instead of one per record.
//  * The block takes kXGVerts consecutive pixels, finds the chords of all of them
//    at once (a warp per vertex), and gathers as many of them as its list holds;
//    the list is then counting-sorted by (vertex, |r| bin).
//  * A class (r1 <= r2) is walked by all warps: 16 neighbours q of bin r2 in the
//    half-warps' registers against two neighbours p of bin r1 a step; steps are
//    dealt evenly over the warps.
//  * Sums are exact integers in two words, which shared memory adds natively: the
//    high one in units of 2^eh as fine as the class's largest record (2^21 units)
//    and the sum of all (2^30) allow, the low one with as many bits below as leave
//    room for all records (xg_scale).  A class is summed so only where that rounds
//    the smallest record of W, whose terms are positive, by at most 2^-21 of itself,
//    and one of typical size of N, whose terms come arbitrarily close to 0, by at
//    most 2^-25 (the FP32 product's own rounding is 2^-24; with 2^-24 for W as well
//    the classes with many records, whose low words are short, go to L2: 2,000 forests
//    on 5 x 4 x 8 bins 328 against 218 ms).  Such a class, one with few
//    records (below kXGDirect a bin) and one whose products leave the FP32 range
//    add their records to L2 as xi3_kernel does; with two blocks per SM the one's
//    reductions in L2 run beside the other's in shared memory.
// What bounds it: the shared-memory pipe (four reductions a record, 25 of 32
// lanes on random bins) and L2's atomics.  Measured (5,000 SDSS-like forests,
// r_max 40, 200,000 bins): xi3_kernel 204 ms,
// this 161 ms; three words 227 ms, one block of 1,024 threads per SM 171 ms, no
// direct classes 185 ms, kXGDirect 3, 12, 20: 160, 161, 186 ms; 64-bit words 449
// ms (emulated).  Smaller grids gain more: 13 x 6^2 bins of 100 classes, 1,300
// forests of a denser sky: 163 -> 54 ms.
// ----------------------------------------------------------------------------
constexpr int kXGThreads = 512;
constexpr int kXGSmem = 113 * 1024;   // shared memory of a block: two per SM
constexpr int kXGVerts = 8;     // vertices a work item
constexpr int kXGBatch = 96;     // most neighbour forests of a vertex
constexpr int kXGMaxR = 16;      // most |r| bins
constexpr int kXGMove = 4;       // list entries a thread moves in the sort (list <= 2,048)
constexpr int kXGClasses = kXGMaxR * (kXGMaxR + 1) / 2;
constexpr double kXGGain = 0.5;  // see x3_group_cap
constexpr int kXGDirect = 6;     // records a bin below which a class goes to L2
constexpr int kXGWords = 5;      // words of a bin: N and W in 2 each, and an odd stride

struct XGLay {
  int cr, cw, ck, hist, ch, end;
};
__host__ __device__ inline XGLay xg_layout(int cap, int nbc) {
  XGLay y;
  int o = 0;
  y.cr = o; o += cap * 16;
  y.cw = o; o += cap * 8;
  y.ck = o; o += cap * 8;
  y.hist = o; o += (nbc * kXGWords * 4 + 15) & ~15;
  y.ch = o; o += kXGVerts * (3 * kXGBatch + 1) * 4;
  y.end = o;
  return y;
}

__device__ __forceinline__ float pow2f(int e) { return __uint_as_float(static_cast<uint32_t>(e + 127) << 23); }

// steps of a class for one vertex: tiles of 16 q, two p a step; within one |r|
// bin (same) tile t meets the p below its end only
__device__ __forceinline__ int xg_steps(int np, int nq, bool same) {
  if (np == 0 || nq == 0) return 0;
  if (!same) return ((nq + 15) >> 4) * ((np + 1) >> 1);
  const int T = (nq + 15) >> 4;
  return nq < 2 ? 0 : 4 * T * (T - 1) + ((nq + 1) >> 1);
}

// Scale of one word pair: records of magnitude up to B and total magnitude up to
// T (both with the FP32 rounding of their own sums) as integers of 2^eh, k bits
// below: the smallest eh with B <= 2^21 2^eh and T <= 2^30 2^eh.
__device__ __forceinline__ int xg_scale(float B, float T) {
  const float u = fmaxf(B * 4.76837158e-7f, T * 9.31322575e-10f);   // 2^-21, 2^-30
  return (u > 0.f) ? static_cast<int>((__float_as_uint(u) >> 23) & 0xFFu) - 126 : 0;   // 2^eh > u
}

__global__ void __launch_bounds__(kXGThreads, 2) xi3_group_kernel(X3Args A, const int32_t* nbr, const int64_t* nstart,
                                                                  int cap, double* sums, unsigned long long* counter,
                                                                  unsigned* err) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ long long s_item;
  __shared__ double s_x[kXGVerts][3], s_u[kXGVerts][3];
  __shared__ float2 s_w[kXGVerts];                       // (w delta, w) of the vertex
  __shared__ int s_f[kXGVerts], s_nb[kXGVerts], s_tot[kXGVerts];
  __shared__ int s_n;                                    // list length
  __shared__ int s_ne, s_nc;                             // sum of the exponents and number of the list's |w delta| > 0
  __shared__ float s_typ;                                // log2 of a typical |N| record
  __shared__ int s_st[kXGVerts * kXGMaxR + 1], s_pos[kXGVerts * kXGMaxR];
  __shared__ int s_steps[kXGClasses], s_recs[kXGClasses];
  // per (vertex, |r| bin): sum and largest |w delta|; sum, largest and smallest w > 0 (infinite without one)
  __shared__ float s_sn[kXGVerts * kXGMaxR], s_mn[kXGVerts * kXGMaxR], s_sw[kXGVerts * kXGMaxR];
  __shared__ float s_mw[kXGVerts * kXGMaxR], s_lw[kXGVerts * kXGMaxR];
  __shared__ int s_eh[kXGClasses];                       // a class's scales, (N + 256) 2^16 + (W + 256); -1: direct
  const int nr = A.n_r, nt = A.n_theta, na = A.n_alpha, nbc = na * nt * nt, ncls = nr * (nr + 1) / 2;
  const XGLay y = xg_layout(cap, nbc);
  float4* cr = reinterpret_cast<float4*>(sm + y.cr);     // r (FP32) and 1 / |r|
  float2* cw = reinterpret_cast<float2*>(sm + y.cw);     // (w delta, w)
  int2* ck = reinterpret_cast<int2*>(sm + y.ck);         // ((vertex << 24) | (|r| bin << 16) | theta bin, forest)
  unsigned* hist = reinterpret_cast<unsigned*>(sm + y.hist);
  int* s_o = reinterpret_cast<int*>(sm + y.ch);          // chords: forest, first pixel, exclusive counts
  int* s_lo = s_o + kXGVerts * kXGBatch;
  int* s_pre = s_lo + kXGVerts * kXGBatch;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  constexpr int nwarps = kXGThreads / 32;
  const double rmax2 = A.r_max * A.r_max;
  const X3Bin bin = x3_bin(A);
  const float half_na = 0.5f * static_cast<float>(na);
  for (int k = tid; k < nbc * kXGWords; k += kXGThreads) hist[k] = 0u;
  for (;;) {
    __syncthreads();
    if (wid == 0) {
      long long it = 0;
      if (lane == 0) it = static_cast<long long>(atomicAdd(counter, static_cast<unsigned long long>(kXGVerts)));
      it = __shfl_sync(0xffffffffu, it, 0);
      if (lane == 0) s_item = it;
      if (lane < kXGVerts) {
        const long long g = it + lane;
        int f = -1;
        if (g < A.n_pix) {
          f = forest_of(A.F, g);
          if (g - A.F.off[f] >= A.F.len[f]) f = -1;    // pixel of a forest that failed the input checks
        }
        s_f[lane] = f;
        if (f >= 0) {
          const double d = A.dist[g], ux = A.F.ux[f], uy = A.F.uy[f], uz = A.F.uz[f];
          s_u[lane][0] = ux; s_u[lane][1] = uy; s_u[lane][2] = uz;
          s_x[lane][0] = d * ux; s_x[lane][1] = d * uy; s_x[lane][2] = d * uz;
          const Pix p = A.pix[g];
          s_w[lane] = make_float2(p.z, p.y);
        }
      }
    }
    __syncthreads();
    if (s_item >= A.n_pix) break;
    for (int v = wid; v < kXGVerts; v += nwarps) {
      const int f = s_f[v];
      const int nb = (f < 0) ? 0 : static_cast<int>(min(nstart[f + 1] - nstart[f], static_cast<int64_t>(kXGBatch)));
      const double di = (f < 0) ? 0.0 : A.dist[s_item + v];
      int carry = 0;
      if (lane == 0) s_pre[v * (kXGBatch + 1)] = 0;
      for (int m0 = 0; m0 < nb; m0 += 32) {
        const int m = m0 + lane;
        int cnt = 0;
        if (m < nb) {
          const int o = nbr[nstart[f] + m];
          const Chord c = chord(A, f, o, di, rmax2);
          s_o[v * kXGBatch + m] = o;
          s_lo[v * kXGBatch + m] = c.lo;
          cnt = c.hi - c.lo;
        }
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int up = __shfl_up_sync(0xffffffffu, cnt, d);
          if (lane >= d) cnt += up;
        }
        cnt += carry;
        if (m < nb) s_pre[v * (kXGBatch + 1) + m + 1] = cnt;
        carry = __shfl_sync(0xffffffffu, cnt, 31);
      }
      if (lane == 0) {
        s_nb[v] = nb;
        s_tot[v] = carry;
      }
    }
    __syncthreads();
    int v1 = 0;
    for (int v0 = 0; v0 < kXGVerts; v0 = v1) {
      // the next vertices whose chords fit the list (a single vertex's always do)
      int sum = 0;
      for (v1 = v0; v1 < kXGVerts && sum + s_tot[v1] <= cap; ++v1) sum += s_tot[v1];
      if (v1 == v0) {   // cannot happen: cap is at least the longest
        if (tid == 0) atomicOr(err, FLAG_X3_CAP);
        v1 = v0 + 1;
        continue;
      }
      const int nkey = (v1 - v0) * nr;
      for (int k = tid; k < nkey; k += kXGThreads) s_pos[k] = 0;
      if (tid == 0) {
        s_n = 0;
        s_ne = 0;
        s_nc = 0;
      }
      __syncthreads();
      // gather, 32 candidates a warp
      int before = 0, ne = 0, nc = 0;
      for (int v = v0; v < v1; ++v) {
        const int tot = s_tot[v], units = (tot + 31) >> 5;
        const int* pre = s_pre + v * (kXGBatch + 1);
        for (int u = (wid - before) & (nwarps - 1); u < units; u += nwarps) {
          const int k = 32 * u + lane;
          bool in = false;
          float4 r4 = make_float4(0.f, 0.f, 0.f, 0.f);
          Pix q = r4;
          int key = 0, o = 0;
          if (k < tot) {
            int lo = 0, hi = s_nb[v] - 1;   // neighbour whose pixels hold candidate k: the last with pre <= k
            while (lo < hi) {
              const int mid = (lo + hi + 1) >> 1;
              if (pre[mid] <= k) lo = mid; else hi = mid - 1;
            }
            o = s_o[v * kXGBatch + lo];
            const int64_t p = A.F.off[o] + s_lo[v * kXGBatch + lo] + (k - pre[lo]);
            int ir, it;
            in = bin.candidate(A, o, p, s_x[v], s_u[v], &r4, &ir, &it);
            if (in) {
              q = A.pix[p];
              key = ((v - v0) << 24) | (ir << 16) | it;
              if (q.z != 0.f) {
                ne += static_cast<int>((__float_as_uint(q.z) >> 23) & 0xFFu) - 127;
                ++nc;
              }
              atomicAdd(&s_pos[(v - v0) * nr + ir], 1);
            }
          }
          const unsigned msk = __ballot_sync(0xffffffffu, in);
          int slot = 0;
          if (lane == 0 && msk) slot = atomicAdd(&s_n, __popc(msk));
          slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(msk & ((1u << lane) - 1u));
          if (in) {   // slot < cap: the chords' pixels fit
            cr[slot] = r4;
            cw[slot] = make_float2(q.z, q.y);
            ck[slot] = make_int2(key, o);
          }
        }
        before += units;
      }
      ne = __reduce_add_sync(0xffffffffu, ne);
      nc = __reduce_add_sync(0xffffffffu, nc);
      if (lane == 0 && nc > 0) {
        atomicAdd(&s_ne, ne);
        atomicAdd(&s_nc, nc);
      }
      __syncthreads();
      // bucket starts (warp 0), typical N record (warp 1)
      if (wid == 0) {
        int carry = 0;
        for (int k0 = 0; k0 < nkey; k0 += 32) {
          const int k = k0 + lane;
          const int c = (k < nkey) ? s_pos[k] : 0;
          int x = c;
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += up;
          }
          if (k < nkey) {
            s_st[k] = carry + x - c;
            s_pos[k] = carry + x - c;
          }
          carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) s_st[nkey] = carry;
      } else if (wid == 1 && lane == 0) {
        int e = 0, c = 0;
        for (int v = v0; v < v1; ++v) {
          const float x = s_w[v].x;
          if (s_f[v] >= 0 && x != 0.f) {
            e += static_cast<int>((__float_as_uint(x) >> 23) & 0xFFu) - 127;
            ++c;
          }
        }
        s_typ = (c > 0 && s_nc > 0) ? 2.f * static_cast<float>(s_ne) / static_cast<float>(s_nc) +
                                          static_cast<float>(e) / static_cast<float>(c) : 0.f;
      }
      __syncthreads();
      // sort the list by (vertex, |r| bin): places first, then the fields; the
      // classes' steps and records meanwhile
      const int n = s_n;
      {
        int pos[kXGMove];
        float4 mr[kXGMove];
#pragma unroll
        for (int e = 0; e < kXGMove; ++e) {
          const int k = tid + e * kXGThreads;
          pos[e] = -1;
          if (k < n) {
            const int key = ck[k].x;
            pos[e] = atomicAdd(&s_pos[(key >> 24) * nr + ((key >> 16) & 0xff)], 1);
            mr[e] = cr[k];
          }
        }
        for (int c = tid; c < ncls; c += kXGThreads) {
          int ra = 0, left = c;
          while (left >= nr - ra) {
            left -= nr - ra;
            ++ra;
          }
          const int rb = ra + left;
          int steps = 0, recs = 0;
          for (int v = 0; v < v1 - v0; ++v) {
            const int np = s_st[v * nr + ra + 1] - s_st[v * nr + ra], nq = s_st[v * nr + rb + 1] - s_st[v * nr + rb];
            steps += xg_steps(np, nq, ra == rb);
            recs += (ra == rb) ? nq * (nq - 1) / 2 : np * nq;
          }
          s_steps[c] = steps;
          s_recs[c] = recs;
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < kXGMove; ++e)
          if (pos[e] >= 0) cr[pos[e]] = mr[e];
        float2 mw[kXGMove];
        int2 mk[kXGMove];
#pragma unroll
        for (int e = 0; e < kXGMove; ++e) {
          const int k = tid + e * kXGThreads;
          if (k < n) {
            mw[e] = cw[k];
            mk[e] = ck[k];
          }
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < kXGMove; ++e)
          if (pos[e] >= 0) {
            cw[pos[e]] = mw[e];
            ck[pos[e]] = mk[e];
          }
      }
      __syncthreads();
      // magnitudes of every bucket, a warp each
      for (int key = wid; key < nkey; key += nwarps) {
        float sn = 0.f, sw = 0.f;
        unsigned mn = 0u, mw = 0u, lw = 0x7F800000u;
        for (int k = s_st[key] + lane; k < s_st[key + 1]; k += 32) {
          const float2 q = cw[k];
          sn += fabsf(q.x);
          sw += q.y;
          mn = max(mn, __float_as_uint(fabsf(q.x)));
          mw = max(mw, __float_as_uint(q.y));
          if (q.y > 0.f) lw = min(lw, __float_as_uint(q.y));
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
          sn += __shfl_xor_sync(0xffffffffu, sn, d);
          sw += __shfl_xor_sync(0xffffffffu, sw, d);
        }
        mn = __reduce_max_sync(0xffffffffu, mn);
        mw = __reduce_max_sync(0xffffffffu, mw);
        lw = __reduce_min_sync(0xffffffffu, lw);
        if (lane == 0) {
          s_sn[key] = sn;
          s_sw[key] = sw;
          s_mn[key] = __uint_as_float(mn);
          s_mw[key] = __uint_as_float(mw);
          s_lw[key] = __uint_as_float(lw);
        }
      }
      __syncthreads();
      for (int c = tid; c < ncls; c += kXGThreads) {
        int ra = 0, left = c;
        while (left >= nr - ra) {
          left -= nr - ra;
          ++ra;
        }
        const int rb = ra + left, recs = s_recs[c];
        s_eh[c] = -1;
        if (recs < kXGDirect * nbc || recs < 1) continue;
        // largest and total magnitude (with mirror weights), smallest W record that is not 0
        float bn = 0.f, bw = 0.f, tn = 0.f, tw = 0.f, lw = INFINITY;
        for (int v = 0; v < v1 - v0; ++v) {
          const float2 wv = s_f[v0 + v] >= 0 ? s_w[v0 + v] : make_float2(0.f, 0.f);
          const int a = v * nr + ra, b = v * nr + rb;
          // (multiplied in the records' order, so that no record is larger or, if not 0, smaller)
          bn = fmaxf(bn, s_mn[a] * (s_mn[b] * fabsf(wv.x)));
          bw = fmaxf(bw, s_mw[a] * (s_mw[b] * wv.y));
          tn += s_sn[a] * (s_sn[b] * fabsf(wv.x));
          tw += s_sw[a] * (s_sw[b] * wv.y);
          if (wv.y > 0.f) lw = fminf(lw, s_lw[a] * (s_lw[b] * wv.y));
        }
        const bool fn = tn == 0.f || (bn > 1e-25f && tn < 1e30f), fw = tw == 0.f || (bw > 1e-25f && tw < 1e30f);
        if (!fn || !fw) continue;   // (sums that are infinite or not numbers among them)
        const int en = xg_scale(2.002f * bn, 1.01f * tn), ew = xg_scale(2.002f * bw, 1.01f * tw);
        const int k = min(21, __clz(recs));
        if (tw != 0.f && !(lw >= pow2f(ew - k + 20))) continue;
        if (tn != 0.f && !(static_cast<float>(en - k + 24) <= s_typ)) continue;
        s_eh[c] = ((en + 256) << 16) | (ew + 256);
      }
      __syncthreads();
      const F2 M2 = f2(kM15, kM15), neg2 = f2(-1.f, -1.f);
      int cls = 0;
      for (int ra = 0; ra < nr; ++ra) {
        for (int rb = ra; rb < nr; ++rb, ++cls) {
          const int S = s_steps[cls];
          if (S == 0) continue;
          const bool same = ra == rb;
          // bits of the low word: its sum over the class's records stays below 2^32
          const int eh = s_eh[cls], bits = min(21, __clz(s_recs[cls]));
          const int en = (eh >> 16) - 256, ew = (eh & 0xffff) - 256;
          const bool direct = eh < 0;
          const F2 sc2 = direct ? 0ull : f2(pow2f(-en), pow2f(-ew)), up2 = f2(pow2f(bits), pow2f(bits));
          double* const base = sums + 2 * (static_cast<int64_t>(ra * nr + rb) * nbc);
          int b = static_cast<int>(static_cast<int64_t>(S) * wid / nwarps);
          int left = static_cast<int>(static_cast<int64_t>(S) * (wid + 1) / nwarps) - b;
          int v = -1, np = 0, nq = 0, p0 = 0, q0 = 0, t = 0;
          // step b of the class: vertex v, tile t, step k of the tile
          int k = b;
          bool find = true;
          while (left > 0) {
            if (find) {
              for (;;) {
                ++v;
                p0 = s_st[v * nr + ra];
                np = s_st[v * nr + ra + 1] - p0;
                q0 = s_st[v * nr + rb];
                nq = s_st[v * nr + rb + 1] - q0;
                const int sv = xg_steps(np, nq, same);
                if (k < sv) break;
                k -= sv;
              }
              t = 0;
              find = false;
            }
            const int lim = same ? min(np, 16 * (t + 1)) : np;
            const int ks = (lim + 1) >> 1;
            if (k >= ks) {
              k -= ks;
              ++t;
              continue;
            }
            const int ql = 16 * t + (lane & 15);
            const bool qv = ql < nq;
            const int q = q0 + min(ql, nq - 1);
            const float4 rq = cr[q];
            const float2 wq = cw[q], wv = s_w[v0 + v];
            const int2 kq = ck[q];
            const float wdq = wq.x * wv.x, wwq = wq.y * wv.y;
            const int tq = kq.x & 0xffff;
            const int m = min(ks - k, left);
            left -= m;
            for (int e = 0; e < m; ++e, ++k) {
              const int pl = 2 * k + (lane >> 4);
              const int p = p0 + min(pl, np - 1);
              const float4 rp = cr[p];
              const float2 wp = cw[p];
              const int2 kp = ck[p];
              const bool on = qv && pl < lim && (!same || pl < ql) && kp.y != kq.y;
              const float ca = (rp.x * rq.x + rp.y * rq.y + rp.z * rq.z) * (rp.w * rq.w);
              const int ia = min(max(static_cast<int>(floorf((ca + 1.0f) * half_na)), 0), na - 1);
              const int tp = kp.x & 0xffff;
              int t1 = tp, t2 = tq;
              float mult = 1.f;
              if (same) {
                t1 = min(tp, tq);
                t2 = max(tp, tq);
                mult = (tp == tq) ? 2.f : 1.f;
              }
              const int l = (ia * nt + t1) * nt + t2;
              const float vn = wp.x * wdq * mult, vw = wp.y * wwq * mult;
              if (direct) {
                const int bb = on ? l : -1;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  const int src = (lane >> 1) + 16 * h;
                  const int b2 = __shfl_sync(0xffffffffu, bb, src);
                  const float n2 = __shfl_sync(0xffffffffu, vn, src), w2 = __shfl_sync(0xffffffffu, vw, src);
                  if (b2 >= 0) red_add_f64_global(base + 2 * static_cast<int64_t>(b2) + (lane & 1), static_cast<double>((lane & 1) ? w2 : n2));
                }
              } else if (on) {
                // floor in units of 2^eh, and the rest, rounded, `bits` below
                const F2 v2 = f2(vn, vw);
                const F2 hm = fma2_rd(v2, sc2, M2);
                const F2 lm = fma2(fma2(v2, sc2, fma2(hm, neg2, M2)), up2, M2);
                const float2 h = unf2(hm), lo = unf2(lm);
                unsigned* w = hist + l * kXGWords;
                atomicAdd(w + 0, __float_as_uint(h.x) - kM15Bits);
                atomicAdd(w + 1, __float_as_uint(lo.x) - kM15Bits);
                atomicAdd(w + 2, __float_as_uint(h.y) - kM15Bits);
                atomicAdd(w + 3, __float_as_uint(lo.y) - kM15Bits);
              }
            }
            if (k == ks) {
              k = 0;
              ++t;
            }
            if (16 * t >= nq) find = true;
          }
          if (!direct) {
            __syncthreads();
            const double inv = pow2(((tid & 1) ? ew : en) - bits);
            for (int k2 = tid; k2 < 2 * nbc; k2 += kXGThreads) {
              unsigned* w = hist + (k2 >> 1) * kXGWords + 2 * (k2 & 1);
              const unsigned h = w[0], lo = w[1];
              if ((h | lo) != 0u) {
                const long long x = (static_cast<long long>(static_cast<int>(h)) << bits) + lo;
                if (x != 0) red_add_f64_global(base + k2, static_cast<double>(x) * inv);
                w[0] = 0u;
                w[1] = 0u;
              }
            }
            __syncthreads();
          }
        }
      }
      __syncthreads();
    }
  }
}

struct X3Count {
  unsigned long long total;   // pixels on the chords of all vertices
  int most, degree;           // of any vertex; most neighbour forests of one
};

// pixels on every main vertex's chords (an upper bound of its neighbours within
// r_max, 1e-2 Mpc/h wider): the longest and the sum, one warp per vertex pixel
__global__ void xi3_count_kernel(X3Args A, const int32_t* nbr, const int64_t* nstart, X3Count* out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const double rmax2 = A.r_max * A.r_max;
  int best = 0;
  unsigned long long total = 0, degree = 0;
  for (int64_t g = warp; g < A.n_pix; g += nw) {
    const int f = forest_of(A.F, g);
    if (g - A.F.off[f] >= A.F.len[f]) continue;
    int cnt = 0;
    for (int64_t e = nstart[f] + lane; e < nstart[f + 1]; e += 32) {
      const Chord c = chord(A, f, nbr[e], A.dist[g], rmax2);
      cnt += c.hi - c.lo;
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    best = max(best, cnt);
    total += cnt;
    degree = max(degree, static_cast<unsigned long long>(nstart[f + 1] - nstart[f]));
  }
  if (lane == 0 && best > 0) {
    atomicMax(&out->most, best);
    atomicMax(&out->degree, static_cast<int>(min(degree, 0x7fffffffull)));
    atomicAdd(&out->total, total);
  }
}

// num, wsum and xi of every bin: the sums of its canonical bin (side-1 key <=
// side-2 key), interleaved (N, W), or, without `sums`, in num and wsum themselves
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
    const double2 v = sums ? reinterpret_cast<const double2*>(sums)[m] : make_double2(num[m], wsum[m]);
    if (sums || m != k) {
      num[k] = v.x;
      wsum[k] = v.y;
    }
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

// List length of the grouped kernel, or 0 where xi3_kernel is the better or the
// only one: the (r1, r2) class has to leave room in shared memory for a list of
// every vertex's neighbours, and a group's records (at most mean^2 / 2 a vertex)
// have to reach half the number of canonical bins (half of all), which are walked
// once a group.  Both kernels, against that ratio: 0.16: 8.0 against 6.8 ms for
// xi3_kernel; 0.29: 4.9 against 5.2; 0.37: 10.3 against 10.1; 1.4: 3.5 against
// 4.8; 2.2: 158 against 204; 3.3: 23.7 against 63 ms.
int x3_group_cap(const X3Args& a, const DevInfo& dev, const X3Count& c) {
  const int64_t nbc = static_cast<int64_t>(a.n_alpha) * a.n_theta * a.n_theta;
  if (a.n_r > kXGMaxR || a.n_theta > 0xffff || c.degree > kXGBatch || c.most < 1 || nbc > 7000) return 0;
  // two blocks per SM (1 KB of each reserved), less 6 KB for the static arrays
  const int room = std::min(dev.smem_optin, kXGSmem) - 6144 - xg_layout(0, static_cast<int>(nbc)).end;
  const int cap = std::min(room / 32 & ~3, kXGMove * kXGThreads);
  if (cap < c.most) return 0;
  const double mean = static_cast<double>(c.total) / static_cast<double>(std::max<int64_t>(a.n_pix, 1));
  const double verts = std::min<double>(kXGVerts, cap / std::max(mean, 1.0));
  const double records = verts * mean * mean / 2, bins = 0.5 * a.n_r * a.n_r * static_cast<double>(nbc);
  return records >= kXGGain * bins ? cap : 0;
}

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
  const size_t o_misc = o; o += 256;
  const size_t o_sums = o;   // (N, W) per bin
  // where the device has no room for the sums beside the caller's num and wsum they go there directly (381 against
  // 204 ms on 5,000 SDSS-like forests)
  cudaError_t e = grow(scratch, scratch_cap, o_sums + static_cast<size_t>(nbins) * 16);
  const bool split = e == cudaErrorMemoryAllocation;
  if (split) e = grow(scratch, scratch_cap, o_sums);
  LYA_TRY(e);
  char* sc = static_cast<char*>(*scratch);
  int32_t* deg = reinterpret_cast<int32_t*>(sc + o_deg);
  int32_t* cur = reinterpret_cast<int32_t*>(sc + o_cur);
  int64_t* start = reinterpret_cast<int64_t*>(sc + o_start);
  int32_t* nbr = reinterpret_cast<int32_t*>(sc + o_nbr);
  double* sums = split ? nullptr : reinterpret_cast<double*>(sc + o_sums);
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(sc + o_misc);
  if (split) {
    LYA_TRY(cudaMemsetAsync(a.num, 0, static_cast<size_t>(nbins) * 8, s));
    LYA_TRY(cudaMemsetAsync(a.wsum, 0, static_cast<size_t>(nbins) * 8, s));
  } else {
    LYA_TRY(cudaMemsetAsync(sums, 0, static_cast<size_t>(nbins) * 16, s));
  }
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
  X3Count* dcount = reinterpret_cast<X3Count*>(sc + o_misc + 64);
  LYA_TRY(cudaMemsetAsync(dcount, 0, sizeof(X3Count), s));
  if (a.n_pix > 0 && nf > 0)
    LYA_COUNT(1), xi3_count_kernel<<<dev.sms * 8, 256, 0, s>>>(a, nbr, start, dcount);
  X3Count count{};
  LYA_TRY(cudaMemcpyAsync(&count, dcount, sizeof(count), cudaMemcpyDeviceToHost, s));
  LYA_TRY(cudaStreamSynchronize(s));
  const int hmax = count.most;
  const int gcap = split ? 0 : x3_group_cap(a, dev, count);
  if (gcap > 0) {
    const int smem = xg_layout(gcap, a.n_alpha * a.n_theta * a.n_theta).end;
    LYA_TRY(set_max_dynamic_smem(reinterpret_cast<const void*>(xi3_group_kernel), smem));
    LYA_COUNT(1), xi3_group_kernel<<<2 * dev.sms, kXGThreads, smem, s>>>(a, nbr, start, gcap, sums, counter, err);
    LYA_TRY(cudaGetLastError());
    LYA_COUNT(1), xi3_finalize_kernel<<<grid_for(nbins, 256), 256, 0, s>>>(sums, a.num, a.wsum, a.xi, a.n_r, a.n_theta,
                                                                          a.n_alpha);
    return cudaGetLastError();
  }
  const int cap_max = (dev.smem_optin - 1024) / per_cand;
  const int cap = std::max(std::min(hmax, cap_max), 256);
  const int smem = cap * per_cand;
  if (smem > dev.smem_optin) return cudaErrorInvalidValue;
  const auto kernel = split ? xi3_kernel<true> : xi3_kernel<false>;
  LYA_TRY(set_max_dynamic_smem(reinterpret_cast<const void*>(kernel), smem));
  int per_sm = 0;
  LYA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kX3Threads, smem));
  if (per_sm < 1) return cudaErrorInvalidValue;
  if (a.n_pix > 0 && nf > 0)
    LYA_COUNT(1), kernel<<<per_sm * dev.sms, kX3Threads, smem, s>>>(a, nbr, start, cap, sums, counter, err);
  LYA_TRY(cudaGetLastError());
  LYA_COUNT(1), xi3_finalize_kernel<<<grid_for(nbins, 256), 256, 0, s>>>(sums, a.num, a.wsum, a.xi, a.n_r, a.n_theta,
                                                                        a.n_alpha);
  return cudaGetLastError();
}

}  // namespace lya
