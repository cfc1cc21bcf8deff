// Pixel-pair histogram of Eq. (2.4): for every forest pair (a, b) and every
// pixel pair (i in a, j in b), bin (r_par, r_perp) and add (w d)_i (w d)_j and
// w_i w_j to the bin (Section 2.1).
//
// Mixed kernel (LYA_PREC_MIXED), persistent, one forest pair per team (a block
// of two warps) at a time:
//  * forest b is staged in the team's shared-memory buffer with coalesced
//    16-byte loads; each warp takes 32 pixels of forest a (one per lane);
//  * separations are FP32 fused multiply-adds on distances relative to a
//    per-forest reference (multiple of 2^-10, so the reference differences and
//    sums entering the pair constants are exact FP32 numbers):
//        r_par/D  = | d~_j * (-c/D) + ((d~_i * c/D) + (ref_a - ref_b) c/D) |
//        r_perp/D =   d~_j *   s/D  + ((d~_i * s/D) + (ref_a + ref_b) s/D)
//  * floor() is an FP32 add rounded toward -inf of 2^23 (the integer lands in
//    the low mantissa bits), so the bin index needs no float->int conversion;
//  * each lane walks j and keeps the current bin's run sums in registers; a
//    run that ends (the bin changed) is held in registers, and the warp adds
//    the held runs to the team's chunk histogram, which covers only the rows
//    of the pair's r_perp band, when a lane that holds one ends another: exact
//    two-word fixed point summed with native 32-bit shared-memory reductions
//    (a lane without a held run aims them at its own dummy word);
//  * every two 32-pixel chunks of forest a (one per warp) the integer sums are
//    folded into the team's compensated FP32 (TwoSum) band accumulator, which
//    survives across consecutive pairs with the same first band row (the pair
//    list is ordered for this) and is added to the FP64 bin sums in global
//    memory when the band changes;
//  * the j loop of each 32-pixel chunk of a is restricted to the pixels that
//    can be in range (distances are sorted; binary searches, one chunk per lane).
// What bounds it: issue slots and fixed latencies (28 warp instructions per
// step of 32 pixel pairs, issue 65-70%), and on the SDSS-like grid, whose runs
// are two pixels long, the shared-memory pipe (81%: 3.6 wavefronts per
// reduction).  A team of two shares 12.7 KB of tables and the staged forest,
// so 9-13 teams (18-26 warps) fit on an SM where 8 single warps did.
// Measured (survey pass): 60,000 SDSS-like forests 624 -> 386 ms, 9,000
// DESI-like forests 414 -> 244 ms.
// FP64 kernel (LYA_PREC_FP64): the same decomposition with FP64 distances,
// separations, products and shared-memory sums, mirroring the oracle's
// operation order: r = |d_i - d_j| * c, x = r * (1/D).
#include <algorithm>
#include <math.h>

#include "lya_internal.cuh"

namespace lya {
namespace {

constexpr int kTeam = 64;         // threads of a team (one block): two warps on one forest pair
// Tables of a team.  A chunk-histogram array holds (K + 1) x (n_par + 1) bins
// (guard row and column) below its last 32 words, one dummy word per lane; an
// accumulator array K x n_par.  The large form holds bands of K = 7 rows of 50
// bins, the small one K = 5 (wider bands are walked in windows).
constexpr int kHcapL = 440, kAcapL = 352;
constexpr int kHcapS = 344, kAcapS = 256;
// The small form is taken where forests are longer than this.  Long forests
// fill shared memory with staged pixels, so the smaller tables let more teams
// in (600 pixels: 11 instead of 9 per SM; DESI-like survey of 9,000 forests
// 244 against 259 ms); short ones gain no team and pay for the bands of 6 and
// 7 rows (207 pixels, SDSS-like survey of 60,000: 414 against 386 ms).
constexpr int kSmallTablesLen = 384;
constexpr uint32_t kM15Bits = 0x4B400000u;   // bits of 1.5 * 2^23
constexpr float kM15 = 12582912.0f;
constexpr int kMaxPar64 = 256;   // largest n_par of the FP64 path
constexpr int kMaxSeg = 1024;    // pixel buffer cap per warp

// Knuth's TwoSum: (hi, lo) += x with the rounding error of hi + x kept in lo.
__device__ __forceinline__ void two_sum(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bp = s - hi;
  lo += (hi - (s - bp)) + (x - bp);
  hi = s;
}

// Exact two-word fixed point.  v (|v| < B) is represented as
// (hi * 2^16 + lo) * 2^-k with q = v * 2^(k-16), hi = floor(q), lo =
// round((q - hi) * 2^16) in [0, 2^16]; sc16 = 2^(k-16) is chosen per forest
// pair so that |q| < 2^21 for every run of in-grid pairs.  Sums of hi and of lo
// are kept in separate 32-bit words (no carries between them), which shared
// memory adds natively; FP32 shared-memory reductions are emulated on this
// part and far slower.

// Two FP32 values in one 64-bit register: one instruction does both lanes'
// fused multiply-adds, each rounded exactly as the scalar one.
using F2 = uint64_t;
__device__ __forceinline__ F2 f2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unf2(F2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ F2 fma2_rd(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// A lane's ended run, held in registers until the warp adds the held runs to
// the chunk histogram.
struct Held {
  uint32_t key;
  float n, w;
  bool on;
};

// Constants of a walk (see chunk_runs).
struct Walk {
  F2 cpsp;           // (-c/D_par, s/D_perp)
  F2 sc;             // fixed-point scales of N and W
  float pmax, tmax;  // clamps of the two floors (guard column and row)
  uint32_t stride, base, guard, twin, tspan, dummy;
};

// Adds every lane's held run to the chunk histogram (four 32-bit reductions
// per lane; a lane without a held run adds to its own dummy word).
template <int HC>
__device__ __forceinline__ void add_held(Held& h, const Walk& k) {
  const F2 m15 = f2(kM15, kM15), nw = f2(h.n, h.w);
  // q = v * sc16 is exact (sc16 is a power of two) and |q| < 2^21
  const F2 hm = fma2_rd(nw, k.sc, m15);                         // 1.5 * 2^23 + floor(q)
  const F2 fr = fma2(nw, k.sc, fma2(hm, f2(-1.f, -1.f), m15));  // q - floor(q), exact
  const F2 lm = fma2(fr, f2(65536.f, 65536.f), m15);              // 1.5 * 2^23 + round(fr * 2^16)
  const float2 hi = unf2(hm), lo = unf2(lm);
  const uint32_t addr = h.on ? k.base + (h.key << 2) : k.dummy;
  asm volatile(
      "{\n\t"
      "red.shared.add.u32 [%0], %1;\n\t"
      "red.shared.add.u32 [%0+%5], %2;\n\t"
      "red.shared.add.u32 [%0+%6], %3;\n\t"
      "red.shared.add.u32 [%0+%7], %4;\n\t}"
      ::"r"(addr), "r"(__float_as_uint(hi.x) - kM15Bits), "r"(__float_as_uint(lo.x) - kM15Bits),
        "r"(__float_as_uint(hi.y) - kM15Bits), "r"(__float_as_uint(lo.y) - kM15Bits), "n"(HC * 4),
        "n"(HC * 8), "n"(HC * 12));
  h.on = false;
}

// One pixel pair of a run walk (see chunk_runs).  A run that ends here is
// held in the lane's registers; the warp adds its held runs to the histogram
// only when some lane that already holds one ends another.  On the DESI-like
// grid a run is about seven pixels long, so the reductions come once per ~6
// steps instead of every step.
template <bool WINDOW, int HC>
__device__ __forceinline__ void run_step(const ulonglong2& q, const Walk& k, F2 ucus, float wdi, float wi,
                                         uint32_t& cur, float& aN, float& aW, Held& held) {
  const float2 r = unf2(fma2(q.x, k.cpsp, ucus));
  const float pf = fminf(__fadd_rd(fabsf(r.x), kMagic), k.pmax);
  const float tf = fminf(__fadd_rd(r.y, kMagic), k.tmax);
  uint32_t key = __float_as_uint(tf) * k.stride + __float_as_uint(pf);
  if (WINDOW) key = ((__float_as_uint(tf) - kMagicBits - k.twin) <= k.tspan) ? key : k.guard;
  const bool chg = key != cur;
  if (__any_sync(0xffffffffu, chg && held.on)) add_held<HC>(held, k);
  const float2 w = unf2(q.y);
  held.key = chg ? cur : held.key;
  held.n = chg ? aN : held.n;
  held.w = chg ? aW : held.w;
  held.on = held.on || chg;
  cur = key;
  // (scalar: packing the two sums costs more moves than the one instruction saves)
  aN = fmaf(wdi, w.x, chg ? 0.f : aN);
  aW = fmaf(wi, w.y, chg ? 0.f : aW);
}

// One 32-pixel chunk of forest a against pixels [jlo, jhi) of the staged
// forest b.  Each lane keeps the current bin and its running sums in
// registers; a run (consecutive j in one bin) that ends is held (see
// run_step) and later added to the shared chunk histogram.  Out-of-grid pairs
// land in the guard row / column (floor clamped with fminf); WINDOW
// additionally sends rows outside [twin, twin + tspan] to the guard.  Pixels
// are read kUnroll at a time before the steps: the reductions write shared
// memory, so a later load cannot be hoisted above them.
template <bool WINDOW, int HC>
__device__ __forceinline__ void chunk_runs(const ulonglong2* buf, int jlo, int jhi, const Walk& k, F2 ucus, float wdi,
                                           float wi) {
  constexpr int kUnroll = 8;
  uint32_t cur = k.guard;
  float aN = 0.f, aW = 0.f;
  Held held{k.guard, 0.f, 0.f, false};
  int j = jlo;
  for (; j + kUnroll <= jhi; j += kUnroll) {
    ulonglong2 q[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) q[u] = buf[j + u];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) run_step<WINDOW, HC>(q[u], k, ucus, wdi, wi, cur, aN, aW, held);
  }
  for (; j < jhi; ++j) run_step<WINDOW, HC>(buf[j], k, ucus, wdi, wi, cur, aN, aW, held);
  // the held runs, then the last run of every lane
  if (__any_sync(0xffffffffu, held.on)) add_held<HC>(held, k);
  held = Held{cur, aN, aW, true};
  add_held<HC>(held, k);
}

// Per-pair scale sc16 = 2^(20 - e) with 2^e <= B < 2^(e+1): every |v| < B
// maps to |q| < 2^21.
__device__ __forceinline__ float fixed_scale(float B) {
  if (!(B > 0.f) || !(B < 1e37f)) return 1.f;
  const int e = static_cast<int>((__float_as_uint(B) >> 23) & 0xFFu) - 127;
  const int ex = 20 - e + 127;
  return __uint_as_float(static_cast<uint32_t>(min(max(ex, 1), 254)) << 23);
}

struct TeamSm {
  uint32_t* h;      // chunk histogram: N hi, N lo, W hi, W lo (HC words each)
  float* acc;       // accumulator: N hi, N lo, W hi, W lo (AC each)
  ulonglong2* buf;  // staged pixels of forest b: {x, x}, {w delta, w}
  uint32_t sN;      // shared address of h
};

// chunk rows [0, nrows) x columns [0, npar) -> accumulator rows [0, nrows)
// (fixed point -> FP32 with the pair's scales); clears the whole chunk
// histogram including the guard row and column.  All threads of the team.
template <int HC, int AC>
__device__ __forceinline__ void fold_chunk(const TeamSm& w, int nrows, int npar, float inv_scN, float inv_scW) {
  __syncthreads();
  const int stride = npar + 1;
  uint32_t* nh = w.h;
  uint32_t* nl = w.h + HC;
  uint32_t* wh = w.h + 2 * HC;
  uint32_t* wl = w.h + 3 * HC;
  float* nhi = w.acc;
  float* nlo = w.acc + AC;
  float* whi = w.acc + 2 * AC;
  float* wlo = w.acc + 3 * AC;
  for (int r = 0; r <= nrows; ++r) {
    for (int p = threadIdx.x; p < stride; p += kTeam) {
      const int k = r * stride + p;
      const uint32_t a1 = nh[k], a2 = nl[k], b1 = wh[k], b2 = wl[k];
      if ((a1 | a2 | b1 | b2) != 0u) {
        if (r < nrows && p < npar) {
          const int a = r * npar + p;
          const float vn = fmaf(static_cast<float>(a2), 1.f / 65536.f, static_cast<float>(static_cast<int32_t>(a1))) * inv_scN;
          const float vw = fmaf(static_cast<float>(b2), 1.f / 65536.f, static_cast<float>(static_cast<int32_t>(b1))) * inv_scW;
          two_sum(nhi[a], nlo[a], vn);
          two_sum(whi[a], wlo[a], vw);
        }
        nh[k] = 0u;
        nl[k] = 0u;
        wh[k] = 0u;
        wl[k] = 0u;
      }
    }
  }
  __syncthreads();
}

// accumulator rows [0, rows) with origin t0 -> FP64 bin sums in global memory
template <int AC>
__device__ __forceinline__ void flush_acc(const TeamSm& w, const XiArgs& A, int rows, int t0, int64_t out_off) {
  __syncthreads();
  const int npar = A.n_par;
  float* nhi = w.acc;
  float* nlo = w.acc + AC;
  float* whi = w.acc + 2 * AC;
  float* wlo = w.acc + 3 * AC;
  for (int r = 0; r < rows; ++r) {
    for (int p = threadIdx.x; p < npar; p += kTeam) {
      const int a = r * npar + p;
      const float h1 = nhi[a], h2 = whi[a];
      if (h1 != 0.f || h2 != 0.f) {
        const int64_t bin = out_off + static_cast<int64_t>(p) * A.n_perp + t0 + r;
        red_add_f64_global(A.num + bin, static_cast<double>(h1) + static_cast<double>(nlo[a]));
        red_add_f64_global(A.wsum + bin, static_cast<double>(h2) + static_cast<double>(wlo[a]));
        nhi[a] = 0.f;
        nlo[a] = 0.f;
        whi[a] = 0.f;
        wlo[a] = 0.f;
      }
    }
  }
  __syncthreads();
}

// Number of entries of the sorted array a[0..n) strictly below v (v NaN -> n).
__device__ __forceinline__ int floats_below(const float* a, int n, float v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Number of staged pixels with distance strictly below v (v NaN -> n).
__device__ __forceinline__ int staged_below(const ulonglong2* buf, int n, float v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (*reinterpret_cast<const float*>(buf + mid) < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Bin rows t0 .. t0 + K - 1 of forest pair (a, b) into the chunk histogram
// (origin t0) and fold them into accumulator rows 0 ..; WINDOW restricts to
// rows [t0, t0 + K) of a wider band whose top is t_hi.
template <bool WINDOW, int HC, int AC>
__device__ void pair_rows(const XiArgs& A, const TeamSm& w, int aidx, int bidx, const Pix* __restrict__ pa,
                          const Pix* __restrict__ pb, int na, int nb, float cp, float sp, float Dc, float Ds, int t0,
                          int K, int t_hi, int seg) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int npar = A.n_par;
  const float fnpar = static_cast<float>(npar), fnperp = static_cast<float>(A.n_perp);
  // fixed-point scales: a run of in-grid pairs (fixed i, one bin) spans less
  // than 2 / cp in distance, so it holds at most 2 / (cp hmin_b) + 1 pixels of b
  const float nrun = 2.f / (cp * A.F.hmin[bidx]) + 1.f;
  const float scN = fixed_scale(A.F.wdmax[aidx] * A.F.wdmax[bidx] * nrun);
  const float scW = fixed_scale(A.F.wmax[aidx] * A.F.wmax[bidx] * nrun);
  const float inv_scN = 1.f / scN, inv_scW = 1.f / scW;
  Walk k;
  k.cpsp = f2(-cp, sp);
  k.sc = f2(scN, scW);
  k.stride = static_cast<uint32_t>(npar + 1);
  // key (M+t)*(npar+1) + (M+p) -> local index (t - t0)*(npar+1) + p
  const uint32_t C = kMagicBits * (k.stride + 1u) + static_cast<uint32_t>(t0) * k.stride;
  k.base = w.sN - 4u * C;
  k.guard = C + static_cast<uint32_t>(npar);   // row 0, guard column
  k.pmax = __uint_as_float(kMagicBits + static_cast<uint32_t>(npar));
  k.tmax = __uint_as_float(kMagicBits + static_cast<uint32_t>(t_hi + 1));
  k.twin = static_cast<uint32_t>(t0);
  k.tspan = static_cast<uint32_t>(K - 1);
  k.dummy = w.sN + 4u * static_cast<uint32_t>(HC - 32 + lane);
  const int nchunk = (na + 31) >> 5;
  for (int j0 = 0; j0 < nb; j0 += seg) {
    const int segn = min(seg, nb - j0);
    for (int q = threadIdx.x; q < segn; q += kTeam) {
      const Pix p = pb[j0 + q];
      w.buf[q] = make_ulonglong2(f2(p.x, p.x), f2(p.z, p.y));
    }
    __syncthreads();
    for (int cb = 0; cb < nchunk; cb += 32) {
      // lane c: the range of b that chunk cb + c can reach (distances are sorted; two binary searches)
      const int i0 = (cb + lane) << 5;
      int jlo = 0, jhi = 0;
      if (i0 < na) {
        const float xf = pa[i0].x, xl = pa[min(i0 + 31, na - 1)].x;
        float dlo = (fmaf(xf, cp, Dc) - fnpar) / cp;
        float dhi = (fmaf(xl, cp, Dc) + fnpar) / cp;
        if (sp > 0.f) dhi = fminf(dhi, (fnperp - fmaf(xf, sp, Ds)) / sp);
        dlo -= fabsf(dlo) * 1e-5f + 1e-2f;
        dhi += fabsf(dhi) * 1e-5f + 1e-2f;
        jlo = staged_below(w.buf, segn, dlo);
        jhi = staged_below(w.buf, segn, dhi);
      }
      // two chunks with work at a time, one per warp, then a fold
      unsigned todo = __ballot_sync(0xffffffffu, jlo < jhi);
      while (todo) {
        const unsigned rest = todo & (todo - 1u);
        const unsigned mine = (wid == 0) ? todo : rest;
        todo = rest & (rest - 1u);
        if (mine) {
          const int c = __ffs(mine) - 1;
          const int i = ((cb + c) << 5) + lane;
          // lanes past the end carry a NaN distance: they only ever hit the guard
          const Pix pi = (i < na) ? pa[i] : make_float4(__int_as_float(0x7fffffff), 0.f, 0.f, 0.f);
          chunk_runs<WINDOW, HC>(w.buf, __shfl_sync(0xffffffffu, jlo, c), __shfl_sync(0xffffffffu, jhi, c), k,
                             f2(fmaf(pi.x, cp, Dc), fmaf(pi.x, sp, Ds)), pi.z, pi.y);
        }
        fold_chunk<HC, AC>(w, K, npar, inv_scN, inv_scW);
      }
    }
    __syncthreads();
  }
}

// HC words per chunk-histogram array, AC entries per accumulator array (see kTables)
template <int HC, int AC>
__global__ void __launch_bounds__(kTeam) xi_mixed_kernel(XiArgs A, int seg, int kmax, int grab) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long s_it;
  // accumulator (4 x AC floats), chunk histogram (4 x HC words), pixel buffer (seg x 16 bytes)
  TeamSm w;
  w.acc = reinterpret_cast<float*>(smem);
  w.h = reinterpret_cast<uint32_t*>(smem + AC * 16);
  w.buf = reinterpret_cast<ulonglong2*>(smem + AC * 16 + HC * 16);
  w.sN = smem_addr(w.h);
  for (int k = threadIdx.x; k < 4 * AC; k += kTeam) w.acc[k] = 0.f;
  for (int k = threadIdx.x; k < 4 * HC; k += kTeam) w.h[k] = 0u;
  const int nperp = A.n_perp;
  const float fnperp = static_cast<float>(nperp);
  // the accumulator holds rows [acc_t0, acc_t0 + kmax) of catalogue acc_off
  int acc_t0 = -1;
  int64_t acc_off = -1;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_it = atomicAdd(A.counter, static_cast<unsigned long long>(grab));
    __syncthreads();
    const unsigned long long it0 = s_it;
    if (it0 >= static_cast<unsigned long long>(A.n_pairs)) break;
    const int64_t it1 = min(static_cast<int64_t>(it0) + grab, A.n_pairs);
    // everything below is uniform over the team
    for (int64_t it = static_cast<int64_t>(it0); it < it1; ++it) {
      const int2 ab = A.pairs[it];
      if (ab.x < 0) continue;   // rejected pair
      const int a = ab.x, b = ab.y;
      const int na = A.F.len[a], nb = A.F.len[b];
      if (na == 0 || nb == 0) continue;
      const float2 cs = A.cs[it];
      const float cp = cs.x, sp = cs.y;
      const Pix* __restrict__ pa = A.pix + A.F.off[a];
      const Pix* __restrict__ pb = A.pix + A.F.off[b];
      const float refa = A.F.dref[a], refb = A.F.dref[b];
      const float Dc = (refa - refb) * cp;
      const float Ds = (refa + refb) * sp;
      // r_perp band from the extreme pixels (r_perp is monotone in both distances)
      const float rt_min = fmaf(pb[0].x, sp, fmaf(pa[0].x, sp, Ds));
      const float rt_max = fmaf(pb[nb - 1].x, sp, fmaf(pa[na - 1].x, sp, Ds));
      if (!(rt_min < fnperp)) continue;
      const int t_lo = static_cast<int>(rt_min);
      const int t_hi = (rt_max < fnperp) ? static_cast<int>(rt_max) : nperp - 1;
      const int K = t_hi - t_lo + 1;
      const int64_t out_off = static_cast<int64_t>(A.F.mock[a]) * A.nb;
      if (K <= kmax) {
        if (t_lo != acc_t0 || out_off != acc_off) {
          if (acc_t0 >= 0) flush_acc<AC>(w, A, kmax, acc_t0, acc_off);
          acc_t0 = t_lo;
          acc_off = out_off;
        }
        pair_rows<false, HC, AC>(A, w, a, b, pa, pb, na, nb, cp, sp, Dc, Ds, t_lo, K, t_hi, seg);
      } else {
        // wide band: windows of kmax rows, each flushed on its own
        if (acc_t0 >= 0) flush_acc<AC>(w, A, kmax, acc_t0, acc_off);
        acc_t0 = -1;
        for (int tw = t_lo; tw <= t_hi; tw += kmax) {
          const int Kw = min(kmax, t_hi - tw + 1);
          pair_rows<true, HC, AC>(A, w, a, b, pa, pb, na, nb, cp, sp, Dc, Ds, tw, Kw, t_hi, seg);
          flush_acc<AC>(w, A, Kw, tw, out_off);
        }
      }
    }
  }
  if (acc_t0 >= 0) flush_acc<AC>(w, A, kmax, acc_t0, acc_off);
}

// ----------------------------------------------------------------------------
// FP64 path
// ----------------------------------------------------------------------------
// FP64 arithmetic is the scarce unit of this part (1.7 fused multiply-adds per
// clock and SM, against 126 in FP32), so the kernel spends it per run of
// pixels in one bin and not per pixel pair, with the results of FP64:
//  * bins: FP32 coordinates with a proven error bound; a pixel pair whose
//    coordinate lies within the bound of a bin edge (about 1 step in 80 holds
//    one) is binned by the definition in FP64, r = |d_i - d_j| * c, x = r * (1/D);
//  * sums: with the forest's FP64 prefix sums P of w and w delta, the pixels
//    [j0, j1) of one run add w_i (P[j1] - P[j0]).  A lane turns w_i P[j] into
//    a 52-bit integer at every run edge (one fused multiply-add with 1.5 2^52)
//    and adds the exact difference of two edges to the team's 64-bit integer
//    histogram, which is added to the FP64 bin sums in global memory per pair.
// Rounding: 2^-52 of the largest w_i P per edge, no error in any sum below the
// bins of a forest pair.  Measured (SDSS-like, 3,000 forests, W and N against
// 64-bit sums): see the error figures at launch_xi_fp64.
struct Fp64Args {
  XiArgs A;
  const double2* dw;    // per packed pixel (d, w delta)
  const double2* pre;   // exclusive prefix sums of (w, w delta): forest f's n + 1 entries from off[f] + f
  const double4_32a* bound;   // per forest: max |w|, max |w delta|, max |prefix of w|, max |prefix of w delta|
  double inv_dpar, inv_dperp;
};

constexpr double kM52 = 6755399441055744.0;   // 1.5 * 2^52
constexpr int kGrab64 = 8;                    // most pairs per work grab

// Power of two 2^(50 - e), 2^e <= B < 2^(e+1): |v| <= B maps below 2^51.
__device__ __forceinline__ double edge_scale(double B) {
  if (!(B > 1e-280) || !(B < 1e280)) return 1.0;
  const int e = static_cast<int>((__double_as_longlong(B) >> 52) & 0x7FF) - 1023;
  return __longlong_as_double(static_cast<long long>(50 - e + 1023) << 52);
}

// 1 / sc of a power of two (no FP64 division)
__device__ __forceinline__ double inv_pow2(double sc) {
  return __longlong_as_double((2046ll << 52) - __double_as_longlong(sc));
}

struct Walk64 {
  float cp, sp;              // c/D_par, s/D_perp
  float hp, ht;              // 1/2 - guard of the two coordinates
  float pmax, tmin, tmax;
  uint32_t stride, base, guard, twin, tspan, dummy;
  double cp64, sp64;
  const float* x;            // staged packed distances of b
  const double2* pre;        // staged prefix sums of b
  const double2* dw;         // b's (d, w delta) in global memory, at the segment
};

struct Lane64 {
  float uc, us;
  double d, w, wd;           // d_i, and w_i, (w delta)_i times the fixed-point scales
  long long eN, eW;          // edge integers at the start of the run to add next
  uint32_t cur, key;
  int j;                     // end of the held run
  bool on;
};

// Adds every lane's held run [previous edge, j) to its bin.
__device__ __forceinline__ void add_run64(Lane64& l, const Walk64& k) {
  const double2 p = k.pre[l.on ? l.j : 0];
  const long long n = __double_as_longlong(fma(l.wd, p.y, kM52));
  const long long w = __double_as_longlong(fma(l.w, p.x, kM52));
  const uint32_t addr = l.on ? k.base + (l.key << 4) : k.dummy;
  const long long dn = l.on ? n - l.eN : 0, dw = l.on ? w - l.eW : 0;
  asm volatile("{\n\tred.shared.add.u64 [%0], %1;\n\tred.shared.add.u64 [%0+8], %2;\n\t}" ::"r"(addr), "l"(dn), "l"(dw));
  l.eN = l.on ? n : l.eN;
  l.eW = l.on ? w : l.eW;
  l.on = false;
}

template <bool WINDOW>
__device__ __forceinline__ void step64(float xj, int j, const Walk64& k, Lane64& l) {
  const float rp = fabsf(fmaf(-xj, k.cp, l.uc));
  const float rt = fmaf(xj, k.sp, l.us);
  const float pm = __fadd_rd(rp, kMagic), tm = __fadd_rd(rt, kMagic);
  const bool near = fabsf((rp - (pm - kMagic)) - 0.5f) > k.hp || fabsf((rt - (tm - kMagic)) - 0.5f) > k.ht;
  const uint32_t tb = __float_as_uint(fminf(WINDOW ? tm : fmaxf(tm, k.tmin), k.tmax));
  uint32_t key = tb * k.stride + __float_as_uint(fminf(pm, k.pmax));
  if (WINDOW) key = (tb - kMagicBits - k.twin <= k.tspan) ? key : k.guard;
  if (__any_sync(0xffffffffu, near)) {
    const double dj = k.dw[j].x;
    const double x = fabs(l.d - dj) * k.cp64, y = (l.d + dj) * k.sp64;
    uint32_t exact = k.guard;
    // pmax and tmax hold n_par and the row past the band
    if (x < static_cast<double>(k.pmax - kMagic) && y < static_cast<double>(k.tmax - kMagic)) {
      const uint32_t t = static_cast<uint32_t>(static_cast<int>(y));
      if (!WINDOW || t - k.twin <= k.tspan)
        exact = (kMagicBits + t) * k.stride + kMagicBits + static_cast<uint32_t>(static_cast<int>(x));
    }
    key = near ? exact : key;
  }
  const bool chg = key != l.cur;
  if (__any_sync(0xffffffffu, chg && l.on)) add_run64(l, k);
  l.key = chg ? l.cur : l.key;
  l.j = chg ? j : l.j;
  l.on = l.on || chg;
  l.cur = key;
}

// Bin rows [t0, t0 + K) of forest pair (a, b) into the FP64 sums; WINDOW
// where the band goes on beyond them (its top row is t_hi).
template <bool WINDOW>
__device__ void pair64(const Fp64Args& P, unsigned long long* hist, double2* pbuf, float* xbuf, int a, int b, int na,
                       int nb, double cp64, double sp64, int t0, int K, int t_hi, int seg, int hcap) {
  const XiArgs& A = P.A;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int npar = A.n_par;
  const float fnpar = static_cast<float>(npar), fnperp = static_cast<float>(A.n_perp);
  const int64_t oa = A.F.off[a], ob = A.F.off[b];
  const Pix* __restrict__ pa = A.pix + oa;
  const Pix* __restrict__ pb = A.pix + ob;
  const float refa = A.F.dref[a], refb = A.F.dref[b];
  Walk64 k;
  k.cp = static_cast<float>(cp64);
  k.sp = static_cast<float>(sp64);
  k.cp64 = cp64;
  k.sp64 = sp64;
  const float Dc = (refa - refb) * k.cp, Ds = (refa + refb) * k.sp;
  // Bounds of the FP32 coordinates' errors, u = 2^-24 and X the largest packed
  // distances: r_par/D: u c/D (4 |ref_a - ref_b| + 3 X_a + 2 X_b) + u (n_par + 2)
  // (rounding of the packed distances, of c/D, of the products and of the two
  // fused multiply-adds); r_perp/D: 9 u (n_perp + 2), its terms being positive.
  const float u = 5.9604645e-8f;
  const float gp = 4.f * u * ((fabsf(refa - refb) + pa[na - 1].x + pb[nb - 1].x) * k.cp + (fnpar + 2.f));
  const float gt = 12.f * u * (fnperp + 2.f);
  k.hp = 0.5f - gp - 1e-7f;
  k.ht = 0.5f - gt - 1e-7f;
  k.stride = static_cast<uint32_t>(npar + 1);
  const uint32_t C = kMagicBits * (k.stride + 1u) + static_cast<uint32_t>(t0) * k.stride;
  const uint32_t h0 = smem_addr(hist);
  k.base = h0 - 16u * C;
  k.guard = C + static_cast<uint32_t>(npar);
  k.pmax = kMagic + fnpar;
  k.tmin = kMagic + static_cast<float>(t0);
  k.tmax = kMagic + static_cast<float>(t_hi + 1);
  k.twin = static_cast<uint32_t>(t0);
  k.tspan = static_cast<uint32_t>(K - 1);
  k.dummy = h0 + 16u * static_cast<uint32_t>(hcap - 32 + lane);
  k.x = xbuf;
  k.pre = pbuf;
  const double4_32a ba = P.bound[a], bb = P.bound[b];
  const double scW = edge_scale(ba.x * bb.z), scN = edge_scale(ba.y * bb.w);
  const double inv_scW = inv_pow2(scW), inv_scN = inv_pow2(scN);
  const int64_t out_off = static_cast<int64_t>(A.F.mock[a]) * A.nb;
  const int nchunk = (na + 31) >> 5;
  for (int j0 = 0; j0 < nb; j0 += seg) {
    const int segn = min(seg, nb - j0);
    for (int q = threadIdx.x; q <= segn; q += kTeam) {
      pbuf[q] = P.pre[ob + b + j0 + q];
      if (q < segn) xbuf[q] = pb[j0 + q].x;
    }
    k.dw = P.dw + ob + j0;
    __syncthreads();
    // batches of 32 chunks (1,024 rows): a bin's integer sum stays below 2^62
    for (int cb = 0; cb < nchunk; cb += 32) {
      const int i0 = (cb + lane) << 5;
      int jlo = 0, jhi = 0;
      if (i0 < na) {
        const float xf = pa[i0].x, xl = pa[min(i0 + 31, na - 1)].x;
        float dlo = (fmaf(xf, k.cp, Dc) - fnpar) / k.cp;
        float dhi = (fmaf(xl, k.cp, Dc) + fnpar) / k.cp;
        if (k.sp > 0.f) dhi = fminf(dhi, (fnperp - fmaf(xf, k.sp, Ds)) / k.sp);
        dlo -= fabsf(dlo) * 1e-5f + 1e-2f;
        dhi += fabsf(dhi) * 1e-5f + 1e-2f;
        jlo = floats_below(xbuf, segn, dlo);
        jhi = floats_below(xbuf, segn, dhi);
      }
      // the chunks with work, in turn to the two warps
      unsigned todo = __ballot_sync(0xffffffffu, jlo < jhi);
      for (int turn = 0; todo; ++turn) {
        const int c = __ffs(todo) - 1;
        todo &= todo - 1u;
        if ((turn & 1) != wid) continue;
        const int jb = __shfl_sync(0xffffffffu, jlo, c), je = __shfl_sync(0xffffffffu, jhi, c);
        const int i = ((cb + c) << 5) + lane;
        const int ic = min(i, na - 1);   // lanes past the end repeat the last pixel with zero weight
        const Pix pi = pa[ic];
        const double2 di = P.dw[oa + ic];
        Lane64 l;
        l.uc = fmaf(pi.x, k.cp, Dc);
        l.us = fmaf(pi.x, k.sp, Ds);
        l.d = di.x;
        l.w = (i < na) ? static_cast<double>(pi.y) * scW : 0.0;
        l.wd = (i < na) ? di.y * scN : 0.0;
        l.cur = l.key = k.guard;
        l.j = jb;
        l.on = false;
        const double2 p0 = pbuf[jb];
        l.eN = __double_as_longlong(fma(l.wd, p0.y, kM52));
        l.eW = __double_as_longlong(fma(l.w, p0.x, kM52));
        int j = jb;
        for (; j + 4 <= je; j += 4) {
          float x[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = xbuf[j + q];
#pragma unroll
          for (int q = 0; q < 4; ++q) step64<WINDOW>(x[q], j + q, k, l);
        }
        for (; j < je; ++j) step64<WINDOW>(xbuf[j], j, k, l);
        if (__any_sync(0xffffffffu, l.on)) add_run64(l, k);
        l.key = l.cur;
        l.j = je;
        l.on = true;
        add_run64(l, k);
      }
      // integer sums -> FP64 bin sums
      __syncthreads();
      for (int q = threadIdx.x; q < (K + 1) * (npar + 1); q += kTeam) {
        const long long n = static_cast<long long>(hist[2 * q]), w = static_cast<long long>(hist[2 * q + 1]);
        if ((n | w) != 0) {
          const int tt = q / (npar + 1), p = q - tt * (npar + 1);
          if (tt < K && p < npar) {
            const int64_t bin = out_off + static_cast<int64_t>(p) * A.n_perp + t0 + tt;
            red_add_f64_global(A.num + bin, static_cast<double>(n) * inv_scN);
            red_add_f64_global(A.wsum + bin, static_cast<double>(w) * inv_scW);
          }
          hist[2 * q] = 0ull;
          hist[2 * q + 1] = 0ull;
        }
      }
      __syncthreads();
    }
  }
}

__global__ void __launch_bounds__(kTeam) xi_fp64_kernel(Fp64Args P, int seg, int kmax, int hcap, int grab) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long s_it;
  __shared__ double2 s_cs[kGrab64];
  const XiArgs& A = P.A;
  // histogram (N, W) interleaved: hcap x 16 bytes | prefix sums (seg + 1) x 16 | packed distances seg x 4
  unsigned long long* hist = reinterpret_cast<unsigned long long*>(smem);
  double2* pbuf = reinterpret_cast<double2*>(smem + static_cast<size_t>(hcap) * 16);
  float* xbuf = reinterpret_cast<float*>(pbuf + seg + 1);
  for (int q = threadIdx.x; q < 2 * hcap; q += kTeam) hist[q] = 0ull;
  const double fnperp = A.n_perp;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_it = atomicAdd(A.counter, static_cast<unsigned long long>(grab));
    __syncthreads();
    const unsigned long long it0 = s_it;
    if (it0 >= static_cast<unsigned long long>(A.n_pairs)) break;
    const int n = static_cast<int>(min(static_cast<int64_t>(grab), A.n_pairs - static_cast<int64_t>(it0)));
    // the grabbed pairs' half-angle factors, one thread each
    if (static_cast<int>(threadIdx.x) < n) {
      const int2 ab = A.pairs[it0 + threadIdx.x];
      double2 cs = make_double2(0.0, 0.0);
      if (ab.x >= 0) {
        const int a = ab.x, b = ab.y;
        const double sx = A.F.ux[a] + A.F.ux[b], sy = A.F.uy[a] + A.F.uy[b], sz = A.F.uz[a] + A.F.uz[b];
        const double dx = A.F.ux[a] - A.F.ux[b], dy = A.F.uy[a] - A.F.uy[b], dz = A.F.uz[a] - A.F.uz[b];
        const double c = 0.5 * sqrt(sx * sx + sy * sy + sz * sz);
        const double s = 0.5 * sqrt(dx * dx + dy * dy + dz * dz);
        cs = make_double2(c * P.inv_dpar, s * P.inv_dperp);
      }
      s_cs[threadIdx.x] = cs;
    }
    __syncthreads();
    for (int q = 0; q < n; ++q) {
      const int2 ab = A.pairs[it0 + q];
      if (ab.x < 0) continue;   // rejected pair
      const int a = ab.x, b = ab.y;
      const int na = A.F.len[a], nb = A.F.len[b];
      if (na == 0 || nb == 0) continue;
      const double cp = s_cs[q].x, sp = s_cs[q].y;
      const double2* da = P.dw + A.F.off[a];
      const double2* db = P.dw + A.F.off[b];
      const double rt_min = (da[0].x + db[0].x) * sp;
      const double rt_max = (da[na - 1].x + db[nb - 1].x) * sp;
      if (!(rt_min < fnperp)) continue;
      const int t_lo = static_cast<int>(rt_min);
      const int t_hi = (rt_max < fnperp) ? static_cast<int>(rt_max) : A.n_perp - 1;
      if (t_hi - t_lo < kmax) {
        pair64<false>(P, hist, pbuf, xbuf, a, b, na, nb, cp, sp, t_lo, t_hi - t_lo + 1, t_hi, seg, hcap);
      } else {
        for (int tw = t_lo; tw <= t_hi; tw += kmax)
          pair64<true>(P, hist, pbuf, xbuf, a, b, na, nb, cp, sp, tw, min(kmax, t_hi - tw + 1), t_hi, seg, hcap);
      }
    }
  }
}

// One warp per forest: FP64 distances and w delta, exclusive prefix sums of w
// and w delta, and the bounds of their fixed-point scales.
__global__ void pack64_kernel(lya_catalog cat, Forests F, int64_t forest_base, double2* dw, double2* pre,
                              double4_32a* bound) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t f = warp; f < cat.n_forests; f += nw) {
    const int64_t gf = forest_base + f;
    const int n = F.len[gf];
    const int64_t o = cat.offsets[f];
    const int64_t g = F.off[gf];
    double2* pf = pre + g + gf;
    double cw = 0.0, cn = 0.0, mw = 0.0, mn = 0.0, mpw = 0.0, mpn = 0.0;
    for (int base = 0; base < n; base += 32) {
      const int k = base + lane;
      double w = 0.0, wd = 0.0;
      if (k < n) {
        w = cat.weight[o + k];
        wd = w * static_cast<double>(cat.delta[o + k]);
        dw[g + k] = make_double2(cat.dist[o + k], wd);
      }
      mw = fmax(mw, fabs(w));
      mn = fmax(mn, fabs(wd));
      double sw = w, sn = wd;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const double ow = __shfl_up_sync(0xffffffffu, sw, d), on = __shfl_up_sync(0xffffffffu, sn, d);
        if (lane >= d) {
          sw += ow;
          sn += on;
        }
      }
      sw += cw;
      sn += cn;
      if (k < n) pf[k + 1] = make_double2(sw, sn);
      mpw = fmax(mpw, fabs(sw));
      mpn = fmax(mpn, fabs(sn));
      cw = __shfl_sync(0xffffffffu, sw, 31);
      cn = __shfl_sync(0xffffffffu, sn, 31);
    }
    mw = warp_max_f64(mw);
    mn = warp_max_f64(mn);
    mpw = warp_max_f64(mpw);
    mpn = warp_max_f64(mpn);
    if (lane == 0) {
      if (n > 0) pf[0] = make_double2(0.0, 0.0);
      bound[gf] = make_double4_32a(mw, mn, mpw, mpn);
    }
  }
}

// In-grid pixel-pair count of every kept pair (same FP32 binning as the
// mixed kernel); one warp per forest pair.
__global__ void pair_stats_kernel(XiArgs A, uint64_t seed, uint64_t thr, int all, StatsOut* out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const float fnpar = static_cast<float>(A.n_par), fnperp = static_cast<float>(A.n_perp);
  unsigned long long my_pairs = 0, my_pix = 0, my_sq = 0;
  for (int64_t k = warp; k < A.n_pairs; k += nw) {
    const int2 ab = A.pairs[k];
    if (ab.x < 0 || !keep_pair(ab.x, ab.y, seed, thr, all)) continue;
    const int na = A.F.len[ab.x], nb = A.F.len[ab.y];
    const float cp = A.cs[k].x, sp = A.cs[k].y;
    const float refa = A.F.dref[ab.x], refb = A.F.dref[ab.y];
    const float Dc = (refa - refb) * cp, Ds = (refa + refb) * sp;
    const Pix* pa = A.pix + A.F.off[ab.x];
    const Pix* pb = A.pix + A.F.off[ab.y];
    unsigned long long cnt = 0;
    for (int i = lane; i < na; i += 32) {
      const float di = pa[i].x;
      const float uc = fmaf(di, cp, Dc), us = fmaf(di, sp, Ds);
      for (int j = 0; j < nb; ++j) {
        const float dj = pb[j].x;
        const float rp = fabsf(fmaf(-dj, cp, uc));
        const float rt = fmaf(dj, sp, us);
        cnt += (rp < fnpar && rt < fnperp) ? 1ull : 0ull;
      }
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    my_pairs += 1;
    my_pix += cnt;
    my_sq += cnt * cnt;
  }
  if (lane == 0 && my_pairs) {
    atomicAdd(&out->pairs, my_pairs);
    atomicAdd(&out->pix, my_pix);
    atomicAdd(&out->pix_sq, my_sq);
  }
}

// Bin-edge flips of the mixed path: for every pixel pair of the kept forest
// pairs, the bin from the mixed kernel's FP32 arithmetic against the bin from
// the FP64 path's arithmetic (FP64 distances of the caller's catalogue, FP64
// half-angle from the unit vectors).  One warp per forest pair.
__global__ void flip_tally_kernel(XiArgs A, const double* dist, double inv_dpar, double inv_dperp,
                                  uint64_t seed, uint64_t thr, int all, FlipOut* out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int npar = A.n_par, nperp = A.n_perp;
  const float fnpar = static_cast<float>(npar), fnperp = static_cast<float>(nperp);
  unsigned long long n64 = 0, nflip = 0;
  double w64 = 0.0, wflip = 0.0;
  for (int64_t k = warp; k < A.n_pairs; k += nw) {
    const int2 ab = A.pairs[k];
    if (ab.x < 0 || !keep_pair(ab.x, ab.y, seed, thr, all)) continue;
    const int a = ab.x, b = ab.y;
    const int na = A.F.len[a], nb = A.F.len[b];
    if (na == 0 || nb == 0) continue;
    const float cp = A.cs[k].x, sp = A.cs[k].y;
    const float refa = A.F.dref[a], refb = A.F.dref[b];
    const float Dc = (refa - refb) * cp, Ds = (refa + refb) * sp;
    const Pix* pa = A.pix + A.F.off[a];
    const Pix* pb = A.pix + A.F.off[b];
    const double* da = dist + A.F.off[a];
    const double* db = dist + A.F.off[b];
    const double sx = A.F.ux[a] + A.F.ux[b], sy = A.F.uy[a] + A.F.uy[b], sz = A.F.uz[a] + A.F.uz[b];
    const double dx = A.F.ux[a] - A.F.ux[b], dy = A.F.uy[a] - A.F.uy[b], dz = A.F.uz[a] - A.F.uz[b];
    const double cp64 = 0.5 * sqrt(sx * sx + sy * sy + sz * sz) * inv_dpar;
    const double sp64 = 0.5 * sqrt(dx * dx + dy * dy + dz * dz) * inv_dperp;
    for (int i = lane; i < na; i += 32) {
      const Pix pi = pa[i];
      const double di = da[i];
      const float uc = fmaf(pi.x, cp, Dc), us = fmaf(pi.x, sp, Ds);
      for (int j = 0; j < nb; ++j) {
        const Pix q = pb[j];
        const float rp = fabsf(fmaf(-q.x, cp, uc));
        const float rt = fmaf(q.x, sp, us);
        const int bin32 = (rp < fnpar && rt < fnperp)
                              ? static_cast<int>(__float_as_uint(__fadd_rd(rp, kMagic)) - kMagicBits) * nperp +
                                    static_cast<int>(__float_as_uint(__fadd_rd(rt, kMagic)) - kMagicBits)
                              : -1;
        const double x = fabs(di - db[j]) * cp64;
        const double y = (di + db[j]) * sp64;
        const int bin64 = (x < npar && y < nperp) ? static_cast<int>(x) * nperp + static_cast<int>(y) : -1;
        const double w = static_cast<double>(pi.y) * static_cast<double>(q.y);
        if (bin64 >= 0) {
          n64 += 1;
          w64 += w;
        }
        if (bin32 != bin64) {
          nflip += 1;
          wflip += w;
        }
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    n64 += __shfl_xor_sync(0xffffffffu, n64, o);
    nflip += __shfl_xor_sync(0xffffffffu, nflip, o);
    w64 += __shfl_xor_sync(0xffffffffu, w64, o);
    wflip += __shfl_xor_sync(0xffffffffu, wflip, o);
  }
  if (lane == 0 && n64 + nflip > 0) {
    atomicAdd(&out->pix, n64);
    atomicAdd(&out->flips, nflip);
    atomicAdd(&out->w, w64);
    atomicAdd(&out->wflip, wflip);
  }
}

__global__ void finalize_kernel(const double* num, const double* wsum, double* xi, int64_t n) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const double w = wsum[k];
    xi[k] = (w != 0.0) ? num[k] / w : 0.0;
  }
}

}  // namespace

int xi_mixed_max_npar() {
  // two chunk-histogram rows (band row and guard row) of n_par + 1 words below the 32 dummy words
  return std::min((kHcapL - 32) / 2 - 1, kAcapL);
}

cudaError_t plan_xi_mixed(const DevInfo& dev, int n_par, int max_len, int grab, XiLaunch* L) {
  if (n_par > xi_mixed_max_npar()) return cudaErrorInvalidValue;
  int seg = ((std::max(max_len, 1) + 31) / 32) * 32;
  if (seg > kMaxSeg) seg = kMaxSeg;   // longer forests are staged in segments
  const bool small = max_len > kSmallTablesLen && (kHcapS - 32) / (n_par + 1) - 1 >= 5 && kAcapS / n_par >= 5;
  L->warps = kTeam / 32;
  L->hcap = small ? kHcapS : kHcapL;
  L->acap = small ? kAcapS : kAcapL;
  L->seg = seg;
  L->grab = grab;
  L->smem = (L->acap + L->hcap + seg) * 16;
  if (L->smem > dev.smem_optin) return cudaErrorInvalidValue;
  const void* fn = small ? reinterpret_cast<const void*>(xi_mixed_kernel<kHcapS, kAcapS>)
                         : reinterpret_cast<const void*>(xi_mixed_kernel<kHcapL, kAcapL>);
  cudaError_t e = set_max_dynamic_smem(fn, L->smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kTeam, L->smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidValue;
  L->blocks = per_sm * dev.sms;
  return cudaSuccess;
}

cudaError_t launch_xi_mixed(const XiArgs& a, const XiLaunch& L, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  if (a.n_pairs == 0) return cudaSuccess;
  // band rows per window: the chunk histogram needs (kmax + 1) x (n_par + 1)
  // entries (guard row and column), the accumulator kmax x n_par
  const int kmax = std::max(1, std::min({a.n_perp, (L.hcap - 32) / (a.n_par + 1) - 1, L.acap / a.n_par}));
  if (L.hcap == kHcapS)
    LYA_COUNT(1), xi_mixed_kernel<kHcapS, kAcapS><<<L.blocks, kTeam, L.smem, s>>>(a, L.seg, kmax, L.grab);
  else
    LYA_COUNT(1), xi_mixed_kernel<kHcapL, kAcapL><<<L.blocks, kTeam, L.smem, s>>>(a, L.seg, kmax, L.grab);
  return cudaGetLastError();
}

cudaError_t launch_xi_fp64(const XiArgs& a, const lya_catalog* cats, int n_cats, const DevInfo& dev,
                           int max_len, double r_par_max, double r_perp_max, XiLaunch* used,
                           cudaStream_t s) {
  if (a.n_par > kMaxPar64) return cudaErrorInvalidValue;
  // FP64 pixels, prefix sums and bounds, built on demand in one temporary buffer
  int64_t npix = 0;
  for (int m = 0; m < n_cats; ++m) npix += cats[m].n_pix;
  const int64_t nf = std::max<int64_t>(a.F.n, 1), np = std::max<int64_t>(npix, 1);
  char* tmp = nullptr;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&tmp), static_cast<size_t>(32 * nf + 16 * (np + nf) + 16 * np), s);
  if (e != cudaSuccess) return e;
  double4_32a* bound = reinterpret_cast<double4_32a*>(tmp);
  double2* pre = reinterpret_cast<double2*>(tmp + 32 * nf);
  double2* dw = pre + np + nf;
  int64_t fb = 0;
  for (int m = 0; m < n_cats; ++m) {
    if (cats[m].n_forests > 0) {
      int64_t blocks = std::min<int64_t>((cats[m].n_forests * 32 + 255) / 256, 65535);
      LYA_COUNT(1), pack64_kernel<<<static_cast<int>(blocks), 256, 0, s>>>(cats[m], a.F, fb, dw, pre, bound);
    }
    fb += cats[m].n_forests;
  }
  Fp64Args P;
  P.A = a;
  P.dw = dw;
  P.pre = pre;
  P.bound = bound;
  P.inv_dpar = static_cast<double>(a.n_par) / r_par_max;
  P.inv_dperp = static_cast<double>(a.n_perp) / r_perp_max;
  int seg = ((std::max(max_len, 1) + 31) / 32) * 32;
  if (seg > kMaxSeg) seg = kMaxSeg;
  // at least one band row and the guard row; 32 dummy entries
  const int hcap = std::max(408, 2 * (a.n_par + 1)) + 32;
  const int kmax = std::min(a.n_perp, (hcap - 32) / (a.n_par + 1) - 1);
  const int smem = hcap * 16 + (seg + 1) * 16 + seg * 4;
  e = set_max_dynamic_smem(reinterpret_cast<const void*>(xi_fp64_kernel), smem);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, xi_fp64_kernel, kTeam, smem);
  if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidValue;
  if (e == cudaSuccess) e = cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s);
  // pairs per grab: one thread each computes the geometry; few at a time where the list is short
  const int teams = per_sm * dev.sms;
  const int grab = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(kGrab64, a.n_pairs / (16 * std::max(teams, 1)))));
  if (e == cudaSuccess && a.n_pairs > 0) {
    LYA_COUNT(1), xi_fp64_kernel<<<teams, kTeam, smem, s>>>(P, seg, kmax, hcap, grab);
    e = cudaGetLastError();
  }
  if (used) {
    used->warps = kTeam / 32;
    used->blocks = teams;
    used->seg = seg;
    used->smem = smem;
    used->hcap = hcap;
    used->grab = grab;
  }
  cudaFreeAsync(tmp, s);
  return e;
}

cudaError_t launch_pair_stats(const XiArgs& a, double p_subsample, uint64_t seed, StatsOut* out,
                              const DevInfo& dev, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(StatsOut), s);
  if (e != cudaSuccess || a.n_pairs == 0 || p_subsample <= 0.0) return e;
  const int all = p_subsample >= 1.0 ? 1 : 0;
  const uint64_t thr = all ? 0 : static_cast<uint64_t>(p_subsample * 18446744073709551616.0);
  LYA_COUNT(1), pair_stats_kernel<<<dev.sms * 8, 256, 0, s>>>(a, seed, thr, all, out);
  return cudaGetLastError();
}

cudaError_t launch_flip_tally(const XiArgs& a, const double* dist, double inv_dpar, double inv_dperp,
                              double p_subsample, uint64_t seed, FlipOut* out, const DevInfo& dev,
                              cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(FlipOut), s);
  if (e != cudaSuccess || a.n_pairs == 0 || p_subsample <= 0.0) return e;
  const int all = p_subsample >= 1.0 ? 1 : 0;
  const uint64_t thr = all ? 0 : static_cast<uint64_t>(p_subsample * 18446744073709551616.0);
  LYA_COUNT(1), flip_tally_kernel<<<dev.sms * 8, 256, 0, s>>>(a, dist, inv_dpar, inv_dperp, seed, thr, all, out);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const double* num, const double* wsum, double* xi, int64_t n,
                            cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  int64_t b = std::min<int64_t>((n + 255) / 256, 4096);
  LYA_COUNT(1), finalize_kernel<<<static_cast<int>(b), 256, 0, s>>>(num, wsum, xi, n);
  return cudaGetLastError();
}

}  // namespace lya
