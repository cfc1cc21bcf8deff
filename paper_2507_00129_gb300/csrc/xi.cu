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
// step of 32 pixel pairs, issue 74-76%), and on the SDSS-like grid, whose runs
// are two pixels long, the shared-memory pipe (77%: 2.9 wavefronts per
// reduction).  A team of two shares 12.7 KB of tables and the staged forest,
// so 9-13 teams (18-26 warps) fit on an SM where 8 single warps did.
// Measured (survey pass): 60,000 SDSS-like forests 624 -> 386 ms, 9,000
// DESI-like forests 414 -> 244 ms; 365 and 238 ms without the reductions of
// guard runs at the ends of a chunk.
// FP64 kernel (LYA_PREC_FP64): the results of FP64 distances, separations and
// products in the oracle's operation order, r = |d_i - d_j| * c, x = r * (1/D);
// see "FP64 path" below.
#include <algorithm>
#include <type_traits>

#include <math.h>

#include "exact.cuh"
#include "fixed.cuh"

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
constexpr int kMaxPar64 = 256;   // largest n_par of the FP64 path
constexpr int kMaxSeg = 1024;    // pixel buffer cap per warp

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

// Bin of a lane's pixel and the pixel {x, x} of b, as the key
// (2^23 bits + row) * (n_par + 1) + (2^23 bits + column).
template <bool WINDOW>
__device__ __forceinline__ uint32_t step_key(F2 xx, const Walk& k, F2 ucus) {
  const float2 r = unf2(fma2(xx, k.cpsp, ucus));
  const float pf = fminf(__fadd_rd(fabsf(r.x), kMagic), k.pmax);
  const float tf = fminf(__fadd_rd(r.y, kMagic), k.tmax);
  const uint32_t key = __float_as_uint(tf) * k.stride + __float_as_uint(pf);
  return (!WINDOW || (__float_as_uint(tf) - kMagicBits - k.twin) <= k.tspan) ? key : k.guard;
}

// One pixel pair of a run walk (see chunk_runs).  A run that ends here is
// held in the lane's registers; the warp adds its held runs to the histogram
// only when some lane that already holds one ends another.  On the DESI-like
// grid a run is about seven pixels long, so the reductions come once per ~6
// steps instead of every step.
template <bool WINDOW, int HC>
__device__ __forceinline__ void run_step(const ulonglong2& q, const Walk& k, F2 ucus, float wdi, float wi,
                                         uint32_t& cur, float& aN, float& aW, Held& held) {
  const uint32_t key = step_key<WINDOW>(q.x, k, ucus);
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
  // the first run starts in the first pixel's bin: ending one of the guard
  // bin there would send all lanes' reductions to one word
  uint32_t cur = step_key<WINDOW>(buf[jlo].x, k, ucus);
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
  // (not of the lanes that have left the grid: their key's column is the guard's)
  held = Held{cur, aN, aW, (cur - (k.guard - (k.stride - 1u))) % k.stride != k.stride - 1u};
  add_held<HC>(held, k);
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
          two_sum_add(nhi[a], nlo[a], vn);
          two_sum_add(whi[a], wlo[a], vw);
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
  // (one pixel has no gap: hmin is then next to 0)
  const float nrun = fminf(2.f / (cp * A.F.hmin[bidx]) + 1.f, static_cast<float>(nb));
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
        jlo = staged_below(w.buf, 0, segn, dlo);
        jhi = staged_below(w.buf, 0, segn, dhi);
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

// HC words per chunk-histogram array, AC entries per accumulator array (see kHcapL)
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
// clock and SM, against 126 in FP32), so the kernel uses it only where a bin
// needs it, with the results of FP64:
//  * bins: FP32 coordinates with a proven error bound; a pixel pair whose
//    coordinate lies within the bound of a bin edge (about 1 step in 80 holds
//    one) is binned by the definition in FP64, r = |d_i - d_j| * c, x = r * (1/D);
//  * products and sums are exact integers (see exact.cuh), except for forest
//    pairs whose values lie too far apart for them (see wide_pair), which a
//    second launch sums in FP64 on the same walk;
//  * the walk goes along the diagonals of the pixel-pair matrix: lane l takes
//    the pairs (i, i + o + l), whose separation changes slowly with i, so a run
//    of pixel pairs in one bin is tens of pairs long on any grid.  A lane that
//    leaves a bin adds its run to the team's 64-bit integer histogram, which
//    is added to the FP64 bin sums in global memory per tile of 256 x 256.
// Rounding: 2^-54 of the forest's largest value per pixel, 2^-51 to 2^-45 of the
// largest product per run (as the sums leave room), to nearest, none in the sums
// below a tile; the run's is at most 2^-36 of the pair's smallest product w_i w_j.
// What bounds it: issue (58%) and latencies of about 55 warp instructions per
// step, of which the key and its edge test take 20, the six multiply-adds 6,
// and the ends of runs (some lane in every second step) a quarter; a third of
// the lanes' pairs lie off the grid at the ends of the diagonals.
// Measured (SDSS-like, 3,000 forests): 370 ms with FP64 arithmetic and shared
// FP64 atomics per pixel pair, 62 ms with FP64 run-edge integers along the
// rows (FP64 pipe 74% busy), 45 ms as it is; the largest relative error of W
// and N against 64-bit sums is that of the first form (6e-15).
struct Fp64Args {
  XiArgs A;
  const double* d;            // per packed pixel: distance
  const int4* v;              // per packed pixel: H, L of w delta, H, L of w
  const double* wd;           // per packed pixel: w delta
  const int2* scale;          // per forest: s of w delta, s of w
  const float4* spread;       // per forest: see Spread64
  unsigned* wide;             // set where a forest pair is left to the FP64 sums
  double inv_dpar, inv_dperp;
};

// Sizes of a forest's values, for w delta and w: log2 of the largest over the
// smallest (rn, rw), and the largest sum of |values| over a tile's pixels in units
// of the largest (qn, qw).  The smallest weight is the smallest that is not 0;
// w delta comes arbitrarily close to 0, so its smallest is that of the largest of
// 32 consecutive pixels (all of them 0 apart, and less than 16 at the forest's end).
using Spread64 = float4;   // (rn, rw, qn, qw)

constexpr int kGrab64 = 8;      // most pairs per work grab
constexpr int kTile64 = 256;    // pixels of a tile edge: a run of 256 products stays below 2^62
constexpr int kPad64 = 40;      // sentinels on both sides of a staged tile of b (a block of 8 rows and 32 diagonals reaches 38 past it)

struct Walk64 {
  float cp, sp;              // c/D_par, s/D_perp
  float hp, ht;              // 1/2 - guard of the two coordinates
  float pmax, tmin, tmax;
  uint32_t stride, base, guard, twin, tspan;
  int shift;                 // bits a run's sum is rounded by before it is added to its bin
  double cp64, sp64;
};

template <class S>
struct Run64 {
  S s;                       // the current run
  S held;                    // an ended run, until the lane ends another
  uint32_t cur, key;         // their bins
  bool in, on;               // the current bin lies in the grid; a run is held
};

// Adds every lane's held run to its bin.
template <class S>
__device__ __forceinline__ void add_run64(Run64<S>& r, const Walk64& k) {
  if (r.on) add_bin64(r.held, k.base + (r.key << 4), k.shift);
  r.on = false;
  __syncwarp();
}

// Bits a run's sum is rounded by: products are below 2^52, and a bin's sum has to
// stay below 2^62.  A bin of a tile holds at most two runs of 2 D_par / (c gap_b) + 1
// pixels per row, and no more than the product of the two tiles' sums.
__device__ __forceinline__ int shift64(const XiArgs& A, const Spread64& a, const Spread64& b, int bi, float cp) {
  const float terms = fminf(fminf(512.f * (2.f / (cp * A.F.hmin[bi]) + 1.f), 65536.f),
                            1.001f * fmaxf(a.z * b.z, a.w * b.w) + 1.f);
  return max(1, 32 - __clz(static_cast<int>(terms)) - 10);
}

// Whether the integers would round a run by more than 2^-36 of the pair's
// smallest product: half of 2^shift against products of 2^(50 - r) and more.
// (Survey weights: r about 9.5 on the SDSS-like and 11 on the DESI-like grid.)
__device__ __forceinline__ bool wide_pair(const Spread64& a, const Spread64& b, int shift) {
  return fmaxf(a.x + b.x, a.y + b.y) + static_cast<float>(shift) > 15.f;
}

// Bin rows [t0, t0 + K) of forest pair (a, b) into the FP64 sums; WINDOW
// where the band goes on beyond them (its top row is t_hi).
template <bool WINDOW, class S>
__device__ void pair64(const Fp64Args& P, unsigned char* smem, int a, int b, int na, int nb, double cp64, double sp64,
                       int shift, int t0, int K, int t_hi, int tile, int hcap) {
  constexpr bool kExact = std::is_same<S, Sum64>::value;   // integers
  const XiArgs& A = P.A;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long* hist = reinterpret_cast<unsigned long long*>(smem);
  int4* av = reinterpret_cast<int4*>(smem + static_cast<size_t>(hcap) * 16);
  int4* bv = av + tile + kPad64;
  float2* au = reinterpret_cast<float2*>(bv + tile + kPad64);
  float* bx = reinterpret_cast<float*>(au + tile) + kPad64;
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
  k.base = smem_addr(hist) - 16u * C;
  k.guard = C + static_cast<uint32_t>(npar);
  k.pmax = kMagic + fnpar;
  k.tmin = kMagic + static_cast<float>(t0);
  k.tmax = kMagic + static_cast<float>(t_hi + 1);
  k.twin = static_cast<uint32_t>(t0);
  k.tspan = static_cast<uint32_t>(K - 1);
  k.shift = shift;
  const int2 ea = P.scale[a], eb = P.scale[b];
  const int64_t out_off = static_cast<int64_t>(A.F.mock[a]) * A.nb;
  // a pixel's (w delta, w): integers, or the FP64 values
  auto value = [&](int64_t g, float w) {
    if (kExact) return P.v[g];
    return pack_f64(P.wd[g], w);
  };
  for (int ia = 0; ia < na; ia += tile) {
    const int ta = min(tile, na - ia);
    for (int jb = 0; jb < nb; jb += tile) {
      const int tb = min(tile, nb - jb);
      // rows up to a multiple of 8 and the padding of b lie at infinite distance, with zero weight
      for (int q = threadIdx.x; q < ((ta + 7) & ~7); q += kTeam) {
        const float x = (q < ta) ? pa[ia + q].x : INFINITY;
        au[q] = (q < ta) ? make_float2(fmaf(x, k.cp, Dc), fmaf(x, k.sp, Ds)) : make_float2(INFINITY, INFINITY);
        av[q] = (q < ta) ? value(oa + ia + q, pa[ia + q].y) : make_int4(0, 0, 0, 0);
      }
      for (int q = static_cast<int>(threadIdx.x) - kPad64; q < tb + kPad64; q += kTeam) {
        const bool in = q >= 0 && q < tb;
        bx[q] = in ? pb[jb + q].x : INFINITY;
        bv[q] = in ? value(ob + jb + q, pb[jb + q].y) : make_int4(0, 0, 0, 0);
      }
      __syncthreads();
      // groups of 32 diagonals j - i = o + lane, in turn to the two warps
      const int ngroup = (ta + tb + 30) >> 5;
      for (int g = wid; g < ngroup; g += kTeam / 32) {
        const int o = 32 * g - (ta - 1);
        // lane m: whether block m of 8 rows can hold an in-grid pixel pair (both coordinates are monotone in
        // the sorted distances; 1e-2 bins cover the FP32 rounding)
        bool work = false;
        {
          const int i0 = 8 * lane, i1 = min(i0 + 7, ta - 1);
          const int jl = max(i0 + o, 0), jh = min(i1 + o + 31, tb - 1);
          if (i0 < ta && jl <= jh) {
            const float2 u0 = au[i0], u1 = au[i1];
            const float xl = bx[jl], xh = bx[jh];
            work = fmaf(-xh, k.cp, u0.x) < fnpar + 1e-2f && fmaf(-xl, k.cp, u1.x) > -fnpar - 1e-2f &&
                   fmaf(xl, k.sp, u0.y) < fnperp + 1e-2f;
          }
        }
        unsigned todo = __ballot_sync(0xffffffffu, work);
        Run64<S> r{S{}, S{}, k.guard, k.guard, false, false};
        for (; todo; todo &= todo - 1u) {
          const int i0 = 8 * (__ffs(todo) - 1);
          const float* px = bx + i0 + o + lane;
          const int4* pv = bv + i0 + o + lane;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float2 ui = au[i0 + q];
            const float xj = px[q];
            const float rp = fabsf(fmaf(-xj, k.cp, ui.x));
            const float rt = fmaf(xj, k.sp, ui.y);
            const float pm = __fadd_rd(rp, kMagic), tm = __fadd_rd(rt, kMagic);
            const bool near = fabsf((rp - (pm - kMagic)) - 0.5f) > k.hp || fabsf((rt - (tm - kMagic)) - 0.5f) > k.ht;
            const uint32_t tbits = __float_as_uint(fminf(WINDOW ? tm : fmaxf(tm, k.tmin), k.tmax));
            uint32_t key = tbits * k.stride + __float_as_uint(fminf(pm, k.pmax));
            if (WINDOW) key = (tbits - kMagicBits - k.twin <= k.tspan) ? key : k.guard;
            if (__any_sync(0xffffffffu, near)) {
              // (near is false for padding: its coordinates are infinite or NaN)
              const int jc = min(max(i0 + q + o + lane, 0), tb - 1);
              const double di = P.d[oa + ia + min(i0 + q, ta - 1)], dj = P.d[ob + jb + jc];
              const double x = fabs(di - dj) * k.cp64, y = (di + dj) * k.sp64;
              uint32_t exact = k.guard;
              // pmax and tmax hold n_par and the row past the band
              if (x < static_cast<double>(k.pmax - kMagic) && y < static_cast<double>(k.tmax - kMagic)) {
                const uint32_t t = static_cast<uint32_t>(static_cast<int>(y));
                if (t - k.twin <= k.tspan)
                  exact = (kMagicBits + t) * k.stride + kMagicBits + static_cast<uint32_t>(static_cast<int>(x));
              }
              key = near ? exact : key;
            }
            const bool chg = key != r.cur;
            if (__any_sync(0xffffffffu, chg)) {
              // (runs off the grid are dropped: all lanes' would go to a few words)
              if (__any_sync(0xffffffffu, chg && r.on && r.in)) add_run64(r, k);
              if (chg) {
                if (r.in) {
                  r.held = r.s;
                  r.key = r.cur;
                  r.on = true;
                }
                r.s = S{};
                r.cur = key;
                const uint32_t q = key - C;   // row * (n_par + 1) + column
                r.in = q < static_cast<uint32_t>(K) * k.stride && q % k.stride != static_cast<uint32_t>(npar);
              }
              __syncwarp();
            }
            const int4 vi = av[i0 + q], vj = pv[q];
            add_products(r.s, vi, vj);
          }
        }
        add_run64(r, k);
        r.held = r.s;
        r.key = r.cur;
        r.on = r.in;
        add_run64(r, k);
      }
      // the tile's sums -> FP64 bin sums
      __syncthreads();
      const double sn = pow2(56 + k.shift - ea.x - eb.x), sw = pow2(56 + k.shift - ea.y - eb.y);
      for (int q = threadIdx.x; q < (K + 1) * (npar + 1); q += kTeam) {
        const long long n = static_cast<long long>(hist[2 * q]), w = static_cast<long long>(hist[2 * q + 1]);
        if ((n | w) != 0) {
          const int tt = q / (npar + 1), p = q - tt * (npar + 1);
          if (tt < K && p < npar) {
            const int64_t bin = out_off + static_cast<int64_t>(p) * A.n_perp + t0 + tt;
            red_add_f64_global(A.num + bin, kExact ? static_cast<double>(n) * sn : __longlong_as_double(n));
            red_add_f64_global(A.wsum + bin, kExact ? static_cast<double>(w) * sw : __longlong_as_double(w));
          }
          hist[2 * q] = 0ull;
          hist[2 * q + 1] = 0ull;
        }
      }
      __syncthreads();
    }
  }
}

// S: Sum64, the forest pairs that the integers serve (the others set P.wide), or
// SumF64, the others.  Both over the whole list.
template <class S>
__global__ void __launch_bounds__(kTeam) xi_fp64_kernel(Fp64Args P, int tile, int kmax, int hcap, int grab) {
  // histogram (N, W) interleaved: hcap x 16 bytes | values of tile a and of tile b | (uc, us) of a | distances of b
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool kExact = std::is_same<S, Sum64>::value;
  if (!kExact && *P.wide == 0u) return;
  __shared__ unsigned long long s_it;
  __shared__ double2 s_cs[kGrab64];
  const XiArgs& A = P.A;
  for (int q = threadIdx.x; q < 2 * hcap; q += kTeam) reinterpret_cast<unsigned long long*>(smem)[q] = 0ull;
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
      const Spread64 ra = P.spread[a], rb = P.spread[b];
      const int shift = shift64(A, ra, rb, b, static_cast<float>(cp));
      if (wide_pair(ra, rb, shift) == kExact) {
        if (kExact && threadIdx.x == 0) *P.wide = 1u;
        continue;
      }
      const double* da = P.d + A.F.off[a];
      const double* db = P.d + A.F.off[b];
      const double rt_min = (da[0] + db[0]) * sp;
      const double rt_max = (da[na - 1] + db[nb - 1]) * sp;
      if (!(rt_min < fnperp)) continue;
      const int t_lo = static_cast<int>(rt_min);
      const int t_hi = (rt_max < fnperp) ? static_cast<int>(rt_max) : A.n_perp - 1;
      if (t_hi - t_lo < kmax) {
        pair64<false, S>(P, smem, a, b, na, nb, cp, sp, shift, t_lo, t_hi - t_lo + 1, t_hi, tile, hcap);
      } else {
        for (int tw = t_lo; tw <= t_hi; tw += kmax)
          pair64<true, S>(P, smem, a, b, na, nb, cp, sp, shift, tw, min(kmax, t_hi - tw + 1), t_hi, tile, hcap);
      }
    }
  }
}

// One warp per forest: distances, w delta, and w delta and w as integers on the
// forest's own power-of-two scales, and their spread.
__global__ void pack64_kernel(lya_catalog cat, Forests F, int64_t forest_base, double* d, double* wd, int4* v,
                              int2* scale, Spread64* spread) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t f = warp; f < cat.n_forests; f += nw) {
    const int64_t gf = forest_base + f;
    const int n = F.len[gf];
    const int64_t o = cat.offsets[f];
    const int64_t g = F.off[gf];
    // largest values; smallest weight; smallest of the 32-pixel segments' largest |w delta|; tiles' sums
    double mw = 0.0, mn = 0.0, lw = INFINITY, ln = INFINITY, qw = 0.0, qn = 0.0, tw = 0.0, tn = 0.0;
    for (int k0 = 0; k0 < n; k0 += 32) {
      if (k0 % kTile64 == 0) tw = tn = 0.0;
      const int k = k0 + lane;
      const double w = (k < n) ? static_cast<double>(cat.weight[o + k]) : 0.0;
      const double x = (k < n) ? fabs(w * static_cast<double>(cat.delta[o + k])) : 0.0;
      mw = fmax(mw, w);
      if (w > 0.0) lw = fmin(lw, w);
      const double top = warp_max_f64(x);
      mn = fmax(mn, top);
      if (top > 0.0 && (n - k0 >= 16 || k0 == 0)) ln = fmin(ln, top);
      tw += w;
      tn += x;
      if (k0 + 32 >= n || (k0 + 32) % kTile64 == 0) {
        qw = fmax(qw, warp_sum_f64(tw));
        qn = fmax(qn, warp_sum_f64(tn));
      }
    }
    mw = warp_max_f64(mw);
    lw = -warp_max_f64(-lw);
    // |value| < 2^(ilogb + 1): scaled below 2^54
    const int en = (mn > 0.0) ? 53 - ilogb(mn) : 0, ew = (mw > 0.0) ? 53 - ilogb(mw) : 0;
    const double sn = pow2(en), sw = pow2(ew);
    for (int k = lane; k < n; k += 32) {
      const double w = cat.weight[o + k], x = w * static_cast<double>(cat.delta[o + k]);
      d[g + k] = cat.dist[o + k];
      wd[g + k] = x;
      const int2 a = split55(x, sn), b = split55(w, sw);
      v[g + k] = make_int4(a.x, a.y, b.x, b.y);
    }
    if (lane == 0) {
      scale[gf] = make_int2(en, ew);
      // (a forest without a segment of its own, its values in the last pixels: as wide as the type)
      const float rn = (mn > 0.0) ? (ln < INFINITY ? log2f(static_cast<float>(mn / ln)) : 128.f) : 0.f;
      const float rw = (mw > 0.0) ? log2f(static_cast<float>(mw / lw)) : 0.f;
      spread[gf] = make_float4(rn, rw, mn > 0.0 ? static_cast<float>(qn / mn) : 0.f, mw > 0.0 ? static_cast<float>(qw / mw) : 0.f);
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
  // FP64 distances and integer pixels, built on demand in one temporary buffer
  int64_t npix = 0;
  for (int m = 0; m < n_cats; ++m) npix += cats[m].n_pix;
  const int64_t nf = (std::max<int64_t>(a.F.n, 1) + 1) & ~int64_t{1}, np = std::max<int64_t>(npix, 1);
  char* tmp = nullptr;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&tmp), static_cast<size_t>(16 + 24 * nf + 32 * np), s);
  if (e != cudaSuccess) return e;
  unsigned* wide = reinterpret_cast<unsigned*>(tmp);
  Spread64* spread = reinterpret_cast<Spread64*>(tmp + 16);
  int2* scale = reinterpret_cast<int2*>(spread + nf);
  int4* v = reinterpret_cast<int4*>(scale + nf);
  double* d = reinterpret_cast<double*>(v + np);
  double* wd = d + np;
  int64_t fb = 0;
  for (int m = 0; m < n_cats; ++m) {
    if (cats[m].n_forests > 0) {
      int64_t blocks = std::min<int64_t>((cats[m].n_forests * 32 + 255) / 256, 65535);
      LYA_COUNT(1), pack64_kernel<<<static_cast<int>(blocks), 256, 0, s>>>(cats[m], a.F, fb, d, wd, v, scale, spread);
    }
    fb += cats[m].n_forests;
  }
  Fp64Args P;
  P.A = a;
  P.d = d;
  P.v = v;
  P.wd = wd;
  P.scale = scale;
  P.spread = spread;
  P.wide = wide;
  P.inv_dpar = static_cast<double>(a.n_par) / r_par_max;
  P.inv_dperp = static_cast<double>(a.n_perp) / r_perp_max;
  const int tile = std::min((std::max(max_len, 1) + 7) & ~7, kTile64);
  // at least one band row and the guard row
  const int hcap = std::max(408, 2 * (a.n_par + 1));
  const int kmax = std::min(a.n_perp, hcap / (a.n_par + 1) - 1);
  const int smem = hcap * 16 + (2 * tile + 2 * kPad64) * 16 + tile * 8 + (tile + 2 * kPad64) * 4;
  e = set_max_dynamic_smem(reinterpret_cast<const void*>(xi_fp64_kernel<Sum64>), smem);
  if (e == cudaSuccess) e = set_max_dynamic_smem(reinterpret_cast<const void*>(xi_fp64_kernel<SumF64>), smem);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, xi_fp64_kernel<Sum64>, kTeam, smem);
  if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidValue;
  if (e == cudaSuccess) e = cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(wide, 0, sizeof(unsigned), s);
  // pairs per grab: one thread each computes the geometry; few at a time where the list is short
  const int teams = per_sm * dev.sms;
  const int grab = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(kGrab64, a.n_pairs / (16 * std::max(teams, 1)))));
  if (e == cudaSuccess && a.n_pairs > 0) {
    LYA_COUNT(1), xi_fp64_kernel<Sum64><<<teams, kTeam, smem, s>>>(P, tile, kmax, hcap, grab);
    e = cudaGetLastError();
    // the forest pairs left by it (the kernel ends at once where there are none)
    if (e == cudaSuccess) e = cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s);
    if (e == cudaSuccess) {
      LYA_COUNT(1), xi_fp64_kernel<SumF64><<<teams, kTeam, smem, s>>>(P, tile, kmax, hcap, grab);
      e = cudaGetLastError();
    }
  }
  if (used) {
    used->warps = kTeam / 32;
    used->blocks = teams;
    used->seg = tile;
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
