// Per-bin weighted means of the pair separations and of the pair distance,
// and pixel-pair counts: the columns a PICCA/Vega fit reads next to xi (the
// paper exports its results for Vega, Appendix A):
//     rpar_mean_A = sum_A w_i w_j r_par / W_A,  rperp_mean_A = sum_A w_i w_j r_perp / W_A,
//     dist_mean_A = sum_A w_i w_j (d_i + d_j) / 2 / W_A,  count_A,
// over the pixel pairs of Eq. (2.4) with the bisector split of Section 2.1.
//
// Bins are the FP32 ones of the mixed path's arithmetic (|d_i - d_j| from the
// packed distances and reference offsets, times cos(theta/2)/D_par).  The
// kernel is described at means_kernel.
#include <math.h>

#include <algorithm>

#include "fixed.cuh"

namespace lya {
namespace {

struct Acc {
  double* W;
  double* WX;
  double* WY;
  double* WD;
  double* WZ;   // sum w_i w_j (z_i + z_j) / 2 (with pixel redshifts)
  unsigned long long* C;
};

constexpr int kTeam = 64;       // threads of a team (one block): two warps on one forest pair
constexpr int kTile = 240;      // pixels of a tile edge: the low words of 57,600 blocks fit 32 bits
constexpr int kPad = 40;        // sentinels on both sides of a staged tile of b (a block of 8 rows reaches 38 past it)
constexpr int kBins = 408;      // bins of the band histogram: (K + 1) x (n_par + 1), guard row and column included

// A lane's current run of pixel pairs in one bin: sums of w_i w_j times
// (1, r_par/D_par), (d_i + d_j, z_i + z_j) and r_perp/D_perp, FP32 over a block
// of at most 8 pairs and two-word fixed point (see fixed.cuh) over blocks.
struct Run {
  F2 wx, sz;
  float y;
  uint32_t h[5], l[5];
  uint32_t cur;         // the run's bin
  int n;                // minus its first row; its pixel pairs once it has ended
  bool in;              // the bin lies in the grid
};

// Closes a block: its FP32 sums go to the run's integer words.
__device__ __forceinline__ void close_pair(F2& v, F2 sc, uint32_t& h0, uint32_t& l0, uint32_t& h1, uint32_t& l1) {
  const F2 m15 = f2(kM15, kM15);
  const F2 hm = fma2_rd(v, sc, m15);
  const F2 fr = fma2(v, sc, fma2(hm, f2(-1.f, -1.f), m15));
  const F2 lm = fma2(fr, f2(65536.f, 65536.f), m15);
  const float2 h = unf2(hm), l = unf2(lm);
  h0 += __float_as_uint(h.x) - kM15Bits;
  h1 += __float_as_uint(h.y) - kM15Bits;
  l0 += __float_as_uint(l.x) - kM15Bits;
  l1 += __float_as_uint(l.y) - kM15Bits;
  v = 0ull;
}

__device__ __forceinline__ void close_one(float& v, float sc, uint32_t& h0, uint32_t& l0) {
  const float hm = __fmaf_rd(v, sc, kM15);
  const float lm = fmaf(fmaf(v, sc, kM15 - hm), 65536.f, kM15);
  h0 += __float_as_uint(hm) - kM15Bits;
  l0 += __float_as_uint(lm) - kM15Bits;
  v = 0.f;
}

// (hi word, low word) -> FP64 value times 2^-e: one FP64 add, the scaling on the exponent
__device__ __forceinline__ double from_fixed(uint32_t h, uint32_t l, int e) {
  const long long v = (static_cast<long long>(static_cast<int32_t>(h)) << 16) + static_cast<long long>(l);
  if (v == 0) return 0.0;
  const double d = __longlong_as_double(v + __double_as_longlong(kM52)) - kM52;
  return __longlong_as_double(__double_as_longlong(d) - (static_cast<long long>(e + 16) << 52));
}

// Bin rows [t0, t0 + K) of forest pair (a, b) into the sums; WINDOW where the
// band goes on beyond them (its top row is t_hi).
template <bool Z, bool WINDOW>
__device__ void pair_means(const MeansArgs& A, const Acc& acc, unsigned char* smem, float* red, int a, int b, int na,
                           int nb, float cP, float sP, int t0, int K, int t_hi, int tile, int bins) {
  constexpr int kWords = Z ? 11 : 9;      // words per bin (odd: neighbouring bins lie in different banks)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t* hist = reinterpret_cast<uint32_t*>(smem);
  float4* bp = reinterpret_cast<float4*>(smem + ((static_cast<size_t>(bins) * kWords * 4 + 15) & ~size_t{15})) + kPad;
  float4* ap = bp + tile + kPad;
  const int npar = A.n_par;
  const float fnpar = static_cast<float>(npar), fnperp = static_cast<float>(A.n_perp);
  const int64_t oa = A.F.off[a], ob = A.F.off[b];
  const Pix* __restrict__ pa = A.pix + oa;
  const Pix* __restrict__ pb = A.pix + ob;
  const float dd = A.F.dref[a] - A.F.dref[b];   // exact: multiples of 2^-10 below 8192
  const float ss = A.F.dref[a] + A.F.dref[b];
  const uint32_t stride = static_cast<uint32_t>(npar + 1);
  const uint32_t C = kMagicBits * (stride + 1u) + static_cast<uint32_t>(t0) * stride;
  const uint32_t base = smem_addr(hist) - 4u * kWords * C;
  const uint32_t guard = C + static_cast<uint32_t>(npar);
  const float pmax = kMagic + fnpar, tmax = kMagic + static_cast<float>(t_hi + 1);
  const uint32_t twin = static_cast<uint32_t>(t0), tspan = static_cast<uint32_t>(K - 1);
  for (int ia = 0; ia < na; ia += tile) {
    const int ta = min(tile, na - ia);
    for (int jb = 0; jb < nb; jb += tile) {
      const int tb = min(tile, nb - jb);
      // rows up to a multiple of 8 and the padding of b lie at infinite distance, with zero weight;
      // of the tile: sums of w^2, smallest weights that are not 0, smallest and largest |z|
      float zm = 0.f, zl = INFINITY, qa = 0.f, qb = 0.f, la = INFINITY, lb = INFINITY;
      for (int q = threadIdx.x; q < ((ta + 7) & ~7); q += kTeam) {
        const Pix p = (q < ta) ? pa[ia + q] : make_float4(INFINITY, 0.f, 0.f, 0.f);
        const float z = (Z && q < ta) ? static_cast<float>(A.zpix[oa + ia + q]) : 0.f;
        ap[q] = make_float4(p.x, z, p.y, 0.f);
        qa = fmaf(p.y, p.y, qa);
        if (p.y != 0.f) la = fminf(la, p.y);
        if (Z) zm = (fabsf(z) < 1e36f) ? fmaxf(zm, fabsf(z)) : INFINITY;   // (a NaN counts as infinite)
        if (Z && z != 0.f) zl = fminf(zl, fabsf(z));
      }
      for (int q = static_cast<int>(threadIdx.x) - kPad; q < tb + kPad; q += kTeam) {
        const bool in = q >= 0 && q < tb;
        const Pix p = in ? pb[jb + q] : make_float4(INFINITY, 0.f, 0.f, 0.f);
        const float z = (Z && in) ? static_cast<float>(A.zpix[ob + jb + q]) : 0.f;
        bp[q] = make_float4(ss + p.x, z, dd - p.x, p.y);   // d_i + d_j = x_i + .x, d_i - d_j = x_i + .z
        qb = fmaf(p.y, p.y, qb);
        if (p.y != 0.f) lb = fminf(lb, p.y);
        if (Z) zm = (fabsf(z) < 1e36f) ? fmaxf(zm, fabsf(z)) : INFINITY;
        if (Z && z != 0.f) zl = fminf(zl, fabsf(z));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        qa += __shfl_xor_sync(0xffffffffu, qa, o);
        qb += __shfl_xor_sync(0xffffffffu, qb, o);
      }
      // (none of them is negative: their bits order like the values)
      la = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(la)));
      lb = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(lb)));
      if (Z) {
        zm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(zm)));
        zl = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(zl)));
      }
      if (lane == 0) {
        float* r = red + 6 * wid;
        r[0] = qa, r[1] = qb, r[2] = la, r[3] = lb, r[4] = zm, r[5] = zl;
      }
      __syncthreads();
      // Fixed-point scales: a run meets every pixel of the tile's rows and columns at most once, so its sum of
      // w_i w_j is at most the geometric mean of the sums of w^2 (Cauchy-Schwarz).  The integers hold 2^-37 of that
      // bound; where it is more than 2^16 of the smallest product (survey weights: 2^13 to 2^15), so that they
      // would round a block by more than 2^-21 of its smallest pair, or the sums leave the fixed point's range,
      // the blocks go to the FP64 sums at once (direct).
      const float bw = 1.001f * sqrtf(red[0] + red[6]) * sqrtf(red[1] + red[7]);
      const float bx = bw * fnpar, by = bw * static_cast<float>(t0 + K), bs = bw * (ss + pa[na - 1].x + pb[nb - 1].x);
      const float scW = fixed_scale(bw), scX = fixed_scale(bx), scY = fixed_scale(by), scS = fixed_scale(bs);
      const float wa = fminf(red[2], red[8]), wb = fminf(red[3], red[9]);   // infinite where all weights are 0
      bool direct = wa < INFINITY && wb < INFINITY &&
                    !(bx < 1e36f && by < 1e36f && bs < 1e36f && bw > 1e-30f && bw <= 65536.f * (wa * wb));
      float scZ = 1.f;
      if (Z) {
        const float zmax = fmaxf(red[4], red[10]), bz = 2.f * bw * zmax;
        direct = direct || !(zmax == 0.f || (zmax <= 16.f * fminf(red[5], red[11]) && bz < 1e36f && (bz == 0.f || bz > 1e-30f)));
        scZ = fixed_scale(bz);
      }
      F2 scWX = f2(scW, scX), scSZ = f2(scS, scZ);
      // (kept from being recomputed inside the walk: 185.6 -> 182.5 ms)
      asm volatile("" : "+l"(scWX), "+l"(scSZ));
      // the end of a block; with `direct` its sums go to the FP64 sums at once,
      // infinities and NaN included
      auto close_block = [&](Run& r) {
        if (direct) {
          const int q = static_cast<int>(r.cur - C), tt = q / (npar + 1), p = q - tt * (npar + 1);
          if (tt < K && p < npar) {
            const int64_t bin = static_cast<int64_t>(p) * A.n_perp + t0 + tt;
            const float2 wx = unf2(r.wx), sz = unf2(r.sz);
            red_add_f64_global(acc.W + bin, wx.x);
            red_add_f64_global(acc.WX + bin, wx.y);
            red_add_f64_global(acc.WY + bin, r.y);
            red_add_f64_global(acc.WD + bin, 0.5 * sz.x);
            if (Z) red_add_f64_global(acc.WZ + bin, 0.5 * sz.y);
          }
          r.wx = r.sz = 0ull;
          r.y = 0.f;
        } else {
          close_pair(r.wx, scWX, r.h[0], r.l[0], r.h[1], r.l[1]);
          close_one(r.y, scY, r.h[2], r.l[2]);
          close_pair(r.sz, scSZ, r.h[3], r.l[3], r.h[4], r.l[4]);
        }
      };
      // the held runs of the lanes that have one -> their bins
      bool on = false;
      auto add_held = [&](Run& r) {
        if (on) {
          close_block(r);
          const uint32_t addr = base + r.cur * (4u * kWords);
          asm volatile(
              "{\n\t"
              "red.shared.add.u32 [%0], %1;\n\tred.shared.add.u32 [%0+4], %2;\n\t"
              "red.shared.add.u32 [%0+8], %3;\n\tred.shared.add.u32 [%0+12], %4;\n\t"
              "red.shared.add.u32 [%0+16], %5;\n\tred.shared.add.u32 [%0+20], %6;\n\t"
              "red.shared.add.u32 [%0+24], %7;\n\tred.shared.add.u32 [%0+28], %8;\n\t"
              "red.shared.add.u32 [%0+32], %9;\n\t}" ::"r"(addr),
              "r"(r.h[0]), "r"(r.l[0]), "r"(r.h[1]), "r"(r.l[1]), "r"(r.h[2]), "r"(r.l[2]), "r"(r.h[3]), "r"(r.l[3]),
              "r"(static_cast<uint32_t>(r.n)));
          if (Z)
            asm volatile("{\n\tred.shared.add.u32 [%0+36], %1;\n\tred.shared.add.u32 [%0+40], %2;\n\t}" ::"r"(addr),
                         "r"(r.h[4]), "r"(r.l[4]));
        }
        on = false;
        __syncwarp();
      };
      // groups of 32 diagonals j - i = o + lane, in turn to the two warps
      const int ngroup = (ta + tb + 30) >> 5;
      for (int g = wid; g < ngroup; g += kTeam / 32) {
        const int o = 32 * g - (ta - 1);
        // lane m: whether block m of 8 rows can hold an in-grid pixel pair (both coordinates are monotone in
        // the sorted distances; 1e-2 bins cover the rounding)
        bool work = false;
        {
          const int i0 = 8 * lane, i1 = min(i0 + 7, ta - 1);
          const int jl = max(i0 + o, 0), jh = min(i1 + o + 31, tb - 1);
          if (i0 < ta && jl <= jh)
            work = (ap[i0].x + bp[jh].z) * cP < fnpar + 1e-2f && (ap[i1].x + bp[jl].z) * cP > -fnpar - 1e-2f &&
                   (ap[i0].x + bp[jl].x) * sP < fnperp + 1e-2f;
        }
        unsigned todo = __ballot_sync(0xffffffffu, work);
        if (!todo) continue;
        const Run none{0ull, 0ull, 0.f, {0u, 0u, 0u, 0u, 0u}, {0u, 0u, 0u, 0u, 0u}, guard, 0, false};
        Run r = none, held = none;
        // the current run of every lane ends before row i
        auto end_runs = [&](int i) {
          if (__any_sync(0xffffffffu, on)) add_held(held);
          held = r;
          held.n += i;
          on = r.in;
          add_held(held);
        };
        int i = -1;
        for (; todo; todo &= todo - 1u) {
          const int ib = 8 * (__ffs(todo) - 1);
          if (i >= 0 && ib != i) {   // blocks without work between: every run ends (its length counts its pairs)
            end_runs(i);
            r = none;
          }
          i = ib;
          const float4* pj = bp + i + o + lane;
#pragma unroll
          for (int q = 0; q < 8; ++q, ++i) {
            const float4 vi = ap[i], vj = pj[q];
            const float xv = fabsf(vi.x + vj.z) * cP;
            const float yv = (vi.x + vj.x) * sP;
            const uint32_t pb_ = __float_as_uint(fminf(__fadd_rd(xv, kMagic), pmax));
            const uint32_t tb_ = __float_as_uint(fminf(__fadd_rd(yv, kMagic), tmax));
            uint32_t key = tb_ * stride + pb_;
            if (WINDOW) key = (tb_ - kMagicBits - twin <= tspan) ? key : guard;
            const bool chg = key != r.cur;
            if (__any_sync(0xffffffffu, chg)) {
              if (__any_sync(0xffffffffu, chg && on && r.in)) add_held(held);
              if (chg) {
                if (r.in) {
                  held = r;
                  held.n += i;
                  on = true;
                }
                r = none;
                r.cur = key;
                r.n = -i;
                r.in = xv < fnpar && yv < fnperp && key != guard;
              }
              __syncwarp();
            }
            const float ww = vi.z * vj.w;
            const F2 w2 = f2(ww, ww);
            r.wx = fma2(w2, f2(1.f, xv), r.wx);
            r.y = fmaf(ww, yv, r.y);
            // (not of the rounded sums x_i + (ref + x_j), z_i + z_j: on a common pixel grid their roundings repeat)
            r.sz = fma2(w2, f2(vi.x, vi.y), fma2(w2, f2(vj.x, vj.y), r.sz));
          }
          close_block(r);
        }
        end_runs(i);
      }
      // integer sums -> FP64 sums
      __syncthreads();
      const int eW = scale_exponent(scW), eX = scale_exponent(scX), eY = scale_exponent(scY);
      const int eS = scale_exponent(scS), eZ = scale_exponent(scZ);
      for (int q = threadIdx.x; q < (K + 1) * (npar + 1); q += kTeam) {
        uint32_t v[kWords], any = 0u;
#pragma unroll
        for (int m = 0; m < kWords; ++m) {
          v[m] = hist[q * kWords + m];
          any |= v[m];
        }
        if (any != 0u) {
          const int tt = q / (npar + 1), p = q - tt * (npar + 1);
          if (tt < K && p < npar) {
            const int64_t bin = static_cast<int64_t>(p) * A.n_perp + t0 + tt;
            if (!direct) {
              red_add_f64_global(acc.W + bin, from_fixed(v[0], v[1], eW));
              red_add_f64_global(acc.WX + bin, from_fixed(v[2], v[3], eX));
              red_add_f64_global(acc.WY + bin, from_fixed(v[4], v[5], eY));
              red_add_f64_global(acc.WD + bin, 0.5 * from_fixed(v[6], v[7], eS));
              if (Z) red_add_f64_global(acc.WZ + bin, 0.5 * from_fixed(v[kWords - 2], v[kWords - 1], eZ));
            }
            if (v[8]) atomicAdd(acc.C + bin, static_cast<unsigned long long>(v[8]));
          }
#pragma unroll
          for (int m = 0; m < kWords; ++m) hist[q * kWords + m] = 0u;
        }
      }
      __syncthreads();
    }
  }
}

// Persistent, one forest pair per team (a block of two warps) at a time, the
// pairs in the list's order.  A tile of up to 240 x 240 pixel pairs is staged
// in shared memory and walked along its diagonals: lane l takes the pairs
// (i, i + o + l), whose separations change slowly with i, so a run of pixel
// pairs in one bin is tens of pairs long (36 on the SDSS-like grid, 66 on the
// DESI-like one, where a run along a row is 2 and 7).  A run's sums of w_i w_j,
// w_i w_j r_par/D_par, w_i w_j r_perp/D_perp, w_i w_j (d_i + d_j) and, with Z,
// w_i w_j (z_i + z_j) are FP32 over at most 8 pairs and two-word fixed point
// beyond; an ended run is held in registers until its lane ends another, and
// then added to the team's band histogram with native 32-bit reductions (runs
// off the grid are dropped: all lanes' would go to one word).  The histogram is
// added to the FP64 sums per tile.
// What bounds it: issue (65%) of about 60 warp instructions per step, a third
// of them at the ends of runs, which some lane has in every second step.
// Eight teams per SM (26 KB each); more teams with smaller tables cost windows.
// Measured (SDSS-like, 15,000 forests, 5.7e10 pixel pairs, with redshifts):
// lanes along the rows with a warp scan and compare-and-swap sums per run
// 777 ms; along the diagonals 261 ms with every run compensated and added at
// once, 237 ms with fixed-point runs, 202 ms held, 160 ms without the runs off
// the grid, 182 ms with the sum of r_perp of its own (from the sum of d_i + d_j
// its rounding differs by 6e-10 on a common pixel grid).
template <bool Z>
__global__ void __launch_bounds__(kTeam, 8) means_kernel(MeansArgs A, Acc acc, int tile, int bins, int kmax, int grab,
                                                      unsigned long long* counter) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long s_it;
  __shared__ float s_red[12];
  constexpr int kWords = Z ? 11 : 9;
  for (int q = threadIdx.x; q < bins * kWords; q += kTeam) reinterpret_cast<uint32_t*>(smem)[q] = 0u;
  const float fnperp = static_cast<float>(A.n_perp);
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_it = atomicAdd(counter, static_cast<unsigned long long>(grab));
    __syncthreads();
    const unsigned long long it0 = s_it;
    if (it0 >= static_cast<unsigned long long>(A.n_pairs)) break;
    const int64_t it1 = min(static_cast<int64_t>(it0) + grab, A.n_pairs);
    for (int64_t it = static_cast<int64_t>(it0); it < it1; ++it) {
      const int2 ab = A.pairs[it];
      if (ab.x < 0 || ab.y < 0) continue;
      const int a = ab.x, b = ab.y;
      const int na = A.F.len[a], nb = A.F.len[b];
      if (na <= 0 || nb <= 0) continue;
      const float2 cs = A.cs[it];
      const Pix* pa = A.pix + A.F.off[a];
      const Pix* pb = A.pix + A.F.off[b];
      const float ss = A.F.dref[a] + A.F.dref[b];
      // r_perp band from the extreme pixels (monotone in both distances, the same arithmetic as the walk)
      const float y0 = (pa[0].x + (ss + pb[0].x)) * cs.y, y1 = (pa[na - 1].x + (ss + pb[nb - 1].x)) * cs.y;
      if (!(y0 < fnperp)) continue;
      const int t_lo = static_cast<int>(y0);
      const int t_hi = (y1 < fnperp) ? static_cast<int>(y1) : A.n_perp - 1;
      if (t_hi - t_lo < kmax) {
        pair_means<Z, false>(A, acc, smem, s_red, a, b, na, nb, cs.x, cs.y, t_lo, t_hi - t_lo + 1, t_hi, tile, bins);
      } else {
        for (int tw = t_lo; tw <= t_hi; tw += kmax)
          pair_means<Z, true>(A, acc, smem, s_red, a, b, na, nb, cs.x, cs.y, tw, min(kmax, t_hi - tw + 1), t_hi, tile,
                              bins);
      }
    }
  }
}

__global__ void means_finalize_kernel(Acc acc, int nb, double d_par, double d_perp, double* wsum, double* rp,
                                      double* rt, double* dm, double* zm, int64_t* count) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nb; k += gridDim.x * blockDim.x) {
    const double w = acc.W[k];
    const bool on = w != 0.0;
    if (wsum) wsum[k] = w;
    rp[k] = on ? d_par * acc.WX[k] / w : 0.0;
    rt[k] = on ? d_perp * acc.WY[k] / w : 0.0;
    dm[k] = on ? acc.WD[k] / w : 0.0;
    if (zm) zm[k] = on ? acc.WZ[k] / w : 0.0;
    count[k] = static_cast<int64_t>(acc.C[k]);
  }
}

int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 1 << 16) b = 1 << 16;
  return static_cast<int>(b);
}

}  // namespace

size_t means_scratch_bytes(int nb) { return 6 * static_cast<size_t>(nb) * 8 + 8; }

// The grids and forest lengths the entry point takes (36 or 44 bytes per bin
// and 16 or 24 per pixel of the longest forest within the size of a block's shared
// memory; the kernel itself needs less).
int means_limit_bytes(int nb, int max_len, bool with_z) {
  const int base = 32 * nb + 4 * ((nb + 1) & ~1);
  return with_z ? base + 8 * nb + 2 * 12 * std::max(max_len, 1) : base + 2 * 8 * std::max(max_len, 1);
}

cudaError_t launch_bin_means(const MeansArgs& a, const DevInfo& dev, void* scratch, double* wsum, double* rpar_mean,
                             double* rperp_mean, double* dist_mean, double* z_mean, int64_t* count, cudaStream_t s) {
  const int nb = a.n_par * a.n_perp;
  const bool with_z = a.zpix != nullptr && z_mean != nullptr;
  Acc acc;
  acc.W = static_cast<double*>(scratch);
  acc.WX = acc.W + nb;
  acc.WY = acc.WX + nb;
  acc.WD = acc.WY + nb;
  acc.WZ = acc.WD + nb;
  acc.C = reinterpret_cast<unsigned long long*>(acc.WZ + nb);
  unsigned long long* counter = acc.C + nb;
  cudaError_t e = cudaMemsetAsync(acc.W, 0, means_scratch_bytes(nb), s);
  if (e != cudaSuccess) return e;
  if (a.n_pairs > 0 && a.F.n > 0) {
    const int tile = std::min((std::max(a.max_len, 1) + 7) & ~7, kTile);
    // at least one band row and the guard row
    const int bins = std::max(kBins, 2 * (a.n_par + 1));
    const int kmax = std::min(a.n_perp, bins / (a.n_par + 1) - 1);
    const int smem = ((bins * (with_z ? 11 : 9) * 4 + 15) & ~15) + (2 * tile + 2 * kPad) * 16;
    const void* fn = with_z ? reinterpret_cast<const void*>(means_kernel<true>)
                            : reinterpret_cast<const void*>(means_kernel<false>);
    e = set_max_dynamic_smem(fn, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kTeam, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int teams = per_sm * dev.sms;
    const int grab = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(8, a.n_pairs / (16 * std::max(teams, 1)))));
    if (with_z) LYA_COUNT(1), means_kernel<true><<<teams, kTeam, smem, s>>>(a, acc, tile, bins, kmax, grab, counter);
    else LYA_COUNT(1), means_kernel<false><<<teams, kTeam, smem, s>>>(a, acc, tile, bins, kmax, grab, counter);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  LYA_COUNT(1), means_finalize_kernel<<<grid_for(nb, 256), 256, 0, s>>>(acc, nb, a.d_par, a.d_perp, wsum, rpar_mean,
                                                                          rperp_mean, dist_mean,
                                                                          with_z ? z_mean : nullptr, count);
  return cudaGetLastError();
}

}  // namespace lya
