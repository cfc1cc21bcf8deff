// Distortion matrix of Eq. (2.6) over the seeded forest-pair subsample
// (Section 2.2), without the O(N^4) contraction.
//
// With eta = I - 1 u^T - x v^T per forest (u = w/W, v = w x/S, Eq. 2.7), one
// forest pair (a, b) adds to D~_AB = sum_{(i,j) in A} w_i w_j sum_{(k,l) in B} eta_ik eta_jl:
//
//   diag(T1)
//   - sum_j w_j (alpha_j alpha_j^T / W_a + beta_j beta_j^T / S_a)         (columns j of b)
//   - sum_i w_i (alpha'_i alpha'_i^T / W_b + beta'_i beta'_i^T / S_b)     (rows i of a)
//   + T1 T1^T/(W_a W_b) + Ty Ty^T/(W_a S_b) + Tx Tx^T/(S_a W_b) + Txy Txy^T/(S_a S_b)
//
// alpha_j[A] = sum_{i:(i,j) in A} w_i, beta_j[A] = sum w_i x_i, alpha'_i, beta'_i
// likewise over j with y = Lambda - Lbar of forest b, T1 = sum_A w_i w_j,
// Tx = sum w_i w_j x_i, Ty = sum w_i w_j y_j, Txy = sum w_i w_j x_i y_j.
//
// Work layout.  All bins a pair touches lie in its r_perp band of K rows
// (r_perp is monotone in both distances), i.e. L = K n_par local bins.  The
// kept pairs are grouped by (first band row, K); a block takes a chunk of
// pairs of one group and keeps the upper triangle of the L x L block of D~
// in shared memory (FP32): each pair's contribution is built there and added
// to the FP64 accumulator G (entries A <= B) with FP64 atomics at the end of
// the pair, so that the sum over pairs is FP64.  The rank-1 terms are applied a
// batch of up to CB vectors (consecutive columns, then rows) at a time:
//  (a1) every thread bins pixel pairs of the batch's vectors and the other
//       forest's pixels within their reach (dm_windows) and marks the local
//       bins; (b) the marks are compacted into the batch's ascending union
//       support S (|S| is a little above one vector's support, because
//       neighbouring columns visit nearly the same bins: 62 on average on
//       SDSS-like forests, 35 on DESI-like ones);
//  (a2) the batch's histograms are summed densely on S with shared atomics;
//       column histograms also feed the T vectors;
//  (d)  each thread owns a 2 x 4 tile of the S x S upper triangle and adds
//       sum_v (a_v a_v^T + b_v b_v^T) over the batch in registers (FP32 FMA,
//       float4 loads), then updates its 8 triangle entries -- no atomics.
// What bounds it: 8.4 batches a pair, each with four block-wide phases of 1,000
// to 4,600 cycles; (d) takes 40% (4 x 4 tiles left three quarters of the
// threads idle at |S| = 62, and 2 x 8 ones half), (a2) 17%, half of it the
// shared atomics, the flush to G 12%.  D on 12,000 SDSS-like forests, 5% of the
// pairs: windows, one division per lane, floors without conversions and four
// phases instead of six a batch 101.9 -> 72 ms, tiles of 2 x 4 (2 x 8: 58.9) and
// V cleared only where used -> 57.7 ms (384, 640, 768, 1024 threads: 61, 60,
// 62, 63).
// Pairs whose band is too wide for shared memory take the same code with the
// triangle replaced by FP64 atomics into G.  Binning uses exactly the FP32
// arithmetic of the xi kernel, so W^DM equals the xi weights of the kept
// pairs up to summation order.
#include <algorithm>
#include <math.h>

#include "fixed.cuh"

namespace lya {
namespace {

constexpr int kDmThreads = 512;
constexpr int kChunk = 32;   // pairs per work unit (each pair is flushed on its own; small units balance the SMs)


// band of a pair: same FP32 arithmetic as the xi kernel
__device__ __forceinline__ bool pair_band(const DmArgs& A, int a, int b, float sp, int* t_lo, int* K) {
  const int na = A.F.len[a], nb = A.F.len[b];
  if (na == 0 || nb == 0) return false;
  const Pix* pa = A.pix + A.F.off[a];
  const Pix* pb = A.pix + A.F.off[b];
  const float Ds = (A.F.dref[a] + A.F.dref[b]) * sp;
  const float fnperp = static_cast<float>(A.n_perp);
  const float rt_min = fmaf(pb[0].x, sp, fmaf(pa[0].x, sp, Ds));
  const float rt_max = fmaf(pb[nb - 1].x, sp, fmaf(pa[na - 1].x, sp, Ds));
  if (!(rt_min < fnperp)) return false;
  const int lo = static_cast<int>(rt_min);
  const int hi = (rt_max < fnperp) ? static_cast<int>(rt_max) : A.n_perp - 1;
  *t_lo = lo;
  *K = hi - lo + 1;
  return true;
}

__global__ void dm_select_kernel(DmArgs A, uint64_t thr, int all, int kfit, int32_t* key,
                                 int32_t* count, int32_t* wide, int32_t* n_wide) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < A.n_pairs;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int2 p = A.pairs[k];
    int32_t kk = -1;
    // the subsample rule sees forest indices local to the pair's catalogue,
    // so a mock's D does not depend on the other mocks of the batch
    const int m = (p.x >= 0) ? A.F.mock[p.x] : 0;
    const int base = (p.x >= 0) ? A.fbase[m] : 0;
    const bool keep = p.x >= 0 && keep_pair(p.x - base, p.y - base, A.seed, thr, all);
    int t_lo, K;
    if (keep && pair_band(A, p.x, p.y, A.cs[k].y, &t_lo, &K)) {
      if (K <= kfit) {
        kk = (m * A.n_perp + t_lo) * kfit + (K - 1);
        atomicAdd(&count[kk], 1);
      } else {
        const int w = atomicAdd(n_wide, 1);
        wide[w] = static_cast<int32_t>(k);
      }
    }
    key[k] = kk;
  }
}

__global__ void dm_scatter_kernel(int64_t n, const int32_t* key, const int64_t* start, int32_t* cursor,
                                  int32_t* order) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t kk = key[k];
    if (kk < 0) continue;
    const int pos = atomicAdd(&cursor[kk], 1);
    order[start[kk] + pos] = static_cast<int32_t>(k);
  }
}

__global__ void chunk_count_kernel(const int32_t* count, int ngroups, int32_t* nchunks) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ngroups; g += gridDim.x * blockDim.x)
    nchunks[g] = (count[g] + kChunk - 1) / kChunk;
}

struct Chunk {
  int32_t begin;   // into order[]
  int32_t n;
  int32_t t0;
  int32_t K;
  int32_t mock;    // catalogue whose accumulator the chunk adds to
};

__global__ void chunk_fill_kernel(const int32_t* count, const int64_t* start, const int64_t* coff,
                                  int ngroups, int kfit, int n_perp, Chunk* chunks) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ngroups; g += gridDim.x * blockDim.x) {
    const int c = count[g];
    for (int q = 0; q * kChunk < c; ++q) {
      Chunk ch;
      ch.begin = static_cast<int32_t>(start[g] + q * kChunk);
      ch.n = min(kChunk, c - q * kChunk);
      ch.t0 = (g / kfit) % n_perp;
      ch.K = g % kfit + 1;
      ch.mock = g / (kfit * n_perp);
      chunks[coff[g] + q] = ch;
    }
  }
}

// vectors per batch: 32 where the band fits in shared memory with them (half
// the block-wide phases per pair), else 16
constexpr int kCB = 16;
constexpr int kCB2 = 32;

// Shared-memory layout of one block (offsets in bytes)
struct Lay {
  int U, T4, V, mark, inv, S, ucs, db, tv, cf, win, misc, end;
};

constexpr int kWin = 16;   // vectors per search window

__host__ __device__ inline int scap_for(int L, int npar, int K, int cb) {
  // union-support capacity: at least one vector's support bound 2 (n_par + K) + 2,
  // with room for the batch's neighbouring vectors
  int c = 2 * (npar + K) + 2;
  c = (cb > kCB) ? 2 * c : c + c / 2;
  if (c > L) c = L;
  return (c + 3) & ~3;
}

// Row stride, in (a, b) entries, of the batch vectors V[cb][.]: at least the
// support capacity rounded up to 16 (the tensor-core tiles read 16-row blocks),
// and 2 modulo 16, i.e. 4 words modulo 32: the histograms of neighbouring
// vectors, one per lane, fall on different banks (8 words modulo 32 instead of
// 4: D on 12,000 SDSS-like forests 106.1 -> 101.9 ms).
__host__ __device__ inline int ldv_for(int scap) { return ((scap + 15) & ~15) + 2; }

__host__ __device__ inline Lay layout(int L, int scap, int max_len, bool global_sink, int cb) {
  auto al = [](int v) { return (v + 15) & ~15; };
  Lay y;
  int o = 0;
  y.U = o;
  if (!global_sink) o += al(static_cast<int>((static_cast<int64_t>(L) * (L + 1) / 2) * 4));
  y.T4 = o; o += al(L * 16);
  y.V = o; o += al(cb * ldv_for(scap) * 8);
  y.mark = o; o += al(L);
  y.inv = o; o += al(L * 2);
  y.S = o; o += al(scap * 4);
  y.ucs = o; o += al(max_len * 8);
  y.db = o; o += al(max_len * 4);
  y.tv = o; o += 2 * al(max_len * 8);
  y.cf = o; o += 2 * al(max_len * 16);
  y.win = o; o += 2 * al((max_len / kWin + 1) * 8);
  y.misc = o; o += 192;
  y.end = o;
  return y;
}

// Bytes by which a band is judged to fit: the triangle, the batch with rows of
// 8 words modulo 32, 23 bytes per local bin and 64 per pixel.  The
// block needs a little less (see layout); whether a pair's vectors are summed
// 32 or 16 at a time, and so the rounding of its FP32 sums, does not follow
// every change of the layout.
__host__ inline int64_t band_bytes(int L, int scap, int max_len, int cb) {
  auto al = [](int64_t v) { return (v + 15) & ~int64_t(15); };
  const int64_t row = ((((scap + 15) & ~15) + 23) & ~31) + 8;
  return al(static_cast<int64_t>(L) * (L + 1) / 2 * 4) + al(L * 16) + 2 * al(cb * row * 4) + al(L) + al(L * 2) +
         al(scap * 4) + 2 * al(max_len * 8) + 3 * al(max_len * 16) + al(L * 4) + 128;
}

__device__ __forceinline__ int tri_rowbase(int r, int L) {
  // index of (r, c), c >= r, in the packed upper triangle is rowbase(r) + c
  return r * (2 * L - r + 1) / 2 - r;
}

// Power of two sc = 2^(29 - e), 2^e <= B < 2^(e+1): sums bounded by B map below 2^30.
__device__ __forceinline__ float word_scale(float B) {
  if (!(B > 0.f) || !(B < 1e37f)) return 1.f;
  const int e = static_cast<int>((__float_as_uint(B) >> 23) & 0xFFu) - 127;
  return __uint_as_float(static_cast<uint32_t>(min(max(29 - e + 127, 1), 254)) << 23);
}

// Bin of pixel pair (i of a, j of b); returns the local bin or -1 if off-grid.
// The floors are FP32 adds of 2^23 rounded toward -inf, as in the xi kernel.
__device__ __forceinline__ int local_bin(float2 u, float dj, float cp, float sp, float fnpar, float fnperp,
                                         int npar, int t0) {
  const float rp = fabsf(fmaf(-dj, cp, u.x));
  const float rt = fmaf(dj, sp, u.y);
  if (rp < fnpar && rt < fnperp) return (static_cast<int>(rt) - t0) * npar + static_cast<int>(rp);
  return -1;
}

// The same for a pixel pair given by (rp, rt) = (fmaf(-dj, cp, u.x), fmaf(dj, sp, u.y)),
// with the floors as FP32 adds of 2^23 rounded toward -inf (a conversion to
// integer runs at a quarter of the rate); corner = bits of both additions and
// the band's first row, see bin_corner.
__device__ __forceinline__ uint32_t bin_corner(int npar, int t0) {
  return 0u - (0x4B000000u + static_cast<uint32_t>(t0)) * static_cast<uint32_t>(npar) - 0x4B000000u;
}
__device__ __forceinline__ bool bin_at(float rp, float rt, float fnpar, float fnperp, uint32_t npar, uint32_t corner,
                                       int* l) {
  rp = fabsf(rp);
  *l = static_cast<int>(__float_as_uint(__fadd_rd(rt, 8388608.0f)) * npar +
                        __float_as_uint(__fadd_rd(rp, 8388608.0f)) + corner);
  return rp < fnpar && rt < fnperp;
}

constexpr int kTileW = 4;   // columns of a tile

// Tile q of 2 rows x kTileW columns of the union support's upper triangle: acc = sum
// over the batch's vectors of a a^T + b b^T.  Tiles of one column block are
// consecutive, so the lanes of a warp read consecutive 16-byte row pairs (4
// shared-memory passes) and the same columns (two broadcasts).
__device__ __forceinline__ void dm_tile(const F2* V, int ldv, int q, int nv, float (&acc)[2][kTileW], int* row, int* col) {
  constexpr int W = kTileW;
  // column block cb has W / 2 (cb + 1) row pairs
  int cb = static_cast<int>((sqrtf(16.f / W * q + 1.f) - 1.f) * 0.5f);
  while (W / 4 * cb * (cb + 1) > q) --cb;
  while (W / 4 * (cb + 1) * (cb + 2) <= q) ++cb;
  *col = W * cb;
  *row = 2 * (q - W / 4 * cb * (cb + 1));
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < W; ++v) acc[u][v] = 0.f;
  const float2 *r = reinterpret_cast<const float2*>(V) + *row, *c = reinterpret_cast<const float2*>(V) + *col;
  auto add = [&](const float4& rr, const float4 (&cc)[W / 2]) {
#pragma unroll
    for (int v = 0; v < W; v += 2) {
      const float4 k = cc[v / 2];
      acc[0][v] = fmaf(rr.y, k.y, fmaf(rr.x, k.x, acc[0][v]));
      acc[1][v] = fmaf(rr.w, k.y, fmaf(rr.z, k.x, acc[1][v]));
      acc[0][v + 1] = fmaf(rr.y, k.w, fmaf(rr.x, k.z, acc[0][v + 1]));
      acc[1][v + 1] = fmaf(rr.w, k.w, fmaf(rr.z, k.z, acc[1][v + 1]));
    }
  };
  constexpr int N = 16 / W;   // vectors in flight
  int vv = 0;
  for (; vv + N <= nv; vv += N, r += N * ldv, c += N * ldv) {
    float4 rr[N], cc[N][W / 2];
#pragma unroll
    for (int e = 0; e < N; ++e) {
      rr[e] = *reinterpret_cast<const float4*>(r + e * ldv);
#pragma unroll
      for (int v = 0; v < W / 2; ++v) cc[e][v] = *reinterpret_cast<const float4*>(c + e * ldv + 2 * v);
    }
#pragma unroll
    for (int e = 0; e < N; ++e) add(rr[e], cc[e]);
  }
  for (; vv < nv; ++vv, r += ldv, c += ldv) {
    float4 cc[W / 2];
#pragma unroll
    for (int v = 0; v < W / 2; ++v) cc[v] = *reinterpret_cast<const float4*>(c + 2 * v);
    add(*reinterpret_cast<const float4*>(r), cc);
  }
}

// Tensor-core form of the rank-1 tiles: C = V^T V over the union support,
// V the batch's [32 x S] matrix (rows: the a vectors, then the b vectors),
// with mma.sync m16n8k8 in TF32 and the 3xTF32 split (x = hi + lo, hi and lo
// TF32; C += lo.hi + hi.lo + hi.hi), which keeps the products at about FP32
// accuracy.  Warp tiles of 16 x 8 entries of the upper triangle (c >= r); each
// lane subtracts its four accumulators from the triangle (entries r <= c only,
// each unordered pair of support entries once).
__device__ __forceinline__ uint32_t tf32_bits(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void mma_tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  hi = tf32_bits(x);
  lo = tf32_bits(x - __uint_as_float(hi));
}

__device__ void dm_tiles_tc(const float* V, int ldv, int ns, int cbn, const int32_t* S, float* U,
                            int L, int wid, int nwarps, int lane) {
  const int g = lane >> 2, t = lane & 3;
  const int R = (ns + 15) >> 4, C8 = (ns + 7) >> 3;
  const int ksteps = (cbn + 7) >> 3;   // vectors [0, cbn) in k steps of 8 (rows past cbn are zero)
  int q = 0;
  for (int rb = 0; rb < R; ++rb) {
    for (int cb = 2 * rb; cb < C8; ++cb, ++q) {
      if (q % nwarps != wid) continue;
      const int r0 = rb * 16, c0 = cb * 8;
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        for (int ks = 0; ks < ksteps; ++ks) {
          const float* v0 = V + (ks * 8 + t) * 2 * ldv + half;   // entry e of vector v: V[(v ldv + e) 2 + half]
          const float* v4 = v0 + 8 * ldv;
          uint32_t ah[4], al[4], bh[2], bl[2];
          split_tf32(v0[2 * (r0 + g)], ah[0], al[0]);
          split_tf32(v0[2 * (r0 + g + 8)], ah[1], al[1]);
          split_tf32(v4[2 * (r0 + g)], ah[2], al[2]);
          split_tf32(v4[2 * (r0 + g + 8)], ah[3], al[3]);
          split_tf32(v0[2 * (c0 + g)], bh[0], bl[0]);
          split_tf32(v4[2 * (c0 + g)], bh[1], bl[1]);
          mma_tf32(acc, al[0], al[1], al[2], al[3], bh[0], bh[1]);
          mma_tf32(acc, ah[0], ah[1], ah[2], ah[3], bl[0], bl[1]);
          mma_tf32(acc, ah[0], ah[1], ah[2], ah[3], bh[0], bh[1]);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = r0 + g + ((e & 2) ? 8 : 0);
        const int c = c0 + 2 * t + (e & 1);
        if (r <= c && c < ns) {
          U[tri_rowbase(S[r], L) + S[c]] -= acc[e];
        }
      }
    }
  }
}

// Subtract a tile from the triangle, or from G with FP64 atomics for wide
// pairs.  S is ascending, so positions r <= c of it are entries of the upper
// triangle.
template <bool GLOBAL>
__device__ __forceinline__ void dm_tile_store(double* G, float* U, const int32_t* S, int g0, int ns, int L, int nbins,
                                              int row, int col, const float (&acc)[2][kTileW]) {
  constexpr int W = kTileW;
  int lc[W];
#pragma unroll
  for (int v = 0; v < W; ++v) lc[v] = S[min(col + v, ns - 1)];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = row + u;
    const int lr = S[min(r, ns - 1)];
    if (!GLOBAL) {
      float* Ur = U + tri_rowbase(lr, L);
      float old[W];   // all loads before the stores
#pragma unroll
      for (int v = 0; v < W; ++v) old[v] = (col + v < ns && r <= col + v) ? Ur[lc[v]] : 0.f;
#pragma unroll
      for (int v = 0; v < W; ++v)
        if (col + v < ns && r <= col + v) Ur[lc[v]] = old[v] - acc[u][v];
    } else {
      double* Gr = G + static_cast<int64_t>(g0 + lr) * nbins + g0;
#pragma unroll
      for (int v = 0; v < W; ++v)
        if (col + v < ns && r <= col + v) red_add_f64_global(Gr + lc[v], -static_cast<double>(acc[u][v]));
    }
  }
}

template <bool GLOBAL>
__device__ __forceinline__ void dm_tiles(const F2* V, int ldv, int nv, double* G, float* U, const int32_t* S, int g0,
                                         int ns, int L, int nbins) {
  constexpr int W = kTileW;
  const int nc = (ns + W - 1) / W;
  for (int q = threadIdx.x; q < W / 4 * nc * (nc + 1); q += kDmThreads) {
    float acc[2][W];
    int row, col;
    dm_tile(V, ldv, q, nv, acc, &row, &col);
    dm_tile_store<GLOBAL>(G, U, S, g0, ns, L, nbins, row, col, acc);
  }
}

// shared-memory arrays of one block
struct Sm {
  float* U;        // triangle of the pair
  float4* T4;      // T1, Tx, Ty, Txy per local bin
  F2* V;           // the batch's vectors, (a, b) entries; fixed-point words while filling
  unsigned char* mark;
  int16_t* inv;
  int32_t* S;
  float2* ucs;     // per pixel of a: (d cp + Dc, d sp + Ds)
  float* db;       // distances of b
  int2* tv_;       // per side: fixed-point terms of the summed-over forest
  float4* cf_;     // per side: coefficients and T weights of the vectors
  int2* win_;      // per side and kWin vectors: range of the summed-over forest in the grid
  int tvn, cfn, winn;   // entries of one side
  int* ns;         // size of the union support
  float* par;      // 2 x 16 scalars of the pair (its own and the next one's)
  __device__ Sm(unsigned char* sm, const Lay& y, int max_len) {
    U = reinterpret_cast<float*>(sm + y.U);
    T4 = reinterpret_cast<float4*>(sm + y.T4);
    V = reinterpret_cast<F2*>(sm + y.V);
    mark = sm + y.mark;
    inv = reinterpret_cast<int16_t*>(sm + y.inv);
    S = reinterpret_cast<int32_t*>(sm + y.S);
    ucs = reinterpret_cast<float2*>(sm + y.ucs);
    db = reinterpret_cast<float*>(sm + y.db);
    tv_ = reinterpret_cast<int2*>(sm + y.tv);
    cf_ = reinterpret_cast<float4*>(sm + y.cf);
    win_ = reinterpret_cast<int2*>(sm + y.win);
    tvn = (y.cf - y.tv) / 16;
    cfn = (y.win - y.cf) / 32;
    winn = (y.misc - y.win) / 16;
    par = reinterpret_cast<float*>(sm + y.misc);
    ns = reinterpret_cast<int*>(sm + y.misc + 128);
  }
  __device__ __forceinline__ int2* tv(int side) const { return tv_ + side * tvn; }
  __device__ __forceinline__ float4* cf(int side) const { return cf_ + side * cfn; }
  __device__ __forceinline__ int2* win(int side) const { return win_ + side * winn; }
};

// scalars of a pair in Sm::par
enum { kScA0, kScB0, kScA1, kScB1, kC11, kCyy, kCxx, kCxy, kIWb, kISb, kIWa, kISa };

struct Pair {
  int na, nb;
  float cp, sp;
  bool ok;
};

// Stage a pair: pixels, fixed-point histogram terms, weights, and the pair's
// FP64 quotients, one per lane of the last warp (every thread computing all
// eight took a fifth of the kernel: FP64 runs at 1.7 lanes a cycle).
__device__ __forceinline__ Pair dm_load(const DmArgs& A, int item, const Sm& m, int par) {
  const int tid = threadIdx.x;
  const int2 pr = A.pairs[item];
  const float2 cs = A.cs[item];
  const int a = pr.x, b = pr.y;
  Pair P;
  P.na = A.F.len[a];
  P.nb = A.F.len[b];
  P.cp = cs.x;
  P.sp = cs.y;
  // staging buffers hold max_len pixels (the longest forest when the pair list
  // was built); a longer forest means the offsets changed in place without a
  // rebuild, and the pair is skipped rather than overrun shared memory
  P.ok = !(P.na > A.max_len || P.nb > A.max_len || P.na == 0 || P.nb == 0);
  if (!P.ok) return P;
  const float refa = A.F.dref[a], refb = A.F.dref[b];
  const float Dc = (refa - refb) * P.cp, Ds = (refa + refb) * P.sp;
  // Histogram terms of the summed-over forest (w, w x) in fixed point, one
  // 32-bit word each: shared memory adds integers natively.  A (vector, bin)
  // sum holds at most 2 / (cp hmin) + 2 pixels (two windows of width 1/cp) of
  // the forest's (one pixel has no gap: hmin is then next to 0).
  const float runa = fminf(2.f / (P.cp * A.F.hmin[a]) + 2.f, static_cast<float>(P.na));
  const float runb = fminf(2.f / (P.cp * A.F.hmin[b]) + 2.f, static_cast<float>(P.nb));
  const float sA0 = word_scale(runa * A.F.wmax[a]), sB0 = word_scale(runa * A.F.wmax[a] * A.F.xmax[a]);
  const float sA1 = word_scale(runb * A.F.wmax[b]), sB1 = word_scale(runb * A.F.wmax[b] * A.F.xmax[b]);
  const Pix* ga = A.pix + A.F.off[a];
  const Pix* gb = A.pix + A.F.off[b];
  for (int k = tid; k < P.na; k += kDmThreads) {
    const Pix p = ga[k];
    m.ucs[k] = make_float2(fmaf(p.x, P.cp, Dc), fmaf(p.x, P.sp, Ds));
    m.tv(0)[k] = make_int2(__float2int_rn(p.y * sA0), __float2int_rn(p.y * p.w * sB0));
    m.cf(1)[k] = make_float4(0.f, 0.f, p.y, p.y * p.w);
  }
  for (int k = tid; k < P.nb; k += kDmThreads) {
    const Pix p = gb[k];
    m.db[k] = p.x;
    m.tv(1)[k] = make_int2(__float2int_rn(p.y * sA1), __float2int_rn(p.y * p.w * sB1));
    m.cf(0)[k] = make_float4(0.f, 0.f, p.y, p.y * p.w);
  }
  float* c = m.par + 16 * par;
  const int t = tid - (kDmThreads - 32);
  if (t >= 0 && t < 8) {
    // 1 / (W_a W_b), 1 / (W_a S_b), 1 / (S_a W_b), 1 / (S_a S_b), 1 / W_b, 1 / S_b, 1 / W_a, 1 / S_a
    const double x = (t < 4) ? (t < 2 ? A.F.wsum[a] : A.F.ssum[a]) : 1.0;
    const double y = (t < 4) ? ((t & 1) ? A.F.ssum[b] : A.F.wsum[b])
                             : (t == 4 ? A.F.wsum[b] : t == 5 ? A.F.ssum[b] : t == 6 ? A.F.wsum[a] : A.F.ssum[a]);
    c[kC11 + t] = (A.eta_mean_slope != 0 && x > 0.0 && y > 0.0) ? static_cast<float>(1.0 / (x * y)) : 0.f;
  }
  if (t == 8) {
    c[kScA0] = 1.f / sA0;
    c[kScB0] = 1.f / sB0;
    c[kScA1] = 1.f / sA1;
    c[kScB1] = 1.f / sB1;
  }
  return P;
}

// Rank-1 coefficients sqrt(w_v / W), sqrt(w_v / S) of the vectors of both
// sides, and for every kWin vectors the range of the other forest's pixels
// that can share the grid with one of them (for one vector r_par is monotone
// in the other pixel and r_perp rises, in FP32 as evaluated, so the two ends
// are found by bisection with the binning's own arithmetic).  About a third of
// the pixel pairs of two SDSS-like forests fall outside.
__device__ __forceinline__ void dm_windows(const DmArgs& A, const Pair& P, const Sm& m, int par) {
  const int tid = threadIdx.x;
  const float* c = m.par + 16 * par;
  const float fnpar = static_cast<float>(A.n_par), fnperp = static_cast<float>(A.n_perp);
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int nvec = side == 0 ? P.nb : P.na, nother = side == 0 ? P.na : P.nb;
    const float iw = c[side == 0 ? kIWa : kIWb], is = c[side == 0 ? kISa : kISb];
    for (int k = tid; k < nvec; k += kDmThreads) {
      const float w = m.cf(side)[k].z;
      m.cf(side)[k].x = sqrtf(w * iw);
      m.cf(side)[k].y = sqrtf(w * is);
    }
    const int ng = (nvec + kWin - 1) / kWin;
    // one thread per end of a range, from the last thread down
    for (int g2 = kDmThreads - 1 - tid; g2 < 2 * ng; g2 += kDmThreads) {
      const int g = g2 >> 1, first = g * kWin, last = min(first + kWin, nvec) - 1;
      int lo = 0, hi = nother;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        // at the vector of the group that reaches furthest down (up) in the other forest
        const float2 u = m.ucs[side == 0 ? mid : ((g2 & 1) ? last : first)];
        const float d = m.db[side == 0 ? ((g2 & 1) ? last : first) : mid];
        const float rp = fmaf(-d, P.cp, u.x);
        bool below;
        if (!(g2 & 1))
          below = side == 0 ? !(rp > -fnpar) : !(rp < fnpar);
        else {
          const float2 uf = m.ucs[side == 0 ? mid : first];
          const float df = m.db[side == 0 ? first : mid];
          below = (side == 0 ? rp < fnpar : rp > -fnpar) && fmaf(df, P.sp, uf.y) < fnperp;
        }
        if (below)
          lo = mid + 1;
        else
          hi = mid;
      }
      reinterpret_cast<int*>(m.win(side))[g2] = lo;
    }
  }
}

// One batch: cbn consecutive vectors from v0 of a side, against the pixels
// [lo, hi) of the other forest.
struct Batch {
  int side, v0, cbn, lo, hi;
};

// the next batch that has pixels in the grid; false after the last one
__device__ __forceinline__ bool next_batch(Batch& B, int v0, int cb, const Pair& P, bool eta, const Sm& m) {
  for (;;) {
    const int nvec = B.side == 0 ? P.nb : P.na;
    if (v0 >= nvec) {
      if (B.side == 1 || !eta) return false;
      B.side = 1;
      v0 = 0;
      continue;
    }
    B.v0 = v0;
    B.cbn = min(cb, nvec - v0);
    B.lo = m.win(B.side)[v0 / kWin].x;
    B.hi = m.win(B.side)[v0 / kWin].y;
    for (int g = v0 / kWin + 1; g * kWin < v0 + B.cbn; ++g) B.hi = max(B.hi, m.win(B.side)[g].y);
    if (B.lo < B.hi) return true;
    v0 += B.cbn;
  }
}

// f(o, l) for the pixel pairs (vector of this thread, pixel o) of a batch that
// are in the grid, l their local bin.  Lanes are consecutive vectors, thread
// groups of CB take every (threads / CB)-th pixel; four loads in flight.
template <int CB, class F>
__device__ __forceinline__ void for_pairs(const Batch& B, const Pair& P, const Sm& m, float fnpar, float fnperp, int npar,
                                          uint32_t corner, F&& f) {
  const int vv = threadIdx.x & (CB - 1);
  constexpr int step = kDmThreads / CB;
  if (vv >= B.cbn) return;
  const float nan = __int_as_float(0x7FC00000);
  int l;
  if (B.side == 0) {
    const float dj = m.db[B.v0 + vv];
    for (int o = B.lo + threadIdx.x / CB; o < B.hi; o += 4 * step) {
      float2 u[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) u[e] = (o + e * step < B.hi) ? m.ucs[o + e * step] : make_float2(nan, nan);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (bin_at(fmaf(-dj, P.cp, u[e].x), fmaf(dj, P.sp, u[e].y), fnpar, fnperp, npar, corner, &l)) f(o + e * step, l);
    }
  } else {
    const float2 u = m.ucs[B.v0 + vv];
    for (int o = B.lo + threadIdx.x / CB; o < B.hi; o += 4 * step) {
      float d[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) d[e] = (o + e * step < B.hi) ? m.db[o + e * step] : nan;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (bin_at(fmaf(-d[e], P.cp, u.x), fmaf(d[e], P.sp, u.y), fnpar, fnperp, npar, corner, &l)) f(o + e * step, l);
    }
  }
}

// The rank-1 terms of one pair, batch by batch, into the triangle (or G), and
// its T vectors.  dirty: entries of V's rows in use by the last batch (the rest
// is zero).  Four block-wide phases a batch: the next batch's marks are
// set in the phase of this one's tiles, whose last round leaves warps idle.
template <bool GLOBAL, int CB>
__device__ void dm_vectors(const DmArgs& A, const Pair& P, double* G, int t0, int L, int scap, const Sm& m, int par,
                           int& dirty) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  constexpr int nwarps = kDmThreads / 32;
  const bool eta = A.eta_mean_slope != 0;
  const int npar = A.n_par, nbins = A.n_par * A.n_perp;
  const int ldv = ldv_for(scap);
  const float fnpar = static_cast<float>(npar), fnperp = static_cast<float>(A.n_perp);
  const uint32_t corner = bin_corner(npar, t0);
  const int g0 = t0 * A.n_par;   // accumulator row of local bin 0 (see dm_finalize_kernel)
  unsigned char* mark = m.mark;
  auto set_marks = [&](const Batch& B) {
    for_pairs<CB>(B, P, m, fnpar, fnperp, npar, corner, [&](int, int l) { mark[l] = 1; });
  };
  auto clear_marks = [&]() {
    for (int k = tid; k < (L + 3) / 4; k += kDmThreads) reinterpret_cast<uint32_t*>(mark)[k] = 0;
  };
  Batch B;
  B.side = 0;
  bool on = next_batch(B, 0, CB, P, eta, m);
  if (!on) return;
  set_marks(B);
  __syncthreads();
  while (on) {
    // compaction of the marks into the ascending union support S and the
    // inverse map: a warp takes 32 local bins and counts the marks below
    // them itself.  The last batch's entries of V are cleared meanwhile.
    for (int l0 = wid * 32; l0 < L; l0 += nwarps * 32) {
      int below = 0;
      for (int k = lane; k < l0 / 4; k += 32) below += __popc(reinterpret_cast<const uint32_t*>(mark)[k]);
      below = __reduce_add_sync(0xffffffffu, below);
      const int l = l0 + lane;
      const bool set = (l < L) && mark[l];
      const unsigned msk = __ballot_sync(0xffffffffu, set);
      if (set) {
        const int pos = below + __popc(msk & ((1u << lane) - 1u));
        if (pos < scap) m.S[pos] = l;
        m.inv[l] = static_cast<int16_t>(pos);
      }
      if (l0 + 32 >= L && lane == 0) *m.ns = below + __popc(msk);
    }
    for (int vv = wid; vv < CB; vv += nwarps)
      for (int k = lane; 2 * k < dirty; k += 32)
        reinterpret_cast<float4*>(m.V + vv * ldv)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    dirty = 0;
    __syncthreads();
    const int ns = *m.ns;
    if (ns > scap) {
      // union too large for the staging arrays: again with half the batch
      clear_marks();
      __syncthreads();
      next_batch(B, B.v0, max(1, B.cbn / 2), P, eta, m);
      set_marks(B);
      __syncthreads();
      continue;
    }
    // histograms on S
    {
      unsigned* row = reinterpret_cast<unsigned*>(m.V + (tid & (CB - 1)) * ldv);
      const int2* tv = m.tv(B.side);
      const int16_t* inv = m.inv;
      for_pairs<CB>(B, P, m, fnpar, fnperp, npar, corner, [&](int o, int l) {
        const int2 t = tv[o];
        const int k = 2 * inv[l];
        atomicAdd(row + k, static_cast<unsigned>(t.x));
        atomicAdd(row + k + 1, static_cast<unsigned>(t.y));
      });
    }
    clear_marks();
    __syncthreads();
    // T vectors (from unscaled column histograms) and scaling by the rank-1
    // coefficients sqrt(w_v / W), sqrt(w_v / S)
    const float4* cf = m.cf(B.side) + B.v0;
    const float isA = m.par[16 * par + (B.side == 0 ? kScA0 : kScA1)];
    const float isB = m.par[16 * par + (B.side == 0 ? kScB0 : kScB1)];
    if (B.side == 0) {
      // item (k, vv) = (bin of S, vector): the vectors of a bin sit in CB
      // consecutive lanes, which sum its four T terms, half of the terms
      // changing lanes at each of the first two steps
      const int vv = tid & (CB - 1);
      const bool actv = vv < B.cbn;
      const float4 c = actv ? cf[vv] : make_float4(0.f, 0.f, 0.f, 0.f);
      for (int k0 = 0; k0 < ns; k0 += kDmThreads / CB) {
        const int k = k0 + tid / CB;
        const bool act = (k < ns) && actv;
        float t[4] = {0.f, 0.f, 0.f, 0.f};
        if (act) {
          const float2 h = unf2(m.V[vv * ldv + k]);
          const float va = static_cast<float>(__float_as_int(h.x)) * isA;
          const float vb = static_cast<float>(__float_as_int(h.y)) * isB;
          t[0] = c.z * va;
          t[1] = c.z * vb;
          t[2] = c.w * va;
          t[3] = c.w * vb;
          m.V[vv * ldv + k] = f2(va * c.x, vb * c.y);
        }
        const bool up1 = vv & (CB / 2), up2 = vv & (CB / 4);
        float x = up1 ? t[2] : t[0], y = up1 ? t[3] : t[1];
        x += __shfl_xor_sync(0xffffffffu, up1 ? t[0] : t[2], CB / 2);
        y += __shfl_xor_sync(0xffffffffu, up1 ? t[1] : t[3], CB / 2);
        float z = up2 ? y : x;
        z += __shfl_xor_sync(0xffffffffu, up2 ? x : y, CB / 4);
#pragma unroll
        for (int o = CB / 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        if (k < ns && (vv & (CB / 4 - 1)) == 0)
          reinterpret_cast<float*>(m.T4 + m.S[k])[vv / (CB / 4)] += z;
      }
    } else {
      for (int vv = wid; vv < B.cbn; vv += nwarps) {
        const float4 c = cf[vv];
        const float ka = c.x, kb = c.y;
        F2* row = m.V + vv * ldv;
        for (int k = lane; k < ns; k += 32) {
          const float2 h = unf2(row[k]);
          row[k] = f2(static_cast<float>(__float_as_int(h.x)) * isA * ka,
                      static_cast<float>(__float_as_int(h.y)) * isB * kb);
        }
      }
    }
    __syncthreads();
    // rank-1 updates of the batch: register tiles of S x S, one per thread,
    // each adding its 8 entries to the triangle
    if (eta) {
      if (!GLOBAL && A.tensor_tiles) {
        dm_tiles_tc(reinterpret_cast<const float*>(m.V), ldv, ns, B.cbn, m.S, m.U, L, wid, nwarps, lane);
      } else {
        dm_tiles<GLOBAL>(m.V, ldv, B.cbn, G, m.U, m.S, g0, ns, L, nbins);
      }
    }
    dirty = ns;
    on = next_batch(B, B.v0 + B.cbn, CB, P, eta, m);
    if (on) set_marks(B);
    __syncthreads();
  }
}

// T1 of a local bin that no pixel pair of this pair has reached: -0, which any
// sum of weights replaces (-0 + 0 is +0)
constexpr uint32_t kUntouched = 0x80000000u;
__device__ __forceinline__ float4 untouched() { return make_float4(__uint_as_float(kUntouched), 0.f, 0.f, 0.f); }

// T terms, diagonal and W: one warp per row r, lanes over c >= r.  The
// pair's whole contribution (its rank-1 terms, already in the triangle, plus
// these) goes to the FP64 accumulator here, and the triangle is cleared, so
// that D~ and W are summed over pairs in FP64 only and nothing of a pair stays
// for the block's next one, which may have other bins in the same words or
// belong to another catalogue.  Rows that no pixel pair touched (kUntouched)
// hold nothing; a row whose T is 0 can (weights that the fixed point of one
// side rounds to 0 and that of the other does not).
template <bool GLOBAL>
__device__ __forceinline__ void dm_flush(const DmArgs& A, double* G, double* wdm, int t0, int L, const Sm& m, int par) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int nwarps = kDmThreads / 32;
  const int g0 = t0 * A.n_par, nbins = A.n_par * A.n_perp;
  const float* pc = m.par + 16 * par;
  const float c11 = pc[kC11], cyy = pc[kCyy], cxx = pc[kCxx], cxy = pc[kCxy];
  for (int r = wid; r < L; r += nwarps) {
    const float4 tr = m.T4[r];
    if (__float_as_uint(tr.x) == kUntouched) continue;
    const float f1 = c11 * tr.x, fy = cyy * tr.z, fx = cxx * tr.y, fxy = cxy * tr.w;
    const int rb = tri_rowbase(r, L);
    // two columns per lane per iteration (independent chains)
    for (int c = r + lane; c < L; c += 64) {
      const int c2 = c + 32;
      const float4 tc = m.T4[c];
      const float4 tc2 = (c2 < L) ? m.T4[c2] : make_float4(0.f, 0.f, 0.f, 0.f);
      float v = f1 * tc.x + fy * tc.z + fx * tc.y + fxy * tc.w;
      const float v2 = f1 * tc2.x + fy * tc2.z + fx * tc2.y + fxy * tc2.w;
      if (c == r) v += tr.x;
      // consecutive lanes add to consecutive entries of the accumulator's row
      double* row = G + static_cast<int64_t>(g0 + r) * nbins + g0;
      if (!GLOBAL) {
        // (r, c), (r, c2) owned by this lane: flush, and clear also where the
        // rank-1 part u and v cancel to exactly 0 (about one entry in 1e7)
        const float u = m.U[rb + c], x = u + v;
        if (x != 0.f) red_add_f64_global(row + c, static_cast<double>(x));
        if (u != 0.f) m.U[rb + c] = 0.f;
        if (c2 < L) {
          const float u2 = m.U[rb + c2], x2 = u2 + v2;
          if (x2 != 0.f) red_add_f64_global(row + c2, static_cast<double>(x2));
          if (u2 != 0.f) m.U[rb + c2] = 0.f;
        }
      } else {
        if (v != 0.f) red_add_f64_global(row + c, static_cast<double>(v));
        if (v2 != 0.f) red_add_f64_global(row + c2, static_cast<double>(v2));
      }
    }
    if (lane == 0) red_add_f64_global(wdm + g0 + r, static_cast<double>(tr.x));
  }
}

template <bool GLOBAL, int CB>
__global__ void __launch_bounds__(kDmThreads, 1) dm_kernel(DmArgs A, const Chunk* chunks,
                                                           const int32_t* n_chunks_dev,
                                                           const int32_t* order, const int32_t* wide,
                                                           const int32_t* n_wide_dev, int scap, int Lalloc,
                                                           int kmin, int kmax, unsigned long long* counter) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ long long s_item;
  const int tid = threadIdx.x;
  const int nbins = A.n_par * A.n_perp;
  const int n_items = GLOBAL ? *n_wide_dev : *n_chunks_dev;
  const Sm m(sm, layout(Lalloc, scap, A.max_len, GLOBAL, CB), A.max_len);
  // clear all accumulators once
  if (!GLOBAL) {
    const int nt = Lalloc * (Lalloc + 1) / 2;
    for (int k = tid; k < nt; k += blockDim.x) m.U[k] = 0.f;
  }
  for (int k = tid; k < Lalloc; k += blockDim.x) {
    m.T4[k] = untouched();
    m.mark[k] = 0;
  }
  for (int k = tid; k < CB * ldv_for(scap); k += blockDim.x) m.V[k] = 0;
  int dirty = 0;
  __syncthreads();
  for (;;) {
    if (tid == 0) s_item = static_cast<long long>(atomicAdd(counter, 1ull));
    __syncthreads();
    const long long item = s_item;
    __syncthreads();
    if (item >= n_items) break;
    int t0, K, first, cnt, mock;
    if (!GLOBAL) {
      const Chunk ch = chunks[item];
      if (ch.K < kmin || ch.K > kmax) continue;   // another launch's band widths (uniform over the block)
      t0 = ch.t0; K = ch.K; first = ch.begin; cnt = ch.n; mock = ch.mock;
    } else {
      const int pi = wide[item];
      const int2 p = A.pairs[pi];
      if (!pair_band(A, p.x, p.y, A.cs[pi].y, &t0, &K)) continue;
      first = 0; cnt = 1; mock = A.F.mock[p.x];
    }
    // accumulators of the chunk's catalogue
    double* G = A.G + static_cast<int64_t>(mock) * nbins * nbins;
    double* wdm = A.wdm + static_cast<int64_t>(mock) * nbins;
    const int L = K * A.n_par;
    // A pair's pixels are loaded while the previous one's triangle is flushed.
    int par = 0;
    Pair P = dm_load(A, GLOBAL ? wide[item] : order[first], m, par);
    __syncthreads();
    for (int q = 0; q < cnt; ++q) {
      if (P.ok) dm_windows(A, P, m, par);
      __syncthreads();
      if (P.ok) dm_vectors<GLOBAL, CB>(A, P, G, t0, L, scap, m, par, dirty);
      Pair N;
      N.ok = false;
      if (!GLOBAL && q + 1 < cnt) N = dm_load(A, order[first + q + 1], m, par ^ 1);
      if (P.ok) dm_flush<GLOBAL>(A, G, wdm, t0, L, m, par);
      __syncthreads();
      if (P.ok)
        for (int k = tid; k < L; k += kDmThreads) m.T4[k] = untouched();
      P = N;
      par ^= 1;
    }
  }
}

// v / w from the rounded reciprocal of w: the product's remainder, exact in a fused
// multiply-add, corrects it to the correctly rounded quotient (Markstein 1990):
// three FP64 operations (a division per entry took three quarters of the kernel).
// near: |w| in 2^-300 .. 2^300; with v = 0 or |v| in 2^-600 .. 2^600 (by its high
// word: FP64 comparisons share the FP64 pipe) no step leaves the normal range.
__device__ __forceinline__ double quotient(double v, double w, double inv, bool near) {
  const uint32_t e = static_cast<uint32_t>(__double2hiint(v)) & 0x7FFFFFFFu;
  if (!near || (e - 0x1A700000u > 0x4B000000u && v != 0.0)) return (w != 0.0) ? v / w : 0.0;
  const double q = v * inv;
  return fma(fma(-q, w, v), inv, q);
}

// D and W from the accumulators, one block per (catalogue, row of D).  The
// accumulators number bin (p, t) as t n_par + p, so that a pair's local bins,
// and with them the 32 lanes of an atomic, are consecutive (L2 takes atomics a
// 32-byte sector at a time); the outputs number it p n_perp + t.
template <bool STAGED>
__global__ void __launch_bounds__(256) dm_finalize_kernel(const double* G, const double* wdm, double* D, double* wout,
                                                          int n_par, int n_perp, int64_t rows) {
  extern __shared__ double frow[];   // the row in the accumulators' numbering
  const int nb = n_par * n_perp;
  for (int64_t q = blockIdx.x; q < rows; q += gridDim.x) {
    const int64_t m = q / nb;
    const int r = static_cast<int>(q - m * nb);
    const int rp = (r % n_perp) * n_par + r / n_perp;
    const double w = wdm[m * nb + rp];
    const double* Gm = G + m * nb * nb;
    auto at = [&](int c) {
      return (c >= rp) ? Gm[static_cast<int64_t>(rp) * nb + c] : Gm[static_cast<int64_t>(c) * nb + rp];
    };
    if (STAGED && w != 0.0) {
      for (int c = threadIdx.x; c < nb; c += blockDim.x) frow[c] = at(c);
      __syncthreads();
    }
    double* out = D + q * nb;
    const double inv = (w != 0.0) ? 1.0 / w : 0.0;
    const bool near = fabs(w) > 4.9e-91 && fabs(w) < 2.0e90;
    for (int c = threadIdx.x; c < nb; c += blockDim.x) {
      const int cp = (c % n_perp) * n_par + c / n_perp;
      const double v = (w != 0.0) ? (STAGED ? frow[cp] : at(cp)) : 0.0;
      out[c] = quotient(v, w, inv, near);
    }
    if (wout && threadIdx.x == 0) wout[q] = w;
    __syncthreads();
  }
}

// first (global) forest index of each catalogue: forests are stored catalogue
// by catalogue, so it is the forest whose predecessor belongs to another one
__global__ void fbase_kernel(Forests F, int32_t* fbase) {
  for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < F.n;
       f += (int64_t)gridDim.x * blockDim.x)
    if (f == 0 || F.mock[f] != F.mock[f - 1]) fbase[F.mock[f]] = static_cast<int32_t>(f);
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

// Work counts of the closed form (one warp per kept forest pair, the D
// kernel's FP32 binning): for every rank-1 vector (column j of b over i of a,
// row i of a over j of b) the number |S_v| of distinct bins it touches, for
// the pair the number |S_pair| of distinct bins of all its pixel pairs, and
// the in-grid pixel pairs.  Bins are marked in lane-private bitmaps of the
// pair's band (word w of lane l at w * 32 + l: no bank conflicts).
__global__ void dm_work_kernel(DmArgs A, uint64_t thr, int all, int words_cap, DmWork* out) {
  extern __shared__ uint32_t wbm[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  uint32_t* mine = wbm + static_cast<size_t>(wid) * 33 * words_cap;
  uint32_t* pbm = mine + 32 * words_cap;
  const int npar = A.n_par;
  const float fnpar = static_cast<float>(npar), fnperp = static_cast<float>(A.n_perp);
  unsigned long long n_pairs = 0, n_pix = 0;
  double sv2 = 0.0, sp2 = 0.0;
  for (int64_t k = warp; k < A.n_pairs; k += nw) {
    const int2 pr = A.pairs[k];
    if (pr.x < 0 || !keep_pair(pr.x, pr.y, A.seed, thr, all)) continue;
    const float2 cs = A.cs[k];
    int t0, K;
    if (!pair_band(A, pr.x, pr.y, cs.y, &t0, &K)) continue;
    const int words = (K * npar + 31) >> 5;
    if (words > words_cap) continue;   // (a band wider than the grid cannot occur)
    const int na = A.F.len[pr.x], nb = A.F.len[pr.y];
    const Pix* pa = A.pix + A.F.off[pr.x];
    const Pix* pb = A.pix + A.F.off[pr.y];
    const float cp = cs.x, sp = cs.y;
    const float Dc = (A.F.dref[pr.x] - A.F.dref[pr.y]) * cp, Ds = (A.F.dref[pr.x] + A.F.dref[pr.y]) * sp;
    for (int w = lane; w < words; w += 32) pbm[w] = 0u;
    __syncwarp();
    for (int side = 0; side < 2; ++side) {
      const int nvec = side == 0 ? nb : na;
      const int nother = side == 0 ? na : nb;
      for (int v0 = 0; v0 < nvec; v0 += 32) {
        const int v = v0 + lane;
        if (v < nvec) {
          for (int w = 0; w < words; ++w) mine[w * 32 + lane] = 0u;
          for (int o = 0; o < nother; ++o) {
            const int i = side == 0 ? o : v;
            const int j = side == 0 ? v : o;
            const float xi = pa[i].x;
            const int l = local_bin(make_float2(fmaf(xi, cp, Dc), fmaf(xi, sp, Ds)), pb[j].x, cp, sp, fnpar,
                                    fnperp, npar, t0);
            if (l >= 0) {
              mine[(l >> 5) * 32 + lane] |= 1u << (l & 31);
              if (side == 0) ++n_pix;
            }
          }
          int cnt = 0;
          for (int w = 0; w < words; ++w) {
            const uint32_t m = mine[w * 32 + lane];
            if (m) {
              cnt += __popc(m);
              atomicOr(&pbm[w], m);
            }
          }
          sv2 += static_cast<double>(cnt) * cnt;
        }
      }
    }
    __syncwarp();
    int c = 0;
    for (int w = lane; w < words; w += 32) c += __popc(pbm[w]);
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) {
      sp2 += static_cast<double>(c) * c;
      n_pairs += 1;
    }
    __syncwarp();
  }
  for (int o = 16; o > 0; o >>= 1) {
    n_pix += __shfl_xor_sync(0xffffffffu, n_pix, o);
    sv2 += __shfl_xor_sync(0xffffffffu, sv2, o);
  }
  if (lane == 0) {
    atomicAdd(&out->pairs, n_pairs);
    atomicAdd(&out->pix, n_pix);
    atomicAdd(&out->sv2, sv2);
    atomicAdd(&out->sp2, sp2);
  }
}

}  // namespace

// single-block exclusive scan (defined in pairs.cu's namespace would be private)
namespace {
__global__ void dm_scan_kernel(const int32_t* in, int64_t n, int64_t* out) {
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
      int64_t v = part[k];
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

__global__ void to_int32_kernel(const int64_t* in, int32_t* out) { *out = static_cast<int32_t>(*in); }
}  // namespace

cudaError_t run_dmat(const DmArgs& a, const DevInfo& dev, void** scratch, size_t* scratch_cap,
                     cudaStream_t s) {
  const int nbins = a.n_par * a.n_perp;
  const int max_len = std::max(a.max_len, 1);
  // largest band that fits in shared memory with batches of 16 vectors (kfit)
  // and with batches of 32 (kfit2 <= kfit)
  auto fits = [&](int K, int cb, int* sc) {
    const int L = K * a.n_par;
    *sc = scap_for(L, a.n_par, K, cb);
    return band_bytes(L, *sc, max_len, cb) <= dev.smem_optin &&
           layout(L, *sc, max_len, false, cb).end + 64 <= dev.smem_optin;
  };
  int kfit = 0, scap = 0, kfit2 = 0, scap2 = 0;
  for (int K = a.n_perp; K >= 1 && kfit == 0; --K)
    if (fits(K, kCB, &scap)) kfit = K;
  for (int K = kfit; K >= 1 && kfit2 == 0; --K)
    if (fits(K, kCB2, &scap2)) kfit2 = K;
  // wide-pair configuration (triangle in global memory)
  const int Lw = a.n_perp * a.n_par;
  const int scapw = scap_for(Lw, a.n_par, a.n_perp, kCB);
  if (layout(Lw, scapw, max_len, true, kCB).end + 64 > dev.smem_optin) return cudaErrorInvalidValue;
  if (kfit == 0) {  // everything goes wide
    kfit = 1;
    scap = scap_for(a.n_par, a.n_par, 1, kCB);
  }

  const int n_mocks = std::max(a.n_mocks, 1);
  if (static_cast<int64_t>(n_mocks) * a.n_perp * kfit > (1 << 30)) return cudaErrorInvalidValue;
  const int ngroups = n_mocks * a.n_perp * kfit;   // (catalogue, first band row, K)
  auto al = [](size_t v) { return (v + 255) & ~size_t(255); };
  const int64_t n = a.n_pairs;
  size_t o = 0;
  const size_t o_key = o; o += al(std::max<int64_t>(n, 1) * 4);
  const size_t o_order = o; o += al(std::max<int64_t>(n, 1) * 4);
  const size_t o_wide = o; o += al(std::max<int64_t>(n, 1) * 4);
  const size_t o_count = o; o += al(ngroups * 4);
  const size_t o_cursor = o; o += al(ngroups * 4);
  const size_t o_start = o; o += al((ngroups + 1) * 8);
  const size_t o_nch = o; o += al(ngroups * 4);
  const size_t o_coff = o; o += al((ngroups + 1) * 8);
  const size_t o_chunks = o; o += al((n / kChunk + ngroups + 1) * sizeof(Chunk));
  const size_t o_fbase = o; o += al(static_cast<size_t>(n_mocks) * 4);
  const size_t o_misc = o; o += al(64);
  LYA_TRY(grow(scratch, scratch_cap, o));
  char* sc = static_cast<char*>(*scratch);
  int32_t* key = reinterpret_cast<int32_t*>(sc + o_key);
  int32_t* order = reinterpret_cast<int32_t*>(sc + o_order);
  int32_t* wide = reinterpret_cast<int32_t*>(sc + o_wide);
  int32_t* count = reinterpret_cast<int32_t*>(sc + o_count);
  int32_t* cursor = reinterpret_cast<int32_t*>(sc + o_cursor);
  int64_t* start = reinterpret_cast<int64_t*>(sc + o_start);
  int32_t* nch = reinterpret_cast<int32_t*>(sc + o_nch);
  int64_t* coff = reinterpret_cast<int64_t*>(sc + o_coff);
  Chunk* chunks = reinterpret_cast<Chunk*>(sc + o_chunks);
  int32_t* fbase = reinterpret_cast<int32_t*>(sc + o_fbase);
  int32_t* misc = reinterpret_cast<int32_t*>(sc + o_misc);   // [0] n_wide, [1] n_chunks
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(sc + o_misc + 16);

  LYA_TRY(cudaMemsetAsync(count, 0, ngroups * 4, s));
  LYA_TRY(cudaMemsetAsync(cursor, 0, ngroups * 4, s));
  LYA_TRY(cudaMemsetAsync(misc, 0, 64, s));
  LYA_TRY(cudaMemsetAsync(a.G, 0, sizeof(double) * nbins * (size_t)nbins * n_mocks, s));
  LYA_TRY(cudaMemsetAsync(a.wdm, 0, sizeof(double) * nbins * (size_t)n_mocks, s));
  LYA_TRY(cudaMemsetAsync(fbase, 0, static_cast<size_t>(n_mocks) * 4, s));
  if (a.F.n > 0) LYA_COUNT(1), fbase_kernel<<<grid_for(a.F.n, 256), 256, 0, s>>>(a.F, fbase);
  DmArgs a2 = a;
  a2.fbase = fbase;
  const int all = a.p_subsample >= 1.0 ? 1 : 0;
  uint64_t thr = 0;
  if (!all && a.p_subsample > 0.0) thr = static_cast<uint64_t>(a.p_subsample * 18446744073709551616.0);
  if (a.p_subsample <= 0.0) return cudaSuccess;  // nothing kept: D = 0, W = 0
  if (n > 0) {
    LYA_COUNT(1), dm_select_kernel<<<grid_for(n, 256), 256, 0, s>>>(a2, thr, all, kfit, key, count, wide, misc);
    LYA_COUNT(1), dm_scan_kernel<<<1, 1024, 0, s>>>(count, ngroups, start);
    LYA_COUNT(1), dm_scatter_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, key, start, cursor, order);
    LYA_COUNT(1), chunk_count_kernel<<<grid_for(ngroups, 256), 256, 0, s>>>(count, ngroups, nch);
    LYA_COUNT(1), dm_scan_kernel<<<1, 1024, 0, s>>>(nch, ngroups, coff);
    LYA_COUNT(1), chunk_fill_kernel<<<grid_for(ngroups, 256), 256, 0, s>>>(count, start, coff, ngroups, kfit,
                                                                           a.n_perp, chunks);
    LYA_COUNT(1), to_int32_kernel<<<1, 1, 0, s>>>(coff + ngroups, misc + 1);
    LYA_TRY(cudaGetLastError());
  }
  // shared-memory triangle: bands of up to kfit2 rows with batches of 32
  // vectors, the wider ones (up to kfit) with batches of 16
  if (kfit2 > 0) {
    const int L = kfit2 * a.n_par;
    const Lay y = layout(L, scap2, max_len, false, kCB2);
    LYA_TRY(set_max_dynamic_smem(reinterpret_cast<const void*>(dm_kernel<false, kCB2>), y.end));
    LYA_TRY(cudaMemsetAsync(counter, 0, 8, s));
    LYA_COUNT(1), dm_kernel<false, kCB2><<<dev.sms, kDmThreads, y.end, s>>>(a2, chunks, misc + 1, order, wide,
                                                                            misc, scap2, L, 1, kfit2, counter);
    LYA_TRY(cudaGetLastError());
  }
  if (kfit2 < kfit) {
    const int L = kfit * a.n_par;
    const Lay y = layout(L, scap, max_len, false, kCB);
    LYA_TRY(set_max_dynamic_smem(reinterpret_cast<const void*>(dm_kernel<false, kCB>), y.end));
    LYA_TRY(cudaMemsetAsync(counter, 0, 8, s));
    LYA_COUNT(1), dm_kernel<false, kCB><<<dev.sms, kDmThreads, y.end, s>>>(a2, chunks, misc + 1, order, wide, misc,
                                                                           scap, L, kfit2 + 1, kfit, counter);
    LYA_TRY(cudaGetLastError());
  }
  // wide pairs
  {
    const Lay y = layout(Lw, scapw, max_len, true, kCB);
    LYA_TRY(set_max_dynamic_smem(reinterpret_cast<const void*>(dm_kernel<true, kCB>), y.end));
    LYA_TRY(cudaMemsetAsync(counter, 0, 8, s));
    LYA_COUNT(1), dm_kernel<true, kCB><<<dev.sms, kDmThreads, y.end, s>>>(a2, chunks, misc + 1, order, wide, misc,
                                                                          scapw, Lw, 1, a.n_perp, counter);
    LYA_TRY(cudaGetLastError());
  }
  return cudaSuccess;
}

cudaError_t launch_dm_finalize(const double* G, const double* wdm, double* D, double* wdm_out, int n_par, int n_perp,
                               int n_mocks, cudaStream_t s) {
  const int64_t rows = static_cast<int64_t>(n_par) * n_perp * n_mocks;
  if (rows == 0) return cudaSuccess;
  const int smem = n_par * n_perp * 8;   // staged up to 48 KB a row (6,144 bins)
  if (smem <= 48 * 1024)
    LYA_COUNT(1), dm_finalize_kernel<true><<<grid_for(rows, 1), 256, smem, s>>>(G, wdm, D, wdm_out, n_par, n_perp, rows);
  else
    LYA_COUNT(1), dm_finalize_kernel<false><<<grid_for(rows, 1), 256, 0, s>>>(G, wdm, D, wdm_out, n_par, n_perp, rows);
  return cudaGetLastError();
}

cudaError_t launch_dm_work(const DmArgs& a, const DevInfo& dev, DmWork* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(DmWork), s);
  if (e != cudaSuccess || a.n_pairs == 0 || a.p_subsample <= 0.0) return e;
  const int all = a.p_subsample >= 1.0 ? 1 : 0;
  const uint64_t thr = all ? 0 : static_cast<uint64_t>(a.p_subsample * 18446744073709551616.0);
  const int words_cap = (a.n_par * a.n_perp + 31) / 32;
  int warps = 8;
  while (warps > 1 && warps * 33 * words_cap * 4 > dev.smem_optin) warps >>= 1;
  const int smem = warps * 33 * words_cap * 4;
  if (smem > dev.smem_optin) return cudaErrorInvalidValue;
  e = set_max_dynamic_smem(reinterpret_cast<const void*>(dm_work_kernel), smem);
  if (e != cudaSuccess) return e;
  LYA_COUNT(1), dm_work_kernel<<<dev.sms * 4, warps * 32, smem, s>>>(a, thr, all, words_cap, out);
  return cudaGetLastError();
}

}  // namespace lya
