// Gradient of L = sum_A g_A xi_A with respect to delta and w (chain rule of
// Eq. 2.4):
//   dL/d delta_i = w_i sum_j gamma_A (w d)_j
//   dL/d w_i     = delta_i sum_j gamma_A (w d)_j - sum_j rho_A w_j
// with gamma_A = g_A / W_A, rho_A = gamma_A xi_A - e_A, j over the in-grid partners
// of i, for L = sum_A g_A xi_A + sum_A e_A W_A (e = 0 unless given).
//
// Each pixel is owned by one warp (work item = 32 consecutive pixels of one
// forest), which walks the forest's full neighbour list (both orientations of
// every stored pair) and gathers gamma/rho from a shared-memory table: no
// atomics, deterministic.  Each pixel pair is binned with the same FP32
// operations, in the same operand roles, as the forward kernel (first forest
// of the stored pair on the "i" side), so forward and backward agree on every
// bin.  The table has a zero guard row and column; pairs that may lie off the
// grid are clamped into them, and the range of a neighbour that lies in the
// grid for all 32 pixels is walked without the clamps.  Per-neighbour FP32
// partial sums are added into two-term (hi, lo) accumulators (Knuth's TwoSum).
// What bounds it: the shared-memory pipe (77%: per visit one broadcast 16-byte
// load and one gathered 8-byte table load).  Neighbours are staged 256 pixels
// at a time, which leaves room for 32 warps per SM, and the separations and the
// two sums are packed FP32 pairs.  Measured (gradient of a DESI-like catalogue
// of 4,000 forests): 70.8 ms with whole neighbours staged (16 warps), 58 ms
// with 256 pixels, 47 ms as it is; shorter segments (192: +1 ms, 128: +7 ms)
// and larger blocks (12 or 16 warps: +0.5 to +3 ms) are slower.
#include <algorithm>

#include "fixed.cuh"

namespace lya {
namespace {

constexpr int kAdjWarps = 8;
constexpr int kAdjSeg = 256;   // staged pixels of a neighbour per warp

// Constants of a visit: the table's address, the pair's factors and the clamps
// into the guard row and column.
struct Visit {
  F2 cpsp;             // (-c/D_par, s/D_perp)
  float pmax, tmax;
  uint32_t stride, tbase;
};

// One pixel pair: acc += (gamma (w delta), rho w).  The separations are
// a * cpsp + b; CLAMP sends pairs off the grid to the zero guard.
template <bool CLAMP>
__device__ __forceinline__ void visit(F2 a, F2 b, F2 wdw, const Visit& k, F2& acc) {
  const float2 r = unf2(fma2(a, k.cpsp, b));
  float pf = __fadd_rd(fabsf(r.x), kMagic), tf = __fadd_rd(r.y, kMagic);
  if (CLAMP) {
    pf = fminf(pf, k.pmax);
    tf = fminf(tf, k.tmax);
  }
  const uint32_t idx = __float_as_uint(pf) * k.stride + __float_as_uint(tf);
  F2 gr;
  asm volatile("ld.shared.b64 %0, [%1];" : "=l"(gr) : "r"(k.tbase + (idx << 3)));
  acc = fma2(gr, wdw, acc);
}

// Pixels [j0, j1) of the staged neighbour.  FIRST: the lane is a first-forest
// pixel (lane = its (uc, us), record = {x, x}); else a second-forest pixel
// (lane = {x, x}, record = (uc, us)).
template <bool FIRST, bool CLAMP>
__device__ __forceinline__ void visits(const ulonglong2* buf, int j0, int j1, F2 lane, const Visit& k, F2& acc) {
#pragma unroll 8
  for (int j = j0; j < j1; ++j) {
    const ulonglong2 q = buf[j];
    if (FIRST) visit<CLAMP>(q.x, lane, q.y, k, acc);
    else visit<CLAMP>(lane, q.x, q.y, k, acc);
  }
}

__global__ void degree_kernel(const int2* pairs, int64_t n, int32_t* deg) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int2 p = pairs[k];
    atomicAdd(&deg[p.x], 1);
    atomicAdd(&deg[p.y], 1);
  }
}

__global__ void adj_fill_kernel(const int2* pairs, int64_t n, const int64_t* start, int32_t* cursor,
                                int2* adj) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int2 p = pairs[k];
    const int pa = atomicAdd(&cursor[p.x], 1);
    adj[start[p.x] + pa] = make_int2(static_cast<int>(k), 1);   // owner is the first forest
    const int pb = atomicAdd(&cursor[p.y], 1);
    adj[start[p.y] + pb] = make_int2(static_cast<int>(k), 0);
  }
}

// Work items (forest, 32-pixel chunk) are laid out in the order of `order`
// (forests in HEALPix-cell order, so consecutive items read overlapping
// neighbour sets from L2), or in index order if it is NULL.
__device__ __forceinline__ int64_t item_forest(const int32_t* order, int64_t k) {
  return order ? static_cast<int64_t>(order[k]) : k;
}

__global__ void chunks_per_forest(Forests F, const int32_t* order, int32_t* nch) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < F.n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = item_forest(order, k);
    nch[k] = (f >= 0) ? (F.len[f] + 31) / 32 : 0;
  }
}

__global__ void item_fill_kernel(Forests F, const int32_t* order, const int64_t* coff, int2* items) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < F.n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = item_forest(order, k);
    if (f < 0) continue;
    const int n = (F.len[f] + 31) / 32;
    for (int c = 0; c < n; ++c) items[coff[k] + c] = make_int2(static_cast<int>(f), c);
  }
}

__global__ void scan1_kernel(const int32_t* in, int64_t n, int64_t* out) {
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

__global__ void __launch_bounds__(kAdjWarps * 32) adjoint_kernel(AdjArgs A, const int2* adj,
                                                                 const int64_t* adj_start,
                                                                 const int2* items,
                                                                 const int64_t* n_items_dev, int seg,
                                                                 unsigned long long* counter) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int npar = A.n_par, nperp = A.n_perp;
  // table entry (p, t) at p * (n_perp + 1) + t; row p = n_par and column
  // t = n_perp are the zero guard
  const int tstride = nperp + 1;
  const int tab_n = (npar + 1) * tstride;
  float2* table = reinterpret_cast<float2*>(sm);
  const int tab_bytes = ((tab_n * 8) + 15) & ~15;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  ulonglong2* buf = reinterpret_cast<ulonglong2*>(sm + tab_bytes + wid * seg * 16);
  for (int k = threadIdx.x; k < tab_n; k += blockDim.x) {
    const int p = k / tstride, t = k - p * tstride;
    float2 e = make_float2(0.f, 0.f);
    if (p < npar && t < nperp) {
      const int bin = p * nperp + t;
      const double w = A.wsum[bin];
      const double g = (w != 0.0) ? A.grad_xi[bin] / w : 0.0;
      // rho = gamma xi - dL/dW (the weight sum's own dependence on w)
      const double r = g * A.xi[bin] - (A.grad_wsum ? A.grad_wsum[bin] : 0.0);
      e = make_float2(static_cast<float>(g), static_cast<float>(r));
    }
    table[k] = e;
  }
  __syncthreads();
  // key (M + p) * tstride + (M + t), M = bits of 2^23, minus this offset is p * tstride + t
  Visit vk;
  vk.stride = static_cast<uint32_t>(tstride);
  vk.tbase = smem_addr(table) - 8u * (kMagicBits * vk.stride + kMagicBits);
  const float fnpar = static_cast<float>(npar), fnperp = static_cast<float>(nperp);
  vk.pmax = __uint_as_float(kMagicBits + static_cast<uint32_t>(npar));
  vk.tmax = __uint_as_float(kMagicBits + static_cast<uint32_t>(nperp));
  const int64_t n_items = *n_items_dev;
  for (;;) {
    unsigned long long it = 0;
    if (lane == 0) it = atomicAdd(counter, 1ull);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= static_cast<unsigned long long>(n_items)) break;
    const int2 item = items[it];
    const int f = item.x;
    const int nf = A.F.len[f];
    const int i = item.y * 32 + lane;
    const bool valid = i < nf;
    // (lanes past the end repeat the last pixel; nothing of them is stored)
    const Pix me = (nf > 0) ? A.pix[A.F.off[f] + min(i, nf - 1)] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float me_first = __shfl_sync(0xffffffffu, me.x, 0), me_last = __shfl_sync(0xffffffffu, me.x, 31);
    const float ref_f = A.F.dref[f];
    float g1h = 0.f, g1l = 0.f, g2h = 0.f, g2l = 0.f;
    const int64_t e0 = adj_start[f], e1 = adj_start[f + 1];
    for (int64_t e = e0; e < e1; ++e) {
      const int2 ent = adj[e];
      const int2 pr = A.pairs[ent.x];
      const float2 cs = A.cs[ent.x];
      const float cp = cs.x, sp = cs.y;
      const bool first = ent.y != 0;
      const int o = first ? pr.y : pr.x;
      const int no = A.F.len[o];
      if (no == 0 || nf == 0) continue;
      const Pix* po = A.pix + A.F.off[o];
      const float ref_o = A.F.dref[o];
      // pair constants with the stored (first, second) roles
      const float ref1 = first ? ref_f : ref_o, ref2 = first ? ref_o : ref_f;
      const float Dc = (ref1 - ref2) * cp, Ds = (ref1 + ref2) * sp;
      vk.cpsp = f2(-cp, sp);
      const float eps = 1e-3f + 1e-5f * (fabsf(Dc) + (me_last + po[no - 1].x) * cp);
      // no pixel pair of this chunk and this neighbour within r_par of each other
      {
        const float lo = first ? fmaf(me_first - po[no - 1].x, cp, Dc) : fmaf(po[0].x - me_last, cp, Dc);
        const float hi = first ? fmaf(me_last - po[0].x, cp, Dc) : fmaf(po[no - 1].x - me_first, cp, Dc);
        if (lo > fnpar + eps || hi < -fnpar - eps) continue;
      }
      const F2 mine = first ? f2(fmaf(me.x, cp, Dc), fmaf(me.x, sp, Ds)) : f2(me.x, me.x);
      F2 acc = 0ull;
      for (int j0 = 0; j0 < no; j0 += seg) {
        const int segn = min(seg, no - j0);
        __syncwarp();
        for (int k = lane; k < segn; k += 32) {
          const Pix q = po[j0 + k];
          buf[k] = make_ulonglong2(first ? f2(q.x, q.x) : f2(fmaf(q.x, cp, Dc), fmaf(q.x, sp, Ds)), f2(q.z, q.y));
        }
        __syncwarp();
        // the range [j0, j3) that some lane can reach and the part [j1, j2) that lies in the grid for all of
        // them: six searches, one per lane (the staged keys ascend)
        float v = 0.f;
        int word = 0;
        if (first) {
          // |uc - x cp| < npar and x sp + us < nperp, x the staged distance
          const float uf = fmaf(me_first, cp, Dc), ul = fmaf(me_last, cp, Dc);
          const float tf = (fnperp - fmaf(me_first, sp, Ds)) / sp, tl = (fnperp - fmaf(me_last, sp, Ds)) / sp;
          const float far = (sp > 0.f) ? 1.f : 0.f;
          v = lane == 0 ? (uf - fnpar) / cp : lane == 1 ? (ul + fnpar) / cp : lane == 2 ? (far != 0.f ? tf : INFINITY)
            : lane == 3 ? (ul - fnpar) / cp : lane == 4 ? (uf + fnpar) / cp : (far != 0.f ? tl : INFINITY);
          const float m = fabsf(v) * 1e-5f + 1e-2f;
          v += (lane == 0 || lane >= 4) ? -m : m;
        } else {
          // |uc - d cp| < npar and d sp + us < nperp, (uc, us) the staged pair
          word = (lane == 2 || lane == 5) ? 1 : 0;
          v = lane == 0 ? fmaf(me_first, cp, -fnpar) : lane == 1 ? fmaf(me_last, cp, fnpar)
            : lane == 2 ? fmaf(-me_first, sp, fnperp) : lane == 3 ? fmaf(me_last, cp, -fnpar)
            : lane == 4 ? fmaf(me_first, cp, fnpar) : fmaf(-me_last, sp, fnperp);
          const float m = fabsf(v) * 1e-5f + 1e-3f;
          v += (lane == 0 || lane >= 4) ? -m : m;
        }
        const int pos = (lane < 6) ? staged_below(buf, word, segn, v) : 0;
        const int lo = __shfl_sync(0xffffffffu, pos, 0);
        const int hi = min(__shfl_sync(0xffffffffu, pos, 1), __shfl_sync(0xffffffffu, pos, 2));
        const int in0 = min(max(__shfl_sync(0xffffffffu, pos, 3), lo), max(hi, lo));
        const int in1 = min(max(min(__shfl_sync(0xffffffffu, pos, 4), __shfl_sync(0xffffffffu, pos, 5)), in0), max(hi, lo));
        if (first) {
          visits<true, true>(buf, lo, in0, mine, vk, acc);
          visits<true, false>(buf, in0, in1, mine, vk, acc);
          visits<true, true>(buf, in1, hi, mine, vk, acc);
        } else {
          visits<false, true>(buf, lo, in0, mine, vk, acc);
          visits<false, false>(buf, in0, in1, mine, vk, acc);
          visits<false, true>(buf, in1, hi, mine, vk, acc);
        }
      }
      const float a1 = unf2(acc).x, a2 = unf2(acc).y;
      two_sum_add(g1h, g1l, a1);
      two_sum_add(g2h, g2l, a2);
    }
    if (valid) {
      const int64_t gi = A.F.off[f] + i - A.pix_base;
      const float s1 = g1h + g1l, s2 = g2h + g2l;
      A.grad_delta[gi] = me.y * s1;
      A.grad_weight[gi] = A.delta[gi] * s1 - s2;
    }
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

cudaError_t run_adjoint(const AdjArgs& a, const DevInfo& dev, void** scratch, size_t* scratch_cap,
                        cudaStream_t s) {
  const int64_t nf = a.F.n;
  const int64_t np = a.n_pairs;
  auto al = [](size_t v) { return (v + 255) & ~size_t(255); };
  // work items (forest, 32-pixel chunk): at most n_pix/32 + n_forests
  const int64_t max_items = a.n_pix / 32 + nf + 1;
  size_t o = 0;
  const size_t o_deg = o; o += al((nf + 1) * 4);
  const size_t o_start = o; o += al((nf + 1) * 8);
  const size_t o_cursor = o; o += al((nf + 1) * 4);
  const size_t o_adj = o; o += al(std::max<int64_t>(2 * np, 1) * 8);
  const size_t o_nch = o; o += al((nf + 1) * 4);
  const size_t o_coff = o; o += al((nf + 1) * 8);
  const size_t o_items = o; o += al(max_items * 8);
  const size_t o_misc = o; o += 256;
  LYA_TRY(grow(scratch, scratch_cap, o));
  char* sc = static_cast<char*>(*scratch);
  int32_t* deg = reinterpret_cast<int32_t*>(sc + o_deg);
  int64_t* start = reinterpret_cast<int64_t*>(sc + o_start);
  int32_t* cursor = reinterpret_cast<int32_t*>(sc + o_cursor);
  int2* adj = reinterpret_cast<int2*>(sc + o_adj);
  int32_t* nch = reinterpret_cast<int32_t*>(sc + o_nch);
  int64_t* coff = reinterpret_cast<int64_t*>(sc + o_coff);
  int2* items = reinterpret_cast<int2*>(sc + o_items);
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(sc + o_misc);
  LYA_TRY(cudaMemsetAsync(deg, 0, (nf + 1) * 4, s));
  LYA_TRY(cudaMemsetAsync(cursor, 0, (nf + 1) * 4, s));
  LYA_TRY(cudaMemsetAsync(counter, 0, 8, s));
  if (np > 0) LYA_COUNT(1), degree_kernel<<<grid_for(np, 256), 256, 0, s>>>(a.pairs, np, deg);
  LYA_COUNT(1), scan1_kernel<<<1, 1024, 0, s>>>(deg, nf, start);
  if (np > 0) LYA_COUNT(1), adj_fill_kernel<<<grid_for(np, 256), 256, 0, s>>>(a.pairs, np, start, cursor, adj);
  LYA_COUNT(1), chunks_per_forest<<<grid_for(nf, 256), 256, 0, s>>>(a.F, a.forder, nch);
  LYA_COUNT(1), scan1_kernel<<<1, 1024, 0, s>>>(nch, nf, coff);
  LYA_COUNT(1), item_fill_kernel<<<grid_for(nf, 256), 256, 0, s>>>(a.F, a.forder, coff, items);
  LYA_TRY(cudaGetLastError());
  const int tab_n = (a.n_par + 1) * (a.n_perp + 1);
  int seg = ((std::max(a.max_len, 1) + 31) / 32) * 32;
  if (seg > kAdjSeg) seg = kAdjSeg;
  const int smem = ((tab_n * 8 + 15) & ~15) + kAdjWarps * seg * 16;
  if (smem > dev.smem_optin) return cudaErrorInvalidValue;
  LYA_TRY(set_max_dynamic_smem(reinterpret_cast<const void*>(adjoint_kernel), smem));
  int per_sm = 0;
  LYA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, adjoint_kernel, kAdjWarps * 32, smem));
  if (per_sm < 1) return cudaErrorInvalidValue;
  LYA_COUNT(1), adjoint_kernel<<<per_sm * dev.sms, kAdjWarps * 32, smem, s>>>(a, adj, start, items, coff + nf, seg,
                                                                counter);
  return cudaGetLastError();
}

}  // namespace lya
