// Tree-level kernels: node statistics, partition of searched nodes, stable
// scatter into the next level, gathers, bootstrap bags, prediction.
//
// Algorithm 2: a node that meets the split condition is searched, split on
// gB, and its two children are grown next; otherwise it becomes a leaf.
// Sec. II-A: leaves predict their majority class (ties: lowest class id);
// regression leaves predict the mean target. The split sets are Eqs. (3)-(4):
// right ("+") iff bin(gB . x) >= b*, i.e. z >= t_b.
//
// Every per-level pass runs over the same kTS-row tiles of the entry-ordered
// level arrays (one CTA per tile), followed by a one-warp-per-node kernel
// where a per-node decision is needed, so shallow levels with a few large
// nodes keep the whole GPU busy. The passes over rows are bound by DRAM, the
// per-node kernels by the chain over a large node's tiles. At 200,000 x 128
// rows, with loads one at a time and 64-bit shared atomics before, and now:
// side of every entry and decision 142 and 47 us a level, scatter 80 and 34,
// statistics 99 and 53, the first gather 128 and 32.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include <type_traits>

#include "slm_internal.cuh"

namespace slm {

namespace {

constexpr int kTT = kTS;  // threads per CTA = rows per tile
constexpr int kNodeWarps = 4;  // nodes per CTA of the per-node kernels

__device__ __forceinline__ int bin_of(float z, float zmin, float inv_w, int B) {
  const float off = __fsub_rn(z, zmin);
  const float pos = __fmul_rn(off, inv_w);
  int b = (int)floorf(pos);
  b = b > B - 1 ? B - 1 : b;
  return b < 0 ? 0 : b;
}

__device__ __forceinline__ int f2ord(float f) {
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7fffffff;
}

// gB . x as one fmaf per feature in increasing order from +0, the same
// sequence the scoring kernels run. Rows of whole 16-byte words (v4) are read
// eight words ahead of their products, a 128-byte line per thread.
__device__ __forceinline__ float project_row(const float* __restrict__ x,
                                             const float* __restrict__ g, int d, bool v4) {
  float acc = 0.0f;
  int j = 0;
  if (v4) {
    constexpr int U = 8;
    for (; j + 4 * U <= d; j += 4 * U) {
      float4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = __ldg(reinterpret_cast<const float4*>(x + j) + u);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        acc = fmaf(v[u].x, g[j + 4 * u], acc);
        acc = fmaf(v[u].y, g[j + 4 * u + 1], acc);
        acc = fmaf(v[u].z, g[j + 4 * u + 2], acc);
        acc = fmaf(v[u].w, g[j + 4 * u + 3], acc);
      }
    }
  }
#pragma unroll 8
  for (; j < d; ++j) acc = fmaf(__ldg(x + j), g[j], acc);
  return acc;
}

// The weight of a tile's entries, in total or per class, in two 32-bit
// halves: a tile's kTS = 256 entries of up to 2^32 - 1 add up to less than
// 2^24 in each (64-bit shared atomics retry in a loop).
struct TileWeight {
  uint32_t lo, hi;
  __device__ __forceinline__ void add(uint32_t w) {
    atomicAdd(&lo, w & 0xffffu);
    if (w >> 16) atomicAdd(&hi, w >> 16);
  }
  __device__ __forceinline__ unsigned long long sum() const {
    return (unsigned long long)lo + ((unsigned long long)hi << 16);
  }
};
// the same over a warp, in every lane
__device__ __forceinline__ unsigned long long warp_weight(uint32_t w) {
  return (unsigned long long)__reduce_add_sync(0xffffffffu, w & 0xffffu) +
         ((unsigned long long)__reduce_add_sync(0xffffffffu, w >> 16) << 16);
}

// Copies the rows of a tile (its thread r: row r of src to row s_to[r] of
// dst), 16 bytes a lane where rows and arrays allow.
__device__ __forceinline__ void copy_rows(const float* __restrict__ src, const int* s_from,
                                          float* __restrict__ dst, const int* s_to, int rows,
                                          int d) {
  const bool v4 = (d & 3) == 0 && ((reinterpret_cast<uintptr_t>(src) |
                                    reinterpret_cast<uintptr_t>(dst)) & 15) == 0;
  auto run = [&](auto* out, const auto* in, int w) {  // w words a row
    using T = std::remove_const_t<std::remove_pointer_t<decltype(out)>>;
    constexpr int U = 8;  // words in flight per thread
    const int step_r = kTT / w, step_j = kTT - step_r * w;
    int r = (int)threadIdx.x / w, j = (int)threadIdx.x - r * w;
    while (r < rows) {
      T v[U];
      int64_t o[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        o[u] = -1;
        if (r < rows) {
          v[u] = __ldg(in + (int64_t)s_from[r] * w + j);
          o[u] = (int64_t)s_to[r] * w + j;
        }
        r += step_r;
        j += step_j;
        if (j >= w) {
          j -= w;
          ++r;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (o[u] >= 0) out[o[u]] = v[u];
    }
  };
  if (v4)
    run(reinterpret_cast<float4*>(dst), reinterpret_cast<const float4*>(src), d >> 2);
  else
    run(dst, src, d);
}

// Block-wide exclusive scan of one int per thread (kTT threads); returns the
// prefix, *total = block sum.
__device__ __forceinline__ int block_excl_scan(int v, int* total, int* sbuf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += u;
  }
  __syncthreads();
  if (lane == 31) sbuf[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int wv = lane < kTT / 32 ? sbuf[lane] : 0;
    int wi = wv;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, wi, off);
      if (lane >= off) wi += u;
    }
    if (lane < kTT / 32) sbuf[lane] = wi - wv;
    if (lane == kTT / 32 - 1) sbuf[kTT / 32] = wi;
  }
  __syncthreads();
  *total = sbuf[kTT / 32];
  return sbuf[warp] + incl - v;
}

// ---- node statistics (per tile, then per node) ------------------------------------

// Per tile of a level node: weighted class counts and weight (integer global
// atomics: order-free), target range (ordered-int atomics) and the tile's
// partial target sums (summed per node in tile order by k_stats_finish).
__global__ void __launch_bounds__(kTT)
    k_stats_tiles(Problem pr, const WorkTile* __restrict__ tiles, LevelAcc acc) {
  const WorkTile wt = tiles[blockIdx.x];
  const int K = pr.K;
  __shared__ TileWeight s_cnt[kMaxClasses];
  __shared__ unsigned long long s_w[kTT / 32];
  __shared__ double s_sy[kTT], s_sq[kTT];
  __shared__ int s_lo, s_hi;
  const bool mse = pr.crit == SLM_MSE;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < kMaxClasses) s_cnt[threadIdx.x] = TileWeight{0u, 0u};
  if (threadIdx.x == 0) {
    s_lo = INT_MAX;
    s_hi = INT_MIN;
  }
  __syncthreads();
  const int r = threadIdx.x;
  double sy = 0.0, sq = 0.0;
  uint32_t w = 0;
  int lo = INT_MAX, hi = INT_MIN;
  if (r < wt.rows) {
    const int64_t e = (int64_t)wt.row0 + r;
    w = pr.w ? pr.w[e] : 1u;
    if (mse) {
      const float yv = pr.y[e];
      sy = (double)w * (double)yv;
      sq = sy * (double)yv;
      lo = hi = f2ord(yv);
    } else {
      s_cnt[pr.lab[e]].add(w);
    }
  }
  const unsigned long long ww = warp_weight(w);
  if (lane == 0) s_w[warp] = ww;
  if (mse) {
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      atomicMin(&s_lo, lo);
      atomicMax(&s_hi, hi);
    }
    s_sy[threadIdx.x] = sy;
    s_sq[threadIdx.x] = sq;
    __syncthreads();
    for (int off = kTT / 2; off > 0; off >>= 1) {  // fixed order: deterministic
      if (threadIdx.x < off) {
        s_sy[threadIdx.x] += s_sy[threadIdx.x + off];
        s_sq[threadIdx.x] += s_sq[threadIdx.x + off];
      }
      __syncthreads();
    }
  } else {
    __syncthreads();
  }
  const int l = wt.node;
  if (threadIdx.x < K && !mse && s_cnt[threadIdx.x].sum())
    atomicAdd(&acc.cls[(int64_t)l * K + threadIdx.x], s_cnt[threadIdx.x].sum());
  if (threadIdx.x == 0) {
    unsigned long long tw = 0;
    for (int i = 0; i < kTT / 32; ++i) tw += s_w[i];
    atomicAdd(&acc.w[l], tw);
    if (mse) {
      acc.tile_s[2 * blockIdx.x] = s_sy[0];
      acc.tile_s[2 * blockIdx.x + 1] = s_sq[0];
    }
    if (mse && s_lo != INT_MAX) {
      atomicMin(&acc.ylo[l], s_lo);
      atomicMax(&acc.yhi[l], s_hi);
    }
  }
}

// One warp per level node: leaf value, splittable flag, parent sums. The
// tiles' target sums are added in tile order, 32 tiles fetched at a time,
// lane 0 the first moments and lane 1 the second (one thread fetching them
// one after the other took 92 us at 200,000 entries).
__global__ void k_stats_finish(Problem pr, const LevelNode* __restrict__ nodes,
                               const int32_t* __restrict__ tile0, int L, LevelAcc acc,
                               TreeArrays tr, int max_depth, double* par,
                               int32_t* splittable) {
  __shared__ double s_t[kNodeWarps][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int l = blockIdx.x * kNodeWarps + warp;
  if (l >= L) return;
  const LevelNode nd = nodes[l];
  const int K = pr.K;
  const unsigned long long nw = acc.w[l];
  const int slot = nd.slot;
  bool pure;
  double sy = 0.0, sq = 0.0;
  if (pr.crit == SLM_MSE) {
    const int t1 = 2 * tile0[l + 1];
    double v = 0.0;
    int o = 2 * tile0[l];
    double n0 = o + lane < t1 ? acc.tile_s[o + lane] : 0.0;
    double n1 = o + 32 + lane < t1 ? acc.tile_s[o + 32 + lane] : 0.0;
    for (; o < t1; o += 64) {
      s_t[warp][lane] = n0;
      s_t[warp][lane + 32] = n1;
      __syncwarp();
      if (o + 64 + lane < t1) n0 = acc.tile_s[o + 64 + lane];
      if (o + 96 + lane < t1) n1 = acc.tile_s[o + 96 + lane];
      const int m = min(64, t1 - o);
      if (lane < 2) {
#pragma unroll 8
        for (int i = lane; i < m; i += 2) v += s_t[warp][i];
      }
      __syncwarp();
    }
    sy = v;
    sq = __shfl_sync(0xffffffffu, v, 1);
  }
  if (lane != 0) return;
  if (pr.crit == SLM_MSE) {
    tr.leaf_value[slot] = nw ? sy / (double)nw : 0.0;
    tr.leaf_class[slot] = -1;
    pure = !(acc.yhi[l] > acc.ylo[l]);
    par[2 * l] = sy;
    par[2 * l + 1] = sq;
  } else {
    int best = 0, nonzero = 0;
    const unsigned long long* c = acc.cls + (int64_t)l * K;
    for (int k = 0; k < K; ++k) {
      if (c[k] > c[best]) best = k;
      nonzero += c[k] > 0;
    }
    tr.leaf_class[slot] = best;
    tr.leaf_value[slot] = 0.0;
    pure = nonzero <= 1;
  }
  tr.kind[slot] = 0;
  tr.weight[slot] = (int64_t)nw;
  tr.bin[slot] = -1;
  splittable[l] = (nd.depth < max_depth) && nw >= 2ull * (unsigned long long)pr.min_leaf &&
                  !pure;
}

// ---- partition (per tile), decision (per node), scatter (per tile) --------------

// Side of every entry of a searched node's tile under its gB: right iff
// bin(gB . x) >= b*. Stores the tile's left-entry count; adds the node's left
// weight and left class counts.
__global__ void __launch_bounds__(kTT)
    k_part_tiles(Problem pr, Swarm sw, const WorkTile* __restrict__ tiles, uint8_t* side,
                 int32_t* tile_left, PartAcc acc) {
  const WorkTile wt = tiles[blockIdx.x];
  const int a = wt.node;
  const EvalRes gb = sw.gb[a];
  const int d = pr.d, K = pr.K;
  extern __shared__ float s_g[];  // [d]
  __shared__ TileWeight s_lk[kMaxClasses];
  __shared__ unsigned long long s_wl[kTT / 32];
  if (!gb.valid) {
    if (threadIdx.x == 0) tile_left[blockIdx.x] = 0;
    return;
  }
  for (int j = threadIdx.x; j < d; j += kTT) s_g[j] = sw.gbest[(int64_t)a * d + j];
  if (threadIdx.x < kMaxClasses) s_lk[threadIdx.x] = TileWeight{0u, 0u};
  __syncthreads();
  const int r = threadIdx.x;
  uint32_t wl = 0;
  int left = 0;
  const bool v4 = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(pr.X) & 15) == 0;
  if (r < wt.rows) {
    const int64_t e = (int64_t)wt.row0 + r;
    const float z = project_row(pr.X + e * d, s_g, d, v4);
    const int b = bin_of(z, gb.zmin, gb.inv_w, pr.B);
    const int right = b >= gb.bin;
    side[e] = (uint8_t)right;
    if (!right) {
      left = 1;
      wl = pr.w ? pr.w[e] : 1u;
      if (pr.crit != SLM_MSE) s_lk[pr.lab[e]].add(wl);
    }
  }
  const unsigned long long ww = warp_weight(wl);
  if ((threadIdx.x & 31) == 0) s_wl[threadIdx.x >> 5] = ww;
  const int n_left = __syncthreads_count(left);
  if (threadIdx.x < K && pr.crit != SLM_MSE && s_lk[threadIdx.x].sum())
    atomicAdd(&acc.lk[(int64_t)a * K + threadIdx.x], s_lk[threadIdx.x].sum());
  if (threadIdx.x == 0) {
    tile_left[blockIdx.x] = n_left;
    unsigned long long tw = 0;
    for (int i = 0; i < kTT / 32; ++i) tw += s_wl[i];
    if (tw) atomicAdd(&acc.wl[a], tw);
  }
}

// One warp per searched node: zero-gain test, internal-node fields, tile
// bases of the scatter. out3[a] = {split?, left entries, right entries}.
__global__ void k_decide(Problem pr, Swarm sw, const NodeDesc* __restrict__ snodes,
                         const int32_t* __restrict__ map, const int32_t* __restrict__ tile0,
                         int A, const int32_t* __restrict__ tile_left, int32_t* tile_base,
                         const unsigned long long* __restrict__ node_cls,
                         const double* __restrict__ par, PartAcc acc, TreeArrays tr,
                         int32_t* out3, int32_t* status) {
  const int lane = threadIdx.x & 31;
  const int a = blockIdx.x * kNodeWarps + (threadIdx.x >> 5);
  if (a >= A) return;
  const NodeDesc nd = snodes[a];
  const EvalRes gb = sw.gb[a];
  const int d = pr.d, K = pr.K;
  int nl_entries = 0;
  const int t1 = tile0[a + 1];
  for (int t0 = tile0[a]; t0 < t1; t0 += 32) {
    const int t = t0 + lane;
    const int v = t < t1 && gb.valid ? tile_left[t] : 0;
    int incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += u;
    }
    if (t < t1) tile_base[t] = nl_entries + incl - v;
    nl_entries += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) {
    out3[3 * a + 1] = nl_entries;
    out3[3 * a + 2] = nd.seg_len - nl_entries;
  }
  if (!gb.valid) {
    if (lane == 0) out3[3 * a] = 0;
    return;
  }
  const int l = map[a];
  const unsigned long long wleft = acc.wl[a];
  const unsigned long long nw = (unsigned long long)(gb.nl + gb.nr);
  if (lane == 0 && wleft != (unsigned long long)gb.nl) atomicExch(status, 2);  // must agree
  // Zero gain: children keep the parent's class mix (Gini and entropy are
  // strictly concave), or the MSE does not drop below the parent's.
  bool no_gain;
  if (pr.crit == SLM_MSE) {
    const double sy = par[2 * l], sq = par[2 * l + 1];
    const double parent = (sq - sy * sy / (double)nw) / (double)nw;
    no_gain = !(gb.loss < parent);
  } else {
    bool differs = false;
    for (int k = lane; k < K; k += 32)
      differs |= acc.lk[(int64_t)a * K + k] * nw != node_cls[(int64_t)l * K + k] * wleft;
    no_gain = !__any_sync(0xffffffffu, differs);
  }
  if (lane == 0) out3[3 * a] = no_gain ? 0 : 1;
  if (no_gain) return;
  const int slot = nd.slot;
#pragma unroll 4
  for (int j = lane; j < d; j += 32)
    tr.dir[(int64_t)slot * d + j] = sw.gbest[(int64_t)a * d + j];
  if (lane != 0) return;
  tr.kind[slot] = 1;
  tr.zmin[slot] = gb.zmin;
  tr.inv_w[slot] = gb.inv_w;
  tr.bin[slot] = gb.bin;
  tr.loss[slot] = gb.loss;
  tr.n_left[slot] = gb.nl;
  tr.n_right[slot] = gb.nr;
}

// Stable scatter of a split node's tile into its children's segments:
// rows, labels / targets, multiplicities and sample ids.
__global__ void __launch_bounds__(kTT)
    k_scatter(Problem pr, const WorkTile* __restrict__ tiles, const uint8_t* __restrict__ side,
              const int32_t* __restrict__ dst, const int32_t* __restrict__ tile_base,
              const int32_t* __restrict__ tile0, const int32_t* __restrict__ idx_cur,
              LevelArrays nx) {
  const WorkTile wt = tiles[blockIdx.x];
  const int a = wt.node;
  const int dl = dst[2 * a], dr = dst[2 * a + 1];
  if (dl < 0) return;
  const int d = pr.d;
  __shared__ int sbuf[kTT / 32 + 1];
  __shared__ int s_src[kTT], s_dst[kTT];
  const int r = threadIdx.x;
  const bool in = r < wt.rows;
  const int64_t e = (int64_t)wt.row0 + r;
  const int is_left = in && !side[e];
  int tot_l;
  const int rank_l = block_excl_scan(is_left, &tot_l, sbuf);
  const int base_l = tile_base[blockIdx.x];
  const int rows_before = ((int)blockIdx.x - tile0[a]) * kTS;  // full tiles
  const int base_r = rows_before - base_l;
  if (in) {
    const int32_t pos = is_left ? dl + base_l + rank_l : dr + base_r + (r - rank_l);
    s_src[r] = (int)e;
    s_dst[r] = pos;
    nx.idx[pos] = idx_cur[e];
    if (nx.lab) nx.lab[pos] = pr.lab[e];
    if (nx.y) nx.y[pos] = pr.y[e];
    if (nx.w) nx.w[pos] = pr.w[e];
  }
  __syncthreads();
  copy_rows(pr.X, s_src, nx.X, s_dst, wt.rows, d);
}

__global__ void __launch_bounds__(kTT)
    k_compact_nonzero(const uint32_t* __restrict__ w_all, int64_t n, int32_t* idx_out,
                      uint32_t* w_out, const int64_t* __restrict__ off, int32_t* counts) {
  const int t = blockIdx.x;
  const uint32_t* w = w_all + (int64_t)t * n;
  __shared__ int sbuf[kTT / 32 + 1];
  const int64_t base = off[t];
  int count = 0;
  for (int64_t s0 = 0; s0 < n; s0 += kTT) {
    const int64_t s = s0 + threadIdx.x;
    const uint32_t ws = s < n ? w[s] : 0u;
    const int nz = ws > 0;
    int tot;
    const int rank = block_excl_scan(nz, &tot, sbuf);
    if (nz) {
      idx_out[base + count + rank] = (int32_t)s;
      w_out[base + count + rank] = ws;
    }
    count += tot;
  }
  if (threadIdx.x == 0) counts[t] = count;
}

// A CTA per R <= kTT entries.
__global__ void __launch_bounds__(kTT)
    k_gather(const float* __restrict__ X, const int32_t* __restrict__ labels,
             const float* __restrict__ y, const int32_t* __restrict__ idx, int64_t E, int d,
             float* Xl, int32_t* lab_l, float* y_l, int R) {
  __shared__ int s_src[kTT], s_dst[kTT];
  const int64_t e0 = (int64_t)blockIdx.x * R;
  const int rows = (int)min((int64_t)R, E - e0);
  if ((int)threadIdx.x < rows) {
    const int64_t e = e0 + threadIdx.x;
    const int s = idx[e];
    s_src[threadIdx.x] = s;
    s_dst[threadIdx.x] = (int)threadIdx.x;
    if (lab_l) lab_l[e] = labels[s];
    if (y_l) y_l[e] = y[s];
  }
  __syncthreads();
  copy_rows(X, s_src, Xl + e0 * d, s_dst, rows, d);
}

// idx[c * stride + i] = i for i < n, c < copies.
__global__ void k_iota(int32_t* idx, int64_t n, int64_t stride, int copies) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * copies) return;
  const int64_t cpy = i / n, r = i - cpy * n;
  idx[cpy * stride + r] = (int32_t)r;
}

__global__ void k_validate(const int32_t* labels, int64_t n, int K, const int32_t* idx,
                           int64_t n_idx, int32_t* status) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (labels && i < n) {
    const int32_t c = labels[i];
    if (c < 0 || c >= K) atomicExch(status, 1);
  }
  if (idx && i < n_idx) {
    const int32_t s = idx[i];
    if (s < 0 || (int64_t)s >= n) atomicExch(status, 1);
  }
}

// Routes rows through every tree (bin rule of scoring). A CTA takes a tile of
// rows, mostly into shared memory; its warps are RB blocks of 32 rows x WT lanes
// of trees: a lane walks one row down trees w, w + WT, ... of each chunk of
// kPredTrees, its leaf ids meeting in shared memory, from which one thread per
// row counts the votes (or adds the leaf values in tree order). Bound by the
// descents' dependent loads (100,000 rows x 32 through 64 trees of depth 8:
// 0.30 ms; one thread per row from global memory, with too few warps, 2.40).
// Features are read 16 bytes at a time (VEC) where d and X's address allow.
//
// F words of a row and of a direction are loaded before any is used, since
// wide rows leave few warps per SM to hide a load behind (ms for 100,000 rows,
// depth 6, left to the compiler and now: 601 features, 4 trees 2.43 and 1.12;
// 680, 2 trees 1.32 and 0.68; 161, 64 trees 5.52 and 3.54; only 400 features
// with 64 trees lost, 5.91 and 6.13). Up to 128 features of 16-byte rows
// (F = 1) there are warps enough and registers count: the loop is the
// compiler's, and its rows' addresses are kept generic (64 features, 64 trees:
// 1.39 ms; 1.44 through shared addresses, 1.53 two words at a time).
// ROWS: where the rows are read. MINB: CTAs per SM that the registers allow.
enum PredRows { kShared, kDirect, kGeneric };
constexpr int kPredTrees = 64;
constexpr int kPredSmem = 96 * 1024;  // rows kept in shared memory up to this

__host__ __device__ inline int pred_stride(int d, bool vec) { return vec ? d + 4 : d | 1; }

template <bool VEC, int F, int ROWS, int MINB>
__global__ void __launch_bounds__(256, MINB)
    k_predict(const float* __restrict__ X, int64_t n, int d, TreeArrays tr, int n_trees, int H,
              int B, int K, int crit, int32_t* class_out, double* value_out, int32_t* leaf_out,
              int RB, int WT, int staged) {
  extern __shared__ __align__(16) float psm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rb = warp % RB, wt = warp / RB, R = 32 * RB;
  const int nct = min(n_trees, kPredTrees);
  int32_t* leaf = reinterpret_cast<int32_t*>(psm);  // [R][nct | 1]
  const int ls = nct | 1;
  float* rows = psm + ((R * ls + 3) & ~3);
  const int stride = pred_stride(d, VEC);
  const int64_t r0 = (int64_t)blockIdx.x * R;
  const int nr = (int)min((int64_t)R, n - r0);
  if (ROWS == kShared || (ROWS == kGeneric && staged)) {
    // every word of the tile on its way at once
    const int w = VEC ? d >> 2 : d, step_r = (int)blockDim.x / w,
              step_c = (int)blockDim.x - step_r * w;
    int r = (int)threadIdx.x / w, c = (int)threadIdx.x - r * w;
    while (r < nr) {
      const float* src = X + (r0 + r) * d + (VEC ? 4 * c : c);
      const uint32_t dst =
          (uint32_t)__cvta_generic_to_shared(rows + r * stride + (VEC ? 4 * c : c));
      if (VEC)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
      else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src));
      r += step_r;
      c += step_c;
      if (c >= w) {
        c -= w;
        ++r;
      }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
  }
  const int rl = rb * 32 + lane;  // this lane's row of the tile
  const bool in = rl < nr;
  const float* x = ROWS == kShared || (ROWS == kGeneric && staged)
                       ? rows + rl * stride
                       : X + (r0 + (in ? rl : 0)) * d;
  const bool tail = (int)threadIdx.x < nr;  // this thread sums up row threadIdx.x
  // x . g as one fmaf per feature in increasing order from +0
  auto dot = [&](const float* __restrict__ g) {
    float acc = 0.0f;
    if constexpr (F == 1) {
#pragma unroll 4
      for (int j = 0; j < d; j += 4) {
        const float4 a = *reinterpret_cast<const float4*>(x + j);
        const float4 b = __ldg(reinterpret_cast<const float4*>(g + j));
        acc = fmaf(a.x, b.x, acc);
        acc = fmaf(a.y, b.y, acc);
        acc = fmaf(a.z, b.z, acc);
        acc = fmaf(a.w, b.w, acc);
      }
    } else {
      using T = std::conditional_t<VEC, float4, float>;
      const T* xv = reinterpret_cast<const T*>(x);
      const T* gv = reinterpret_cast<const T*>(g);
      const int w = VEC ? d >> 2 : d;
      auto ld = [&](int j) { return ROWS == kDirect ? __ldg(xv + j) : xv[j]; };
      auto add = [&](const T& a, const T& b) {
        if constexpr (VEC) {
          acc = fmaf(a.x, b.x, acc);
          acc = fmaf(a.y, b.y, acc);
          acc = fmaf(a.z, b.z, acc);
          acc = fmaf(a.w, b.w, acc);
        } else {
          acc = fmaf(a, b, acc);
        }
      };
      int j = 0;
      for (; j + F <= w; j += F) {
        T a[F], b[F];
#pragma unroll
        for (int i = 0; i < F; ++i) {
          a[i] = ld(j + i);
          b[i] = __ldg(gv + j + i);
        }
#pragma unroll
        for (int i = 0; i < F; ++i) add(a[i], b[i]);
      }
      for (; j < w; ++j) add(ld(j), __ldg(gv + j));
    }
    return acc;
  };
  int votes[kMaxClasses];
  for (int k = 0; k < kMaxClasses; ++k) votes[k] = 0;
  double vsum = 0.0;
  for (int t0 = 0; t0 < n_trees; t0 += kPredTrees) {
    const int nt = min(kPredTrees, n_trees - t0);
    if (in)
      for (int t = wt; t < nt; t += WT) {
        const int64_t base = (int64_t)(t0 + t) * H;
        int h = 0;
        while (h < H && __ldg(tr.kind + base + h) == 1) {
          const int64_t slot = base + h;
          const float* g = tr.dir + slot * d;
          const float zmin = __ldg(tr.zmin + slot), inv_w = __ldg(tr.inv_w + slot);
          const int eb = __ldg(tr.bin + slot);
          const float acc = dot(g);
          h = bin_of(acc, zmin, inv_w, B) >= eb ? 2 * h + 2 : 2 * h + 1;
        }
        leaf[rl * ls + t] = h;
      }
    __syncthreads();
    if (leaf_out)
      for (int q = threadIdx.x; q < nr * nt; q += blockDim.x) {
        const int r = q / nt, t = q - r * nt;
        leaf_out[(r0 + r) * n_trees + t0 + t] = leaf[r * ls + t];
      }
    if (tail) {
      const int32_t* lf = leaf + threadIdx.x * ls;
#pragma unroll 4
      for (int t = 0; t < nt; ++t) {
        const int64_t slot = (int64_t)(t0 + t) * H + lf[t];
        if (crit == SLM_MSE)
          vsum += __ldg(tr.leaf_value + slot);
        else
          votes[__ldg(tr.leaf_class + slot)] += 1;
      }
    }
    __syncthreads();  // the leaf ids are read
  }
  if (!tail) return;
  const int64_t s = r0 + threadIdx.x;
  if (crit == SLM_MSE) {
    if (value_out) value_out[s] = vsum / (double)n_trees;
    if (class_out) class_out[s] = -1;
  } else {
    int best = 0;
    for (int k = 1; k < K; ++k)
      if (votes[k] > votes[best]) best = k;
    if (class_out) class_out[s] = best;
    if (value_out) value_out[s] = (double)best;
  }
}


// ---- feature pre-screen (Sec. III-B, Algorithm 2) --------------------------------

// pos[a][p][j] = 1 if p == j else 0: particle k of every node is the unit
// vector e_k (its projection is feature k itself).
__global__ void k_unit_positions(float* pos, int A, int Pp, int d) {
  const int64_t total = (int64_t)A * Pp * d;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t pj = i % ((int64_t)Pp * d);
    pos[i] = (pj / d == pj % d) ? 1.0f : 0.0f;
  }
}

// zmm[i] = (INT_MAX, INT_MIN): empty ordered-int ranges.
__global__ void k_range_reset(int32_t* zmm, int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    zmm[2 * i] = INT_MAX;
    zmm[2 * i + 1] = INT_MIN;
  }
}

// Xs[e][j] = X[e][feat[a][j]] for the rows of each tile of node a.
__global__ void k_gather_cols(const float* __restrict__ X, int d,
                              const int32_t* __restrict__ feat, int n,
                              const WorkTile* __restrict__ tiles, float* Xs) {
  const WorkTile wt = tiles[blockIdx.x];
  const int32_t* f = feat + (int64_t)wt.node * n;
  for (int i = threadIdx.x; i < wt.rows * n; i += blockDim.x) {
    const int r = i / n, j = i - r * n;
    const int64_t e = (int64_t)wt.row0 + r;
    Xs[e * n + j] = X[e * d + f[j]];
  }
}

// gfull[a][k] = gs[a][j] where feat[a][j] = k, else 0.
__global__ void k_lift(const float* __restrict__ gs, const int32_t* __restrict__ feat, int n,
                       int d, float* gfull) {
  const int a = blockIdx.x;
  for (int k = threadIdx.x; k < d; k += blockDim.x) gfull[(int64_t)a * d + k] = 0.0f;
  __syncthreads();
  for (int j = threadIdx.x; j < n; j += blockDim.x)
    gfull[(int64_t)a * d + feat[(int64_t)a * n + j]] = gs[(int64_t)a * n + j];
}

}  // namespace

cudaError_t launch_node_stats(const Problem& pr, const LevelNode* nodes, int L,
                              const WorkTile* tiles, int n_tiles, const int32_t* tile0,
                              LevelAcc acc, TreeArrays tr, int max_depth, double* par,
                              int32_t* splittable, cudaStream_t st) {
  if (L <= 0) return cudaSuccess;
  if (n_tiles > 0) k_stats_tiles<<<n_tiles, kTT, 0, st>>>(pr, tiles, acc);
  cudaError_t e = cudaGetLastError();
  if (e) return e;
  k_stats_finish<<<(L + kNodeWarps - 1) / kNodeWarps, 32 * kNodeWarps, 0, st>>>(pr, nodes, tile0, L, acc, tr, max_depth,
                                                  par, splittable);
  return cudaGetLastError();
}

cudaError_t launch_partition(const Problem& pr, const Swarm& sw, const WorkTile* tiles,
                             int n_tiles, uint8_t* side, int32_t* tile_left, PartAcc acc,
                             cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  k_part_tiles<<<n_tiles, kTT, sizeof(float) * pr.d, st>>>(pr, sw, tiles, side, tile_left,
                                                            acc);
  return cudaGetLastError();
}

cudaError_t launch_decide(const Problem& pr, const Swarm& sw, const NodeDesc* snodes,
                          const int32_t* map, const int32_t* tile0, int A,
                          const int32_t* tile_left, int32_t* tile_base,
                          const unsigned long long* node_cls, const double* par,
                          PartAcc acc, TreeArrays tr, int32_t* out3, int32_t* status,
                          cudaStream_t st) {
  if (A <= 0) return cudaSuccess;
  k_decide<<<(A + kNodeWarps - 1) / kNodeWarps, 32 * kNodeWarps, 0, st>>>(pr, sw, snodes, map, tile0, A, tile_left,
                                            tile_base, node_cls, par, acc, tr, out3, status);
  return cudaGetLastError();
}

cudaError_t launch_scatter(const Problem& pr, const WorkTile* tiles, int n_tiles,
                           const uint8_t* side, const int32_t* dst, const int32_t* tile_base,
                           const int32_t* tile0, const int32_t* idx_cur, LevelArrays next,
                           cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  k_scatter<<<n_tiles, kTT, 0, st>>>(pr, tiles, side, dst, tile_base, tile0, idx_cur, next);
  return cudaGetLastError();
}

cudaError_t launch_compact_nonzero(const uint32_t* w_all, int n_trees, int64_t n,
                                   int32_t* idx_out, uint32_t* w_out, const int64_t* off,
                                   int32_t* counts, cudaStream_t st) {
  if (n_trees <= 0) return cudaSuccess;
  k_compact_nonzero<<<n_trees, kTT, 0, st>>>(w_all, n, idx_out, w_out, off, counts);
  return cudaGetLastError();
}

cudaError_t launch_gather(const float* X, const int32_t* labels, const float* y,
                          const int32_t* idx, int64_t E, int d, float* Xl, int32_t* lab_l,
                          float* y_l, cudaStream_t st) {
  const int64_t total = E * d;
  if (total <= 0) return cudaSuccess;
  // Fewer entries a CTA (a multiple of 4: rows stay on 16 bytes) while that
  // fills more SMs, down to about two words a thread: 1,000 rows x 1000 on four
  // CTAs added 20 us to a scoring call of 157.
  int R = kTT;
  while (R > 4 && (E + R - 1) / R < 2 * sm_count() && (int64_t)R * d > 2 * kTT) R /= 2;
  k_gather<<<(unsigned)((E + R - 1) / R), kTT, 0, st>>>(X, labels, y, idx, E, d, Xl, lab_l, y_l,
                                                       R);
  return cudaGetLastError();
}

cudaError_t launch_iota(int32_t* idx, int64_t n, int64_t stride, int copies,
                        cudaStream_t st) {
  const int64_t total = n * copies;
  if (total <= 0) return cudaSuccess;
  k_iota<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(idx, n, stride, copies);
  return cudaGetLastError();
}

cudaError_t launch_validate(const int32_t* labels, int64_t n, int K, const int32_t* idx,
                            int64_t n_idx, int32_t* status, cudaStream_t st) {
  const int64_t m = (labels && n > n_idx) ? n : n_idx;
  if (m <= 0) return cudaSuccess;
  k_validate<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(labels, n, K, idx, n_idx, status);
  return cudaGetLastError();
}

cudaError_t launch_predict(const float* X, int64_t n, int d, TreeArrays tr, int n_trees,
                           int H, int B, int K, int crit, int32_t* class_out,
                           double* value_out, int32_t* leaf_out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const bool vec = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  // as many warps over a tile's trees as there are trees, up to eight; the
  // rest take more rows, as far as they fit
  int WT = 1;
  while (WT < 8 && WT < n_trees) WT *= 2;
  int RB = 8 / WT;
  const int ls = (n_trees < kPredTrees ? n_trees : kPredTrees) | 1;
  auto smem = [&](int rb, bool staged) {
    return sizeof(float) * ((size_t)((32 * rb * ls + 3) & ~3) +
                            (staged ? (size_t)32 * rb * pred_stride(d, vec) : 0));
  };
  while (RB > 1 && smem(RB, true) > 48 * 1024) RB /= 2;
  // few rows: smaller tiles, on more SMs
  const int n_sm = sm_count();
  while (RB > 1 && (n + 32 * RB - 1) / (32 * RB) < n_sm) RB /= 2;
  // Rows are staged while 32 of them fit. A single tree walks a row about
  // once per level and gains little: in batches of more tiles than the SMs hold
  // its wide rows are read where they are (100,000 rows, staged and direct: 200
  // features 0.17 and 0.16 ms, 512 0.45 to 0.76 and 0.45, 601 2.4 and 0.75; but
  // 128 0.12 and 0.16, 5,000 rows of 601 0.16 and 0.28).
  const bool few = (n + 31) / 32 <= n_sm * (int64_t)(227 * 1024 / smem(1, true));
  const size_t most = few || n_trees > 1 ? (size_t)kPredSmem : (size_t)(vec ? 24 : 56) * 1024;
  const bool staged = smem(1, true) <= most;
  const size_t sm = smem(RB, staged);
  auto* f = !vec ? (staged ? k_predict<false, 8, kShared, 8> : k_predict<false, 8, kDirect, 6>)
            : d <= 128 ? k_predict<true, 1, kGeneric, 0>
            : staged   ? k_predict<true, 4, kShared, 5>
                       : k_predict<true, 2, kDirect, 6>;
  if (sm > 48 * 1024)
    if (cudaError_t e = allow_smem((const void*)f, (int)sm)) return e;
  f<<<(unsigned)((n + 32 * RB - 1) / (32 * RB)), 32 * RB * WT, sm, st>>>(
      X, n, d, tr, n_trees, H, B, K, crit, class_out, value_out, leaf_out, RB, WT, staged);
  return cudaGetLastError();
}

cudaError_t launch_unit_positions(float* pos, int A, int Pp, int d, cudaStream_t st) {
  const int64_t total = (int64_t)A * Pp * d;
  if (total <= 0) return cudaSuccess;
  const int64_t blocks = (total + 255) / 256;
  k_unit_positions<<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, st>>>(pos, A, Pp, d);
  return cudaGetLastError();
}

cudaError_t launch_range_reset(int32_t* zmm, int64_t count, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  const int64_t blocks = (count + 255) / 256;
  k_range_reset<<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, st>>>(zmm, count);
  return cudaGetLastError();
}

cudaError_t launch_gather_cols(const float* X, int d, const int32_t* feat, int n,
                               const WorkTile* tiles, int n_tiles, float* Xs, cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  k_gather_cols<<<(unsigned)n_tiles, 256, 0, st>>>(X, d, feat, n, tiles, Xs);
  return cudaGetLastError();
}

cudaError_t launch_lift(const float* gs, const int32_t* feat, int A, int n, int d, float* gfull,
                        cudaStream_t st) {
  if (A <= 0) return cudaSuccess;
  k_lift<<<(unsigned)A, 256, 0, st>>>(gs, feat, n, d, gfull);
  return cudaGetLastError();
}

// ---- SLR Boost: the boosting rounds' elementwise steps --------------------------

namespace {

// A sum over n values in a fixed order, whatever the GPU: chain c of 1024
// adds values c, c + 1024, ... in turn, a shuffle tree adds the 32 chains of a
// group and another the 32 groups. Each group is a CTA of one warp (the
// double-precision lanes of 32 SMs instead of one); k_sum_finish adds the
// groups.
constexpr int kSumChains = 1024;
enum SumOf { kSumF, kSumSqDiff, kSumD };

template <int OF>
__global__ void __launch_bounds__(32)
    k_sum_part(const float* __restrict__ y, const float* __restrict__ F,
               const double* __restrict__ v, int64_t n, double* part) {
  double s = 0.0;
#pragma unroll 8
  for (int64_t i = blockIdx.x * 32 + threadIdx.x; i < n; i += kSumChains) {
    if (OF == kSumF) s += (double)y[i];
    if (OF == kSumD) s += v[i];
    if (OF == kSumSqDiff) {
      const double di = (double)y[i] - (double)F[i];
      s += di * di;
    }
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// The mean of n values from their groups' sums, as double and / or float.
__global__ void __launch_bounds__(32)
    k_sum_finish(const double* __restrict__ part, int64_t n, double* out, float* fout) {
  double s = part[threadIdx.x];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if (threadIdx.x == 0) {
    if (out) *out = s / (double)n;
    if (fout) *fout = (float)(s / (double)n);
  }
}

// F[i] = *base.
__global__ void k_boost_init(float* F, const float* __restrict__ base, int64_t n) {
  const float b = *base;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    F[i] = b;
}

__global__ void k_boost_residual(const float* __restrict__ y, const float* __restrict__ F,
                                 float* r, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    r[i] = __fsub_rn(y[i], F[i]);
}

// F[i*K + k] += eta * (float)v_i, one rounding per operation.
__global__ void k_boost_update(float* F, const double* __restrict__ v, float eta, int64_t n,
                               int K, int k) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    F[i * K + k] = __fadd_rn(F[i * K + k], __fmul_rn(eta, (float)v[i]));
}

// Softmax of one row of K scores in double: its maximum and the sum of
// exp(F_k - max) over k ascending.
__device__ __forceinline__ void softmax_row(const float* f, int K, double* mx, double* s) {
  double m = (double)f[0];
  for (int k = 1; k < K; ++k) m = (double)f[k] > m ? (double)f[k] : m;
  double t = 0.0;
  for (int k = 0; k < K; ++k) t += exp((double)f[k] - m);
  *mx = m;
  *s = t;
}

// R[k*n + i] = (float)([labels_i == k] - p_ik), p the softmax of F's row i.
__global__ void k_softmax_residual(const float* __restrict__ F, const int32_t* __restrict__ lab,
                                   int64_t n, int K, float* R) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float* f = F + i * K;
    double mx, sum;
    softmax_row(f, K, &mx, &sum);
    const int y = lab[i];
    for (int k = 0; k < K; ++k)
      R[(int64_t)k * n + i] = (float)((y == k ? 1.0 : 0.0) - exp((double)f[k] - mx) / sum);
  }
}

// v[i] = -log p_{i, labels_i} (log-sum-exp form) in double.
__global__ void k_boost_ce(const float* __restrict__ F, const int32_t* __restrict__ lab, int64_t n,
                           int K, double* v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float* f = F + i * K;
    double mx, sum;
    softmax_row(f, K, &mx, &sum);
    v[i] = -(((double)f[lab[i]] - mx) - log(sum));
  }
}

// class_out[i] = argmax over k of F[i*K + k], ties to the lower class.
__global__ void k_argmax_rows(const float* __restrict__ F, int64_t n, int K, int32_t* cls) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float* f = F + i * K;
    int b = 0;
    for (int k = 1; k < K; ++k)
      if (f[k] > f[b]) b = k;
    cls[i] = b;
  }
}

__global__ void k_fill_f(float* F, float v, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    F[i] = v;
}

unsigned elementwise_blocks(int64_t n) {
  const int64_t b = (n + 255) / 256;
  return (unsigned)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

}  // namespace

cudaError_t launch_boost_init(const float* y, int64_t n, float* F, float* base_out, double* part,
                              cudaStream_t st) {
  if (n <= 0) return cudaErrorInvalidValue;
  k_sum_part<kSumF><<<32, 32, 0, st>>>(y, nullptr, nullptr, n, part);
  k_sum_finish<<<1, 32, 0, st>>>(part, n, nullptr, base_out);
  k_boost_init<<<elementwise_blocks(n), 256, 0, st>>>(F, base_out, n);
  return cudaGetLastError();
}

cudaError_t launch_boost_mse(const float* y, const float* F, int64_t n, double* out, double* part,
                             cudaStream_t st) {
  if (n <= 0) return cudaErrorInvalidValue;
  k_sum_part<kSumSqDiff><<<32, 32, 0, st>>>(y, F, nullptr, n, part);
  k_sum_finish<<<1, 32, 0, st>>>(part, n, out, nullptr);
  return cudaGetLastError();
}

cudaError_t launch_boost_residual(const float* y, const float* F, float* r, int64_t n,
                                  cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_boost_residual<<<elementwise_blocks(n), 256, 0, st>>>(y, F, r, n);
  return cudaGetLastError();
}

cudaError_t launch_boost_update(float* F, const double* v, float eta, int64_t n,
                                cudaStream_t st, int K, int k) {
  if (n <= 0) return cudaSuccess;
  k_boost_update<<<elementwise_blocks(n), 256, 0, st>>>(F, v, eta, n, K, k);
  return cudaGetLastError();
}

cudaError_t launch_softmax_residual(const float* F, const int32_t* labels, int64_t n, int K,
                                    float* R, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_softmax_residual<<<elementwise_blocks(n), 256, 0, st>>>(F, labels, n, K, R);
  return cudaGetLastError();
}

cudaError_t launch_boost_ce(const float* F, const int32_t* labels, int64_t n, int K,
                            double* out, double* v, double* part, cudaStream_t st) {
  if (n <= 0) return cudaErrorInvalidValue;
  k_boost_ce<<<elementwise_blocks(n), 256, 0, st>>>(F, labels, n, K, v);
  k_sum_part<kSumD><<<32, 32, 0, st>>>(nullptr, nullptr, v, n, part);
  k_sum_finish<<<1, 32, 0, st>>>(part, n, out, nullptr);
  return cudaGetLastError();
}

cudaError_t launch_argmax_rows(const float* F, int64_t n, int K, int32_t* cls,
                               cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_argmax_rows<<<elementwise_blocks(n), 256, 0, st>>>(F, n, K, cls);
  return cudaGetLastError();
}

cudaError_t launch_fill_f(float* F, float v, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_fill_f<<<elementwise_blocks(n), 256, 0, st>>>(F, v, n);
  return cudaGetLastError();
}

}  // namespace slm
