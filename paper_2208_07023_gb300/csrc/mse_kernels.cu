// Histogram and threshold scan of unweighted regression searches
// (Sec. II-A, Eqs. 3-4 with the squared error): the scores of block_scan_mse,
// bit for bit, at a fraction of its shared-memory atomics and double
// precision.
//
// What bounded the exact histogram (k_hist_mse) was not reading memory: each
// (entry, particle) pair cost seven shared atomics to random banks (about 10
// adds per clock per SM), and each of the B - 1 edges three double-precision
// divisions, on a GPU with two double-precision lanes per clock per SM:
// 5,000 clocks per (node, particle), whatever the node's size. Here:
//
//  1. The histogram holds, per bin, the number of entries and the sum of the
//     centred target rounded to 30 bits (Problem::mq). Both fit two 32-bit
//     counters, so a pair costs two shared atomics; in nodes with long slices
//     every lane has its own copy of a bin (32 copies), and no two lanes of a
//     warp meet in a bank.
//  2. The edge that minimises the squared error maximises
//     G = D^2 / (n_l n_r), D = S_l - n_l S / n (S: sums of the target): the
//     between-children sum of squares. From the rounded sums each edge gets
//     an interval [G_lo, G_hi] that holds its exact G and the rounding of its
//     exact double-precision loss (see mse_interval). An edge whose G_hi is
//     below the largest G_lo cannot be the argmin.
//  3. In a search only a loss strictly below the particle's best so far has
//     any effect (pbest step, and with it the gbest step: gB is never worse
//     than any pbest). When the largest G_hi shows that no edge gets there,
//     the particle is done: its score is recorded as "no improvement"
//     (invalid). Adaptive PSO and the BF16 form compare every particle's
//     score, and the first evaluation sets the bests: there every particle
//     goes on.
//  4. The remaining edges (mostly one) are scored exactly: their left sums
//     of both 64-bit fixed-point moments by a masked pass over the entries (no
//     atomics, order-free), then block_scan_mse's double expression, one lane
//     per edge.
//
// k_mse_hist takes a (node, particle) per cluster of CTAs; k_mse_warp takes
// one per warp, for levels of many small nodes.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <limits.h>

#include <algorithm>
#include <type_traits>

#include "device_util.cuh"
#include "philox.cuh"
#include "scan_util.cuh"
#include "slm_internal.cuh"

namespace slm {
namespace {

// A counter pair of one (bin, copy): word A = entries (12 bits) + 2^12 x the
// sum of the targets' low 9 bits, word B = the sum of their upper 21 bits.
// Up to 2048 entries per copy: 2048 < 2^12, 2048 (2^9 - 1) < 2^20 and
// 2048 (2^21 - 1) < 2^32.
constexpr int kMqCntBits = 12, kMqLoBits = 9;
constexpr int kMqEntries = 2048;
constexpr int kMqOffset = 1 << 29;  // targets are stored as q + 2^29, |q| <= 2^28 + 1
// Entries of a slice for 32 copies (lane l takes every 32nd 16-byte group:
// at most ceil(65000 / 128) 4 + 1 = 2033 entries per copy) and for 8 copies,
// whose merge is cheaper on short slices (at most 1,100 per copy).
constexpr int kMseSlice = 65000;
constexpr int kMseSliceFew = 8192;
constexpr int kMseMaxCluster = 16;
constexpr int kMseWarps = kThreads / 32;
constexpr int kMseGroup = 4;  // edges scored per masked pass
// Slack of G for the double-precision rounding of two losses, in squared
// target units: the loss expression's error is below 2^-49 of the node's
// second moment, which is at most 2^56 n units (|q| <= 2^28).
constexpr float kMseSlack = 2048.0f;

__device__ __forceinline__ int mse_dvec(int d) { return (d + 3) & ~3; }

// The mean of the rounded targets, S / n to within 0.51: a float quotient,
// then one of its exact remainder.
__device__ __forceinline__ long long mse_mean(long long S, uint32_t n) {
  const float fn = (float)n;
  const long long q0 = __float2ll_rn(__fdividef(__ll2float_rn(S), fn));
  const long long r = S - q0 * (long long)n;
  return q0 + __float2ll_rn(__fdividef(__ll2float_rn(r), fn));
}

// [lo, hi] holding G = D^2 / (nl nr) of an edge, in squared units of the
// rounded targets. The sums S_l and S carry at most half a unit per entry
// and mu half a unit per entry more: D is within 1.51 nl of S_l - nl mu; the
// float conversions and products are within 2^-21.
__device__ __forceinline__ void mse_interval(long long sl, uint32_t nl, uint32_t nr, long long mu,
                                             float* lo, float* hi) {
  const float ad = fabsf(__ll2float_rn(sl - (long long)nl * mu));
  const float e = 2.0f * (float)nl + ad * 0x1p-22f;
  const float inv = __fdividef(1.0f, (float)nl * (float)nr);
  const float l = fmaxf(ad - e, 0.0f), h = ad + e;
  *lo = l * l * inv * (1.0f - 0x1p-19f);
  *hi = h * h * inv * (1.0f + 0x1p-19f);
}

// block_scan_mse's loss of one edge: s, q the left sums of both moments.
__device__ __forceinline__ double mse_loss(uint32_t nl, uint32_t nr, long long s, long long q,
                                           long long stot, long long qtot, double f1, double f2) {
  const double sl = (double)s * f1, ql = (double)q * f2;
  const double sr = (double)(stot - s) * f1;
  const double qr = (double)(qtot - q) * f2;
  const double sse_l = ql - sl * sl / (double)nl;
  const double sse_r = qr - sr * sr / (double)nr;
  return (sse_l + sse_r) / (double)(nl + nr);
}

// The G an edge must reach to get below `loss` (rounded down): no edge with
// G_hi + kMseSlack under it can.
__device__ __forceinline__ float mse_needed(const MseNode& nd, double loss, double n) {
  return __double2float_rd((nd.base - loss * n) * nd.inv);
}

struct MseEdge {
  long long s, q;  // left sums of the moments
  uint32_t nl;
  int e;
};

// ---- one (node, particle) per cluster ---------------------------------------------

struct MseScratch {
  uint32_t cnt[kMaxBins];
  long long sq[kMaxBins];
  uint32_t wc[kMseWarps];
  long long ws[kMseWarps];
  uint32_t wlo[kMseWarps], whi[kMseWarps];
  int wn[kMseWarps];
  uint16_t list[kMaxBins];
  // the pass ranks take part in: edges, whether another pass follows
  int dec_n, dec_more, dec_e[kMseGroup];
  unsigned long long acc_s[kMseGroup], acc_q[kMseGroup];
  unsigned int acc_n[kMseGroup];
  EvalRes pb, gb;
  int imp, last;
};

template <int C>
__global__ void __launch_bounds__(kThreads, 3)
    k_mse_hist(Problem pr, Swarm sw, const NodeDesc* __restrict__ nodes,
               const int32_t* __restrict__ list, int t, int do_update) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ MseScratch sc;
  const cg::cluster_group cl = cg::this_cluster();
  pdl_trigger();
  const int S = (int)cl.num_blocks();
  const int rank = (int)cl.block_rank();
  const int a = list ? list[blockIdx.x / S] : (int)blockIdx.x / S;
  const int p = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int B = pr.B, d = pr.d;
  const NodeDesc nd = nodes[a];
  const int dv = mse_dvec(d);
  uint32_t* hA = reinterpret_cast<uint32_t*>(smem);  // [B][C]
  uint32_t* hB = hA + B * C;
  // also the top-k selection's scratch, once the counters are merged
  const int words = max(2 * B * C, (int)((sizeof(EvalRes) + 8) * pr.P / 4));
  float* c1u = reinterpret_cast<float*>(hA + ((words + 3) & ~3));
  float* s2u = c1u + dv;
  float* xrow = s2u + dv;
  float* vrow = xrow + dv;
  float* prow = vrow + dv;
  const bool upd = do_update && rank == 0;
  const bool premove = upd && sw.ic && t < sw.T;
  const bool force = !do_update || t == 0 || sw.apso;

  for (int i = threadIdx.x; i < (2 * B * C) / 4; i += kThreads)
    reinterpret_cast<uint4*>(hA)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (premove) {
    const uint32_t k0 = (uint32_t)sw.co.seed, k1 = (uint32_t)(sw.co.seed >> 32);
    for (int q = threadIdx.x; q < ((d + 3) >> 2); q += kThreads) {
      const U4 r1 = philox4x32_10(nd.uid, (uint32_t)(t + 1), (uint32_t)p,
                                  (uint32_t)q | (kR1 << 24), k0, k1);
      const U4 r2 = philox4x32_10(nd.uid, (uint32_t)(t + 1), (uint32_t)p,
                                  (uint32_t)q | (kR2 << 24), k0, k1);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (4 * q + c < d) {
          c1u[4 * q + c] = __fmul_rn(sw.co.c1, uniform24(r1.v[c]));
          s2u[4 * q + c] = __fmul_rn(sw.co.c2, uniform24(r2.v[c]));
        }
    }
  }
  __syncthreads();  // the zeroed counters, before any binning
  pdl_wait();
  const int64_t ci = (int64_t)a * pr.Pp + p;
  int* zz = sw.zmm + ci * 2;
  const int chunk = ((nd.seg_len + S - 1) / S + 3) & ~3;
  const int r_begin = min(nd.seg_len, rank * chunk);
  const int r_end = min(nd.seg_len, r_begin + chunk);
  const int64_t e0 = nd.seg_start + r_begin;
  const float* zs = sw.z + (int64_t)p * pr.Ez + e0;
  const uint32_t* us = pr.mq + e0;
  const long long* m1 = pr.m1 + e0;
  const long long* m2 = pr.m2 + e0;
  const int n = r_end - r_begin;
  const bool g16 = (e0 & 3) == 0;  // 16-byte loads: groups of four entries
  const int n4 = g16 ? n >> 2 : 0;
  // Two sets of U groups per thread, one on its way while the other is
  // binned (with one set of four a thread waited out a memory round trip
  // every 16 entries: 75 us on 200,000 entries x 64 particles).
  constexpr int U = 2;
  struct Groups {
    float4 z[U];
    uint4 u[U];
  } ga, gc;
  auto load_groups = [&](Groups& q, int g0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int g = g0 + u * kThreads;
      if (g < n4) {
        q.z[u] = __ldcg(reinterpret_cast<const float4*>(zs) + g);
        q.u[u] = __ldg(reinterpret_cast<const uint4*>(us) + g);
      }
    }
  };
  load_groups(ga, threadIdx.x);
  const int64_t prow0 = ci * d;
  float need = 0.0f;
  if (upd) {
    constexpr int kResWords = (int)(sizeof(EvalRes) / 4);
    const int64_t gi = (int64_t)((t + 1) & 1) * sw.n_nodes + a;
    if (threadIdx.x < kResWords)
      cp_async4(reinterpret_cast<uint32_t*>(&sc.pb) + threadIdx.x,
                reinterpret_cast<const uint32_t*>(sw.pb + ci) + threadIdx.x, 4);
    else if (threadIdx.x >= 32 && threadIdx.x < 32 + kResWords && sw.imp)
      cp_async4(reinterpret_cast<uint32_t*>(&sc.gb) + (threadIdx.x - 32),
                reinterpret_cast<const uint32_t*>(sw.gb + gi) + (threadIdx.x - 32), 4);
    for (int j = threadIdx.x; j < d; j += kThreads) {
      cp_async4(xrow + j, sw.pos + prow0 + j, 4);
      if (premove) {
        cp_async4(vrow + j, sw.vel + prow0 + j, 4);
        cp_async4(prow + j, sw.pbest + prow0 + j, 4);
      }
    }
    cp_async_commit();
    if (!force) need = __ldcg(sw.gneed + ci);
  }
  float zmin = 0.f, inv_w = 0.f;
  bool ok = false;
  {
    const int lo_o = __ldcg(zz), hi_o = __ldcg(zz + 1);
    if (lo_o != INT_MAX) {
      const float lo = ord2f(lo_o), hi = ord2f(hi_o);
      inv_w = __fdiv_rn((float)B, __fsub_rn(hi, lo));
      zmin = lo;
      ok = (hi > lo) && isfinite(inv_w);
    }
  }
  // ---- binning of this rank's slice
  if (ok) {
    const int cp = lane & (C - 1);
    auto add = [&](float z, uint32_t u) {
      const int i = bin_of(z, zmin, inv_w, B) * C + cp;
      atomicAdd(hA + i, 1u | ((u & ((1u << kMqLoBits) - 1u)) << kMqCntBits));
      atomicAdd(hB + i, u >> kMqLoBits);
    };
    auto bin_groups = [&](const Groups& q, int g0) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (g0 + u * kThreads >= n4) break;
        add(q.z[u].x, q.u[u].x);
        add(q.z[u].y, q.u[u].y);
        add(q.z[u].z, q.u[u].z);
        add(q.z[u].w, q.u[u].w);
      }
    };
    for (int g0 = threadIdx.x; g0 < n4; g0 += 2 * U * kThreads) {
      load_groups(gc, g0 + U * kThreads);
      bin_groups(ga, g0);
      load_groups(ga, g0 + 2 * U * kThreads);
      bin_groups(gc, g0 + U * kThreads);
    }
    for (int i = (n4 << 2) + (int)threadIdx.x; i < n; i += kThreads)
      add(__ldcg(zs + i), __ldg(us + i));
  }
  __syncthreads();
  // ---- the copies of bin b (thread b) into its count and exact sum; the
  // 16-byte chunks of a bin in a rotated order, so that eight consecutive
  // lanes read distinct banks
  const int b = threadIdx.x;
  uint32_t cnt = 0;
  long long sq = 0;
  if (b < B) {
    uint32_t lo = 0;
    unsigned long long hi = 0;
    const uint4* pa = reinterpret_cast<const uint4*>(hA + b * C);
    const uint4* pb4 = reinterpret_cast<const uint4*>(hB + b * C);
    constexpr int Q = C / 4;
    const int rot = Q == 8 ? lane : lane >> 2;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const uint4 x = pa[(i + rot) & (Q - 1)], y = pb4[(i + rot) & (Q - 1)];
      constexpr uint32_t m = (1u << kMqCntBits) - 1u;
      cnt += (x.x & m) + (x.y & m) + (x.z & m) + (x.w & m);
      lo += (x.x >> kMqCntBits) + (x.y >> kMqCntBits) + (x.z >> kMqCntBits) +
            (x.w >> kMqCntBits);
      hi += (unsigned long long)y.x + y.y;
      hi += (unsigned long long)y.z + y.w;
    }
    sq = (long long)lo + (long long)(hi << kMqLoBits) - (long long)cnt * kMqOffset;
  }
  if (S > 1) {
    if (b < B) {
      sc.cnt[b] = cnt;
      sc.sq[b] = sq;
    }
    cl.sync();  // every rank's bins are complete
    if (rank == 0 && b < B) {
#pragma unroll
      for (int r = 1; r < kMseMaxCluster; ++r)
        if (r < S) {
          cnt += cl.map_shared_rank(sc.cnt, r)[b];
          sq += cl.map_shared_rank(sc.sq, r)[b];
        }
    }
  }
  const MseNode mn = pr.mnode[a];
  EvalRes res = invalid_res();
  // exact scores of the edges in sc.dec_e: this rank's masked sums into rank 0
  auto masked_edges = [&](auto edges, int nc) {
    constexpr int N = decltype(edges)::value;
    int ed[N];
#pragma unroll
    for (int c = 0; c < N; ++c) ed[c] = c < nc ? sc.dec_e[c] : 0;
    unsigned long long as[N] = {}, aq[N] = {};
    uint32_t an[N] = {};
    auto take = [&](float z, long long v1, long long v2) {
      const int bz = bin_of(z, zmin, inv_w, B);
#pragma unroll
      for (int c = 0; c < N; ++c)
        if (bz < ed[c]) {
          as[c] += (unsigned long long)v1;
          aq[c] += (unsigned long long)v2;
          an[c] += 1u;
        }
    };
    if (ok) {
#pragma unroll 2
      for (int g = threadIdx.x; g < n4; g += kThreads) {
        const float4 z4 = __ldcg(reinterpret_cast<const float4*>(zs) + g);
        const longlong2 a0 = __ldg(reinterpret_cast<const longlong2*>(m1) + 2 * g);
        const longlong2 a1 = __ldg(reinterpret_cast<const longlong2*>(m1) + 2 * g + 1);
        const longlong2 b0 = __ldg(reinterpret_cast<const longlong2*>(m2) + 2 * g);
        const longlong2 b1 = __ldg(reinterpret_cast<const longlong2*>(m2) + 2 * g + 1);
        take(z4.x, a0.x, b0.x);
        take(z4.y, a0.y, b0.y);
        take(z4.z, a1.x, b1.x);
        take(z4.w, a1.y, b1.y);
      }
      for (int i = (n4 << 2) + (int)threadIdx.x; i < n; i += kThreads)
        take(__ldcg(zs + i), __ldg(m1 + i), __ldg(m2 + i));
    }
    unsigned long long* ds = S > 1 ? cl.map_shared_rank(sc.acc_s, 0) : sc.acc_s;
    unsigned long long* dq = S > 1 ? cl.map_shared_rank(sc.acc_q, 0) : sc.acc_q;
    unsigned int* dn = S > 1 ? cl.map_shared_rank(sc.acc_n, 0) : sc.acc_n;
#pragma unroll
    for (int c = 0; c < N; ++c) {
      if (c >= nc) break;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        as[c] += __shfl_xor_sync(0xffffffffu, as[c], off);
        aq[c] += __shfl_xor_sync(0xffffffffu, aq[c], off);
      }
      an[c] = __reduce_add_sync(0xffffffffu, an[c]);
      if (lane == 0) {
        atomicAdd(ds + c, as[c]);
        atomicAdd(dq + c, aq[c]);
        atomicAdd(dn + c, an[c]);
      }
    }
  };
  auto masked_pass = [&](int nc) {  // (mostly one edge)
    if (nc == 1)
      masked_edges(std::integral_constant<int, 1>{}, 1);
    else
      masked_edges(std::integral_constant<int, kMseGroup>{}, nc);
  };
  auto all_sync = [&] {
    if (S > 1)
      cl.sync();
    else
      __syncthreads();
  };
  if (rank != 0) {
    for (;;) {
      cl.sync();  // rank 0 has read this rank's bins and set the edges to score
      const int nc = sc.dec_n, more = sc.dec_more;
      if (nc == 0) return;
      masked_pass(nc);
      cl.sync();  // the sums are in rank 0
      if (!more) return;
    }
  }

  // ---- rank 0: prefix sums, the edges' intervals, the edges left
  uint32_t nl = cnt;
  long long sl = sq;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t uc = __shfl_up_sync(0xffffffffu, nl, off);
    const long long us2 = __shfl_up_sync(0xffffffffu, sl, off);
    if (lane >= off) {
      nl += uc;
      sl += us2;
    }
  }
  if (lane == 31) {
    sc.wc[warp] = nl;
    sc.ws[warp] = sl;
  }
  __syncthreads();
  uint32_t ntot = 0;
  long long stot = 0;
#pragma unroll
  for (int w = 0; w < kMseWarps; ++w) {
    const uint32_t c = sc.wc[w];
    const long long s = sc.ws[w];
    if (w < warp) {
      nl += c;
      sl += s;
    }
    ntot += c;
    stot += s;
  }
  const uint32_t nr = ntot - nl;
  const bool valid = ok && b <= B - 2 && cnt != 0 && nl >= (uint32_t)pr.min_leaf &&
                     nr >= (uint32_t)pr.min_leaf && nr > 0;
  float glo = 0.0f, ghi = 0.0f;
  if (valid) mse_interval(sl, nl, nr, mse_mean(stot, ntot), &glo, &ghi);
  {
    // (non-negative floats order like their bit patterns)
    const uint32_t ml = __reduce_max_sync(0xffffffffu, __float_as_uint(glo));
    const uint32_t mh = __reduce_max_sync(0xffffffffu, valid ? __float_as_uint(ghi) + 1u : 0u);
    if (lane == 0) {
      sc.wlo[warp] = ml;
      sc.whi[warp] = mh;
    }
  }
  __syncthreads();
  uint32_t mlo = 0, mhi = 0;
#pragma unroll
  for (int w = 0; w < kMseWarps; ++w) {
    mlo = max(mlo, sc.wlo[w]);
    mhi = max(mhi, sc.whi[w]);
  }
  // (mhi = 0: no admissible edge)
  const bool go = mhi != 0 && (force || mn.full ||
                               !(__uint_as_float(mhi - 1u) + kMseSlack < need));
  int ncand = 0;
  {
    bool cand = go && valid && (mn.full || ghi + kMseSlack >= __uint_as_float(mlo));
    const unsigned bal = __ballot_sync(0xffffffffu, cand);
    if (lane == 0) sc.wn[warp] = __popc(bal);
    __syncthreads();
    int before = 0;
#pragma unroll
    for (int w = 0; w < kMseWarps; ++w) {
      if (w < warp) before += sc.wn[w];
      ncand += sc.wn[w];
    }
    if (cand) sc.list[before + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(b + 1);
    // constant targets: every loss is exactly zero and the lowest edge wins
    if (mn.flat && ncand > 1) ncand = 1;
    __syncthreads();
  }
  // ---- exact scores, kMseGroup edges a pass, in increasing edge order
  double best = 0.0;
  int bb = -1;
  uint32_t bnl = 0;
  for (int c0 = 0;; c0 += kMseGroup) {
    const int nc = min(kMseGroup, ncand - c0);
    const int more = c0 + kMseGroup < ncand;
    if (threadIdx.x < S) {  // into every rank's shared memory
      MseScratch* o = S > 1 ? cl.map_shared_rank(&sc, (int)threadIdx.x) : &sc;
      o->dec_n = nc;
      o->dec_more = more;
      for (int c = 0; c < nc; ++c) o->dec_e[c] = sc.list[c0 + c];
    }
    if (threadIdx.x >= 32 && threadIdx.x < 32 + kMseGroup) {
      sc.acc_s[threadIdx.x - 32] = 0ull;
      sc.acc_q[threadIdx.x - 32] = 0ull;
      sc.acc_n[threadIdx.x - 32] = 0u;
    }
    all_sync();
    if (nc <= 0) break;
    masked_pass(nc);
    all_sync();
    if (warp == 0) {
      const bool in = lane < nc;
      double l = 0.0;
      uint32_t cn = 0;
      int ce = -1;
      if (in) {
        cn = sc.acc_n[lane];
        ce = sc.dec_e[lane];
        l = mse_loss(cn, ntot - cn, (long long)sc.acc_s[lane], (long long)sc.acc_q[lane], mn.S,
                     mn.Q, pr.mscale[2 * a], pr.mscale[2 * a + 1]);
      }
      // lanes in edge order: a later edge wins only by a smaller loss
      for (int c = 0; c < nc; ++c) {
        const double ol = __shfl_sync(0xffffffffu, l, c);
        const int oe = __shfl_sync(0xffffffffu, ce, c);
        const uint32_t on = __shfl_sync(0xffffffffu, cn, c);
        if (bb < 0 || ol < best) {
          best = ol;
          bb = oe;
          bnl = on;
        }
      }
    }
    if (!more) break;
    __syncthreads();  // the pass's sums and edges are read
  }
  cp_async_wait<0>();  // the tail's prefetched inputs
  __syncthreads();

  // ---- score, range reset, pbest step, the next move's gB-independent terms
  if (threadIdx.x == 0) {
    if (bb >= 0) {
      res.valid = 1;
      res.bin = bb;
      res.nl = bnl;
      res.nr = ntot - bnl;
      res.loss = best;
    }
    if (ok) {
      res.zmin = zmin;
      res.inv_w = inv_w;
    }
    store_score(sw, ci, res);
    zz[0] = INT_MAX;  // ready for the next iteration
    zz[1] = INT_MIN;
    int imp = 0;
    if (do_update) {
      if (sw.imp && res.valid && (t == 0 || better(res, sc.gb, pr.crit)))
        atomicOr(sw.imp + (int64_t)(t & 1) * sw.n_nodes + a, 1);
      imp = (t == 0) || better(res, sc.pb, pr.crit);
      if (imp) {
        sw.pb[ci] = res;
        sw.gneed[ci] = res.valid ? mse_needed(mn, res.loss, (double)ntot)
                                 : __int_as_float(0xff800000);  // -inf: any edge improves
      }
    }
    sc.imp = imp;
  }
  if (sw.tk_sel) {
    // the reduced pass of the BF16 form: the last CTA of the node to score
    // its particle selects the node's top k (the counters are free by now)
    __threadfence();  // this CTA's score write before the count
    __syncthreads();
    if (threadIdx.x == 0) sc.last = atomicAdd(&sw.done[a], 1) + 1 == pr.P;
    __syncthreads();
    if (sc.last) {
      __threadfence();
      topk_select(pr, sw, a, smem);
      if (threadIdx.x == 0) sw.done[a] = 0;
    }
  }
  if (!do_update) return;
  __syncthreads();
  const bool imp = sc.imp;
  if (imp || premove)
    for (int j = threadIdx.x; j < d; j += kThreads) {
      const float x = xrow[j];
      if (imp) sw.pbest[prow0 + j] = x;  // the position is kept on improvement
      if (premove) {
        // ic = omega v + (c1 r1)(pB - x); pB is x itself after an improvement
        const float pbv = imp ? x : prow[j];
        sw.ic[prow0 + j] = __fadd_rn(__fmul_rn(sw.co.inertia, vrow[j]),
                                     __fmul_rn(c1u[j], __fsub_rn(pbv, x)));
        sw.s2[prow0 + j] = s2u[j];
      }
    }
}

// ---- one (node, particle) per warp -------------------------------------------------

struct MseWarpScratch {
  MseEdge job[kMseWarps][kMseGroup];
  int nc[kMseWarps];
  double best[kMseWarps];
  int bb[kMseWarps];
  uint32_t bnl[kMseWarps];
  int last;
};

// Most bins per lane of the warp scan, and log2 of the bins per lane.
constexpr int kBpl = kMaxBins / 32;
__host__ __device__ inline int mse_bpl_log2(int B) {
  return B <= 32 ? 0 : B <= 64 ? 1 : B <= 128 ? 2 : 3;
}

// Nodes of at most kMqEntries entries: a CTA takes eight particles of a node,
// a warp each; the warp's histogram has one copy. The double-precision
// losses of all eight warps' edges are evaluated together, one lane each (a
// warp-wide double-precision instruction costs the same for one lane as
// for 32).
__global__ void __launch_bounds__(kThreads, 4)
    k_mse_warp(Problem pr, Swarm sw, const NodeDesc* __restrict__ nodes,
               const int32_t* __restrict__ list, int t, int do_update) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ MseWarpScratch sc;
  pdl_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int a = list ? list[blockIdx.x] : (int)blockIdx.x;
  const int p = blockIdx.y * kMseWarps + warp;
  const NodeDesc nd = nodes[a];
  const int B = pr.B;
  const bool force = !do_update || t == 0 || sw.apso;
  // lane l scans bins l bpl .. l bpl + bpl - 1 (bpl a power of two); the
  // lanes' words are an odd stride apart against bank conflicts
  const int sh = mse_bpl_log2(B), bpl = 1 << sh, stride = bpl | 1;
  uint32_t* hA = reinterpret_cast<uint32_t*>(smem) + warp * 64 * stride;
  uint32_t* hB = hA + 32 * stride;
  for (int i = lane; i < 64 * stride; i += 32) hA[i] = 0u;
  __syncwarp();
  pdl_wait();
  const bool in_p = p < pr.P;
  const int64_t ci = (int64_t)a * pr.Pp + p;
  int* zz = sw.zmm + ci * 2;
  float zmin = 0.f, inv_w = 0.f;
  bool ok = false;
  if (in_p) {
    const int lo_o = __ldcg(zz), hi_o = __ldcg(zz + 1);
    if (lo_o != INT_MAX) {
      const float lo = ord2f(lo_o), hi = ord2f(hi_o);
      inv_w = __fdiv_rn((float)B, __fsub_rn(hi, lo));
      zmin = lo;
      ok = (hi > lo) && isfinite(inv_w);
    }
  }
  const float need = in_p && !force ? __ldcg(sw.gneed + ci) : 0.0f;
  const MseNode mn = pr.mnode[a];
  const int n = nd.seg_len;
  const float* zs = sw.z + (int64_t)(in_p ? p : 0) * pr.Ez + nd.seg_start;
  const uint32_t* us = pr.mq + nd.seg_start;
  const long long* m1 = pr.m1 + nd.seg_start;
  const long long* m2 = pr.m2 + nd.seg_start;
  const bool g16 = (nd.seg_start & 3) == 0;
  const int n4 = g16 ? n >> 2 : 0;
  if (ok) {
    auto add = [&](float z, uint32_t u) {
      const int bz = bin_of(z, zmin, inv_w, B);
      const int i = (bz >> sh) * stride + (bz & (bpl - 1));
      atomicAdd(hA + i, 1u | ((u & ((1u << kMqLoBits) - 1u)) << kMqCntBits));
      atomicAdd(hB + i, u >> kMqLoBits);
    };
    constexpr int U = 2;
    struct Groups {
      float4 z[U];
      uint4 u[U];
    } ga, gc;
    auto load = [&](Groups& q, int g0) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int g = g0 + 32 * u;
        if (g < n4) {
          q.z[u] = __ldcg(reinterpret_cast<const float4*>(zs) + g);
          q.u[u] = __ldg(reinterpret_cast<const uint4*>(us) + g);
        }
      }
    };
    auto bin_groups = [&](const Groups& q, int g0) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (g0 + 32 * u >= n4) break;
        add(q.z[u].x, q.u[u].x);
        add(q.z[u].y, q.u[u].y);
        add(q.z[u].z, q.u[u].z);
        add(q.z[u].w, q.u[u].w);
      }
    };
    load(ga, lane);
    for (int g0 = lane; g0 < n4; g0 += 64 * U) {
      load(gc, g0 + 32 * U);
      bin_groups(ga, g0);
      load(ga, g0 + 64 * U);
      bin_groups(gc, g0 + 32 * U);
    }
    for (int i = (n4 << 2) + lane; i < n; i += 32) add(__ldcg(zs + i), __ldg(us + i));
  }
  __syncwarp();
  // ---- prefix sums over the bins, lane l holding bins l bpl .. l bpl + bpl - 1
  uint32_t cv[kBpl];
  uint32_t csum = 0;
  long long ssum = 0, sv[kBpl];
#pragma unroll
  for (int i = 0; i < kBpl; ++i) {
    cv[i] = 0;
    sv[i] = 0;
    if (i < bpl) {
      const uint32_t x = hA[lane * stride + i], y = hB[lane * stride + i];
      cv[i] = x & ((1u << kMqCntBits) - 1u);
      sv[i] = (long long)(x >> kMqCntBits) + ((long long)y << kMqLoBits) -
              (long long)cv[i] * kMqOffset;
      csum += cv[i];
      ssum += sv[i];
    }
  }
  uint32_t nl = csum;
  long long sl = ssum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t uc = __shfl_up_sync(0xffffffffu, nl, off);
    const long long us2 = __shfl_up_sync(0xffffffffu, sl, off);
    if (lane >= off) {
      nl += uc;
      sl += us2;
    }
  }
  const uint32_t ntot = __shfl_sync(0xffffffffu, nl, 31);
  const long long stot = __shfl_sync(0xffffffffu, sl, 31);
  const long long mu = ntot ? mse_mean(stot, ntot) : 0;
  nl -= csum;
  sl -= ssum;
  float gh[kBpl];
  uint32_t mlo = 0, mhi = 0;
#pragma unroll
  for (int i = 0; i < kBpl; ++i) {
    gh[i] = -1.0f;
    if (i < bpl) {
      nl += cv[i];
      sl += sv[i];
      const int b = lane * bpl + i;
      const uint32_t nr = ntot - nl;
      if (b <= B - 2 && cv[i] != 0 && nl >= (uint32_t)pr.min_leaf &&
          nr >= (uint32_t)pr.min_leaf && nr > 0) {
        float glo;
        mse_interval(sl, nl, nr, mu, &glo, &gh[i]);
        mlo = max(mlo, __float_as_uint(glo));
        mhi = max(mhi, __float_as_uint(gh[i]) + 1u);
      }
    }
  }
  mlo = __reduce_max_sync(0xffffffffu, mlo);
  mhi = __reduce_max_sync(0xffffffffu, mhi);
  const bool go = ok && mhi != 0 &&
                  (force || mn.full || !(__uint_as_float(mhi - 1u) + kMseSlack < need));
  // ---- exact scores of the edges left, kMseGroup of every warp a pass:
  // bit i of `mine` = this lane's edge of bin l bpl + i
  uint32_t mine = 0;
  if (go) {
#pragma unroll
    for (int i = 0; i < kBpl; ++i)
      if (i < bpl && gh[i] >= 0.0f && (mn.full || gh[i] + kMseSlack >= __uint_as_float(mlo)))
        mine |= 1u << i;
  }
  if (lane == 0) sc.bb[warp] = -1;
  bool first = true;
  while (__syncthreads_or(mine != 0 && (first || !mn.flat))) {
    // the next edges in increasing order
    int nc = 0, ed[kMseGroup];
#pragma unroll
    for (int c = 0; c < kMseGroup; ++c) {
      ed[c] = 0;
      const unsigned bal = __ballot_sync(0xffffffffu, mine != 0);
      if (bal && (first || !mn.flat) && (c == 0 || !mn.flat)) {
        const int src = __ffs(bal) - 1;
        const int low = __ffs(mine) - 1;
        ed[c] = src * bpl + __shfl_sync(0xffffffffu, low, src) + 1;
        if (lane == src) mine &= mine - 1;
        ++nc;
      }
    }
    auto masked_edges = [&](auto edges) {
      constexpr int N = decltype(edges)::value;
      unsigned long long as[N] = {}, aq[N] = {};
      uint32_t an[N] = {};
      auto take = [&](float z, long long v1, long long v2) {
        const int bz = bin_of(z, zmin, inv_w, B);
#pragma unroll
        for (int c = 0; c < N; ++c)
          if (bz < ed[c]) {
            as[c] += (unsigned long long)v1;
            aq[c] += (unsigned long long)v2;
            an[c] += 1u;
          }
      };
#pragma unroll 1
      for (int g = lane; g < n4; g += 32) {
        const float4 z4 = __ldcg(reinterpret_cast<const float4*>(zs) + g);
        const longlong2 a0 = __ldg(reinterpret_cast<const longlong2*>(m1) + 2 * g);
        const longlong2 a1 = __ldg(reinterpret_cast<const longlong2*>(m1) + 2 * g + 1);
        const longlong2 b0 = __ldg(reinterpret_cast<const longlong2*>(m2) + 2 * g);
        const longlong2 b1 = __ldg(reinterpret_cast<const longlong2*>(m2) + 2 * g + 1);
        take(z4.x, a0.x, b0.x);
        take(z4.y, a0.y, b0.y);
        take(z4.z, a1.x, b1.x);
        take(z4.w, a1.y, b1.y);
      }
      for (int i = (n4 << 2) + lane; i < n; i += 32)
        take(__ldcg(zs + i), __ldg(m1 + i), __ldg(m2 + i));
#pragma unroll
      for (int c = 0; c < N; ++c) {
        if (c >= nc) break;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          as[c] += __shfl_xor_sync(0xffffffffu, as[c], off);
          aq[c] += __shfl_xor_sync(0xffffffffu, aq[c], off);
        }
        an[c] = __reduce_add_sync(0xffffffffu, an[c]);
        if (lane == 0) sc.job[warp][c] = MseEdge{(long long)as[c], (long long)aq[c], an[c], ed[c]};
      }
    };
    if (nc == 1)  // (most often)
      masked_edges(std::integral_constant<int, 1>{});
    else if (nc > 1)
      masked_edges(std::integral_constant<int, kMseGroup>{});
    if (lane == 0) sc.nc[warp] = nc;
    first = false;
    __syncthreads();
    if (warp == 0) {  // lane 4 w + c: edge c of warp w
      const int w = lane >> 2, c = lane & 3;
      const bool in = c < sc.nc[w];
      double l = 0.0;
      MseEdge j{0, 0, 0, -1};
      if (in) {
        j = sc.job[w][c];
        const uint32_t nt = (uint32_t)nd.seg_len;  // unweighted: every entry counts one
        l = mse_loss(j.nl, nt - j.nl, j.s, j.q, mn.S, mn.Q, pr.mscale[2 * a],
                     pr.mscale[2 * a + 1]);
      }
      // lanes in edge order: a later edge wins only by a smaller loss
      double bl = l;
      int be = j.e;
      uint32_t bn = j.nl;
#pragma unroll
      for (int k = 1; k < kMseGroup; ++k) {
        const double ol = __shfl_sync(0xffffffffu, l, (lane & ~3) + k);
        const int oe = __shfl_sync(0xffffffffu, j.e, (lane & ~3) + k);
        const uint32_t on = __shfl_sync(0xffffffffu, j.nl, (lane & ~3) + k);
        if (k < sc.nc[w] && ol < bl) {
          bl = ol;
          be = oe;
          bn = on;
        }
      }
      if (c == 0 && in && (sc.bb[w] < 0 || bl < sc.best[w])) {
        sc.best[w] = bl;
        sc.bb[w] = be;
        sc.bnl[w] = bn;
      }
    }
  }
  __syncthreads();  // the warps' results
  if (in_p) {
    EvalRes res = invalid_res();
    if (sc.bb[warp] >= 0) {
      res.valid = 1;
      res.bin = sc.bb[warp];
      res.nl = sc.bnl[warp];
      res.nr = ntot - sc.bnl[warp];
      res.loss = sc.best[warp];
    }
    if (ok) {
      res.zmin = zmin;
      res.inv_w = inv_w;
    }
    if (lane == 0) {
      store_score(sw, ci, res);
      zz[0] = INT_MAX;  // ready for the next iteration
      zz[1] = INT_MIN;
      if (do_update) mark_improvement(pr, sw, a, t, res);
    }
    if (do_update) {
      if (pbest_step(pr, sw, a, p, t, res) && lane == 0)
        sw.gneed[ci] = res.valid ? mse_needed(mn, res.loss, (double)ntot)
                                 : __int_as_float(0xff800000);  // -inf: any edge improves
      if (sw.ic && t < sw.T) {
        __syncwarp();  // the pbest row the lanes just wrote
        premove_particle(pr, sw, nd.uid, a, t, p);
      }
    }
  }
  if (sw.tk_sel) {
    // the reduced pass of the BF16 form: the node's last CTA selects its top k
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      const int np = min(kMseWarps, pr.P - (int)blockIdx.y * kMseWarps);
      sc.last = atomicAdd(&sw.done[a], np) + np == pr.P;
    }
    __syncthreads();
    if (sc.last) {
      __threadfence();
      topk_select(pr, sw, a, smem);
      if (threadIdx.x == 0) sw.done[a] = 0;
    }
  }
}

size_t topk_bytes(const Problem& pr) { return ((sizeof(EvalRes) + 8) * (size_t)pr.P + 15) & ~(size_t)15; }

size_t mse_hist_smem(const Problem& pr, int C) {
  const size_t counters = std::max(sizeof(uint32_t) * 2 * (size_t)pr.B * C, topk_bytes(pr));
  return counters + sizeof(float) * 5 * (size_t)((pr.d + 3) & ~3);
}

size_t mse_warp_smem(const Problem& pr) {
  const size_t stride = (size_t)(1 << mse_bpl_log2(pr.B)) | 1;
  return std::max(sizeof(uint32_t) * 64 * stride * kMseWarps, topk_bytes(pr));
}

const void* mse_fn(int C) {
  return C == 32 ? (const void*)k_mse_hist<32> : (const void*)k_mse_hist<8>;
}

// Copies per bin for slices of `slice` entries.
int mse_copies_for(int64_t slice) { return slice <= kMseSliceFew ? 8 : 32; }
// Longest slice of a node of max_len entries in S slices (which start on
// multiples of 4).
int64_t mse_launch_slice(int64_t max_len, int S) { return (max_len + S - 1) / S + 4; }

// The fewest slices that a node's counters take.
int64_t mse_min_split(int64_t max_len) {
  return std::max<int64_t>(1, (max_len + kMseSlice - 5) / (kMseSlice - 4));
}
// Clusters of S CTAs of the kernel with C copies that run at once.
int mse_clusters(const Problem& pr, int C, int S) {
  const void* f = mse_fn(C);
  const size_t smem = mse_hist_smem(pr, C);
  int n = 0;
  if (allow_smem(f, (int)smem) || allow_cluster(f) ||
      active_clusters(&n, f, kThreads, smem, S)) {
    (void)cudaGetLastError();
    return S <= 8 ? 1 : 0;  // (8: the portable size)
  }
  return n;
}

}  // namespace

bool mse_lazy_ok(const Problem& pr) {
  return pr.crit == SLM_MSE && !pr.w && pr.mq && pr.mnode && pr.B >= 2 && pr.B <= kMaxBins;
}

int mse_warp_max() { return kMqEntries; }

cudaError_t prepare_mse_lazy(const Problem& pr) {
  for (int C : {8, 32}) {
    if (cudaError_t e = allow_smem(mse_fn(C), (int)mse_hist_smem(pr, C))) return e;
    if (cudaError_t e = allow_cluster(mse_fn(C))) return e;
  }
  return allow_smem((const void*)k_mse_warp, (int)mse_warp_smem(pr));
}

bool mse_lazy_fits(const Problem& pr, int64_t max_len) {
  const int64_t S = mse_min_split(max_len);
  return S <= kMseMaxCluster && mse_clusters(pr, 32, (int)S) > 0;
}

int mse_lazy_split(const Problem& pr, int A, int64_t max_len) {
  // As many slices as one wave of clusters takes, since the last CTA's exact
  // pass ends the launch: as many clusters as the device holds at once (of 7
  // CTAs 59, of 6 74: 64 particles on 80,000 entries, 51 iterations, 2.08 ms
  // with 7 slices and 1.78 with 6). Above 8 CTAs a cluster needs a quarter of
  // them to spare (32 particles on 20,000 entries: 1.14 ms with 12 slices, of
  // which 36 fit, and 0.96 with 9). Slices of at least 1,400 entries, above 8
  // of 2,048; two short ones never pay (4,597 entries, 16 particles: 0.83 ms
  // with 3, 0.88 with 2; 3,732: 0.79 with one, 0.82 with 2).
  const int64_t pairs = (int64_t)A * pr.P;
  const int least = (int)mse_min_split(max_len);
  int S = max_len < 3 * 1400 ? 1 : (int)std::min<int64_t>(8, max_len / 1400);
  S = (int)std::max<int64_t>({least, S, std::min<int64_t>(kMseMaxCluster, max_len / 2048)});
  for (; S > least; --S) {
    const int64_t n = mse_clusters(pr, mse_copies_for(mse_launch_slice(max_len, S)), S);
    if (S > 8 ? 3 * n >= 4 * pairs : n >= pairs) break;
  }
  return S;
}

cudaError_t launch_mse_lazy(const Problem& pr, const Swarm& sw, const NodeDesc* nodes, int A,
                            int64_t max_len, int S, int t, int do_update, cudaStream_t st,
                            const int32_t* list) {
  if (A <= 0) return cudaSuccess;
  if (S < mse_min_split(max_len) || S > kMseMaxCluster) return cudaErrorInvalidValue;
  const int C = mse_copies_for(mse_launch_slice(max_len, S));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(A * S), (unsigned)pr.P, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = mse_hist_smem(pr, C);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  void* args[] = {(void*)&pr, (void*)&sw, (void*)&nodes, (void*)&list, (void*)&t,
                  (void*)&do_update};
  return cudaLaunchKernelExC(&cfg, mse_fn(C), args);
}

cudaError_t launch_mse_warp(const Problem& pr, const Swarm& sw, const NodeDesc* nodes,
                            const int32_t* list, int n_nodes, int t, int do_update,
                            cudaStream_t st) {
  if (n_nodes <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n_nodes, (unsigned)((pr.P + kMseWarps - 1) / kMseWarps), 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = mse_warp_smem(pr);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mse_warp, pr, sw, nodes, list, t, do_update);
}

}  // namespace slm
