// Learned swarm proposal: node statistics, a 3-layer network (bfloat16
// weights, FP32 accumulation), its loss gradient, Adam, and the seeded
// initial swarm.
//
// The network maps a node's statistics s (per-class mean offsets and feature
// variances, padded to 256 features x 20 classes + 1: 5376 inputs) to a
// direction mu (256) and 64 spread radii: h1 = relu(s W1 + b1),
// h2 = relu(h1 W2 + b2), o = h2 W3 + b3. A search seeded by it starts particle
// i at sigma (mu_hat + rho_i u_i / |u_i|) (mu_hat = mu / |mu| over the node's d
// features, rho_i = softplus(o[256 + i]), u_i uniform in [-1, 1)^d from the
// swarm stream), instead of uniformly in [-1, 1)^d (Sec. III-A's "preset
// range"). The paper has no learned proposal; this is a way to start the
// swarm near a good direction.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include "device_util.cuh"
#include "philox.cuh"
#include "slm_internal.cuh"

namespace slm {
namespace {

constexpr int kD = kPropD, kK = kPropK, kIn = kPropIn, kH = kPropH, kP = kPropP, kOut = kPropOut;

// ---- node statistics ------------------------------------------------------------

__global__ void k_stats_yinit(int32_t* yr, int A) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a < A) {
    yr[2 * a] = INT_MAX;
    yr[2 * a + 1] = INT_MIN;
  }
}

// Regression groups: the node's y range (ordered ints) per node.
__global__ void k_stats_yrange(Problem pr, const NodeDesc* __restrict__ nodes, int32_t* yr,
                               int splits) {
  const int a = blockIdx.x;
  const NodeDesc nd = nodes[a];
  int lo = INT_MAX, hi = INT_MIN;
  for (int64_t r = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; r < nd.seg_len;
       r += (int64_t)splits * blockDim.x) {
    const int o = f2ord(pr.y[nd.seg_start + r]);
    lo = min(lo, o);
    hi = max(hi, o);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, off));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, off));
  }
  if ((threadIdx.x & 31) == 0 && lo != INT_MAX) {
    atomicMin(&yr[2 * a], lo);
    atomicMax(&yr[2 * a + 1], hi);
  }
}

// Group of an entry: its class, or (regression) the quarter of the node's y
// range, in float with one rounding per operation.
__device__ __forceinline__ int stat_group(const Problem& pr, int64_t e, const int32_t* yr, int a) {
  if (pr.lab) return pr.lab[e];
  const float lo = ord2f(yr[2 * a]), hi = ord2f(yr[2 * a + 1]);
  if (!(hi > lo)) return 0;
  int g = (int)floorf(__fmul_rn(4.0f, __fdiv_rn(__fsub_rn(pr.y[e], lo), __fsub_rn(hi, lo))));
  return g > 3 ? 3 : (g < 0 ? 0 : g);
}

// Grid (node, 32-feature slice, row split); warp w of a block takes rows w,
// w + 8, ... of its split. Per class: sum w (x - x0); per feature: sum w (x -
// x0), sum w (x - x0)^2, with x0 the node's first row (a shift against
// cancellation). Folded into acc[A][K + 2][d] and wk[A][K] in double.
__global__ void __launch_bounds__(256)
    k_stats_accum(Problem pr, const NodeDesc* __restrict__ nodes, const int32_t* yr, int K,
                  int splits, double* acc, double* wk) {
  __shared__ float s_acc[8][kK + 2][32];
  __shared__ float s_w[8][kK];
  const int a = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const NodeDesc nd = nodes[a];
  const int d = pr.d;
  const int j = blockIdx.y * 32 + lane;
  for (int k = 0; k < K + 2; ++k) s_acc[warp][k][lane] = 0.0f;
  if (lane < K) s_w[warp][lane] = 0.0f;
  __syncwarp();
  const float x0 = (j < d && nd.seg_len > 0) ? pr.X[(int64_t)nd.seg_start * d + j] : 0.0f;
  for (int64_t r = (int64_t)blockIdx.z * 8 + warp; r < nd.seg_len; r += (int64_t)splits * 8) {
    const int64_t e = nd.seg_start + r;
    const float w = pr.w ? (float)pr.w[e] : 1.0f;
    const int g = stat_group(pr, e, yr, a);
    if (j < d) {
      const float t = pr.X[e * d + j] - x0;
      s_acc[warp][g][lane] += w * t;
      s_acc[warp][K][lane] += w * t;
      s_acc[warp][K + 1][lane] += w * t * t;
    }
    if (lane == 0 && blockIdx.y == 0) s_w[warp][g] += w;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < (K + 2) * 32; i += blockDim.x) {
    const int k = i / 32, l = i % 32, jj = blockIdx.y * 32 + l;
    if (jj >= d) continue;
    float s = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += s_acc[w][k][l];
    atomicAdd(&acc[((int64_t)a * (K + 2) + k) * d + jj], (double)s);
  }
  if (blockIdx.y == 0 && threadIdx.x < K) {
    float s = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += s_w[w][threadIdx.x];
    atomicAdd(&wk[(int64_t)a * K + threadIdx.x], (double)s);
  }
}

// stats[a][k*256 + j] = class mean offset, stats[a][20*256 + j] = variance.
__global__ void k_stats_final(int d, int K, const double* __restrict__ acc,
                              const double* __restrict__ wk, float* stats) {
  const int a = blockIdx.x;
  float* st = stats + (int64_t)a * kIn;
  const double* ac = acc + (int64_t)a * (K + 2) * d;
  double W = 0.0;
  for (int k = 0; k < K; ++k) W += wk[(int64_t)a * K + k];
  for (int i = threadIdx.x; i < kIn; i += blockDim.x) {
    const int k = i / kD, j = i % kD;
    float v = 0.0f;
    if (j < d && W > 0.0) {
      const double m = ac[(int64_t)K * d + j] / W;  // shifted mean
      if (k == kK) {
        v = (float)fmax(0.0, ac[(int64_t)(K + 1) * d + j] / W - m * m);
      } else if (k < K) {
        const double wkk = wk[(int64_t)a * K + k];
        v = wkk > 0.0 ? (float)(ac[(int64_t)k * d + j] / wkk - m) : 0.0f;
      }
    }
    st[i] = v;
  }
}

// ---- network ---------------------------------------------------------------------

// What the products do with their sums: nothing, add the bias, add it and
// clip at zero, or keep where the layer's activation was positive (the
// backward of the clip; `aux` = the activations).
enum Epi { kPlain, kBias, kBiasRelu, kReluMask };

template <int EPI>
__device__ __forceinline__ float epilogue(float v, const float* aux, int64_t m, int n, int ldc) {
  if (EPI == kBias || EPI == kBiasRelu) v += aux[n];
  if (EPI == kBiasRelu) v = fmaxf(v, 0.0f);
  if (EPI == kReluMask) v = aux[m * ldc + n] > 0.0f ? v : 0.0f;
  return v;
}

__device__ __forceinline__ float4 ld4(const float* p) {
  return __ldg(reinterpret_cast<const float4*>(p));
}
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                     __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}

// C[M x N] = op(A) op(B). op(A)(m, k) = TA ? A[k lda + m] : A[m lda + k];
// op(B)(k, n) = TB ? B[n ldb + k] : B[k ldb + n]; N, the row strides and the
// untransposed K are multiples of 4. T x T tiles, R x R outputs per thread
// (rows ty + D i, columns tx + D j), KS-deep K steps through two shared-memory
// stages (the next step's 16-byte loads in flight while one computes), each
// operand in shared memory as it lies in memory, so that its 16-byte pieces
// are stored whole: [row][k] where k is contiguous, else [k][row]. Every
// output is one FP32 chain over k in increasing order, whatever the tile, so
// both shapes give the same bits.
// A batch of 64 has eight 64 x 64 tiles in the first layer (K = 5376), which
// took 0.7 ms on eight SMs; 16 x 16 tiles spread it over 128, where the
// chain's own latency (5376 dependent FMAs of 4 clocks: 10 us) is the floor.
template <bool TA, bool TB, typename BT, int EPI, int T, int R, int KS>
__global__ void __launch_bounds__((T / R) * (T / R))
    k_gemm(int M, int N, int K, const float* __restrict__ A, int lda, const BT* __restrict__ B,
           int ldb, const float* __restrict__ aux, float* __restrict__ C, int ldc) {
  constexpr int D = T / R, NT = D * D, NV = T * KS / 4 / NT;
  static_assert(T * KS % (4 * NT) == 0 && KS % 4 == 0, "tile");
  // words of an operand's stage: [k][T + 4] or [T][KS + 4]
  constexpr int SA = TA ? KS * (T + 4) : T * (KS + 4), SB = TB ? T * (KS + 4) : KS * (T + 4);
  __shared__ __align__(16) float As[2][SA], Bs[2][SB];
  const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
  const int tx = threadIdx.x % D, ty = threadIdx.x / D;
  // this thread's 16-byte pieces of a step: 4 along k of one row (kc), or 4
  // along the rows at one k
  auto place = [](bool kc, int v, int* row, int* k) {
    const int id = (int)threadIdx.x + v * NT;
    *row = kc ? id / (KS / 4) : 4 * (id % (T / 4));
    *k = kc ? 4 * (id % (KS / 4)) : id / (T / 4);
  };
  float4 av[NV], bv[NV];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      int r, k;
      place(!TA, v, &r, &k);
      av[v] = make_float4(0, 0, 0, 0);
      if (k0 + k < K && m0 + r < M)
        av[v] = TA ? ld4(A + (int64_t)(k0 + k) * lda + m0 + r)
                   : ld4(A + (int64_t)(m0 + r) * lda + k0 + k);
      place(TB, v, &r, &k);
      bv[v] = make_float4(0, 0, 0, 0);
      if (k0 + k < K && n0 + r < N)
        bv[v] = TB ? ld4(B + (int64_t)(n0 + r) * ldb + k0 + k)
                   : ld4(B + (int64_t)(k0 + k) * ldb + n0 + r);
    }
  };
  auto store = [&](int st) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      int r, k;
      place(!TA, v, &r, &k);
      *reinterpret_cast<float4*>(&As[st][TA ? k * (T + 4) + r : r * (KS + 4) + k]) = av[v];
      place(TB, v, &r, &k);
      *reinterpret_cast<float4*>(&Bs[st][TB ? r * (KS + 4) + k : k * (T + 4) + r]) = bv[v];
    }
  };
  // four consecutive k of this thread's i-th row (of T, at base t + D i)
  auto read = [](const float* s, bool kc, int row, int k, float (&v)[4]) {
    if (kc) {
      const float4 x = *reinterpret_cast<const float4*>(s + row * (KS + 4) + k);
      v[0] = x.x;
      v[1] = x.y;
      v[2] = x.z;
      v[3] = x.w;
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = s[(k + c) * (T + 4) + row];
    }
  };
  float acc[R][R] = {};
  fetch(0);
  store(0);
  __syncthreads();
  int st = 0;
  for (int k0 = 0; k0 < K; k0 += KS, st ^= 1) {
    const bool more = k0 + KS < K;
    if (more) fetch(k0 + KS);
#pragma unroll 4
    for (int kk = 0; kk < KS; kk += 4) {
      float xs[R][4], ys[R][4];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        read(As[st], !TA, ty + D * i, kk, xs[i]);
        read(Bs[st], TB, tx + D * i, kk, ys[i]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < R; ++j) acc[i][j] = fmaf(xs[i][c], ys[j][c], acc[i][j]);
    }
    if (more) store(st ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int m = m0 + ty + D * i;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int n = n0 + tx + D * j;
      if (m < M && n < N) C[(int64_t)m * ldc + n] = epilogue<EPI>(acc[i][j], aux, m, n, ldc);
    }
  }
}

// A layer's forward product on few rows: C[M x N] = A[M x K] B[K x N] (+ bias,
// clipped), 16 x 16 tiles, two adjacent outputs per thread, operands through
// a ring of kFwdStages shared-memory stages of 128 k (asynchronous copies, two
// stages in flight while one computes). K and N are multiples of 16. One FP32
// chain per output over k in increasing order: k_gemm's bits. The chain is
// what bounds it (K = 5376: 5376 dependent FMAs of 4 clocks, 10 us); with
// k_gemm's two register-staged steps of 64 the first layer took 95 us, most
// of it waiting for each step's loads; 33 us now at 64 rows (40 with four k of
// the loop unrolled instead of 128): the loads, conversions and 2 FMAs per k are
// issued by only 4 warps per SM. More stages or operands read further ahead
// change nothing.
constexpr int kFwdK = 128, kFwdStages = 3;
constexpr int kFwdA = 16 * (kFwdK + 4);          // floats: [16 rows][128 k + 4]
constexpr int kFwdBytes = kFwdA * 4 + kFwdK * 16 * 2;  // and [128 k][16 columns] bfloat16

template <int EPI>
__global__ void __launch_bounds__(128)
    k_gemm_fwd(int M, int N, int K, const float* __restrict__ A, const __nv_bfloat16* __restrict__ B,
               const float* __restrict__ bias, float* __restrict__ C) {
  __shared__ __align__(16) unsigned char sm[kFwdStages][kFwdBytes];
  const int m0 = blockIdx.y * 16, n0 = blockIdx.x * 16;
  const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  const int ns = (K + kFwdK - 1) / kFwdK;
  auto stage = [&](int s) {
    if (s < ns) {
      float* a = reinterpret_cast<float*>(sm[s % kFwdStages]);
      unsigned char* b = sm[s % kFwdStages] + kFwdA * 4;
      const int k0 = s * kFwdK, kc = min(kFwdK, K - k0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {  // 16 rows x 32 pieces
        const int id = (int)threadIdx.x + 128 * i, r = id >> 5, k = 4 * (id & 31);
        const bool in = k < kc && m0 + r < M;
        cp_async16(a + r * (kFwdK + 4) + k, in ? A + (int64_t)(m0 + r) * K + k0 + k : A,
                   in ? 16 : 0);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {  // 128 k x 2 pieces
        const int id = (int)threadIdx.x + 128 * i, k = id >> 1, h = id & 1;
        const bool in = k < kc;
        cp_async16(b + k * 32 + 16 * h, in ? B + (int64_t)(k0 + k) * N + n0 + 8 * h : B,
                   in ? 16 : 0);
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < kFwdStages - 1; ++s) stage(s);
  float c0 = 0.0f, c1 = 0.0f;
  for (int s = 0; s < ns; ++s) {
    cp_async_wait<kFwdStages - 2>();
    __syncthreads();  // stage s is in place; every thread is done with s - 1
    stage(s + kFwdStages - 1);
    const float* a = reinterpret_cast<const float*>(sm[s % kFwdStages]) + ty * (kFwdK + 4);
    const uint32_t* b =
        reinterpret_cast<const uint32_t*>(sm[s % kFwdStages] + kFwdA * 4) + tx;
    const int kc = min(kFwdK, K - s * kFwdK);
#pragma unroll 32
    for (int k = 0; k < kc; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(a + k);
      const uint32_t w0 = b[8 * k], w1 = b[8 * k + 8], w2 = b[8 * k + 16], w3 = b[8 * k + 24];
      c0 = fmaf(x.x, __uint_as_float(w0 << 16), c0);
      c1 = fmaf(x.x, __uint_as_float(w0 & 0xffff0000u), c1);
      c0 = fmaf(x.y, __uint_as_float(w1 << 16), c0);
      c1 = fmaf(x.y, __uint_as_float(w1 & 0xffff0000u), c1);
      c0 = fmaf(x.z, __uint_as_float(w2 << 16), c0);
      c1 = fmaf(x.z, __uint_as_float(w2 & 0xffff0000u), c1);
      c0 = fmaf(x.w, __uint_as_float(w3 << 16), c0);
      c1 = fmaf(x.w, __uint_as_float(w3 & 0xffff0000u), c1);
    }
  }
  const int m = m0 + ty, n = n0 + 2 * tx;
  if (m < M)
    *reinterpret_cast<float2*>(C + (int64_t)m * N + n) =
        make_float2(epilogue<EPI>(c0, bias, m, n, N), epilogue<EPI>(c1, bias, m, n + 1, N));
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sh[i];
  return s;
}

// Two sums over the block's threads, each block_sum's (the warps' butterflies,
// then the warps in order); the warps from `active` on hold zeros.
struct Sums2 {
  double v[2][8], s[2];
};
__device__ __forceinline__ double2 block_sum2(double a, double b, int active, Sums2& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < active) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, off);
      b += __shfl_xor_sync(0xffffffffu, b, off);
    }
  }
  if (lane == 0) {
    sh.v[0][warp] = warp < active ? a : 0.0;
    sh.v[1][warp] = warp < active ? b : 0.0;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int i = 0; i < 8; ++i) s += sh.v[threadIdx.x][i];
    sh.s[threadIdx.x] = s;
  }
  __syncthreads();
  return make_double2(sh.s[0], sh.s[1]);
}

// One block (256 threads) per sample r: its loss (added into *loss, already
// divided by N) and dL/do (divided by N) in double. Bound by the double
// pipes (two lanes per clock per SM): the sums run in pairs, added up by one
// warp, and only warps with features of the sample divide (64 samples of 64
// features: 19.6 us with every warp summing and dividing, 14.6 now).
__global__ void __launch_bounds__(256)
    k_mlp_loss(const float* __restrict__ O, const int32_t* __restrict__ dims,
               const float* __restrict__ targets, int N, float* dO, double* loss) {
  __shared__ Sums2 sh0, sh1, sh2;
  const int r = blockIdx.x, j = threadIdx.x;
  const float* o = O + (int64_t)r * kOut;
  const float* a = targets + (int64_t)r * kD;
  const int d = dims[r], wd = (d + 31) >> 5;  // warps with features
  const double oj = j < d ? (double)o[j] : 0.0, aj = j < d ? (double)a[j] : 0.0;
  const double2 cm = block_sum2(oj * aj, oj * oj, wd, sh0);
  const double c = cm.x, mm = cm.y;
  const double q = mm + 1e-12, sg = c >= 0.0 ? 1.0 : -1.0;
  const double nm = sqrt(mm);
  double mh = 0.0, uj = 0.0;
  if (j < d) {
    mh = mm > 0.0 ? oj / nm : 0.0;
    uj = mh - sg * aj;
  }
  const double2 uh = block_sum2(uj * uj, mh * uj, wd, sh1);
  const double delta = mm > 0.0 ? sqrt(uh.x) : 1.0, hu = uh.y;
  // spread: radii i < 64 on threads 0..63
  double pin = 0.0, dld = 0.0;
  if (j < kP) {
    const double tau = (j + 0.5) / kP;
    const double x = (double)o[kD + j];
    const double rho = x > 30.0 ? x : log1p(exp(x));
    const double u = delta - rho;
    pin = u >= 0.0 ? tau * u : (tau - 1.0) * u;
    dld = (u >= 0.0 ? tau : tau - 1.0) / kP;
    const double dl_drho = (u >= 0.0 ? -tau : 1.0 - tau) / kP;
    dO[(int64_t)r * kOut + kD + j] = (float)(dl_drho / (1.0 + exp(-x)) / N);
  }
  const double2 sd = block_sum2(pin, dld, (kP + 31) >> 5, sh2);
  const double spread = sd.x, dl_ddelta = sd.y;
  float g32 = 0.0f;
  if (j < d) {
    double g = -2.0 * c * aj / q + 2.0 * c * c * oj / (q * q);
    if (mm > 0.0 && delta > 0.0) g += dl_ddelta * (uj - mh * hu) / (nm * delta);
    g32 = (float)(g / N);
  }
  dO[(int64_t)r * kOut + j] = g32;
  if (j == 0) atomicAdd(loss, (1.0 - c * c / q + spread / kP) / N);
}

// The bias gradients: column sums over the batch's rows of dO, dH2 and dH1,
// one thread per column.
__global__ void __launch_bounds__(64)
    k_bias_grads(const float* __restrict__ dO, const float* __restrict__ dH2,
                 const float* __restrict__ dH1, int rows, float* b3, float* b2, float* b1) {
  const int c0 = blockIdx.x * blockDim.x + threadIdx.x;
  if (c0 >= kOut + 2 * kH) return;
  const int l = c0 < kOut ? 0 : c0 < kOut + kH ? 1 : 2;
  const int n = l == 0 ? kOut : kH, c = l == 0 ? c0 : (c0 - kOut) % kH;
  const float* X = l == 0 ? dO : l == 1 ? dH2 : dH1;
  float s = 0.0f;
#pragma unroll 32
  for (int r = 0; r < rows; ++r) s += X[(int64_t)r * n + c];
  (l == 0 ? b3 : l == 1 ? b2 : b1)[c] = s;
}

// One Adam step (Kingma and Ba, 2015) on parameters i .. i + 3 of the packed
// arrays (W1 | b1 | W2 | b2 | W3 | b3, n in all); c1 = 1 - b1^t, c2 = 1 - b2^t.
// wb: the packed bfloat16 weights the network computes with (W1 | W2 | W3).
__global__ void __launch_bounds__(256)
    k_adam(float* w, float* m, float* v, const float* __restrict__ g, __nv_bfloat16* wb, int64_t n,
           float lr, float b1, float b2, float eps, float c1, float c2) {
  const int64_t i = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  const float4 g4 = *reinterpret_cast<const float4*>(g + i);
  float4 m4 = *reinterpret_cast<const float4*>(m + i);
  float4 v4 = *reinterpret_cast<const float4*>(v + i);
  float4 w4 = *reinterpret_cast<const float4*>(w + i);
  auto step = [&](float gi, float& mi, float& vi, float& wi) {
    mi = b1 * mi + (1.0f - b1) * gi;
    vi = b2 * vi + (1.0f - b2) * gi * gi;
    wi = wi - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  };
  step(g4.x, m4.x, v4.x, w4.x);
  step(g4.y, m4.y, v4.y, w4.y);
  step(g4.z, m4.z, v4.z, w4.z);
  step(g4.w, m4.w, v4.w, w4.w);
  *reinterpret_cast<float4*>(m + i) = m4;
  *reinterpret_cast<float4*>(v + i) = v4;
  *reinterpret_cast<float4*>(w + i) = w4;
  // the layer that holds element i (every boundary is a multiple of 4)
  constexpr int64_t n1 = (int64_t)kIn * kH, n2 = (int64_t)kH * kH, n3 = (int64_t)kH * kOut;
  int64_t o = -1;
  if (i < n1) o = i;
  else if (i >= n1 + kH && i < n1 + kH + n2) o = i - kH;
  else if (i >= n1 + n2 + 2 * kH && i < n1 + n2 + n3 + 2 * kH) o = i - 2 * kH;
  if (o >= 0) {
    uint2 u;
    u.x = pack_bf16x2(w4.x, w4.y);
    u.y = pack_bf16x2(w4.z, w4.w);
    *reinterpret_cast<uint2*>(wb + o) = u;
  }
}

__global__ void k_to_bf16(const float* __restrict__ w, __nv_bfloat16* wb, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) wb[i] = __float2bfloat16_rn(w[i]);
}

// Glorot-uniform weights from Philox: entry i of layer L is (2u - 1) lim,
// u from counter (L, i / 4, 0, purpose 8 << 24), lane i mod 4.
__global__ void k_glorot(float* w, int64_t n, uint32_t layer, float lim, uint64_t seed) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const U4 r = philox4x32_10(layer, (uint32_t)(i >> 2), 0u, 8u << 24, (uint32_t)seed,
                             (uint32_t)(seed >> 32));
  w[i] = (2.0f * uniform24(r.v[i & 3]) - 1.0f) * lim;
}

// ---- seeded swarm ----------------------------------------------------------------

// Particle i of node uid at sigma (mu_hat + rho u / |u|), u_j = 2 U - 1 of
// the swarm stream (purpose 6, iteration 0), sigma = sqrt(d / 3) (the expected
// norm of a uniform start in [-1, 1)^d, so the start velocities keep their
// relative size; the loss is scale-invariant): one rounding per operation,
// |u| = sqrt of a sequential fused multiply-add sum of squares.
__device__ void seed_particle(uint64_t seed, uint32_t uid, int i, int d, const float* mu_hat,
                              float rho, float* pos) {
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  float acc = 0.0f;
  for (int q = 0; q < (d + 3) / 4; ++q) {
    const U4 r = philox4x32_10(uid, 0u, (uint32_t)i, (uint32_t)q | (6u << 24), k0, k1);
    for (int c = 0; c < 4 && 4 * q + c < d; ++c) {
      const float u = __fsub_rn(__fmul_rn(2.0f, uniform24(r.v[c])), 1.0f);
      acc = fmaf(u, u, acc);
    }
  }
  const float nrm = __fsqrt_rn(acc);
  const float sigma = __fsqrt_rn(__fdiv_rn((float)d, 3.0f));
  for (int q = 0; q < (d + 3) / 4; ++q) {
    const U4 r = philox4x32_10(uid, 0u, (uint32_t)i, (uint32_t)q | (6u << 24), k0, k1);
    for (int c = 0; c < 4 && 4 * q + c < d; ++c) {
      const int j = 4 * q + c;
      const float u = __fsub_rn(__fmul_rn(2.0f, uniform24(r.v[c])), 1.0f);
      const float qv = nrm > 0.0f ? __fdiv_rn(u, nrm) : 0.0f;
      pos[j] = __fmul_rn(sigma, __fadd_rn(mu_hat[j], __fmul_rn(rho, qv)));
    }
  }
}

__global__ void k_seed_positions(uint64_t seed, uint32_t uid, int P, int d,
                                 const float* __restrict__ mu_hat, const float* __restrict__ rho,
                                 float* pos) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < P) seed_particle(seed, uid, i, d, mu_hat, rho[i], pos + (int64_t)i * d);
}

// The initial swarm of each node from the network's output prop[a][OUT]:
// positions seeded around sigma mu_hat, velocities 0.1 U[-1,1) as for random
// starts, ranges / bests reset (as k_swarm_init).
__global__ void __launch_bounds__(256)
    k_swarm_seed_init(Problem pr, Swarm sw, const NodeDesc* __restrict__ nodes, SwarmCoef co,
                      const float* __restrict__ prop) {
  __shared__ float s_mu[kD];
  __shared__ float s_rho[kP];
  __shared__ double sh[8];
  const int a = blockIdx.x;
  const uint32_t uid = nodes[a].uid;
  const int d = pr.d, d4 = (d + 3) >> 2;
  const float* o = prop + (int64_t)a * kOut;
  const float oj = (int)threadIdx.x < d ? o[threadIdx.x] : 0.0f;
  const double nrm = sqrt(block_sum((double)oj * oj, sh));
  if ((int)threadIdx.x < d) s_mu[threadIdx.x] = nrm > 0.0 ? (float)(oj / nrm) : 0.0f;
  if (threadIdx.x < kP) {
    const float x = o[kD + threadIdx.x];
    s_rho[threadIdx.x] = x > 30.0f ? x : log1pf(expf(x));
  }
  __syncthreads();
  float* pos = sw.pos + (int64_t)a * pr.Pp * d;
  float* vel = sw.vel + (int64_t)a * pr.Pp * d;
  const uint32_t k0 = (uint32_t)co.seed, k1 = (uint32_t)(co.seed >> 32);
  for (int p = threadIdx.x; p < pr.Pp; p += blockDim.x) {
    if (p < pr.P) {
      seed_particle(co.seed, uid, p, d, s_mu, s_rho[p % kP], pos + (int64_t)p * d);
    } else {
      for (int j = 0; j < d; ++j) pos[(int64_t)p * d + j] = 0.0f;
    }
    int* z = sw.zmm + ((int64_t)a * pr.Pp + p) * 2;
    z[0] = INT_MAX;
    z[1] = INT_MIN;
  }
  for (int e = threadIdx.x; e < pr.Pp * d4; e += blockDim.x) {
    const int p = e / d4, q = e - p * d4;
    const U4 rv = philox4x32_10(uid, 0u, (uint32_t)p, (uint32_t)q | (kInitV << 24), k0, k1);
    for (int c = 0; c < 4; ++c) {
      const int j = 4 * q + c;
      if (j >= d) break;
      vel[(int64_t)p * d + j] =
          p < pr.P ? __fmul_rn(0.1f, __fsub_rn(__fmul_rn(2.0f, uniform24(rv.v[c])), 1.0f))
                   : 0.0f;
    }
  }
  __syncthreads();
  if (sw.posb) {
    const int dp4 = pr.dp >> 2;
    for (int e = threadIdx.x; e < pr.Pp * dp4; e += blockDim.x) {
      const int p = e / dp4, j0 = 4 * (e - p * dp4);
      float v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = j0 + c < d ? pos[(int64_t)p * d + j0 + c] : 0.0f;
      store_posb4(sw.posb, pr.Pp, pr.dp, a, p, j0, v);
    }
  }
  if (threadIdx.x == 0) {
    sw.gb[a] = invalid_res();
    sw.gb[gridDim.x + a] = invalid_res();
    sw.gpart[a] = 0;
    sw.giter[a] = 0;
    if (sw.apso) sw.apso[a] = ApsoState{1, 0, co.c1, co.c2, co.inertia};
  }
}

template <typename T>
__global__ void k_gather_rows(const T* __restrict__ src, int64_t cols, const int32_t* __restrict__ idx,
                              int b, T* dst) {
  const int r = blockIdx.y;
  const T* s = src + (int64_t)idx[r] * cols;
  T* o = dst + (int64_t)r * cols;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < cols;
       c += (int64_t)gridDim.x * blockDim.x)
    o[c] = s[c];
}

__global__ void k_acc_double(double* acc, const double* __restrict__ v) { *acc += *v; }

// 64 x 64 tiles from one CTA per SM on, 16 x 16 below.
template <bool TA, bool TB, typename BT, int EPI>
cudaError_t gemm(int M, int N, int K, const float* A, int lda, const BT* B, int ldb,
                 const float* aux, float* C, int ldc, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  auto tiles = [&](int t) { return dim3((unsigned)((N + t - 1) / t), (unsigned)((M + t - 1) / t)); };
  const dim3 g = tiles(64), s = tiles(16);
  if ((int64_t)g.x * g.y >= sm_count() || s.y > 65535)
    k_gemm<TA, TB, BT, EPI, 64, 4, 16><<<g, 256, 0, st>>>(M, N, K, A, lda, B, ldb, aux, C, ldc);
  else
    k_gemm<TA, TB, BT, EPI, 16, 1, 64><<<s, 256, 0, st>>>(M, N, K, A, lda, B, ldb, aux, C, ldc);
  return cudaGetLastError();
}

unsigned blocks(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ---- launchers -------------------------------------------------------------------

cudaError_t launch_node_stats(const Problem& pr, const NodeDesc* nodes, int A,
                              int64_t max_len, int K, int32_t* yr, double* acc, double* wk,
                              float* stats, int n_sm, cudaStream_t st) {
  if (A <= 0) return cudaSuccess;
  cudaError_t e;
  const int fy = (pr.d + 31) / 32;
  // row splits so that the whole batch is a few waves of CTAs
  int splits = (int)((int64_t)4 * n_sm / ((int64_t)A * fy));
  splits = splits < 1 ? 1 : splits;
  const int by_rows = (int)((max_len + 255) / 256);
  splits = splits < by_rows ? splits : (by_rows < 1 ? 1 : by_rows);
  if ((e = cudaMemsetAsync(acc, 0, sizeof(double) * (size_t)A * (K + 2) * pr.d, st))) return e;
  if ((e = cudaMemsetAsync(wk, 0, sizeof(double) * (size_t)A * K, st))) return e;
  if (!pr.lab) {
    k_stats_yinit<<<blocks(A), 256, 0, st>>>(yr, A);
    k_stats_yrange<<<dim3((unsigned)A, (unsigned)splits), 256, 0, st>>>(pr, nodes, yr, splits);
  }
  k_stats_accum<<<dim3((unsigned)A, (unsigned)fy, (unsigned)splits), 256, 0, st>>>(
      pr, nodes, yr, K, splits, acc, wk);
  k_stats_final<<<(unsigned)A, 256, 0, st>>>(pr.d, K, acc, wk, stats);
  return cudaGetLastError();
}

// A layer's forward product: few rows by k_gemm_fwd (below one 64 x 64 tile
// per SM), else k_gemm.
template <int EPI>
cudaError_t gemm_fwd(int M, int N, int K, const float* A, const __nv_bfloat16* B,
                     const float* bias, float* C, cudaStream_t st) {
  const int64_t tiles = (int64_t)((N + 63) / 64) * ((M + 63) / 64);
  if (M <= 0) return cudaSuccess;
  if (tiles >= sm_count()) return gemm<false, false, __nv_bfloat16, EPI>(M, N, K, A, K, B, N, bias, C, N, st);
  k_gemm_fwd<EPI><<<dim3((unsigned)(N / 16), (unsigned)((M + 15) / 16)), 128, 0, st>>>(
      M, N, K, A, B, bias, C);
  return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const MlpParams& m, const float* S, int N, MlpWork w,
                               cudaStream_t st) {
  static_assert(kIn % 16 == 0 && kH % 16 == 0 && kOut % 16 == 0, "k_gemm_fwd's tiles");
  cudaError_t e;
  if ((e = gemm_fwd<kBiasRelu>(N, kH, kIn, S, m.W1b, m.b1, w.H1, st))) return e;
  if ((e = gemm_fwd<kBiasRelu>(N, kH, kH, w.H1, m.W2b, m.b2, w.H2, st))) return e;
  return gemm_fwd<kBias>(N, kOut, kH, w.H2, m.W3b, m.b3, w.O, st);
}

cudaError_t launch_mlp_loss_grad(const MlpParams& m, const float* S, const int32_t* dims,
                                 const float* targets, int N, MlpWork w, MlpGrads g,
                                 double* loss, cudaStream_t st) {
  cudaError_t e;
  if ((e = launch_mlp_forward(m, S, N, w, st))) return e;
  if ((e = cudaMemsetAsync(loss, 0, sizeof(double), st))) return e;
  k_mlp_loss<<<(unsigned)N, 256, 0, st>>>(w.O, dims, targets, N, w.dO, loss);
  // layer 3: gW3 = H2^T dO, gb3 = colsum dO, dH2 = dO W3^T (x relu')
  if ((e = gemm<true, false, float, kPlain>(kH, kOut, N, w.H2, kH, w.dO, kOut, nullptr, g.W3, kOut, st)))
    return e;
  if ((e = gemm<false, true, __nv_bfloat16, kReluMask>(N, kH, kOut, w.dO, kOut, m.W3b, kOut, w.H2,
                                                      w.dH2, kH, st)))
    return e;
  // layer 2
  if ((e = gemm<true, false, float, kPlain>(kH, kH, N, w.H1, kH, w.dH2, kH, nullptr, g.W2, kH, st)))
    return e;
  if ((e = gemm<false, true, __nv_bfloat16, kReluMask>(N, kH, kH, w.dH2, kH, m.W2b, kH, w.H1, w.dH1,
                                                      kH, st)))
    return e;
  // layer 1
  if ((e = gemm<true, false, float, kPlain>(kIn, kH, N, S, kIn, w.dH1, kH, nullptr, g.W1, kH, st)))
    return e;
  k_bias_grads<<<blocks(kOut + 2 * kH, 64), 64, 0, st>>>(w.dO, w.dH2, w.dH1, N, g.b3, g.b2, g.b1);
  return cudaGetLastError();
}

cudaError_t launch_adam(MlpParams& m, MlpState& s, const MlpGrads& g, int t, float lr,
                        cudaStream_t st) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = (float)(1.0 - pow(0.9, t)), c2 = (float)(1.0 - pow(0.999, t));
  // parameters, gradients and moments are packed alike (slm_proposal_create)
  const int64_t n = (m.b3 + kOut) - m.W1;
  k_adam<<<blocks(n / 4), 256, 0, st>>>(m.W1, s.mW1, s.vW1, g.W1, m.W1b, n, lr, b1, b2, eps, c1,
                                        c2);
  return cudaGetLastError();
}

cudaError_t launch_mlp_sync_bf16(const MlpParams& m, cudaStream_t st) {
  k_to_bf16<<<blocks((int64_t)kIn * kH), 256, 0, st>>>(m.W1, m.W1b, (int64_t)kIn * kH);
  k_to_bf16<<<blocks((int64_t)kH * kH), 256, 0, st>>>(m.W2, m.W2b, (int64_t)kH * kH);
  k_to_bf16<<<blocks((int64_t)kH * kOut), 256, 0, st>>>(m.W3, m.W3b, (int64_t)kH * kOut);
  return cudaGetLastError();
}

cudaError_t launch_mlp_init(const MlpParams& m, uint64_t seed, cudaStream_t st) {
  cudaError_t e;
  const int64_t n1 = (int64_t)kIn * kH, n2 = (int64_t)kH * kH, n3 = (int64_t)kH * kOut;
  k_glorot<<<blocks(n1), 256, 0, st>>>(m.W1, n1, 1u, sqrtf(6.0f / (kIn + kH)), seed);
  k_glorot<<<blocks(n2), 256, 0, st>>>(m.W2, n2, 2u, sqrtf(6.0f / (kH + kH)), seed);
  k_glorot<<<blocks(n3), 256, 0, st>>>(m.W3, n3, 3u, sqrtf(6.0f / (kH + kOut)), seed);
  if ((e = cudaMemsetAsync(m.b1, 0, sizeof(float) * kH, st))) return e;
  if ((e = cudaMemsetAsync(m.b2, 0, sizeof(float) * kH, st))) return e;
  if ((e = cudaMemsetAsync(m.b3, 0, sizeof(float) * kOut, st))) return e;
  return launch_mlp_sync_bf16(m, st);
}

cudaError_t launch_gather_rows(const float* src, int64_t cols, const int32_t* idx, int b,
                               float* dst, cudaStream_t st) {
  if (b <= 0) return cudaSuccess;
  k_gather_rows<float><<<dim3(blocks(cols < 4096 ? cols : 4096), (unsigned)b), 256, 0, st>>>(
      src, cols, idx, b, dst);
  return cudaGetLastError();
}

cudaError_t launch_gather_rows(const int32_t* src, int64_t cols, const int32_t* idx, int b,
                               int32_t* dst, cudaStream_t st) {
  if (b <= 0) return cudaSuccess;
  k_gather_rows<int32_t><<<dim3(blocks(cols < 4096 ? cols : 4096), (unsigned)b), 256, 0, st>>>(
      src, cols, idx, b, dst);
  return cudaGetLastError();
}

cudaError_t launch_acc_double(double* acc, const double* v, cudaStream_t st) {
  k_acc_double<<<1, 1, 0, st>>>(acc, v);
  return cudaGetLastError();
}

cudaError_t launch_seed_positions(uint64_t seed, uint32_t uid, int P, int d, const float* mu_hat,
                                  const float* rho, float* pos, cudaStream_t st) {
  if (P <= 0) return cudaSuccess;
  k_seed_positions<<<blocks(P, 64), 64, 0, st>>>(seed, uid, P, d, mu_hat, rho, pos);
  return cudaGetLastError();
}

cudaError_t launch_swarm_seed_init(const Problem& pr, const Swarm& sw, const NodeDesc* nodes,
                                   int A, SwarmCoef co, const float* prop, cudaStream_t st) {
  if (A <= 0) return cudaSuccess;
  k_swarm_seed_init<<<(unsigned)A, 256, 0, st>>>(pr, sw, nodes, co, prop);
  return cudaGetLastError();
}

}  // namespace slm
