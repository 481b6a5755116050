// The projection z = X_node . x_p of a search's iteration (Sec. II-A, Eq. 1)
// from blocked rows, with the swarm move folded in (Sec. III-A, Eq. pso-1 and
// Algorithm 1) or from positions a separate kernel moved.
//
// Blocked rows. A search reads its rows T + 1 times, so they are laid out once
// for these reads (k_block_rows): blocks of 32 rows of one node, feature-major
// ([d][32] floats, rows past the node zero), node a's first block at row
// seg_start + 32 a of the array. A block streams through shared memory as
// whole 2 KB chunks without an address computed per row, whatever d is, and a
// thread's four consecutive rows at one feature are one 16-byte word: two
// pairs of rows for the packed FP32 multiply-add (fma.rn.f32x2: two
// independent FMAs, each rounded as fmaf; half the issue slots, which with
// shared-memory reads and address arithmetic were what bounded the earlier
// row-major kernel, at 2.2 instructions per FMA).
//
// Units. A warp takes a block and the 8 QP particles of a slice (thread tile 8
// rows x QP particles: every x pair meets QP particles, every position 8 rows),
// or PB warps share the slice. A CTA takes a contiguous run of blocks in
// (node, slice, block) order, so its warps read one set of positions, in
// shared memory, feature-major. Every z is the sequential fused multiply-add
// over the features in increasing order, for every shape.
//
// Fold. An iteration t of a folded search is two launches: k_step (gbest step
// of evaluation t-1, the move to x_t, z and the per-particle ranges) and a
// histogram kernel (bins, threshold scan, pbest step, and the gB-independent
// terms of the next move). The move needs gB, which needs every particle's
// score, so every CTA that projects a node takes the node's gbest step itself
// (a warp argmin over P scores) and forms its slice's new positions from the
// terms the histogram kernel left: x' = x + (ic + s2 (gB - x)). The CTA
// holding the slice's first block writes x' and v' back (into the other of two
// position buffers, so the other CTAs still read x), and slice 0's the gbest
// records, exactly as k_move would.
#include <cuda_runtime.h>
#include <float.h>
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <cmath>

#include "device_util.cuh"
#include "slm_internal.cuh"

namespace slm {
namespace {

constexpr int kStepMaxPosBytes = 96 * 1024;  // a slice's positions in shared memory
constexpr int kBR = 32;                      // rows of a block
constexpr int kSC = 16;                      // features of a staged chunk (2 KB)
constexpr int kStepStages = 3;               // a warp's ring of chunks
// Warps of a CTA and registers of a thread. Folded: one CTA per SM, so that a
// node's positions and move terms (48 KB at P = d = 64) are read once per SM;
// 120 registers leave room for the histogram kernel's CTAs beside it, whose
// programmatic launch then overlaps (8 warps, two CTAs per SM: the
// 50,000 x 64 tree 17.5 ms instead of 15.9). Unfolded: two CTAs per SM, so
// that one's change of node overlaps the other's products, with small rings:
// the carveout they leave to L1 is the one the histogram kernel beside them
// runs with, and its entries' labels and targets hit there (with 96 KB rings
// two SLM Boost rounds took 83 ms instead of 72).
constexpr int kFoldWarps = 12, kProjWarps = 8;
constexpr int kFoldRegs = 120, kFoldRegsWide = 152, kProjRegs = 128;  // wide: QP > 6

// Two packed FP32 fused multiply-adds, each rounded to nearest like fmaf.
__device__ __forceinline__ void fma2(uint64_t& c, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;\n" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;\n" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
// (lo, hi) -> (hi, lo)
__device__ __forceinline__ uint64_t swap2(uint64_t v) {
  const float2 f = unpack2(v);
  return pack2(f.y, f.x);
}

// Where particle r (0 .. 8 QP - 1) of a warp's slice sits in the row of
// feature k. Lane group g (8 of them) owns particles 4g .. 4g + 3 of the
// first 32 and W g .. W g + W - 1 of the rest (W = QP - 4, or QP below 4);
// the groups' words are permuted by a key that changes every four features,
// so that the 16-byte move stores of one particle's features spread over the
// banks while a warp's reads at one feature stay distinct.
template <int QP>
__device__ __forceinline__ int pos_slot(int r, int k) {
  const int key = (k >> 2) & 7;
  if (QP >= 4 && r < 32) return (((r >> 2) ^ key) << 2) + (r & 3);
  constexpr int W = QP >= 4 ? (QP > 4 ? QP - 4 : 1) : QP, B0 = QP >= 4 ? 32 : 0;
  const int q = r - B0;
  return B0 + ((q / W) ^ key) * W + q % W;
}

// The blocked rows; one CTA per 256-row tile (which starts a multiple of 256
// rows into its node), a warp per block. Bound by DRAM (204 MB at 200,000 x
// 128 rows: 41 us).
__global__ void __launch_bounds__(256)
    k_block_rows(const float* __restrict__ X, int d, const WorkTile* __restrict__ tiles,
                 float* __restrict__ Xt) {
  __shared__ float s[8][32][33];
  const WorkTile wt = tiles[blockIdx.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r0 = warp * 32;
  if (r0 >= wt.rows) return;
  const int nr = min(32, wt.rows - r0);
  float* out = Xt + ((int64_t)wt.row0 + r0 + 32 * (int64_t)wt.node) * d;
  for (int k0 = 0; k0 < d; k0 += 32) {
    const int kc = min(32, d - k0);
    float v[32];  // 32 loads on their way (8: 125 us at 200,000 x 128 rows)
    const float* x = X + ((int64_t)wt.row0 + r0) * d + k0 + lane;
#pragma unroll
    for (int r = 0; r < 32; ++r) v[r] = r < nr && lane < kc ? __ldg(x + (int64_t)r * d) : 0.0f;
#pragma unroll
    for (int r = 0; r < 32; ++r) s[warp][r][lane] = v[r];
    __syncwarp();
#pragma unroll 8
    for (int k = 0; k < 32; ++k)
      if (k < kc) out[(int64_t)(k0 + k) * 32 + lane] = s[warp][lane][k];
    __syncwarp();
  }
}

template <int QP, int PB, bool FOLD>
__global__ void __launch_bounds__(32 * (FOLD ? kFoldWarps : kProjWarps))
    __maxnreg__(FOLD ? (QP > 6 ? kFoldRegsWide : kFoldRegs) : kProjRegs) k_step(Problem pr, Swarm sw, const float* pos_prev, const NodeDesc* __restrict__ nodes, int A,
           const StepRun* __restrict__ runs, int n_slices, uint32_t inv_d, int t) {
  constexpr int NW = FOLD ? kFoldWarps : kProjWarps, NT = 32 * NW;
  constexpr int PW = 8 * QP;             // particles of a warp
  constexpr int PU = PW * PB;            // particles of a slice
  constexpr int RB = NW / PB;            // row warps
  constexpr int NS = kStepStages;
  // Features of an unrolled turn: a whole chunk. (Folded, us a launch with 8, 16:
  // 12.6, 11.3 on 7,321 x 23 rows, 17.7, 17.2 on 50,000 x 64, 16.8, 16.1 on
  // 30,011 x 50; unfolded with 8: 87 instead of 78 on 200,000 x 128. A turn of 4
  // for the rest of a chunk costs the others registers: 85 there.)
  constexpr int TF = 16;
  constexpr int W = QP >= 4 ? QP - 4 : QP;  // particles per lane beyond the first four
  // Ranges are exchanged once per (node, slice) where two registers a particle
  // are free, else after each block (64 trees on 100,000 x 32 rows, P = 48:
  // 219 us instead of 253; with QP = 8 they spill: 112 us instead of 99 in
  // the first levels of SLM Boost, and the folded kernels lose 2%).
  constexpr bool kRun = !FOLD && QP <= 6;
  static_assert(RB * PB == NW && QP >= 1 && QP <= 8 && PU <= 64, "tile shape");
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_lo[64], s_hi[64];  // ordered-int range of each particle of the slice
  __shared__ int s_best;
  const int d = pr.d, Pp = pr.Pp, P = pr.P;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rg = lane & 3, pg = lane >> 2;  // rows 4 rg.. and 16 + 4 rg..; particle group
  // (rotated by CTA, so that the warps that take one block more fall on
  // different schedulers of an SM)
  const int rw = (warp + blockIdx.x) % RB, pbk = warp / RB;
  float* xs = sm + warp * (NS * kSC * kBR);           // this warp's ring of chunks
  float* ps = sm + NW * NS * kSC * kBR;               // [PB][d][PW] positions
  float* gs = ps + (size_t)PU * d;                    // the node's gB (d floats)
  pdl_trigger();
  const StepRun run = runs[blockIdx.x];
  const int nk = (d + kSC - 1) / kSC;

  // ---- the warp's chunks in order: blocks rw, rw + RB, ... of each (node,
  // slice) of the run, the features of a block in chunks
  int f_node = run.node, f_slice = run.slice, f_left = run.count;
  int f_b = 0, f_end = 0;         // the open (node, slice)'s next block and end
  const float* f_src = pr.Xt;     // this lane's place in the open block's next chunk
  int f_rem = 0;                  // floats of the block from there on
  const int blk_floats = kBR * d;
  auto f_open = [&](int first) {  // blocks of the open (node, slice)
    const NodeDesc nd = nodes[f_node];
    const int nb = (nd.seg_len + kBR - 1) / kBR;
    const int take = min(f_left, nb - first);
    f_b = first + rw;
    f_end = first + take;
    f_left -= take;
    f_src = pr.Xt + ((int64_t)nd.seg_start + 32 * (int64_t)f_node + (int64_t)f_b * kBR) * d +
            4 * lane;
    f_rem = blk_floats - 4 * lane;
  };
  f_open(run.blk);
  float* f_dst = xs + 4 * lane;
  float* const f_dst_end = f_dst + NS * kSC * kBR;
  auto stage = [&] {
    while (f_b >= f_end && f_left > 0) {  // the next (node, slice)
      if (++f_slice == n_slices) {
        f_slice = 0;
        ++f_node;
      }
      f_open(0);
    }
    if (f_b < f_end) {
#pragma unroll
      for (int i = 0; i < kSC * kBR / 128; ++i)
        if (f_rem > 128 * i) cp_async16(f_dst + 128 * i, f_src + 128 * i, 16);
      f_src += kSC * kBR;
      f_rem -= kSC * kBR;
      if (f_rem + 4 * lane <= 0) {  // (the same for every lane) the next block
        const int used = blk_floats - 4 * lane - f_rem;
        f_b += RB;
        f_src += (int64_t)RB * blk_floats - used;
        f_rem += used;
      }
    }
    cp_async_commit();
    f_dst += kSC * kBR;
    if (f_dst == f_dst_end) f_dst -= NS * kSC * kBR;
  };

  if (threadIdx.x < 64) {
    s_lo[threadIdx.x] = INT_MAX;
    s_hi[threadIdx.x] = INT_MIN;
  }
  // Within a search the blocked rows and runs are written before the first
  // iteration's launch, so iterations t > 0 start fetching them before the
  // previous kernel's results are visible.
  if (t > 0)
#pragma unroll 1
    for (int s = 0; s < NS - 1; ++s) stage();
  // positions of particles past the swarm stay zero
  for (int i = threadIdx.x; i < PU * d; i += NT) ps[i] = 0.0f;
  touch(sw.pos);
  touch(sw.z);
  touch(sw.zmm);
  touch(sw.node_step);
  if (FOLD) {
    touch(pos_prev);
    touch(sw.vel);
    touch(sw.gbest);
    touch(sw.cur);
    touch(sw.gb);
    touch(sw.trace);
    touch(sw.ic);
    touch(sw.s2);
    touch(sw.imp);
    touch(sw.keys);
  }
  touch(pr.crit);
  touch((int)pr.Ez);
  __syncthreads();
  pdl_wait();
  if (t == 0)
#pragma unroll 1
    for (int s = 0; s < NS - 1; ++s) stage();

  // A slice's rows [particle][feature] start on 16 bytes whatever d is (its
  // first particle is a multiple of 8) and are read and moved four words at a
  // time; with d % 4 == 0 the four belong to one particle. f / d of a word
  // index f < 2^17 by the launcher's factor.
  const bool vec = (d & 3) == 0;
  auto quot = [](int e, uint32_t inv) { return inv ? (int)__umulhi((uint32_t)e, inv) : e; };
  auto put = [&](int pl, int k, float v) {  // particle pl of the slice
    const int pb = pl / PW;
    ps[(pb * d + k) * PW + pos_slot<QP>(pl - pb * PW, k)] = v;
  };
  // words 4 e .. 4 e + 3 of the slice's rows, np particles
  auto put4 = [&](int e, int np, const float4& v) {
    int pl = quot(4 * e, inv_d), j = 4 * e - pl * d;
    if (vec) {
      put(pl, j, v.x);
      put(pl, j + 1, v.y);
      put(pl, j + 2, v.z);
      put(pl, j + 3, v.w);
      return;
    }
    const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (pl < np) put(pl, j, w[c]);
      if (++j == d) {
        j = 0;
        ++pl;
      }
    }
  };

  // The positions of node a's slice (particles pg0 .. pg0 + PU - 1) for
  // iteration t in ps; desig: this CTA holds the slice's first block.
  auto node_positions = [&](int a, int pg0, bool desig) {
    const int64_t nb = (int64_t)a * Pp * d;
    const int np = min(P, pg0 + PU) - pg0;  // the slice's particles
    const int64_t o0 = nb + (int64_t)pg0 * d;
    const int n4 = (np * d + 3) >> 2;
    if (!FOLD || t == 0 || sw.node_step) {  // another kernel moved the swarm
      const float* src = (FOLD ? pos_prev : sw.pos) + o0;
#pragma unroll 4
      for (int e = threadIdx.x; e < n4; e += NT)
        put4(e, np, __ldcg(reinterpret_cast<const float4*>(src) + e));
      __syncthreads();
      return;
    }
    if constexpr (FOLD) {
      const bool desig0 = desig && pg0 == 0;
      // All inputs in flight before any is used: the slice's positions of
      // t - 1 and move terms, the recorded gB, and (warp 0) the node's scores
      // (two per lane), improvement flag and gbest score.
      constexpr int kPre = 3;
      float4 xa[kPre], ia[kPre], sa[kPre];
      auto load_terms = [&](int e0) {
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
          const int e = e0 + u * NT;
          if (e < n4) {
            xa[u] = __ldcg(reinterpret_cast<const float4*>(pos_prev + o0) + e);
            ia[u] = __ldcg(reinterpret_cast<const float4*>(sw.ic + o0) + e);
            sa[u] = __ldcg(reinterpret_cast<const float4*>(sw.s2 + o0) + e);
          }
        }
      };
      const float* gb_row = sw.gbest + (int64_t)a * d;
      if (warp == 0) {
        // gbest step of evaluation t - 1 (k_move's rule and double
        // buffering): nothing when no particle beat gB in evaluation t - 1;
        // else the particle of the smallest loss key where that decides (no
        // other within 8 ulps of it, nor gB), else by the exact records
        const EvalRes* cur = sw.cur + (int64_t)a * Pp;
        const EvalRes* gold_at = sw.gb + (int64_t)(t & 1) * A + a;
        const int flag =
            t == 1 || !sw.imp ? 1 : __ldcg(sw.imp + (int64_t)((t - 1) & 1) * A + a);
        const uint64_t* kp = sw.keys + (int64_t)a * Pp;
        const uint64_t k0 = lane < P ? __ldcg(kp + lane) : ~0ull;
        const uint64_t k1 = lane + 32 < P ? __ldcg(kp + lane + 32) : ~0ull;
        const double gl = __ldcg(&gold_at->loss);
        const int gv = __ldcg(&gold_at->valid);
        load_terms(threadIdx.x);
        int bi = -1;
        if (flag != 0) {
          const uint64_t km = k0 < k1 ? k0 : k1;
          const uint32_t h = __reduce_min_sync(0xffffffffu, (uint32_t)(km >> 32));
          const uint32_t l = __reduce_min_sync(
              0xffffffffu, (uint32_t)(km >> 32) == h ? (uint32_t)km : 0xffffffffu);
          const uint64_t kmin = ((uint64_t)h << 32) | l;
          const uint64_t near = kmin > ~0ull - 8 ? ~0ull : kmin + 8;
          const unsigned n0 = __ballot_sync(0xffffffffu, k0 <= near);
          const unsigned n1 = __ballot_sync(0xffffffffu, k1 <= near);
          const uint64_t kg = gv ? loss_key(gl) : ~0ull;
          if (t > 1 && __popc(n0) + __popc(n1) == 1 && near < kg) {
            bi = n0 ? __ffs(n0) - 1 : 31 + __ffs(n1);
          } else {
            const EvalRes gold = ldcg_res(gold_at);
            int ci = -1;
            EvalRes ce = invalid_res(), be = gold;
            for (int p = lane; p < P; p += 32)
              gbest_consider(pr, gold, t - 1, p, ldcg_res(cur + p), &ci, &ce);
            bi = gbest_select(pr, ci, ce, &be);
          }
        }
        if (lane == 0) {
          s_best = bi;
          if (desig0) {
            if (sw.imp) sw.imp[(int64_t)(t & 1) * A + a] = 0;  // evaluation t's flag
            const EvalRes g = ldcg_res(bi >= 0 ? cur + bi : gold_at);
            sw.gb[(int64_t)((t - 1) & 1) * A + a] = g;
            if (bi >= 0) {
              sw.gpart[a] = bi;
              sw.giter[a] = t - 1;
            }
            if (sw.trace)
              sw.trace[(int64_t)a * (sw.T + 1) + (t - 1)] =
                  g.valid ? g.loss : __longlong_as_double(0x7ff0000000000000LL);
          }
        }
      } else {
        load_terms(threadIdx.x);
        for (int j = threadIdx.x - 32; j < d; j += NT - 32) gs[j] = __ldcg(gb_row + j);
      }
      __syncthreads();
      // After a gbest change gB is the new best particle's position of t - 1
      // (it beat every pbest, so its own pbest became that position).
      const int bi = s_best;
      if (bi >= 0) {
        if (n4 <= kPre * NT && bi >= pg0 && bi < pg0 + np && vec) {
#pragma unroll
          for (int u = 0; u < kPre; ++u) {  // from the thread that holds it
            const int e = threadIdx.x + u * NT, j = 4 * e - (bi - pg0) * d;
            if (e < n4 && j >= 0 && j < d) {
              *reinterpret_cast<float4*>(gs + j) = xa[u];
              if (desig0) *reinterpret_cast<float4*>(sw.gbest + (int64_t)a * d + j) = xa[u];
            }
          }
        } else {
          for (int j = threadIdx.x; j < d; j += NT) {
            const float g = __ldcg(pos_prev + nb + (int64_t)bi * d + j);
            gs[j] = g;
            if (desig0) sw.gbest[(int64_t)a * d + j] = g;
          }
        }
        __syncthreads();
      }
      // x' = x + (ic + s2 (gB - x)), v' = ic + s2 (gB - x), one rounding each
      auto move1 = [](float x, float ic, float s2, float g, float* v) {
        *v = __fadd_rn(ic, __fmul_rn(s2, __fsub_rn(g, x)));
        return __fadd_rn(x, *v);
      };
      for (int e0 = threadIdx.x; e0 < n4; e0 += kPre * NT) {
        if (e0 != (int)threadIdx.x) load_terms(e0);
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
          const int e = e0 + u * NT;
          if (e >= n4) break;
          const float4 x = xa[u], ic = ia[u], s2 = sa[u];
          float4 g;
          {
            int j = 4 * e - quot(4 * e, inv_d) * d;
            if (vec) {
              g = *reinterpret_cast<const float4*>(gs + j);
            } else {
              auto next = [&] {
                const float v = gs[j];
                j = j + 1 == d ? 0 : j + 1;
                return v;
              };
              g.x = next();
              g.y = next();
              g.z = next();
              g.w = next();
            }
          }
          float4 vn, xn;
          xn.x = move1(x.x, ic.x, s2.x, g.x, &vn.x);
          xn.y = move1(x.y, ic.y, s2.y, g.y, &vn.y);
          xn.z = move1(x.z, ic.z, s2.z, g.z, &vn.z);
          xn.w = move1(x.w, ic.w, s2.w, g.w, &vn.w);
          if (desig) {  // (words past the last particle are padding)
            reinterpret_cast<float4*>(sw.pos + o0)[e] = xn;
            reinterpret_cast<float4*>(sw.vel + o0)[e] = vn;
          }
          put4(e, np, xn);
        }
      }
      __syncthreads();
    }
  };

  // the CTA's range of each particle of node a's slice, into the node's
  auto flush_ranges = [&](int a, int pg0) {
    if ((int)threadIdx.x < PU && s_lo[threadIdx.x] != INT_MAX) {
      int* zz = sw.zmm + ((int64_t)a * Pp + pg0 + threadIdx.x) * 2;
      atomicMin(zz, s_lo[threadIdx.x]);
      atomicMax(zz + 1, s_hi[threadIdx.x]);
      s_lo[threadIdx.x] = INT_MAX;
      s_hi[threadIdx.x] = INT_MIN;
    }
  };
  // particle j of this lane, of the slice
  auto my_particle = [&](int j) {
    return pbk * PW +
           (QP >= 4 ? (j < 4 ? 4 * pg + j : 32 + W * pg + j - 4) : W * pg + j);
  };

  const bool z16 = ((reinterpret_cast<uintptr_t>(sw.z) | (uintptr_t)pr.Ez * 4) & 15) == 0;
  int slot = 0;
  int a = run.node, slice = run.slice, left = run.count, first = run.blk;
  while (left > 0) {
    const NodeDesc nd = nodes[a];
    const int nb = (nd.seg_len + kBR - 1) / kBR;
    const int take = min(left, nb - first);
    const int pg0 = slice * PU;
    node_positions(a, pg0, first == 0);
    // this lane's ranges of its particles, over the warp's blocks (kRun) or a
    // block
    constexpr int QR = (QP + 3) & ~3;  // particles of the range exchange
    float lo[QR], hi[QR];
    auto reset_ranges = [&] {
#pragma unroll
      for (int j = 0; j < QR; ++j) {
        lo[j] = FLT_MAX;
        hi[j] = -FLT_MAX;
      }
    };
    auto exchange_ranges = [&] {
      // The four lanes that share these particles (rg) exchange ranges,
      // halving their particles each time: every lane ends with QR / 4
      // particles' ranges over all the warp's rows (3 QR / 2 shuffles; a
      // reduction of each particle by every lane takes 4 QR).
#pragma unroll
      for (int j = 0; j < QR / 2; ++j) {
        const bool up = rg & 1;
        const float sl = up ? lo[j] : lo[j + QR / 2], sh = up ? hi[j] : hi[j + QR / 2];
        const float kl = up ? lo[j + QR / 2] : lo[j], kh = up ? hi[j + QR / 2] : hi[j];
        lo[j] = fminf(kl, __shfl_xor_sync(0xffffffffu, sl, 1));
        hi[j] = fmaxf(kh, __shfl_xor_sync(0xffffffffu, sh, 1));
      }
#pragma unroll
      for (int j = 0; j < QR / 4; ++j) {
        const bool up = rg & 2;
        const float sl = up ? lo[j] : lo[j + QR / 4], sh = up ? hi[j] : hi[j + QR / 4];
        const float kl = up ? lo[j + QR / 4] : lo[j], kh = up ? hi[j + QR / 4] : hi[j];
        lo[j] = fminf(kl, __shfl_xor_sync(0xffffffffu, sl, 2));
        hi[j] = fmaxf(kh, __shfl_xor_sync(0xffffffffu, sh, 2));
        const int jj = (rg & 1) * (QR / 2) + (rg >> 1) * (QR / 4) + j;
        const int pl = my_particle(jj);
        if (jj < QP && pg0 + pl < P) {
          atomicMin(&s_lo[pl], f2ord(lo[j]));
          atomicMax(&s_hi[pl], f2ord(hi[j]));
        }
      }
    };
    if (kRun) reset_ranges();
    for (int b = first + rw; b < first + take; b += RB) {
      uint64_t acc[4][QP];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < QP; ++j) acc[i][j] = 0ull;
      const float* ar0 = ps + pbk * d * PW;
      // One feature's operands: rows 4 rg .. + 3 and 16 + 4 rg .. + 3 in pairs
      // (x0, x1), the positions in pairs (a0, a1). A pair of rows meets a pair
      // of positions in two packed multiply-adds, straight (x0 a0, x1 a1) and
      // crossed (x0 a1, x1 a0): one swap per pair of positions instead of a
      // copy of every position into both halves, which took the multiply-add
      // pipe as long as half of the products did. (An odd last position is
      // copied.)
      struct Operands {
        ulonglong2 x0, x1;
        uint64_t a[(QP + 1) / 2];
      };
      for (int c = 0; c < nk; ++c) {
        cp_async_wait<NS - 2>();
        __syncwarp();  // the chunk is in place; every lane is done with the last one
        const float* xr = xs + slot * (kSC * kBR) + 4 * rg;
        slot = slot + 1 == NS ? 0 : slot + 1;
        const int k0 = c * kSC;
        const float* ar = ar0 + k0 * PW;
        auto read = [&](Operands& o, int k, int key) {
          o.x0 = *reinterpret_cast<const ulonglong2*>(xr + k * kBR);
          o.x1 = *reinterpret_cast<const ulonglong2*>(xr + k * kBR + 16);
          const float* ak = ar + k * PW;
          constexpr int J0 = QP >= 4 ? 4 : 0;
          if constexpr (QP >= 4) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(ak + ((pg ^ key) << 2));
            o.a[0] = v.x;
            o.a[1] = v.y;
          }
          if constexpr (W == 4) {
            const ulonglong2 v =
                *reinterpret_cast<const ulonglong2*>(ak + 32 + ((pg ^ key) << 2));
            o.a[2] = v.x;
            o.a[3] = v.y;
          } else if constexpr (W == 2) {
            o.a[J0 / 2] = *reinterpret_cast<const uint64_t*>(ak + 8 * J0 + ((pg ^ key) << 1));
          } else if constexpr (W == 3) {
            const float* aw = ak + 8 * J0 + (pg ^ key) * W;
            o.a[J0 / 2] = pack2(aw[0], aw[1]);
            o.a[J0 / 2 + 1] = pack2(aw[2], aw[2]);
          } else if constexpr (W == 1) {
            const float v = ak[8 * J0 + (pg ^ key)];
            o.a[J0 / 2] = pack2(v, v);
          }
        };
        auto feature = [&](const Operands& o) {
#pragma unroll
          for (int m = 0; m < QP / 2; ++m) {
            const uint64_t as = swap2(o.a[m]);
            fma2(acc[0][2 * m], o.x0.x, o.a[m]);
            fma2(acc[1][2 * m], o.x0.y, o.a[m]);
            fma2(acc[2][2 * m], o.x1.x, o.a[m]);
            fma2(acc[3][2 * m], o.x1.y, o.a[m]);
            fma2(acc[0][2 * m + 1], o.x0.x, as);
            fma2(acc[1][2 * m + 1], o.x0.y, as);
            fma2(acc[2][2 * m + 1], o.x1.x, as);
            fma2(acc[3][2 * m + 1], o.x1.y, as);
          }
          if constexpr (QP & 1) {
            fma2(acc[0][QP - 1], o.x0.x, o.a[QP / 2]);
            fma2(acc[1][QP - 1], o.x0.y, o.a[QP / 2]);
            fma2(acc[2][QP - 1], o.x1.x, o.a[QP / 2]);
            fma2(acc[3][QP - 1], o.x1.y, o.a[QP / 2]);
          }
        };
        const int kc = min(kSC, d - k0);
        Operands o[2];
        const int key0 = (k0 >> 2) & 7;  // (a chunk's keys do not wrap)
        read(o[0], 0, key0);
        stage();  // into the slot of the chunk before this one
        // TF features a turn, the next one's operands read ahead
        int k = 0;
#pragma unroll 1
        for (; k + TF <= kc; k += TF) {
          const int key = key0 + (k >> 2);
#pragma unroll
          for (int i = 0; i < TF; ++i) {
            if (i + 1 < TF)
              read(o[(i + 1) & 1], k + i + 1, key + ((i + 1) >> 2));
            else if (k + TF < kc)
              read(o[0], k + TF, key + TF / 4);
            feature(o[i & 1]);
          }
        }
#pragma unroll 1
        for (; k < kc; ++k) {
          feature(o[0]);
          if (k + 1 < kc) read(o[0], k + 1, key0 + ((k + 1) >> 2));
        }
      }
      // block complete: its ranges into the lane's, z out (16 bytes a store
      // where the block is whole and aligned)
      const int nr = min(kBR, nd.seg_len - b * kBR);
      const int64_t zrow = (int64_t)nd.seg_start + b * kBR;
      const bool whole = nr == kBR;
      const bool v16 = z16 && whole && (zrow & 3) == 0;
      if (!kRun) reset_ranges();
      float* zp = sw.z + (int64_t)(pg0 + my_particle(0)) * pr.Ez + zrow + 4 * rg;
#pragma unroll
      for (int j = 0; j < QP; ++j) {
        const int p = pg0 + my_particle(j);
        if (j > 0) zp += j == 4 && QP > 4 ? (int64_t)(my_particle(4) - my_particle(3)) * pr.Ez : pr.Ez;
        // rows' pairs of particle j: the straight sums' halves of its own
        // parity and the crossed sums' of the other (an odd last particle has
        // both halves)
        auto rows = [&](const uint64_t (&c)[QP]) {
          if (j == QP - 1 && (QP & 1)) return unpack2(c[j]);
          const float2 s0 = unpack2(c[j & ~1]), s1 = unpack2(c[j | 1]);
          return (j & 1) ? make_float2(s1.x, s0.y) : make_float2(s0.x, s1.y);
        };
        const float2 v0 = rows(acc[0]), v1 = rows(acc[1]), v2 = rows(acc[2]), v3 = rows(acc[3]);
        if (whole) {
          lo[j] = fminf(lo[j], fminf(fminf(fminf(v0.x, v0.y), fminf(v1.x, v1.y)),
                               fminf(fminf(v2.x, v2.y), fminf(v3.x, v3.y))));
          hi[j] = fmaxf(hi[j], fmaxf(fmaxf(fmaxf(v0.x, v0.y), fmaxf(v1.x, v1.y)),
                               fmaxf(fmaxf(v2.x, v2.y), fmaxf(v3.x, v3.y))));
        }
        if (v16) {
          if (p < P) {
            *reinterpret_cast<float4*>(zp) = make_float4(v0.x, v0.y, v1.x, v1.y);
            *reinterpret_cast<float4*>(zp + 16) = make_float4(v2.x, v2.y, v3.x, v3.y);
          }
        } else {
          const float v[8] = {v0.x, v0.y, v1.x, v1.y, v2.x, v2.y, v3.x, v3.y};
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int off = (i & 3) + 16 * (i >> 2);
            if (4 * rg + off < nr) {
              if (!whole) {
                lo[j] = fminf(lo[j], v[i]);
                hi[j] = fmaxf(hi[j], v[i]);
              }
              if (p < P) zp[off] = v[i];
            }
          }
        }
      }
      if (!kRun) exchange_ranges();
    }
    if (kRun && rw < take) exchange_ranges();
    __syncthreads();  // every warp's ranges are in; the positions are read
    flush_ranges(a, pg0);
    left -= take;
    first = 0;
    if (++slice == n_slices) {
      slice = 0;
      ++a;
    }
  }
}

// The projection of few particles (slices of 8): a thread takes two rows and
// all 8, so every x is read once, straight from the blocked rows (8 bytes per
// lane, eight features on their way while eight are multiplied), and a slice's
// positions at one feature are two broadcast words. A warp takes two blocks
// at a time. Bound by waiting for the rows: the FP32 re-scores of the BF16
// form, 200,000 x 128 rows and 8 particles (102 MB), take 33 us of an iteration
// (24.8 captured by themselves; four blocks a warp 36), by the row-major kernel
// (row tiles through shared memory) 39.
constexpr int kFewWarps = 8, kFewP = 8, kFewF = 8;
constexpr int kFewBlocks = 2;  // blocks of a warp

__global__ void __launch_bounds__(32 * kFewWarps, 3)
    k_project_few(Problem pr, Swarm sw, const NodeDesc* __restrict__ nodes,
                  const StepRun* __restrict__ runs, int n_slices) {
  constexpr int NT = 32 * kFewWarps;
  extern __shared__ __align__(16) float sm[];  // [d][8] positions
  __shared__ int s_lo[kFewP], s_hi[kFewP];
  const int d = pr.d, P = pr.P;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int blk = lane >> 4, rl = 2 * (lane & 15);  // this lane's block of the two, its rows
  pdl_trigger();
  const StepRun run = runs[blockIdx.x];
  const bool z16 = ((reinterpret_cast<uintptr_t>(sw.z) | (uintptr_t)pr.Ez * 4) & 15) == 0;
  const int nc = (d + kFewF - 1) / kFewF;  // chunks of features
  if (threadIdx.x < kFewP) {
    s_lo[threadIdx.x] = INT_MAX;
    s_hi[threadIdx.x] = INT_MIN;
  }
  pdl_wait();
  int a = run.node, slice = run.slice, left = run.count, first = run.blk;
  while (left > 0) {
    const NodeDesc nd = nodes[a];
    const int nb = (nd.seg_len + kBR - 1) / kBR;
    const int take = min(left, nb - first);
    const int pg0 = slice * kFewP, np = min(P - pg0, kFewP);
    const float* src = sw.pos + ((int64_t)a * pr.Pp + pg0) * d;
    for (int i = threadIdx.x; i < kFewP * d; i += NT) {
      const int q = i / d, k = i - q * d;
      sm[k * kFewP + q] = q < np ? __ldcg(src + i) : 0.0f;
    }
    __syncthreads();
    float lo[kFewP], hi[kFewP];
#pragma unroll
    for (int q = 0; q < kFewP; ++q) {
      lo[q] = FLT_MAX;
      hi[q] = -FLT_MAX;
    }
    for (int u = kFewBlocks * warp; u < take; u += kFewBlocks * kFewWarps) {
      const int b = first + u + blk;  // this lane's block
      const bool in = u + blk < take;
      const float* x = pr.Xt +
                       ((int64_t)nd.seg_start + 32 * (int64_t)a + (int64_t)b * kBR) * d + rl;
      float2 v[2][kFewF];
      auto load = [&](float2 (&w)[kFewF], int c) {
#pragma unroll
        for (int i = 0; i < kFewF; ++i) {
          const int k = c * kFewF + i;
          w[i] = in && k < d ? __ldcg(reinterpret_cast<const float2*>(x + (int64_t)k * kBR))
                             : make_float2(0.f, 0.f);
        }
      };
      // rows in pairs, straight and crossed with the particles' pairs (see
      // k_step): acc[2 j] = (r0 p0, r1 p1), acc[2 j + 1] = (r1 p0, r0 p1)
      uint64_t acc[kFewP];
#pragma unroll
      for (int q = 0; q < kFewP; ++q) acc[q] = 0ull;
      auto multiply = [&](const float2 (&w)[kFewF], int c) {
        const float* ps = sm + c * kFewF * kFewP;
        const int kc = d - c * kFewF;  // (a product past d could turn -0 into 0)
#pragma unroll
        for (int i = 0; i < kFewF; ++i) {
          if (i >= kc) break;
          const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(ps + i * kFewP);
          const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(ps + i * kFewP + 4);
          const uint64_t av[4] = {a0.x, a0.y, a1.x, a1.y};
          const uint64_t x = pack2(w[i].x, w[i].y), y = pack2(w[i].y, w[i].x);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            fma2(acc[2 * j], x, av[j]);
            fma2(acc[2 * j + 1], y, av[j]);
          }
        }
      };
      load(v[0], 0);
      for (int c = 0; c < nc; c += 2) {
        load(v[1], c + 1);
        multiply(v[0], c);
        if (c + 1 >= nc) break;
        load(v[0], c + 2);
        multiply(v[1], c + 1);
      }
      const int nr = in ? min(kBR, nd.seg_len - b * kBR) : 0;
      const int64_t zrow = (int64_t)nd.seg_start + (int64_t)b * kBR + rl;
      const bool v8 = z16 && nr == kBR && (zrow & 1) == 0;
#pragma unroll
      for (int q = 0; q < kFewP; ++q) {
        const float2 s0 = unpack2(acc[q & ~1]), s1 = unpack2(acc[q | 1]);
        const float r0 = (q & 1) ? s1.y : s0.x, r1 = (q & 1) ? s0.y : s1.x;
        float* zp = sw.z + (int64_t)(pg0 + q) * pr.Ez + zrow;
        if (rl < nr) {
          lo[q] = fminf(lo[q], r0);
          hi[q] = fmaxf(hi[q], r0);
          if (!v8 && q < np) zp[0] = r0;
        }
        if (rl + 1 < nr) {
          lo[q] = fminf(lo[q], r1);
          hi[q] = fmaxf(hi[q], r1);
          if (!v8 && q < np) zp[1] = r1;
        }
        if (v8 && q < np) *reinterpret_cast<float2*>(zp) = make_float2(r0, r1);
      }
    }
    if (kFewBlocks * warp < take) {  // (the warp had blocks)
#pragma unroll
      for (int q = 0; q < kFewP; ++q) {
        const int l = __reduce_min_sync(0xffffffffu, f2ord(lo[q]));
        const int h = __reduce_max_sync(0xffffffffu, f2ord(hi[q]));
        if (lane == q) {
          atomicMin(&s_lo[q], l);
          atomicMax(&s_hi[q], h);
        }
      }
    }
    __syncthreads();  // every warp's ranges are in; the positions are read
    if ((int)threadIdx.x < np && s_lo[threadIdx.x] != INT_MAX) {
      int* zz = sw.zmm + ((int64_t)a * pr.Pp + pg0 + threadIdx.x) * 2;
      atomicMin(zz, s_lo[threadIdx.x]);
      atomicMax(zz + 1, s_hi[threadIdx.x]);
      s_lo[threadIdx.x] = INT_MAX;
      s_hi[threadIdx.x] = INT_MIN;
    }
    left -= take;
    first = 0;
    if (++slice == n_slices) {
      slice = 0;
      ++a;
    }
  }
}

// Tile shapes of a folded search's padded swarm: particles per thread and
// particle warps. Shapes 0-2 take every particle in a unit, on 384, 192 or 96
// rows of the CTA; shapes 3-5 take half of them (two slices of a swarm of 32
// or 64), so a short node is spread over twice the CTAs with half the move
// and projection each.
bool step_shape(const Problem& pr, int sh, int* QP, int* PB) {
  const int Pp = pr.Pp;
  if (Pp % 16 || Pp < 16 || Pp > 64 || sh < 0 || sh >= kStepShapeCount) return false;
  const int pu = sh < 3 ? Pp : Pp / 2;
  if ((sh >= 3 && Pp != 32 && Pp != 64) || pu % 16) return false;
  *PB = 1 << (sh % 3);
  if (pu == 48) {
    *QP = (pr.P + 7) / 8;  // 5 or 6
    return *PB == 1;
  }
  *QP = pu / 8 / *PB;
  return *QP >= 1;
}

// The unfolded projection's slices of a long batch: the fewest of at most 64
// particles whose positions fit, each shared by as many warps (1, 2 or 4) as
// leaves a row warp for each of the `blocks` of a node: small nodes' blocks
// would leave the other warps idle.
bool proj_shape(const Problem& pr, int64_t blocks, int* QP, int* PB) {
  for (int n = (pr.P + 63) / 64; n <= pr.P; ++n) {
    const int q = ((pr.P + n - 1) / n + 7) / 8;
    if ((size_t)8 * q * pr.d * sizeof(float) <= (size_t)kStepMaxPosBytes) {
      *PB = 1;
      while (*PB < 4 && blocks * *PB * 2 <= kProjWarps && q > *PB) *PB *= 2;
      *QP = (q + *PB - 1) / *PB;
      return true;
    }
    if (q == 1) break;
  }
  return false;
}

size_t step_smem(int d, int pu, int warps) {
  return sizeof(float) * ((size_t)warps * kStepStages * kSC * kBR + (size_t)pu * d +
                          (size_t)((d + 3) & ~3));
}

const void* step_fn(int QP, int PB) {
  switch (QP * 16 + PB) {
    case 8 * 16 + 1: return (const void*)k_step<8, 1, true>;
    case 6 * 16 + 1: return (const void*)k_step<6, 1, true>;
    case 5 * 16 + 1: return (const void*)k_step<5, 1, true>;
    case 4 * 16 + 1: return (const void*)k_step<4, 1, true>;
    case 4 * 16 + 2: return (const void*)k_step<4, 2, true>;
    case 2 * 16 + 1: return (const void*)k_step<2, 1, true>;
    case 2 * 16 + 2: return (const void*)k_step<2, 2, true>;
    case 2 * 16 + 4: return (const void*)k_step<2, 4, true>;
    case 1 * 16 + 1: return (const void*)k_step<1, 1, true>;
    case 1 * 16 + 2: return (const void*)k_step<1, 2, true>;
    case 1 * 16 + 4: return (const void*)k_step<1, 4, true>;
    default: return nullptr;
  }
}

const void* proj_fn(int QP, int PB) {
  switch (QP * 16 + PB) {
    case 1 * 16 + 1: return (const void*)k_step<1, 1, false>;
    case 2 * 16 + 1: return (const void*)k_step<2, 1, false>;
    case 3 * 16 + 1: return (const void*)k_step<3, 1, false>;
    case 4 * 16 + 1: return (const void*)k_step<4, 1, false>;
    case 5 * 16 + 1: return (const void*)k_step<5, 1, false>;
    case 6 * 16 + 1: return (const void*)k_step<6, 1, false>;
    case 7 * 16 + 1: return (const void*)k_step<7, 1, false>;
    case 8 * 16 + 1: return (const void*)k_step<8, 1, false>;
    case 1 * 16 + 2: return (const void*)k_step<1, 2, false>;
    case 2 * 16 + 2: return (const void*)k_step<2, 2, false>;
    case 3 * 16 + 2: return (const void*)k_step<3, 2, false>;
    case 4 * 16 + 2: return (const void*)k_step<4, 2, false>;
    case 1 * 16 + 4: return (const void*)k_step<1, 4, false>;
    case 2 * 16 + 4: return (const void*)k_step<2, 4, false>;
    default: return nullptr;
  }
}

}  // namespace

bool step_ok(const Problem& pr) {
  int QP = 0, PB = 0;
  return step_shape(pr, 0, &QP, &PB) &&
         (size_t)8 * QP * PB * pr.d * sizeof(float) <= (size_t)kStepMaxPosBytes;
}

namespace {
void fill_config(const Problem& pr, const void* fn, int QP, int PB, int warps, StepConfig* c) {
  c->fn = fn;
  c->qp = QP;
  c->pb = PB;
  c->slices = (pr.P + 8 * QP * PB - 1) / (8 * QP * PB);
  c->threads = 32 * warps;
  c->row_warps = warps / PB;
  c->smem = step_smem(pr.d, 8 * QP * PB, warps);
}
}  // namespace

bool step_config(const Problem& pr, int sh, StepConfig* c) {
  int QP = 0, PB = 0;
  if (!step_shape(pr, sh, &QP, &PB)) return false;
  fill_config(pr, step_fn(QP, PB), QP, PB, kFoldWarps, c);
  return c->fn != nullptr;
}

// Few blocks leave most warps of the widest slices idle, and each of the rest
// with all the products of its particles in turn: such batches take narrower
// slices, a warp each. The estimate is the clocks of the longest CTA: its
// (node, slice) pairs, each its warps' blocks one after another (12 clocks per
// feature and particle of a thread and 50 of latency), or the issue slots of
// its SM (8, and 24 a feature), and the pairs' positions. Constants fitted to
// 282 batches (1 to 1,000 nodes of 50 to 100,000 rows, 8 to 300 features,
// 24 to 250 particles): the pick is within 1 % of the fastest shape in the mean,
// and never 3 % slower than the widest slices or the row-major kernel. Of
// these 81 were slower with the widest slices than row-major: one node of 1,000
// x 128 rows, P = 100, 31 iterations 0.76 ms row-major, 0.97 with slices of 56
// and 0.64 with 13 of 8; 16 nodes of 190 x 128 rows, P = 100: 1.85, 1.96, 1.63.
bool proj_config(const Problem& pr, int A, int64_t blocks, int n_sm, StepConfig* c) {
  int QP = 0, PB = 0;
  const double bn = (double)std::max<int64_t>(1, blocks / std::max(A, 1));  // of a node
  if (!proj_shape(pr, (int64_t)bn, &QP, &PB)) return false;
  auto estimate = [&](const StepConfig& q) {
    if (prepare_step(q) != cudaSuccess) return -1.0;
    const double pairs = (double)A * q.slices, g = step_grid(q, n_sm);
    if (g <= 0) return -1.0;
    double k = 1, m = bn, ctas = g;  // pairs of a CTA, blocks of each, CTAs
    if (pairs <= g) {
      m = std::ceil(bn / std::floor(g / pairs));
      ctas = pairs * std::ceil(bn / m);
    } else {
      k = pairs / g;
    }
    const double lat = k * std::ceil(m / q.row_warps) * pr.d * (12.0 * q.qp + 50.0);
    const double thr =
        k * m * q.pb * std::ceil(ctas / n_sm) / 4.0 * pr.d * (8.0 * q.qp + 24.0);
    return std::max(lat, thr) + k * 8.0 * q.qp * q.pb * pr.d / 10.0;
  };
  fill_config(pr, proj_fn(QP, PB), QP, PB, kProjWarps, c);
  double best = 0.95 * estimate(*c);  // (a narrower slice has to be clearly faster)
  // (with more pairs the blocks of one pair follow those of another, and the
  // nodes of a tree's level differ in size: a 30,011 x 50 regression tree's
  // level of some 250 nodes lost 5 us of 16 an iteration)
  const bool few = 4 * (int64_t)A * c->slices <= step_grid(*c, n_sm);
  for (int q = 1; few && q <= 8; ++q) {
    StepConfig n;
    if ((size_t)8 * q * pr.d * sizeof(float) > (size_t)kStepMaxPosBytes) break;
    fill_config(pr, proj_fn(q, 1), q, 1, kProjWarps, &n);
    const double e = estimate(n);
    if (e > 0.0 && e < best) {
      best = e;
      *c = n;
    }
  }
  return c->fn != nullptr;
}

bool few_config(const Problem& pr, StepConfig* c) {
  c->fn = nullptr;
  c->qp = 1;
  c->pb = 1;
  c->slices = (pr.P + kFewP - 1) / kFewP;
  c->threads = 32 * kFewWarps;
  c->row_warps = kFewWarps;
  c->smem = sizeof(float) * (size_t)pr.d * kFewP;
  if (c->smem > (size_t)kStepMaxPosBytes) return false;
  c->fn = (const void*)k_project_few;
  return true;
}

cudaError_t launch_project_few(const StepConfig& c, const Problem& pr, const Swarm& sw,
                               const NodeDesc* nodes, const StepRun* runs, int n_runs,
                               cudaStream_t st) {
  if (n_runs <= 0) return cudaSuccess;
  if (!pr.Xt) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n_runs, 1, 1);
  cfg.blockDim = dim3((unsigned)c.threads, 1, 1);
  cfg.dynamicSmemBytes = c.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_project_few, pr, sw, nodes, runs, c.slices);
}

cudaError_t prepare_step(const StepConfig& c) { return allow_smem(c.fn, (int)c.smem); }

int step_grid(const StepConfig& c, int n_sm) {
  int per_sm = 0;
  if (occupancy(&per_sm, c.fn, c.threads, c.smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * n_sm;
}

int64_t step_rows_floats(const Problem& pr, int A) { return (pr.E + 32 * (int64_t)A) * pr.d; }

cudaError_t launch_block_rows(const Problem& pr, const WorkTile* tiles, int n_tiles, float* Xt,
                              cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  k_block_rows<<<(unsigned)n_tiles, 256, 0, st>>>(pr.X, pr.d, tiles, Xt);
  return cudaGetLastError();
}

cudaError_t launch_step(const StepConfig& c, const Problem& pr, const Swarm& sw,
                        const float* pos_prev, const NodeDesc* nodes, int A, const StepRun* runs,
                        int n_runs, int t, cudaStream_t st) {
  if (n_runs <= 0) return cudaSuccess;
  if (!pr.Xt) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n_runs, 1, 1);
  cfg.blockDim = dim3((unsigned)c.threads, 1, 1);
  cfg.dynamicSmemBytes = c.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n_slices = c.slices;
  // ceil(2^32 / v): __umulhi(e, .) = e / v exactly for e v < 2^32; 0 (no
  // factor of 32 bits) for v = 1
  auto factor = [](uint32_t v) {
    return v > 1 ? (uint32_t)(((1ull << 32) + v - 1) / v) : 0u;
  };
  uint32_t inv_d = factor((uint32_t)pr.d);
  void* args[] = {(void*)&pr, (void*)&sw, (void*)&pos_prev, (void*)&nodes, (void*)&A,
                  (void*)&runs, (void*)&n_slices, (void*)&inv_d, (void*)&t};
  return cudaLaunchKernelExC(&cfg, c.fn, args);
}

}  // namespace slm
