// The tree phases of large trees in the scaled forms: a warp per node (tree.cuh: a CTA per node).
//
// What bounds them: below the subtree roots there are many more nodes than the chip has warps, so a node's latency
// is hidden by the other warps of its SM, and what counts is how many nodes an SM holds at once. A warp here reads
// its block from global memory straight into registers and keeps only the vectors in shared memory (256 bytes a
// vector), with no barrier inside a level; a CTA of tree.cuh takes one node at a time with all its warps, needs
// 10 KB a CTA for its blocks (four CTAs beside the dense stream) and idles half of its warps where a step has fewer
// tasks than warps (k = 16, up to eight vectors). One launch per phase; a CTA owns a subtree of T levels,
// the nodes above it are climbed with a ticket per level, the second CTA to arrive at a parent taking it.
// 2D n = 2^20, int16 with FP32 bases, phases in order, tree.cuh -> here: upsweep / downsweep of one vector 118 / 86 -> 84 /
// 48 us, of four 228 / 150 -> 112 / 70, of eight 297 / 183 -> 175 / 165.
#pragma once
#include <algorithm>

#include "mixed.cuh"

namespace h2 {

constexpr int kWarpTreeWarps = 8, kWarpTreeMaxVectors = 8;
// Whether a pass of up to nvb vectors (1, 2, 4 or 8) over a tree of depth q takes these kernels. Measured, product in us,
// tree.cuh / these, int16 codes with FP32 bases, then fp16 codes and bases, k = 16, 64-point leaves:
//   vectors             1                      2                      4                       8
//   depth 10     105/112  100/135       118/133  114/149      149/145  151/170        188/223   166/210
//   depth 11     143/147  150/180       164/174  163/192      231/194  238/221        308/325   260/291
//   depth 12     217/209  234/242       254/247  254/256      391/299  400/318        537/499   445/422
//   depth 14     686/643  756/741       846/790  856/831    1292/1036 1331/1058     1812/1671 1432/1331
// k = 9: 270 -> 260 at depth 12, one vector; k = 25: 576 -> 625 (above 16 rows a warp takes one column at a time).
inline bool warp_tree(int q, int k, int nvb, bool bases_fp32) {
  if (k > 16 || nvb > kWarpTreeMaxVectors) return false;
  return q >= (nvb == 4 ? 11 : nvb <= 2 && !bases_fp32 ? 13 : 12);
}
// The same for a batch, all of whose members' trees count. fp16, 32-point leaves, product in us, tree.cuh / these: 64
// members of 4,096 .. 32,768 points (some 40,000 leaves), 1, 2, 4, 8 vectors 2539/2459, 2812/2766, 3078/2928, 2530/2075;
// 128 members of 4,096 .. 131,072, 1 to 16 vectors 13853/12352. The tree phases of 32 members of 1,024 .. 16,384 (some
// 8,000 leaves) took as long a warp per node as they do here.
constexpr int64_t kWarpTreeBatchLeaves = 1 << 14;
inline bool warp_tree_batch(int64_t leaves, int k) { return k <= 16 && leaves >= kWarpTreeBatchLeaves; }
// levels of the CTAs' subtrees: two CTAs an SM; opt: the tuner's choice (one or two levels more)
inline int warp_tree_levels(int q, int sms, int opt) {
  int L = 0;
  while ((1 << L) < 2 * sms) L++;
  return q - std::max(0, std::min(L, q) - opt);
}

// leaf j's 16-bit parts for passes of up to four vectors (a batch's; a function of its own: few launches want them, and its
// registers would be the projection's; as a call in the variant of eight vectors it took 40 us more at 2D n = 2^20)
template <int F>
__device__ __noinline__ void leaf_parts_w(const MatDesc* D, int64_t j, int s, const float* xs, int spad, const unsigned* vmax) {
  TreeParamsM P{};
  P.nv = D->nv;
  P.D = D;
  TreeOpM<F>::parts(P, j, s, xs, 1, spad, vmax, threadIdx.x & 31, 32);
}

// the leaf's x (convert: from the product's own x, whose FP32 copy and 16-bit parts are left here) times V_j^T
template <int F, int NVB>
__device__ __forceinline__ void project_leaf_w(const TreeParamsM& P, int LR, int64_t j, int lane, float* wbuf, unsigned* vmax,
                                               bool convert) {
  const int64_t leaf0 = ((int64_t)1 << P.q) - 1, off = P.leaf_off[j];
  const int sj = (int)(P.leaf_off[j + 1] - off), spad = (sj + 3) & ~3;
  float* xj = P.x4 + P.xp4_off[j] * P.nv;
  if (convert) {
    // every load of the chunk is issued before any store (the stores could alias x for the compiler)
    float xr[NVB][2];
#pragma unroll
    for (int v = 0; v < NVB; v++)
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int a = lane + 32 * h;
        xr[v][h] = (v < P.nv && a < sj) ? x_load(P.x, P.xy32, off + v * P.ldx + a) : 0.f;  // padding is zero
      }
    const bool parts = TreeOpM<F>::want_parts(P);  // (in a batch also for members of few vectors)
#pragma unroll
    for (int v = 0; v < NVB; v++) {
      if (v >= P.nv) break;
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int a = lane + 32 * h;
        if (a < spad) {
          xj[v * spad + a] = xr[v][h];
          wbuf[v * spad + a] = xr[v][h];
        }
      }
      if (parts) {
        const unsigned m = __reduce_max_sync(0xFFFFFFFFu, max(TreeOpM<F>::abs_bits(xr[v][0]), TreeOpM<F>::abs_bits(xr[v][1])));
        if (lane == 0) vmax[v] = m;
      }
    }
    __syncwarp();
    if constexpr (NVB > 4) {
      if (parts) TreeOpM<F>::parts(P, j, sj, wbuf, 1, spad, vmax, lane, 32);
    } else {
      if (parts) leaf_parts_w<F>(P.D, j, sj, wbuf, spad, vmax);
    }
  } else {
    stage_vectors(wbuf, xj, P.nv * spad, lane);  // the FP32 copy of x(j), padding zero
  }
  float acc[1][NVB];
#pragma unroll
  for (int v = 0; v < NVB; v++) acc[0][v] = 0.f;
  warp_mv_m<F, 1, NVB>(static_cast<const typename CodeT<F>::T*>(P.Vt) + P.vt_off[j], P.vscale[j], P.k, sj, LR, wbuf, spad, P.nv,
                       acc, lane);
  __syncwarp();
  group_reduce_m(acc, LR);
  store_node_m<1, NVB, false>(P.xhat + (leaf0 + j) * P.nv * P.kp, P.k, P.kp, LR, P.nv, acc, lane);
}

// parent p of the upsweep for vectors v0 .. v0 + nw - 1 (nw <= NVB); CG: a child was written by another CTA
template <int F, int NVB, bool CG>
__device__ __forceinline__ void up_node_w(const TreeParamsM& P, int LR, int64_t p, int lane, float* wbuf, int v0, int nw) {
  float acc[1][NVB];
#pragma unroll
  for (int v = 0; v < NVB; v++) acc[0][v] = 0.f;
  for (int64_t ch = 2 * p + 1; ch <= 2 * p + 2; ch++) {
    stage_vectors<CG>(wbuf, P.xhat + (ch * P.nv + v0) * P.kp, nw * P.kp, lane);
    warp_mv_m<F, 1, NVB>(TreeOpM<F>::Ft(P, ch), TreeOpM<F>::bF(P, ch), P.k, P.k, LR, wbuf, P.kp, nw, acc, lane);
    __syncwarp();
  }
  group_reduce_m(acc, LR);
  store_node_m<1, NVB, false>(P.xhat + (p * P.nv + v0) * P.kp, P.k, P.kp, LR, nw, acc, lane);
}

// leaf projection and the whole upsweep (Alg. 2, Eq. 2): CTA b works on subtree jobs[b].y of matrix jobs[b].x (without jobs:
// subtree b of the only matrix); the matrices of fewer than nvlo or more than NVB vectors are left to another launch
template <int F, int NVB>
__global__ void __launch_bounds__(kWarpTreeWarps * 32, NVB == 2 ? 4 : 0) k_upsweep_warps(const MatDesc* __restrict__ mats,
                                                                        const int2* __restrict__ jobs, int nvlo, int Tmax, int convert) {
  __shared__ __align__(16) float wstage[kWarpTreeWarps][NVB * 64];
  __shared__ unsigned vmax[kWarpTreeWarps][16];
  __shared__ int second;
  const int2 job = jobs ? jobs[blockIdx.x] : make_int2(0, (int)blockIdx.x);
  const TreeParamsM P = tree_params(mats[job.x]);
  if (P.nv < nvlo || P.nv > NVB) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, LR = P.D->LR, T = min(Tmax, P.q), L = P.q - T;
  float* wbuf = wstage[warp];
  const int64_t sub = job.y;
  for (int t = warp; t < 1 << T; t += kWarpTreeWarps)
    project_leaf_w<F, NVB>(P, LR, (sub << T) + t, lane, wbuf, vmax[warp], convert != 0);
  __syncthreads();
  for (int lvl = P.q - 1; lvl >= L; lvl--) {
    const int64_t node0 = ((int64_t)1 << lvl) - 1 + (sub << (lvl - L));
    const int nn = 1 << (lvl - L);
    if (nn >= kWarpTreeWarps || P.nv == 1) {  // a warp per node, all vectors
      for (int t = warp; t < nn; t += kWarpTreeWarps) up_node_w<F, NVB, false>(P, LR, node0 + t, lane, wbuf, 0, P.nv);
    } else {  // fewer nodes than warps: a warp per node and vector
      for (int u = warp; u < nn * P.nv; u += kWarpTreeWarps)
        up_node_w<F, 1, false>(P, LR, node0 + u % nn, lane, wbuf, u / nn, 1);
    }
    __syncthreads();
  }
  __threadfence();
  __syncthreads();
  // climb while this CTA arrives second at the parent; a warp per vector
  int64_t node = ((int64_t)1 << L) - 1 + sub;
  while (node > 0) {
    const int64_t par = (node - 1) / 2;
    if (threadIdx.x == 0) {
      second = atomicAdd(P.ticket + par, 1) == 1;
      if (second) P.ticket[par] = 0;  // both arrivals are in: reset for the next product
    }
    __syncthreads();
    if (!second) break;
    __threadfence();
    if (warp < P.nv) up_node_w<F, 1, true>(P, LR, par, lane, wbuf, warp, 1);
    __threadfence();
    __syncthreads();
    node = par;
  }
}

// child ch of the downsweep for vectors v0 .. v0 + nw - 1: yhat_ch += E_ch yhat_parent
template <int F, int NVB>
__device__ __forceinline__ void down_node_w(const TreeParamsM& P, int LR, int64_t ch, int lane, float* wbuf, int v0, int nw) {
  float acc[1][NVB];
#pragma unroll
  for (int v = 0; v < NVB; v++) acc[0][v] = 0.f;
  stage_vectors(wbuf, P.yhat + (((ch - 1) / 2) * P.nv + v0) * P.kp, nw * P.kp, lane);
  warp_mv_m<F, 1, NVB>(TreeOpM<F>::E(P, ch), TreeOpM<F>::bE(P, ch), P.k, P.k, LR, wbuf, P.kp, nw, acc, lane);
  __syncwarp();
  group_reduce_m(acc, LR);
  store_node_m<1, NVB, true>(P.yhat + (ch * P.nv + v0) * P.kp, P.k, P.kp, LR, nw, acc, lane);
}

// leaf j's expansion (Eq. 4): a lane owns rows lane and lane + 32, eight columns' loads before their use
template <int F, int NVB>
__device__ __forceinline__ void expand_leaf_w(const TreeParamsM& P, int64_t j, int lane, float* wbuf, bool assign) {
  using Op = TreeOpM<F>;
  const typename Op::Leaf l = Op::leaf_u(P, j);
  stage_vectors(wbuf, P.yhat + ((((int64_t)1 << P.q) - 1 + j) * P.nv) * P.kp, P.nv * P.kp, lane);
  const typename Op::A* U = reinterpret_cast<const typename Op::A*>(Op::U(P, l));
  int roff[2], cs = l.s;
#pragma unroll
  for (int r = 0; r < 2; r++) {
    roff[r] = lane + 32 * r;
    Op::u_layout(P, l, lane + 32 * r, roff[r], cs);
  }
  float acc[2][NVB];
#pragma unroll
  for (int r = 0; r < 2; r++)
#pragma unroll
    for (int v = 0; v < NVB; v++) acc[r][v] = 0.f;
  for (int nu0 = 0; nu0 < P.k; nu0 += 8) {
    float u[8][2];
#pragma unroll
    for (int c = 0; c < 8; c++)
#pragma unroll
      for (int r = 0; r < 2; r++)
        u[c][r] = lane + 32 * r < l.s && nu0 + c < P.k ? code_to_f<F>(__ldg(U + roff[r] + cs * (nu0 + c))) : 0.f;
#pragma unroll
    for (int c = 0; c < 8; c++) {
      if (nu0 + c >= P.k) break;
#pragma unroll
      for (int v = 0; v < NVB; v++) {
        const float yv = v < P.nv ? wbuf[v * P.kp + nu0 + c] : 0.f;
        acc[0][v] = fmaf(u[c][0], yv, acc[0][v]);
        acc[1][v] = fmaf(u[c][1], yv, acc[1][v]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 2; r++)
#pragma unroll
    for (int v = 0; v < NVB; v++)
      if (lane + 32 * r < l.s && v < P.nv) Op::ystore(P, l, v, lane + 32 * r, l.bU * acc[r][v], assign);
  __syncwarp();  // wbuf is reused by the warp's next leaf
}

// the whole downsweep (Alg. 4, Eq. 5); expand as tree_down
template <int F, int NVB>
__global__ void __launch_bounds__(kWarpTreeWarps * 32, NVB == 8 ? 3 : 4) k_downsweep_warps(const MatDesc* __restrict__ mats,
                                                                        const int2* __restrict__ jobs, int nvlo, int Tmax, int expand) {
  __shared__ float path[2][NVB][64];
  __shared__ __align__(16) float wstage[kWarpTreeWarps][NVB * 64];
  const int2 job = jobs ? jobs[blockIdx.x] : make_int2(0, (int)blockIdx.x);
  const TreeParamsM P = tree_params(mats[job.x]);
  if (P.nv < nvlo || P.nv > NVB) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, LR = P.D->LR, T = min(Tmax, P.q), L = P.q - T;
  float* wbuf = wstage[warp];
  const int64_t sub = job.y, root = ((int64_t)1 << L) - 1 + sub;
  // the path from the root to the subtree's root, recomputed by every CTA, a warp per vector (only the subtree's
  // own root is stored: the nodes above belong to several CTAs)
  if (L > 0 && warp < P.nv) {
    int cur = 0;
    for (int r = lane; r < P.k; r += 32) path[0][warp][r] = P.yhat[(int64_t)warp * P.kp + r];
    __syncwarp();
    for (int l = 1; l <= L; l++) {
      const int64_t a = ((root + 1) >> (L - l)) - 1;
      float acc[1][1] = {{0.f}};
      warp_mv_m<F, 1, 1>(TreeOpM<F>::E(P, a), TreeOpM<F>::bE(P, a), P.k, P.k, LR, path[cur][warp], 64, 1, acc, lane);
      group_reduce_m(acc, LR);
      if (lane < P.k && lane < LR) {
        float* at = P.yhat + (a * P.nv + warp) * P.kp + lane;
        const float val = acc[0][0] + *at;
        if (l == L) *at = val;
        else path[cur ^ 1][warp][lane] = val;
      }
      __syncwarp();
      cur ^= 1;
    }
  }
  __syncthreads();
  for (int lvl = L + 1; lvl <= P.q; lvl++) {
    const int64_t node0 = ((int64_t)1 << lvl) - 1 + (sub << (lvl - L));
    const int nn = 1 << (lvl - L);
    if (nn >= kWarpTreeWarps || P.nv == 1) {
      for (int t = warp; t < nn; t += kWarpTreeWarps) down_node_w<F, NVB>(P, LR, node0 + t, lane, wbuf, 0, P.nv);
    } else {
      for (int u = warp; u < nn * P.nv; u += kWarpTreeWarps) down_node_w<F, 1>(P, LR, node0 + u % nn, lane, wbuf, u / nn, 1);
    }
    __syncthreads();
  }
  if (expand)  // the leaves' yhat is final
    for (int t = warp; t < 1 << T; t += kWarpTreeWarps) expand_leaf_w<F, NVB>(P, (sub << T) + t, lane, wbuf, expand == 2);
}

}  // namespace h2
