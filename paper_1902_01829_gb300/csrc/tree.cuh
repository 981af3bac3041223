// The tree phases of the product (leaf projection, upsweep, downsweep, leaf expansion), one launch
// each, shared by the FP64 form (double-float arithmetic, hmv_fp64.cuh) and the scaled forms
// (mixed.cuh). `Op` supplies the element types, the arithmetic and where a node's blocks are.
//
// What bounds them: latency. The bytes are about a hundredth of the product's, but an output at the
// root hangs on q dependent levels. A CTA owns the subtree below one node of level L and takes its
// leaves and nodes one after another, all warps on each block:
//  - every step is the same piece of code, "rows += A x" for a block A in shared memory: a step runs
//    once per level, and an unrolled copy per use spent more time on instruction fetches than on
//    arithmetic (17 us for the first 64 x 64 FP64 nodes of a level).
//  - nothing in a step waits for global memory: the next block is copied into shared memory (cp.async)
//    while the current one is multiplied, its scale and the next leaf's x are loaded a step ahead, the
//    leaves' offsets sit in a table, and the vectors of a CTA's own nodes stay in shared memory. (Each
//    dependent load cost a step 700 cycles, a third of it.)
//  - above L the upsweep goes on in clusters of eight CTAs, whose nodes' vectors pass through distributed
//    shared memory with a cluster barrier per level; a node's xhat is stored after that barrier, so
//    that the barrier does not wait for the store. Above the cluster, one ticket per five levels: the last
//    of up to 32 clusters below a node computes the levels up to it, its CTAs sharing each level's
//    nodes. One ticket per level (fence, atomic, reload through L2) cost 2.5 us a level.
//  - the downsweep's path from the root to the subtree is recomputed by every CTA.
// Measured (upsweep with the vectors' conversion / downsweep with expansion, phases in order, us; one warp per node and a
// ticket per level before): 2D n = 50,001 FP64, 16 vectors 294 / 184 -> 89 / 55; 2D n = 2^16 int16, 16 vectors 68 / 41 ->
// 46 / 35; 3D n = 2^14 bf16, k = 64, 16 vectors 160 / 62 -> 77 / 41; 3D n = 2^16 int16, 8 vectors 203 / 157 -> 78 / 58;
// 3D n = 2^14 FP64, one vector 169 / 69 -> 83 / 49. Where the nodes outnumber the chip's warps a warp per node is the better
// one: tree_warps.cuh, for the scaled forms. A step is still bound by the length of its instruction
// chain (about 4.5 cycles an instruction, one warp per scheduler): 2,000 cycles.
#pragma once
#include <cooperative_groups.h>
#include <cstdint>
#include <cuda_runtime.h>

namespace h2 {

namespace cg = cooperative_groups;

constexpr int kTreeClusterLog = 3, kTreeCluster = 1 << kTreeClusterLog;  // CTAs (subtrees) per cluster of the upsweep

// With fewer subtrees (2^L) than a cluster has CTAs, subtree s is on rank s << tree_spread(L): a level of nn
// nodes is climbed on ranks 0, 8 / nn, ..., the subtrees' roots like the levels above them.
__host__ __device__ constexpr int tree_spread(int L) { return L < kTreeClusterLog ? kTreeClusterLog - L : 0; }

// warps per CTA: a step has (rows / 8) x (vectors / 4) tasks of a warp
template <int NVB>
__host__ __device__ constexpr int tree_warps() { return NVB >= 4 ? 8 : 4; }
// vectors of a task, and the stride of a row's vectors in shared memory (16-byte groups of four)
template <int NVB>
__host__ __device__ constexpr int tree_slice() { return NVB < 4 ? NVB : 4; }
template <int NVB>
__host__ __device__ constexpr int tree_vstride() { return NVB >= 8 ? NVB + 4 : NVB; }

// elements of a k-row vector area (a multiple of 16 bytes)
template <int NVB>
__host__ __device__ constexpr int tree_area(int k) { return (k * tree_vstride<NVB>() + 3) & ~3; }

// Dynamic shared memory of a tree CTA: nbuf block buffers of `block` bytes, two vector areas of 64 rows
// (a leaf's points, a pair of children, a path node), then 2 + T vector areas of k rows, the leaf table,
// the leaves' maxima and a flag.
struct TreeSmem {
  int block, nbuf, table, bytes;
};
template <class Op, int NVB>
__host__ __device__ inline TreeSmem tree_smem(int k, int block_entries, int T) {
  TreeSmem S;
  S.block = (block_entries * (int)sizeof(typename Op::A) + 15) & ~15;
  // one buffer where two would leave one CTA per SM (64 x 64 FP64 pairs), or, for passes of up to four
  // vectors, would not fit beside the dense stream's CTA (kTreeReserve)
  S.nbuf = S.block <= (NVB >= 8 ? 32768 : 10240) ? 2 : 1;
  S.table = (S.nbuf * S.block + (2 * 64 * tree_vstride<NVB>() + (2 + T) * tree_area<NVB>(k)) * (int)sizeof(typename Op::V) + 15) & ~15;
  S.bytes = S.table + (((1 << T) * (int)sizeof(typename Op::Leaf) + 15) & ~15) + 16 + 3 * 64;
  return S;
}
// i / k for i < 4096, k <= 64, as a multiplication (m = div_magic(k))
__device__ __forceinline__ unsigned div_magic(int k) { return (1u << 19) / (unsigned)k + 1u; }
__device__ __forceinline__ int div_by(int i, unsigned m) { return (int)(((unsigned)i * m) >> 19); }
// entries of the largest block a tree kernel copies: a leaf's 64 x k (panel layout: and its pads) or two transfers
__host__ __device__ inline int tree_block_entries(int k, int64_t kks, bool panel) {
  const int leaf = 64 * k + (panel ? 64 : 0), pair = (int)(2 * kks);
  return leaf > pair ? leaf : pair;
}

// the same for the downsweep: a leaf's 64 x k or one transfer
__host__ __device__ inline int tree_down_entries(int k, int64_t kks, bool panel) {
  const int leaf = 64 * k + (panel ? 64 : 0);
  return leaf > kks ? leaf : (int)kks;
}

// copy `bytes` (a multiple of Op::kCopy, both ends so aligned) into shared memory, asynchronously
template <int W>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src) {
  if (W == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(W) : "memory");
}
template <int W, int THREADS>
__device__ __forceinline__ void copy_block(unsigned char* dst, const void* src, int bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  const unsigned char* s = static_cast<const unsigned char*>(src);
#pragma unroll 4
  for (int i = threadIdx.x * W; i < bytes; i += THREADS * W) cp_async<W>(d + i, s + i);
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One step's product for a task: acc[v] = sum_b (sum_c A_b(row, c) x_b(c, v0 + v)), entry (row, c) of block b
// at A + b * abs + roff + c * cs in shared memory, the vectors at x_b + c * VS. Lane (rl, g) of a warp owns
// row 8 rb + rl and the columns g, g + 4, ...; the sums over g are joined by shuffles, every lane of a row
// ends with its totals. Vectors past nv multiply whatever their slots hold and are dropped by the caller.
template <class Op, int NVB>
__device__ __forceinline__ void tree_product(const typename Op::A* A, int abs, int roff, int cs, bool ok, int C, int NB,
                                             const typename Op::V* x0, const typename Op::V* x1, int v0,
                                             typename Op::Blk b0, typename Op::Blk b1,
                                             typename Op::Acc (&acc)[tree_slice<NVB>()]) {
  using V = typename Op::V;
  constexpr int VW = tree_slice<NVB>(), VS = tree_vstride<NVB>();
  const int g = (threadIdx.x >> 3) & 3;
#pragma unroll 1
  for (int b = 0; b < NB; b++) {
    typename Op::Acc p[VW] = {};
    const typename Op::Blk blk = b ? b1 : b0;
    const V* x = (b ? x1 : x0) + v0;
    const typename Op::A* a = A + b * abs + roff;
#pragma unroll Op::kUnroll
    for (int c = g; c < C; c += 4) {
      V xv[VW];
      if constexpr (VW == 4) {
        const float4* src = reinterpret_cast<const float4*>(x + c * VS);
#pragma unroll
        for (int i = 0; i < (int)sizeof(V); i += 4) reinterpret_cast<float4*>(xv)[i / 4] = src[i / 4];
      } else {
#pragma unroll
        for (int v = 0; v < VW; v++) xv[v] = x[c * VS + v];
      }
      const auto e = Op::prep(ok ? a[c * cs] : Op::none(), blk);
#pragma unroll
      for (int v = 0; v < VW; v++) Op::fma(p[v], e, xv[v]);
    }
#pragma unroll
    for (int v = 0; v < VW; v++) {
      Op::scale(p[v], blk);
      if (b) Op::add(acc[v], p[v]);
      else acc[v] = p[v];
    }
  }
#pragma unroll
  for (int off = 8; off < 32; off <<= 1)
#pragma unroll
    for (int v = 0; v < VW; v++) Op::add(acc[v], Op::shfl_xor(acc[v], off));
}

// element v of acc for lane group g: the four lanes of a row write four vectors at once
template <class Op, int VW>
__device__ __forceinline__ typename Op::Acc tree_pick(const typename Op::Acc (&acc)[VW], int g) {
  typename Op::Acc r = acc[0];
#pragma unroll
  for (int v = 1; v < VW; v++)
    if (g == v) r = acc[v];
  return r;
}

// Leaf projection and the whole upsweep (Alg. 2, Eq. 2) of subtree `sub` (active: this CTA has one; a CTA
// without passes its cluster's first subtree and takes part in the barriers only). Subtrees are on the
// clusters' ranks in order, eight to a cluster (fewer in all: tree_spread). The subtree's steps
// follow a binary counter: leaf, leaf, their parent, leaf, ... convert: x(j) is copied into the product's
// own layout and type here (else a kernel before this one did it).
// CLUSTER false: the CTA climbs alone, with a ticket per level. A cluster needs room on eight SMs of a GPC at
// once and found none beside the dense stream until that had ended (2D n = 2^17, one vector: upsweep done
// after 86 us of 92 beside it; alone 25), so passes whose phases overlap take this variant.
template <class Op, int NVB, bool CLUSTER>
__device__ __forceinline__ void tree_up(const typename Op::P& P, int64_t sub, bool active, bool convert, int T_smem,
                                        int block_entries) {
  using V = typename Op::V;
  using Blk = typename Op::Blk;
  using Leaf = typename Op::Leaf;
  constexpr int VW = tree_slice<NVB>(), VS = tree_vstride<NVB>(), TW = tree_warps<NVB>(), TH = TW * 32;
  constexpr int XN = (64 * NVB + TH - 1) / TH;
  extern __shared__ __align__(16) unsigned char tree_dyn[];
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int CLOG = CLUSTER ? kTreeClusterLog : 0, CS = 1 << CLOG;
  const int k = P.k, nv = P.nv, T = P.q - P.L, rank = CLUSTER ? (int)cluster.block_rank() : 0;
  auto group_sync = [&] {
    if constexpr (CLUSTER) cluster.sync();
    else __syncthreads();
  };
  const TreeSmem S = tree_smem<Op, NVB>(k, block_entries, T_smem);
  V* xbuf = reinterpret_cast<V*>(tree_dyn + S.nbuf * S.block);  // two areas of 64 rows
  V* nodes = xbuf + 2 * 64 * VS;                                // right results (by depth parity), then left ones by depth
  Leaf* table = reinterpret_cast<Leaf*>(tree_dyn + S.table);
  int* won_s = reinterpret_cast<int*>(tree_dyn + S.bytes - 16);
  unsigned* vmax = reinterpret_cast<unsigned*>(tree_dyn + S.bytes - 16 - 3 * 64);  // max |x| per vector of a leaf, three leaves in turn
  const int warp = threadIdx.x >> 5, rl = threadIdx.x & 7, g = (threadIdx.x >> 3) & 3;
  const int64_t j0 = sub << T, leaf0 = ((int64_t)1 << P.q) - 1, vs = (int64_t)nv * P.kp;
  const int kr = (k + 7) / 8, krl = 32 - __clz(kr - 1), ns = (nv + VW - 1) / VW, nt = ns << krl;
  const unsigned kdiv = div_magic(k);
  const int AS = tree_area<NVB>(k);

  bool parts = false;  // the dense phase wants the vectors as 16-bit parts too
  if constexpr (Op::kParts) parts = convert && Op::want_parts(P);
  typename Op::X xr[XN];  // the next leaf's x: point tid % 64 of vectors tid / 64 + (TH / 64) i
  const int xa = threadIdx.x & 63, xv0 = threadIdx.x >> 6;
  int buf = 0;
  Blk nb0{}, nb1{};  // the next step's scales
  // start the loads a step needs: leaf t and its x, or the transfers of node par's children
  auto fetch_leaf = [&](int t, int to) {
    const Leaf lf = table[t];
    nb0 = nb1 = lf.bV;
    copy_block<Op::kCopy, TH>(tree_dyn + to * S.block, Op::Vt(P, lf), Op::copy_bytes(k * lf.s));
#pragma unroll
    for (int i = 0; i < XN; i++) {
      const int v = xv0 + (TH / 64) * i;
      xr[i] = (v < nv && xa < lf.s) ? Op::xload(P, lf, v, xa, convert) : typename Op::X{};
    }
  };
  auto fetch_node = [&](int64_t par, int to) {
    nb0 = Op::bF(P, 2 * par + 1);
    nb1 = Op::bF(P, 2 * par + 2);
    copy_block<Op::kCopy, TH>(tree_dyn + to * S.block, Op::Ft(P, 2 * par + 1), Op::copy_bytes((int)(2 * P.kks)));
  };

  // ---- climb state: level l of the step towards level up below ancestor anc. A level of nn nodes below anc
  // is on ranks 0, 8 / nn, ... (nn <= 8) or nn / 8 per rank; cv: where a rank's last result is (the same
  // place on every rank), from_global: the step's first level takes its children from other clusters.
  int l = P.L, up = P.L - min(P.L, CLOG);
  int64_t anc = sub >> (P.L - up), cnode = 0, pend = -1;
  int crem = 0, cstep = 1;
  bool from_global = false, climbing = !active;
  V* cv = T == 0 ? nodes : xbuf;
  // xhat of this rank's last node, stored once its cluster barrier is past
  auto store_pending = [&]() {
    if (pend < 0) return;
    for (int i = threadIdx.x; i < nv * k; i += TH) {
      const int v = div_by(i, kdiv), r = i - v * k;
      P.xhat[pend * vs + v * P.kp + r] = cv[r * VS + v];
    }
    pend = -1;
  };
  // the next node of the climb for this CTA (its loads started, its children complete), or -1
  auto climb_next = [&]() -> int64_t {
    if (crem > 0) {
      crem--;
      return ++cnode;
    }
    for (;;) {
      if (l == up) {
        if (up == 0) {
          group_sync();  // no CTA ends while another may read its shared memory
          store_pending();
          return -1;
        }
        const int steps = (up + 4) / 5, St = CLUSTER ? (up + steps - 1) / steps : 1;
        up -= St;
        anc >>= St;
        __syncthreads();
        store_pending();
        group_sync();
        if (rank == 0 && threadIdx.x == 0) {
          int* t = P.ticket + ((int64_t)1 << up) - 1 + anc;
          __threadfence();  // the cluster's xhat stores (ordered before this by its barrier) before the ticket
          const int won = atomicAdd(t, 1) == (1 << St) - 1;
          if (won) *t = 0;  // all arrivals are in: reset for the next product
          __threadfence();  // order the others' xhat (published before their tickets) before our reads
          if constexpr (CLUSTER) {
            for (int r = 0; r < CS; r++) *cluster.map_shared_rank(won_s, r) = won;
          } else {
            *won_s = won;
          }
        }
        group_sync();
        if (!*won_s) return -1;
        from_global = true;
      } else {
        from_global = false;
      }
      l--;
      const int nn = 1 << (l - up), per = max(1, nn / CS);
      cstep = max(1, CS / nn);
      const bool mine = rank % cstep == 0;
      cnode = ((int64_t)1 << l) - 1 + (anc << (l - up)) + rank / cstep * per;
      if (mine) fetch_node(cnode, buf);
      if (!from_global || per > 1) group_sync();  // the children's vectors on every rank
      store_pending();
      if (mine) {
        crem = per - 1;
        return cnode;
      }
      cv = from_global || cv != nodes ? nodes : xbuf;  // (where the active ranks leave this level's results)
    }
  };

  if (active) {
    for (int i = threadIdx.x; i < (1 << T); i += TH) table[i] = Op::leaf_v(P, j0 + i);
    if (threadIdx.x < 48) vmax[threadIdx.x] = 0u;
    __syncthreads();
  }
  int t = 0, d = 0;
  int64_t node = leaf0 + j0;
  if (active) fetch_leaf(0, 0);
  else if ((node = climb_next()) < 0) return;
  auto slot = [&](int tt, int dd) { return nodes + (((tt >> dd) & 1) ? (dd & 1) : 2 + dd) * AS; };
#pragma unroll 1
  for (;;) {
    const V *x0, *x1;
    V* out;
    int C = k, NB = 2;
    const Blk b0 = nb0, b1 = nb1;
    bool store = true;
    if (!climbing) {
      out = d < T ? slot(t, d) : cv;
      if (d == 0) {  // leaf: its x into shared memory and the product's own layout
        const Leaf lf = table[t];
        const int sp = Op::spad(lf.s);
        V* xs = xbuf + (t & 1) * 64 * VS;
#pragma unroll
        for (int i = 0; i < XN; i++) {
          const int v = xv0 + (TH / 64) * i;
          if (v < nv) {  // (the same for the whole warp)
            const V val = Op::xvalue(P, xr[i], v);
            if (xa < lf.s) xs[xa * VS + v] = val;
            if (convert && xa < sp) Op::xstore(P, lf, sp, v, xa, val);  // (the padding is zero)
            if constexpr (Op::kParts) {
              if (parts) {
                const unsigned m = __reduce_max_sync(0xFFFFFFFFu, xa < lf.s ? Op::abs_bits(val) : 0u);
                if ((threadIdx.x & 31) == 0) atomicMax(vmax + 16 * (t % 3) + v, m);
              }
            }
          }
        }
        // cleared for the next leaf: its last reader was the leaf before the last one, a barrier ago
        if (parts && threadIdx.x < 16) vmax[16 * ((t + 1) % 3) + threadIdx.x] = 0u;
        x0 = x1 = xs;
        C = lf.s;
        NB = 1;
      } else {
        x0 = slot(t & ~(1 << (d - 1)), d - 1);
        x1 = slot(t, d - 1);
      }
      if (d == T) {
        store = false;  // after the first cluster barrier
        pend = node;
        if (P.L == 0) store = true, pend = -1;
      }
    } else if (from_global) {  // the children's vectors through L2
      const int64_t ch = 2 * node + 1;
      for (int i = threadIdx.x; i < 2 * nv * k; i += TH) {
        const int b = i >= nv * k, r = i - b * nv * k, v = div_by(r, kdiv), c = r - v * k;
        xbuf[b * 64 * VS + c * VS + v] = __ldcg(P.xhat + (ch + b) * vs + v * P.kp + c);
      }
      x0 = xbuf;
      x1 = xbuf + 64 * VS;
      out = cv = nodes;
      if (crem > 0) out = nodes;
      else if (cstep == 1 && (1 << (l - up)) > CS) out = nodes + AS;  // the second of a pair
      store = (1 << (l - up)) > CS;
      if (!store) pend = node;
    } else {
      x0 = cv;
      if (cstep == 1) {  // both children on this rank: a pair's two results
        x1 = nodes + AS;
      } else if constexpr (CLUSTER) {  // the right child from the rank cstep / 2 further on
        const float4* src = reinterpret_cast<const float4*>(cluster.map_shared_rank(cv, rank + cstep / 2));
        float4* dst = reinterpret_cast<float4*>(nodes + AS);
        for (int i = threadIdx.x; i < AS * (int)sizeof(V) / 16; i += TH) dst[i] = src[i];
        x1 = nodes + AS;
      }
      out = cv = cv == nodes ? xbuf : nodes;
      pend = node;
      store = false;
    }
    cp_async_wait();
    __syncthreads();
    const int cur = buf;
    auto fetch_next = [&](int to) {  // the step after this one, where it is known already
      if (climbing) {
        if (crem > 0) fetch_node(cnode + 1, to);
      } else if (d < T && ((t >> d) & 1)) {
        fetch_node(((int64_t)1 << (P.q - d - 1)) - 1 + ((j0 + t) >> (d + 1)), to);
      } else if (t + 1 < (1 << T)) {
        fetch_leaf(t + 1, to);
      }
    };
    if (S.nbuf == 2) fetch_next(buf = cur ^ 1);
    if constexpr (Op::kParts) {
      if (parts && !climbing && d == 0) Op::parts(P, j0 + t, C, x0, VS, 1, vmax + 16 * (t % 3), threadIdx.x, TH);
    }
    const typename Op::A* A = reinterpret_cast<const typename Op::A*>(tree_dyn + cur * S.block);
#pragma unroll 1
    for (int u = warp; u < nt; u += TW) {
      const int rb = u & ((1 << krl) - 1), v0 = (u >> krl) * VW, row = 8 * rb + rl;
      if (rb >= kr) continue;
      typename Op::Acc acc[VW];
      tree_product<Op, NVB>(A, (int)P.kks, row, k, row < k, C, NB, x0, x1, v0, b0, b1, acc);
      const int v = v0 + g;
      if (g < VW && row < k && v < nv) {
        const V val = Op::value(tree_pick<Op, VW>(acc, g));
        if (store) P.xhat[node * vs + v * P.kp + row] = val;
        out[row * VS + v] = val;
      }
    }
    if (S.nbuf == 1) {
      __syncthreads();
      fetch_next(0);
    } else if (climbing && crem > 0) {
      __syncthreads();  // the children's area is rewritten by the next node
    }
    if (!climbing) {
      if (d < T && ((t >> d) & 1)) {
        d++;
        node = ((int64_t)1 << (P.q - d)) - 1 + ((j0 + t) >> d);
        continue;
      }
      if (t + 1 < (1 << T)) {
        t++;
        d = 0;
        node = leaf0 + j0 + t;
        continue;
      }
      climbing = true;
    }
    if ((node = climb_next()) < 0) return;
  }
}

// The whole downsweep (Alg. 4, Eq. 5) of subtree `sub`: yhat_c += E_c yhat_parent along the path from the
// root to the subtree's root (its nodes are shared with other CTAs, so their sums stay in this CTA's shared
// memory), then over the subtree in pre-order; only the leaves' yhat is written back. expand: after a leaf,
// its basis U_j is multiplied with its yhat (Eq. 4) and the rows go to Op::ystore (2: assigned, 1: added).
template <class Op, int NVB>
__device__ __forceinline__ void tree_down(const typename Op::P& P, int64_t sub, int expand, int T_smem, int block_entries) {
  using V = typename Op::V;
  using Blk = typename Op::Blk;
  using Leaf = typename Op::Leaf;
  constexpr int VW = tree_slice<NVB>(), VS = tree_vstride<NVB>(), TW = tree_warps<NVB>(), TH = TW * 32;
  constexpr int ON = (64 * NVB + TH - 1) / TH;
  extern __shared__ __align__(16) unsigned char tree_dyn[];
  const int k = P.k, nv = P.nv, L = P.L, T = P.q - L;
  const TreeSmem S = tree_smem<Op, NVB>(k, block_entries, T_smem);
  V* own = reinterpret_cast<V*>(tree_dyn + S.nbuf * S.block);  // two areas: the node's own yhat
  V* slots = own + 2 * 64 * VS;                                // path parity 0, 1; then depths 1 .. T
  Leaf* table = reinterpret_cast<Leaf*>(tree_dyn + S.table);
  const int warp = threadIdx.x >> 5, rl = threadIdx.x & 7, g = (threadIdx.x >> 3) & 3;
  const int64_t vs = (int64_t)nv * P.kp, root = ((int64_t)1 << L) - 1 + sub;
  const int ns = (nv + VW - 1) / VW;
  const unsigned kdiv = div_magic(k);
  const int AS = tree_area<NVB>(k);
  // step (dep, n): dep <= 0 the path's node of level L + dep (n unused), dep > 0 node n of the subtree's
  // level dep; expanding: leaf n's expansion
  int dep = L > 0 ? 1 - L : 0, n = 0, buf = 0;
  bool expanding = false;
  auto node_of = [&](int dp, int nn) {
    return dp <= 0 ? ((root + 1) >> -dp) - 1 : ((int64_t)1 << (L + dp)) - 1 + (sub << dp) + nn;
  };
  auto slot_of = [&](int dp) { return slots + (dp <= 0 ? ((L + dp) & 1) : 1 + dp) * AS; };
  // on to the next step; false: none
  auto advance = [&]() -> bool {
    if (!expanding && dep >= T && expand) return expanding = true;
    expanding = false;
    if (dep < T) {
      dep++;
      n = dep == 1 ? 0 : 2 * n;
      return true;
    }
    while (dep > 0 && (n & 1)) {
      n >>= 1;
      dep--;
    }
    if (dep <= 0) return false;
    n++;
    return true;
  };
  V on[ON];  // the next node's own yhat: entry threadIdx.x + TH i of [v][row]
  Blk nb{};
  auto fetch = [&](int to) {  // start the loads of step (dep, n, expanding)
    if (expanding) {
      const Leaf& lf = table[n];
      nb = lf.bU;
      copy_block<Op::kCopy, TH>(tree_dyn + to * S.block, Op::U(P, lf), Op::u_bytes(P, lf));
      return;
    }
    const int64_t a = node_of(dep, n);
    nb = Op::bE(P, a);
    copy_block<Op::kCopy, TH>(tree_dyn + to * S.block, Op::E(P, a), Op::copy_bytes((int)P.kks));
#pragma unroll
    for (int i = 0; i < ON; i++) {
      const int e = threadIdx.x + TH * i, v = div_by(e, kdiv);
      on[i] = e < nv * k ? P.yhat[a * vs + v * P.kp + (e - v * k)] : V{};
    }
  };
  if (expand) {
    for (int i = threadIdx.x; i < (1 << T); i += TH) table[i] = Op::leaf_u(P, (sub << T) + i);
  }
  for (int i = threadIdx.x; i < nv * k; i += TH) {  // the root's yhat
    const int v = div_by(i, kdiv), r = i - v * k;
    slot_of(-L)[r * VS + v] = P.yhat[v * P.kp + r];
  }
  __syncthreads();
  if (L == 0 && !advance()) return;  // the subtree's root is the root: its first child, or (one leaf) its expansion
  fetch(0);
#pragma unroll 1
  for (;;) {
    const bool ex = expanding;
    const int dp = dep, j = n, cur = buf;
    const int64_t a = node_of(dp, n);
    const Blk blk = nb;
    V* ow = own + (cur & 1) * 64 * VS;
    if (!ex) {
#pragma unroll
      for (int i = 0; i < ON; i++) {
        const int e = threadIdx.x + TH * i, v = div_by(e, kdiv);
        if (e < nv * k) ow[(e - v * k) * VS + v] = on[i];
      }
    }
    cp_async_wait();
    __syncthreads();
    const V* x = ex ? slot_of(dp) : slot_of(dp - 1);
    V* out = slot_of(dp);
    const int rows = ex ? table[j].s : k;
    const bool more = advance();
    if (S.nbuf == 2 && more) fetch(buf = cur ^ 1);
    const typename Op::A* A = reinterpret_cast<const typename Op::A*>(tree_dyn + cur * S.block);
    const int kr = (rows + 7) / 8, krl = 32 - __clz(kr - 1);
#pragma unroll 1
    for (int u = warp; u < ns << krl; u += TW) {
      const int rb = u & ((1 << krl) - 1), v0 = (u >> krl) * VW, row = 8 * rb + rl, v = v0 + g;
      if (rb >= kr) continue;
      int roff = row, cs = rows;
      if (ex) Op::u_layout(P, table[j], row, roff, cs);
      typename Op::Acc acc[VW];
      tree_product<Op, NVB>(A, 0, roff, cs, row < rows, k, 1, x, x, v0, blk, blk, acc);
      if (g < VW && row < rows && v < nv) {
        typename Op::Acc r = tree_pick<Op, VW>(acc, g);
        if (ex) {
          Op::ystore(P, table[j], v, row, r, expand == 2);
        } else {
          Op::add_value(r, ow[row * VS + v]);
          const V val = Op::value(r);
          out[row * VS + v] = val;
          if (dp == T) P.yhat[a * vs + v * P.kp + row] = val;
        }
      }
    }
    if (!more) return;
    if (S.nbuf == 1) {
      __syncthreads();
      fetch(0);
    }
  }
}

}  // namespace h2
