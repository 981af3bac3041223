// FP64 plain-form kernels of the H^2 matrix-vector product (Sec. 4.2 - 4.4): the tree phases
// (tree.cuh with double-float arithmetic), the coupling phase and the per-vector scale.
//
// Each phase is a sum of column-major block products "rows += A_block * x_cols":
//   leaf projection  xhat_j  = V_j^T x(j)            A = V_j^T (stored transposed)
//   upsweep          xhat_p  = sum_c F_c^T xhat_c    A = F_c^T (stored transposed)   Eq. 2
//   coupling         yhat_i  = sum_j S_ij xhat_j     A = S_ij                        Eq. 3
//   downsweep        yhat_c += E_c yhat_p            A = E_c                         Eq. 5
// A lane owns output rows, consecutive lanes read consecutive rows of a column (coalesced), the
// column's input entry is a broadcast, and products accumulate in double-float. Loads of several
// columns are issued before any of them is used, so a warp keeps many in flight.
//
// Range: every block is split with its exponent offset o (a' = a * 2^-o, see
// df64.cuh) and x is scaled per vector by 2^-vexp[v], so that x, xhat and yhat
// hold values of magnitude at most about 1 (bounds computed by h2_create).
//
// Workspace layouts (float2 = double-float hi, lo; kp = k rounded up to even):
//   x2    leaf j's chunk at xp_off[j] * nv: [v][spad_j] (spad = leaf size rounded up to even)
//   xhat  [(node * nv + v) * kp + row]   vector trees of Sec. 4.2 - 4.4
//   yhat  same as xhat
#pragma once
#include "df64.cuh"
#include "mma_fp64.cuh"
#include "tree.cuh"

namespace h2 {

constexpr int kWarps = 4;  // warps per CTA for the per-node kernels

// Row mapping of a warp over an R-row block: lane = g * LR + rl owns rows
// rl + 32 r (r < RPL) and columns col = g, g + G, ... with G = 32 / LR groups.
// RPL = 2 requires LR = 32 (R <= 64); RPL = 1 allows LR = 1 .. 32 (R <= LR).
// xin is read with plain loads
template <int RPL, int NVB>
__device__ __forceinline__ void warp_mv(const double* __restrict__ A, int o, int R, int C, int LR, const float2* xin,
                                             int64_t xstride, int nv, float (&s)[RPL][NVB], float (&c)[RPL][NVB], int lane) {
  constexpr int UB = (NVB <= 2) ? 8 : (NVB <= 4 ? 4 : 2);  // columns whose loads are issued together
  const int G = 32 / LR;
  const int g = lane / LR, rl = lane - g * LR;
  for (int col0 = g; col0 < C; col0 += UB * G) {
    double a[UB][RPL];
    float2 xv[UB][NVB];
#pragma unroll
    for (int u = 0; u < UB; u++) {
      const int col = col0 + u * G;
#pragma unroll
      for (int r = 0; r < RPL; r++) {
        const int row = rl + 32 * r;
        a[u][r] = (col < C && row < R) ? __ldg(A + row + (int64_t)R * col) : 0.0;
      }
#pragma unroll
      for (int v = 0; v < NVB; v++)
        xv[u][v] = (col < C && v < nv) ? xin[v * xstride + col] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < UB; u++) {
#pragma unroll
      for (int r = 0; r < RPL; r++) {
        float ah, al;
        split_f64(a[u][r], o, ah, al);
#pragma unroll
        for (int v = 0; v < NVB; v++) df_fma(s[r][v], c[r][v], ah, al, xv[u][v].x, xv[u][v].y);
      }
    }
  }
}

// (S, C) += (s, c) elementwise, (s, c) = 0
template <int RPL, int NVB>
__device__ __forceinline__ void acc_fold(float (&S)[RPL][NVB], float (&C)[RPL][NVB], float (&s)[RPL][NVB],
                                         float (&c)[RPL][NVB]) {
#pragma unroll
  for (int r = 0; r < RPL; r++)
#pragma unroll
    for (int v = 0; v < NVB; v++) df_fold(S[r][v], C[r][v], s[r][v], c[r][v]);
}

template <int RPL, int NVB>
__device__ __forceinline__ void acc_zero(float (&s)[RPL][NVB], float (&c)[RPL][NVB]) {
#pragma unroll
  for (int r = 0; r < RPL; r++)
#pragma unroll
    for (int v = 0; v < NVB; v++) s[r][v] = c[r][v] = 0.f;
}

// sum the partial results of the G column groups (lanes rl, rl + LR, ...)
template <int RPL, int NVB>
__device__ __forceinline__ void group_reduce(float (&s)[RPL][NVB], float (&c)[RPL][NVB], int LR) {
  for (int off = LR; off < 32; off <<= 1) {
#pragma unroll
    for (int r = 0; r < RPL; r++)
#pragma unroll
      for (int v = 0; v < NVB; v++) {
        const float s2 = __shfl_xor_sync(0xFFFFFFFFu, s[r][v], off);
        const float c2 = __shfl_xor_sync(0xFFFFFFFFu, c[r][v], off);
        df_add(s[r][v], c[r][v], s2, c2);
      }
  }
}

// ---------------------------------------------------------------- tree phases, one launch each
struct TreeParams {
  const double* Vt;        // leaf j: k x size_j (V_j^T)
  const double* Ft;        // node h >= 1: F_h^T
  const double* Et;        // node h >= 1: E_h
  const int64_t* leaf_off;
  const int64_t* xp_off;
  const double* x;         // pass input, ldx
  int64_t ldx;
  float2* x2;              // split x (padded leaf layout)
  float2* xhat;
  float2* yhat;
  int* ticket;             // one counter per node above level L, zero between products
  const int* oV;           // leaf j: exponent offset of V_j (projection)
  const int* oF;           // node h >= 1: exponent offset of F_h (upsweep into the parent)
  const int* oE;           // node h >= 1: exponent offset of E_h (downsweep from the parent)
  const int* vexp;         // per vector of the pass: x enters scaled by 2^-vexp[v]
  int64_t kks;             // doubles from a node's transfer matrix to the next node's
  int k, kp, q, L, nv;
  // passes whose dense phase is k_dense_oz: the vectors' digits (xks K steps per leaf)
  int oz, xks;
  unsigned char* xd;
  // the leaf expansion: U_j at dmat + u_off[j], its exponent offset, the rows' output exponent; added to y
  // (atomically) when the dense phase runs beside the tree phases, else assigned
  int add;
  const char* dmat;
  const int64_t* u_off;
  const int* oU;
  const int* eY;
  double* y;
  int64_t ldy;
};

// tree.cuh's arithmetic for the FP64 form: double-float vectors, FP64 entries split with their
// block's exponent offset
struct TreeOp64 {
  using P = TreeParams;
  using A = double;
  using V = float2;
  using Blk = int;
  struct Acc {
    float s, c;
  };
  static constexpr int kCopy = 8, kUnroll = 4;
  static __device__ __forceinline__ double none() { return 0.0; }
  static __device__ __forceinline__ float2 prep(double a, int o) {
    float2 e;
    split_f64(a, o, e.x, e.y);
    return e;
  }
  static __device__ __forceinline__ void fma(Acc& p, float2 e, float2 x) { df_fma(p.s, p.c, e.x, e.y, x.x, x.y); }
  static __device__ __forceinline__ void scale(Acc&, int) {}
  static __device__ __forceinline__ void add(Acc& p, const Acc& q) { df_add(p.s, p.c, q.s, q.c); }
  static __device__ __forceinline__ void add_value(Acc& p, float2 v) { df_add(p.s, p.c, v.x, v.y); }
  static __device__ __forceinline__ Acc shfl_xor(const Acc& p, int off) {
    return Acc{__shfl_xor_sync(0xFFFFFFFFu, p.s, off), __shfl_xor_sync(0xFFFFFFFFu, p.c, off)};
  }
  static __device__ __forceinline__ float2 value(const Acc& p) { return df_norm(p.s, p.c); }
  static __device__ __forceinline__ int spad(int s) { return s + (s & 1); }
  struct Leaf {
    int64_t off, xp, uoff;  // first point; offsets of the split x (per vector slot) and of U_j
    int s, bV, bU, eY;      // points; exponent offsets of V_j and U_j; the rows' output exponent
  };
  static __device__ __forceinline__ Leaf leaf_v(const P& T, int64_t j) {
    Leaf l{};
    l.off = T.leaf_off[j];
    l.s = (int)(T.leaf_off[j + 1] - l.off);
    l.xp = T.xp_off[j];
    l.bV = T.oV[j];
    return l;
  }
  static __device__ __forceinline__ Leaf leaf_u(const P& T, int64_t j) {
    Leaf l{};
    l.off = T.leaf_off[j];
    l.s = (int)(T.leaf_off[j + 1] - l.off);
    l.uoff = T.u_off[j];
    l.bU = T.oU[j];
    l.eY = T.eY[j];
    return l;
  }
  static __device__ __forceinline__ const double* Vt(const P& T, const Leaf& l) { return T.Vt + l.off * T.k; }
  static __device__ __forceinline__ const double* Ft(const P& T, int64_t h) { return T.Ft + (h - 1) * T.kks; }
  static __device__ __forceinline__ const double* E(const P& T, int64_t h) { return T.Et + (h - 1) * T.kks; }
  static __device__ __forceinline__ int bF(const P& T, int64_t h) { return T.oF[h]; }
  static __device__ __forceinline__ int bE(const P& T, int64_t h) { return T.oE[h]; }
  using X = double;
  static __device__ __forceinline__ double xload(const P& T, const Leaf& l, int v, int a, bool) {
    return __ldg(T.x + v * T.ldx + l.off + a);
  }
  static __device__ __forceinline__ float2 xvalue(const P& T, double x, int v) { return f64_to_df(scale2(x, -T.vexp[v])); }
  static __device__ __forceinline__ void xstore(const P& T, const Leaf& l, int sp, int v, int a, float2 x) {
    T.x2[l.xp * T.nv + v * sp + a] = x;
  }
  static constexpr bool kParts = true;
  static __device__ __forceinline__ bool want_parts(const P& T) { return T.oz != 0; }
  static __device__ __forceinline__ unsigned abs_bits(float2 x) { return __float_as_uint(x.x) & 0x7FFFFFFFu; }
  // leaf j's vectors as digits (mma_fp64.cuh); arguments as TreeOpM::parts
  static __device__ __forceinline__ void parts(const P& T, int64_t j, int s, const float2* xs, int cs, int vs,
                                               const unsigned* vmax, int tid, int threads) {
    const int nh = T.nv > 8 ? 2 : 1;
    unsigned char* chunk = T.xd + j * xd_chunk_bytes(T.xks, nh);
    // |x| 2^(54 - ex) <= 0x7F7F7F7F7F7F7F, the digits' range: the exponent of the largest |x|, one more where its
    // fraction leaves no room
    auto ex = [&](int v) { return max((int)(vmax[v] >> 23) - ((vmax[v] & 0x7FFFFFu) < 0x7D0000u ? 127 : 126), kXdMinExp); };
    for (int i = tid; i < ((s + 15) >> 4) * 32 * nh; i += threads) {
      const int ln = i & 31, u = i >> 5, ks = nh == 2 ? u >> 1 : u, half = nh == 2 ? u & 1 : 0;
      const int v = (ln >> 2) + 8 * half, c0 = 16 * ks + (ln & 3);
      const float up = __int_as_float((127 - (v < T.nv ? ex(v) : 0)) << 23);  // 2^-ex; 2^(54 - ex) may be no float
      uint32_t lo[4], hi[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int c = c0 + 4 * q;
        const float2 x = (v < T.nv && c < s) ? xs[c * cs + v * vs] : make_float2(0.f, 0.f);
        const long long n = __float2ll_rn(x.x * up * 0x1p54f) + __float2ll_rn(x.y * up * 0x1p54f) + 0x80808080808080LL;
        lo[q] = (uint32_t)n;
        hi[q] = (uint32_t)((unsigned long long)n >> 32);
      }
      uint32_t d0[kXdDigits], d1[kXdDigits];
      digit_pairs(lo[0], hi[0], lo[1], hi[1], d0);
      digit_pairs(lo[2], hi[2], lo[3], hi[3], d1);
      uint2* dst = reinterpret_cast<uint2*>(chunk + kXdScale + u * kXdStep + ln * 8);
#pragma unroll
      for (int p = 0; p < kXdDigits; p++) dst[32 * p] = make_uint2(d0[p], d1[p]);
    }
    // (a chunk with an infinity or NaN: kXdNaN makes its vector's sums NaN)
    if (tid < 16)
      reinterpret_cast<int*>(chunk)[tid] = tid >= T.nv ? kXdMinExp : vmax[tid] >= 0x7F800000u ? kXdNaN : ex(tid);
  }
  static __device__ __forceinline__ int copy_bytes(int entries) { return 8 * entries; }
  static __device__ __forceinline__ const char* U(const P& T, const Leaf& l) { return T.dmat + l.uoff; }
  static __device__ __forceinline__ int u_bytes(const P& T, const Leaf& l) { return 8 * l.s * T.k; }
  static __device__ __forceinline__ void u_layout(const P&, const Leaf&, int, int&, int&) {}
  static __device__ __forceinline__ void ystore(const P& T, const Leaf& l, int v, int row, const Acc& a, bool assign) {
    double* y = T.y + v * T.ldy + l.off + row;
    const double val = scale2(df_to_f64(a.s, a.c), l.eY + T.vexp[v]);
    if (assign) *y = val;
    else atomicAdd(y, val);
  }
};

template <int NVB>
__global__ void __cluster_dims__(kTreeCluster) __launch_bounds__(tree_warps<NVB>() * 32) k_upsweep_tree(TreeParams P) {
  const int spread = tree_spread(P.L);
  const bool active = (blockIdx.x & ((1 << spread) - 1)) == 0;
  tree_up<TreeOp64, NVB, true>(P, active ? blockIdx.x >> spread : 0, active, true, P.q - P.L, tree_block_entries(P.k, P.kks, false));
}

template <int NVB>
__global__ void __launch_bounds__(tree_warps<NVB>() * 32) k_downsweep_tree(TreeParams P) {
  tree_down<TreeOp64, NVB>(P, blockIdx.x, P.add ? 1 : 2, P.q - P.L, tree_down_entries(P.k, P.kks, false));
}

// ---------------------------------------------------------------- coupling, all levels
// yhat_i = sum_{b in row i} S_b xhat_{col(b)}   (Eq. 3, Alg. 3). A CTA of kWarps warps takes one
// segment, a run of blocks of one node row, and its warps take the segment's blocks in turn; the
// warps' sums meet in shared memory. Most rows are one segment. Where the matrix has few long rows
// (3D, upper levels, small n) a row is cut into several segments (coupling_segments): each leaves
// its partial sum in `part`, and the row's last segment to finish (ticket per row) adds them in
// order, so the result does not depend on the order of arrival.
// What bounds it: HBM at few vectors, as long as enough 16-byte loads are in flight. One warp per
// row left 3D n = 2^14 (511 rows of up to 150 blocks of 32 KB) with 511 warps on the chip and the
// longest row as the kernel's time: 972 us against 87 us of HBM time; split as above 180 us, and 146 as below.
//
// k = 2H with H a power of two: lane = g * H + h owns rows 2h, 2h + 1 of every block,
// read as one 16-byte load per column; column groups g = 0 .. G-1 (G = 32 / H)
// take a run of columns each (xhat in pairs). The warp's blocks are walked in batches of CB
// columns per lane, two batches in flight: the next batch's matrix and xhat
// loads are issued before the current batch is multiplied. Blocks are padded
// to kkp doubles; Sco[b] = (column node, exponent offset) of block b. Every node row
// is written (zero when it has no blocks). A lane's products form chains of
// at most 64 (kFoldProducts) that are folded into a long-term pair, so the
// FP32 sum of the small parts never runs over a whole row.
// Passes of more than four vectors run slices of four (grid y): 16 vectors in one warp took 255 registers and
// left 8 warps an SM; four slices split every entry four times but hold twice the warps (2D n = 50,001, 16 vectors:
// 234 -> 204 us; 3D n = 4,096, 13 vectors: 150 -> 89; slices of two: 240 and 87).
// SAFE: some coupling entry is zero or below 2^-103 after its offset (zero-safe split).
constexpr int kFoldProducts = 64;

struct __align__(16) CouplingSeg {
  int row, b0, nb;  // node row; first block; blocks
  int base;         // the row's first slot in `part` (and its ticket); unused when parts = 1
  int seg, parts;   // this segment of the row, and how many the row has
  int pad[2];
};

struct CouplingParams {
  const double* S;
  const int2* Sco;
  const CouplingSeg* segs;
  const float2* xhat;
  float2* yhat;
  float2* part;   // [slot][v][kp], the segments of split rows
  int* ticket;    // [slot base][4], a counter per vector slice, zero between products
  int kkp, k, kp, LR, nv;
};

// the CTA's warps have left their sums in red[warp][v][64]: add them, then store the row (or add up
// the row's segments when this is the last of them)
template <int NVB>
__device__ __forceinline__ void coupling_finish(const CouplingParams& P, const CouplingSeg& sg, float2 (*red)[NVB][64],
                                                int* last) {
  __syncthreads();
  const int k = P.k, kp = P.kp, v0 = blockIdx.y * NVB, nv = min(P.nv - v0, NVB);
  const int64_t stride = (int64_t)P.nv * kp;
  float2* row = P.yhat + sg.row * stride + v0 * kp;
  float2* mine = sg.parts == 1 ? row : P.part + (sg.base + sg.seg) * stride + v0 * kp;
  for (int t = threadIdx.x; t < nv * k; t += kWarps * 32) {
    const int v = t / k, r = t - v * k;
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; w++) df_add(s, c, red[w][v][r].x, red[w][v][r].y);
    mine[v * kp + r] = df_norm(s, c);
  }
  if (sg.parts == 1) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    int* ticket = P.ticket + 4 * (int64_t)sg.base + blockIdx.y;
    *last = atomicAdd(ticket, 1) == sg.parts - 1;
    if (*last) *ticket = 0;  // every segment has arrived: reset for the next product
  }
  __syncthreads();
  if (!*last) return;
  __threadfence();
  for (int t = threadIdx.x; t < nv * k; t += kWarps * 32) {
    const int v = t / k, r = t - v * k;
    const float2* src = P.part + sg.base * stride + (v0 + v) * kp + r;
    float s = 0.f, c = 0.f;
#pragma unroll 4
    for (int p = 0; p < sg.parts; p++) {
      const float2 a = __ldcg(src + p * stride);
      df_add(s, c, a.x, a.y);
    }
    row[v * kp + r] = df_norm(s, c);
  }
}

// k = K = 16, 32 or 64: nothing to test, since the lanes' columns fill the block. From K = 32 on the four warps take a
// quarter of every block's columns each (a block to a warp left them waiting for the one with a block more, a
// sixth of the kernel's time); at 16 a block is one or two batches, and a warp takes it whole. Bound by issue slots
// (about 0.6 of them used, 12 operations of each product in double-float): with k known only at run time, a column of
// 3D n = 2^14 took 80 instructions; phase 180 -> 146 us, n = 10,004 with four vectors 406 -> 256, 2D n = 50,001
// with 16 vectors 204 -> 150.
template <int K, int NVB, bool SAFE>
__global__ void __launch_bounds__(kWarps * 32) k_coupling(CouplingParams P) {
  constexpr int CB = NVB <= 2 ? 4 : 2, H = K / 2, G = 32 / H, CW = K >= 32 ? K / kWarps : K, CPL = CW / G, NCB = CPL / CB;
  constexpr int STEP = K >= 32 ? 1 : kWarps;  // from a warp's block to its next
  constexpr int FB = kFoldProducts / CB;      // batches per chain
  static_assert(G * H == 32 && CPL * G == CW && NCB * CB == CPL && FB % 2 == 0, "k_coupling: column split");
  __shared__ float2 red[kWarps][NVB][64];
  __shared__ int last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const CouplingSeg sg = P.segs[blockIdx.x];
  const int v0 = blockIdx.y * NVB, nv = min(P.nv - v0, NVB);  // this CTA's vectors
  const int g = lane / H, h = lane % H;
  const int col0 = g * CPL + (K >= 32 ? warp * CW : 0);  // the lane's first column
  const int first = sg.b0 + (K >= 32 ? 0 : warp), end = sg.b0 + sg.nb;
  const int nbatch = first < end ? (end - first + STEP - 1) / STEP * NCB : 0;
  float s[2][NVB], c[2][NVB], S2[2][NVB], C2[2][NVB];
  acc_zero(s, c);
  acc_zero(S2, C2);
  int xo[NVB];  // (a slice's missing vectors repeat its last one; their sums are not stored)
#pragma unroll
  for (int v = 0; v < NVB; v++) xo[v] = (v0 + min(v, nv - 1)) * K + col0;
  // the next batch's place: block b, columns cb CB ..; the block's column node and offset are read a block ahead
  int b = first, cb = 0;
  int2 co = nbatch > 0 ? __ldg(P.Sco + b) : make_int2(0, 0), cn = b + STEP < end ? __ldg(P.Sco + b + STEP) : co;
  const double* A = P.S + (int64_t)b * (K * K) + 2 * h + K * col0;
  const float2* X = P.xhat + (int64_t)co.x * P.nv * K;

  double2 a0[CB], a1[CB];
  float4 x0[CB / 2][NVB], x1[CB / 2][NVB];
  int o0 = 0, o1 = 0;
  auto load = [&](double2(&a)[CB], float4(&xv)[CB / 2][NVB], int& o) {
    o = co.y;
#pragma unroll
    for (int u = 0; u < CB; u++) a[u] = __ldg(reinterpret_cast<const double2*>(A + K * u));
#pragma unroll
    for (int u = 0; u < CB / 2; u++)
#pragma unroll
      for (int v = 0; v < NVB; v++) xv[u][v] = __ldg(reinterpret_cast<const float4*>(X + xo[v] + 2 * u));
    A += K * CB;
    X += CB;
    if (++cb == NCB) {
      cb = 0;
      b += STEP;
      A += STEP * K * K - CPL * K;
      co = cn;
      if (b + STEP < end) cn = __ldg(P.Sco + b + STEP);
      X = P.xhat + (int64_t)co.x * P.nv * K;
    }
  };
  auto compute = [&](const double2(&a)[CB], const float4(&xv)[CB / 2][NVB], int o) {
#pragma unroll
    for (int u = 0; u < CB; u++) {
      float h0, l0, h1, l1;
      if (SAFE) {
        split_f64(a[u].x, o, h0, l0);
        split_f64(a[u].y, o, h1, l1);
      } else {
        split_f64_fast(a[u].x, o, h0, l0);
        split_f64_fast(a[u].y, o, h1, l1);
      }
#pragma unroll
      for (int v = 0; v < NVB; v++) {
        const float4 x = xv[u / 2][v];
        const float xh = u % 2 ? x.z : x.x, xl = u % 2 ? x.w : x.y;
        df_fma(s[0][v], c[0][v], h0, l0, xh, xl);
        df_fma(s[1][v], c[1][v], h1, l1, xh, xl);
      }
    }
  };
  if (nbatch > 0) load(a0, x0, o0);
  for (int bt = 0; bt < nbatch; bt += 2) {
    if (bt + 1 < nbatch) load(a1, x1, o1);
    compute(a0, x0, o0);
    if (bt + 2 < nbatch) load(a0, x0, o0);
    if (bt + 1 < nbatch) compute(a1, x1, o1);
    if ((bt + 2) % FB == 0) acc_fold(S2, C2, s, c);
  }
  acc_fold(S2, C2, s, c);
#pragma unroll
  for (int r = 0; r < 2; r++)
#pragma unroll
    for (int v = 0; v < NVB; v++) {
      s[r][v] = S2[r][v];
      c[r][v] = C2[r][v];
    }
  // sum the column groups (lanes h, h + H, ...)
  for (int off = H; off < 32; off <<= 1) {
#pragma unroll
    for (int r = 0; r < 2; r++)
#pragma unroll
      for (int v = 0; v < NVB; v++) {
        const float s2 = __shfl_xor_sync(0xFFFFFFFFu, s[r][v], off);
        const float c2 = __shfl_xor_sync(0xFFFFFFFFu, c[r][v], off);
        df_add(s[r][v], c[r][v], s2, c2);
      }
  }
  if (g == 0) {
#pragma unroll
    for (int v = 0; v < NVB; v++) {
      red[warp][v][2 * h] = make_float2(s[0][v], c[0][v]);
      red[warp][v][2 * h + 1] = make_float2(s[1][v], c[1][v]);
    }
  }
  coupling_finish<NVB>(P, sg, red, &last);
}

// k = 2, 4 or 8: columns g, g + G, ... with lanes beyond k columns idle; every bound is tested
template <int NVB, bool SAFE>
__global__ void __launch_bounds__(kWarps * 32) k_coupling_small(CouplingParams P) {
  constexpr int CB = NVB <= 2 ? 4 : 2;
  __shared__ float2 red[kWarps][NVB][64];
  __shared__ int last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const CouplingSeg sg = P.segs[blockIdx.x];
  const int k = P.k, kp = P.kp, v0 = blockIdx.y * NVB, nv = min(P.nv - v0, NVB);  // this CTA's vectors
  const double* __restrict__ S = P.S;
  const int2* __restrict__ Sco = P.Sco;
  const float2* __restrict__ xhat = P.xhat;
  const int H = k >> 1, G = 32 / H;
  const int g = lane / H, h = lane - g * H;
  const bool active = g < G;            // lanes beyond G * H idle
  const int cpl = (k + G - 1) / G;      // columns per lane per block
  const int ncb = (cpl + CB - 1) / CB;  // batches per block
  const int b0 = sg.b0 + warp;          // this warp's blocks: b0, b0 + kWarps, ...
  const int nbatch = warp < sg.nb ? ((sg.nb - warp + kWarps - 1) / kWarps) * ncb : 0;
  constexpr int FB = kFoldProducts / CB;  // batches per chain
  float s[2][NVB], c[2][NVB], S2[2][NVB], C2[2][NVB];
  acc_zero(s, c);
  acc_zero(S2, C2);

  double2 a0[CB], a1[CB];
  float2 x0[CB][NVB], x1[CB][NVB];
  int o0 = 0, o1 = 0;
  auto load = [&](int bt, double2(&a)[CB], float2(&xv)[CB][NVB], int& o) {
    const int bl = bt / ncb, cb = bt - bl * ncb, b = b0 + kWarps * bl;
    const double* A = S + (int64_t)b * P.kkp;
    const int2 co = __ldg(Sco + b);
    const float2* X = xhat + ((int64_t)co.x * P.nv + v0) * kp;
    o = co.y;
#pragma unroll
    for (int u = 0; u < CB; u++) {
      const int col = g + G * (cb * CB + u);
      const bool ok = active && col < k;
      a[u] = ok ? __ldg(reinterpret_cast<const double2*>(A + 2 * h + k * col)) : make_double2(0.0, 0.0);
#pragma unroll
      for (int v = 0; v < NVB; v++) xv[u][v] = (ok && v < nv) ? __ldg(X + v * kp + col) : make_float2(0.f, 0.f);
    }
  };
  auto compute = [&](const double2(&a)[CB], const float2(&xv)[CB][NVB], int o) {
#pragma unroll
    for (int u = 0; u < CB; u++) {
      float h0, l0, h1, l1;
      if (SAFE) {
        split_f64(a[u].x, o, h0, l0);
        split_f64(a[u].y, o, h1, l1);
      } else {
        split_f64_fast(a[u].x, o, h0, l0);
        split_f64_fast(a[u].y, o, h1, l1);
      }
#pragma unroll
      for (int v = 0; v < NVB; v++) {
        df_fma(s[0][v], c[0][v], h0, l0, xv[u][v].x, xv[u][v].y);
        df_fma(s[1][v], c[1][v], h1, l1, xv[u][v].x, xv[u][v].y);
      }
    }
  };
  if (nbatch > 0) load(0, a0, x0, o0);
  for (int bt = 0; bt < nbatch; bt += 2) {
    if (bt + 1 < nbatch) load(bt + 1, a1, x1, o1);
    compute(a0, x0, o0);
    if (bt + 2 < nbatch) load(bt + 2, a0, x0, o0);
    if (bt + 1 < nbatch) compute(a1, x1, o1);
    if ((bt + 2) % FB == 0) acc_fold(S2, C2, s, c);
  }
  acc_fold(S2, C2, s, c);
#pragma unroll
  for (int r = 0; r < 2; r++)
#pragma unroll
    for (int v = 0; v < NVB; v++) {
      s[r][v] = S2[r][v];
      c[r][v] = C2[r][v];
    }
  // sum the column groups (lanes h, h + H, ...)
  for (int off = H; off < 32; off <<= 1) {
#pragma unroll
    for (int r = 0; r < 2; r++)
#pragma unroll
      for (int v = 0; v < NVB; v++) {
        const float s2 = __shfl_xor_sync(0xFFFFFFFFu, s[r][v], off);
        const float c2 = __shfl_xor_sync(0xFFFFFFFFu, c[r][v], off);
        df_add(s[r][v], c[r][v], s2, c2);
      }
  }
  if (g == 0) {
#pragma unroll
    for (int v = 0; v < NVB; v++) {
      red[warp][v][2 * h] = make_float2(s[0][v], c[0][v]);
      red[warp][v][2 * h + 1] = make_float2(s[1][v], c[1][v]);
    }
  }
  coupling_finish<NVB>(P, sg, red, &last);
}

// Any other k: the generic row mapping of warp_mv, one block at a time (each
// block's chain folded into the row's long-term pair).
template <int RPL, int NVB>
__global__ void __launch_bounds__(kWarps * 32) k_coupling_generic(CouplingParams P) {
  __shared__ float2 red[kWarps][NVB][64];
  __shared__ int last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const CouplingSeg sg = P.segs[blockIdx.x];
  const int k = P.k, kp = P.kp, LR = P.LR, v0 = blockIdx.y * NVB, nv = min(P.nv - v0, NVB);
  float s[RPL][NVB], c[RPL][NVB], S2[RPL][NVB], C2[RPL][NVB];
  acc_zero(s, c);
  acc_zero(S2, C2);
  for (int b = sg.b0 + warp; b < sg.b0 + sg.nb; b += kWarps) {
    const int2 co = P.Sco[b];
    warp_mv<RPL, NVB>(P.S + (int64_t)b * P.kkp, co.y, k, k, LR, P.xhat + ((int64_t)co.x * P.nv + v0) * kp, kp, nv, s, c, lane);
    acc_fold(S2, C2, s, c);
  }
  group_reduce(S2, C2, LR);
  if (lane < LR) {
#pragma unroll
    for (int r = 0; r < RPL; r++)
#pragma unroll
      for (int v = 0; v < NVB; v++) red[warp][v][lane + 32 * r] = make_float2(S2[r][v], C2[r][v]);
  }
  coupling_finish<NVB>(P, sg, red, &last);
}

// ---------------------------------------------------------------- per-vector scale
// vexp[v] = s with max_i |x[i, v]| * 2^-s < 1 (frexp exponent; 0 for a zero or
// non-finite maximum), so that the pass works on x * 2^-s. Each block writes
// its maxima to partial[block][v]; the last block to finish (atomic ticket)
// reduces them and resets the ticket for the next launch. A thread keeps
// eight loads in flight; one round covers n = 2^20 on 152 blocks.
constexpr int kScaleBlocks = 152, kScaleThreads = 1024, kScaleUnroll = 8;
__device__ __forceinline__ unsigned long long abs_bits(double a) { return (unsigned long long)__double_as_longlong(fabs(a)); }
// zero_y (or null): zeroed for the products whose phases add into it.
__global__ void __launch_bounds__(kScaleThreads) k_vec_scale(const double* __restrict__ x, int64_t ldx, int64_t n, int nv,
                                                            unsigned long long* partial, unsigned* ticket, int* vexp,
                                                            double* zero_y, int64_t ldy) {
  __shared__ unsigned long long wmax[kScaleThreads / 32][16];
  __shared__ int last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * kScaleThreads;
  if (zero_y)
    for (int v = 0; v < nv; v++)
      for (int64_t i = (int64_t)blockIdx.x * kScaleThreads + threadIdx.x; i < n; i += stride) zero_y[v * ldy + i] = 0.0;
  for (int v = 0; v < nv; v++) {
    const double* xv = x + v * ldx;
    unsigned long long m = 0;
    int64_t i = (int64_t)blockIdx.x * kScaleThreads + threadIdx.x;
    for (; i + (kScaleUnroll - 1) * stride < n; i += kScaleUnroll * stride) {
      double a[kScaleUnroll];
#pragma unroll
      for (int u = 0; u < kScaleUnroll; u++) a[u] = __ldcs(xv + i + u * stride);
#pragma unroll
      for (int u = 0; u < kScaleUnroll; u++) m = max(m, abs_bits(a[u]));
    }
    for (; i < n; i += stride) m = max(m, abs_bits(__ldcs(xv + i)));
    for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
    if (lane == 0) wmax[warp][v] = m;
  }
  __syncthreads();
  if (threadIdx.x < nv) {
    unsigned long long m = 0;
    for (int w = 0; w < kScaleThreads / 32; w++) m = max(m, wmax[w][threadIdx.x]);
    partial[blockIdx.x * 16 + threadIdx.x] = m;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int v = warp; v < nv; v += kScaleThreads / 32) {
    unsigned long long m = 0;
#pragma unroll 4
    for (int b = lane; b < (int)gridDim.x; b += 32) m = max(m, __ldcg(partial + b * 16 + v));
    for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
    if (lane == 0) vexp[v] = vec_exponent(m);
  }
  if (threadIdx.x == 0) *ticket = 0u;
}

}  // namespace h2
