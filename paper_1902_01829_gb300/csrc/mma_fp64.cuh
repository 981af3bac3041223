// Dense near field of the FP64 plain form for passes of more than four vectors, on the tensor cores:
//   y(i) += sum_j D_ij x(j)     (Sec. 2.2; y(i) holds U_i yhat_i from the downsweep)
// by integer slicing (the Ozaki scheme: Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", 2012): every entry becomes seven signed
// 8-bit digits, digit products are exact in FP16 MMAs, and their sums are exact in the FP32 accumulators.
//
//   a = 2^(ea - 54) sum_i d_i 2^(8 (6 - i)),  |a| <= 0x7F7F7F7F7F7F7F 2^(ea - 54) over the block,   i = 0 .. 6
//   x = 2^(ex - 54) sum_j e_j 2^(8 (6 - j)),  the same over a leaf's chunk of one vector
// so a block's entries are held to 2^-55 of its largest, where the double-float kernel cuts each at 2^-46 of
// itself: a block takes this form if it has no zeros and its entries lie within 2^9 of 2^(ea + 1), and none of them
// is then held in fewer bits. Any other block ("wide") is multiplied in double-float by the same warps
// (oz_wide_block), so that an entry far below its block's largest, in a row that sees no other, keeps its bits.
// The vectors' entries are held to 2^-54 of their chunk's largest, whatever they span: without zeros every row
// of a digit block weighs that largest entry with 2^-9 of the block's at least, so the cut is below
// 64 2^9 2^-54 of sum_j |a_ij| |x_j|, and 2^-50 of it where a row's entries are alike. The 21 products with
// i + j <= 5 are summed by weight: |d e| <= 2^14, 64 columns and at most 6 pairs stay below 2^23, exact for every
// weight; the seven of weight 6 join weight 5's at 2^-8, the rest (2^-56 of the largest product each) is left out.
// A block's six sums are joined in double-float (the upper four exactly) and added to the row's running pairs, so
// blocks of any magnitude meet as in the double-float kernel.
//
// What bounds it: at 16 vectors a 64 x 64 block cost the FP32 pipes 65,536 double-float products of 11
// instructions, 8,800 cycles an SM (which a wide block still takes); 896 MMAs take 1,792, slicing its 4,096 entries
// about 800 issue slots, and its 32 KB 1,400 at the copy bandwidth. Measured, 2D n = 50,001 (48- and 49-point leaves),
// 16 vectors: six digits 837 -> 404 us in the dense phase, error against 64 bits 2.6e-14 -> 2.1e-14 (weight 6 left
// out: 7e-14; the sums joined without the third exact step: 1e-13); seven digits with the vectors' fragments loaded
// one at a time (60 bytes of spills less) 397 -> 375 us, error 2.0e-14. 4,200 cycles a block are
// still the chain of slicing, loads and MMAs of three warps a scheduler, not a pipe.
//
// Y^T = X^T D^T as in mma_dense.cuh: the vectors' digits are the A operand, written in fragment order by
// the upsweep; a lane slices the entries it loads from the item's stage into B fragments. The dense
// stream's items and roles: a producer warp, twelve consumer warps, each taking 16-row quarters of blocks
// in turn.
#pragma once
#include "mma_dense.cuh"
#include "stream_fp64.cuh"

namespace h2 {

// digits of a leaf's vectors: 16 exponents ex (ints), then per K step of 16 points and half of eight vectors seven
// digits of 256 bytes, lane (g, t)'s entries (vector g + 8 half; points t, t + 4, t + 8, t + 12) at 8 (4 g + t)
constexpr int kXdScale = 64, kXdDigits = 7, kXdStep = kXdDigits * 256;
constexpr int kXdMinExp = -120;   // smallest ex: a chunk further below its vector's largest entry keeps this unit
constexpr int kXdNaN = 1 << 20;  // as an exponent: the chunk's vector has an entry that is not finite
__host__ __device__ constexpr int xd_chunk_bytes(int ksteps, int halves) { return kXdScale + ksteps * halves * kXdStep; }

constexpr int kOzWarps = 12;  // a multiple of 1 .. 4: a warp keeps to one 16-row quarter of the rows
constexpr int kOzRedStride = 18;  // float2 per vector of a warp's 16 rows (padded against bank conflicts)
constexpr int kOzRed = kOzWarps * 16 * kOzRedStride * 8;
constexpr int kOzStage = kStageHeader + kStageMat + xd_chunk_bytes(4, 2);
constexpr int kOzStages = (kSmemLimit - 256 - kOzRed) / kOzStage;
constexpr int kOzSmem = kOzStages * kOzStage + 256 + kOzRed;
static_assert(kOzStages >= 3, "at least three stages");
static_assert(kOzStage % 16 == 0, "stage alignment");

// v = (a as an integer multiple of 2^(ea - 54), rounded to nearest) + 0x80808080808080: the digits are its
// bytes minus 128. E = ea + 1031: |a| < 2^(ea + 1) has a biased FP64 exponent of ea + 1023 at most. lo: low 32
// bits, hi: the rest. The block's entries are normal; a zero (a column or row past the block) gives digits
// of no meaning, which meet zeros or are not stored.
__device__ __forceinline__ void slice_f64(double a, int E, uint32_t& lo, uint32_t& hi) {
  const uint32_t h = (uint32_t)__double2hiint(a), l = (uint32_t)__double2loint(a);
  const int s = min(E - (int)((h >> 20) & 0x7FFu), 31);  // |a| 2^(55 - ea): the value with one bit below the unit (s >= 8)
  const uint32_t mh = __funnelshift_l(l, h, 11) | 0x80000000u, ml = l << 11;
  uint32_t vl = __funnelshift_r(ml, mh, s), vh = mh >> s;
  // round: (v + 1) >> 1, then the sign, then the digits' bias
  asm("add.cc.u32 %0, %0, 1;\n\taddc.u32 %1, %1, 0;" : "+r"(vl), "+r"(vh));
  vl = __funnelshift_r(vl, vh, 1);
  vh >>= 1;
  if (h >> 31) asm("sub.cc.u32 %0, 0, %0;\n\tsubc.u32 %1, 0, %1;" : "+r"(vl), "+r"(vh));
  asm("add.cc.u32 %0, %0, 0x80808080;\n\taddc.u32 %1, %1, 0x808080;" : "+r"(vl), "+r"(vh));
  lo = vl;
  hi = vh;
}

// digit bytes -> fp16 pairs: byte b of p in the low half, byte b + 1 in the high half, minus 128
// (0x6400 | b is the fp16 of 1024 + b)
template <int B>
__device__ __forceinline__ uint32_t digit_pair(uint32_t p) {
  const uint32_t v = __byte_perm(p, 0x64646464u, B == 0 ? 0x4140 : 0x4342);
  const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&v), __float2half2_rn(-1152.f));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// the seven digits (from the top) of two sliced values as fp16 pairs
__device__ __forceinline__ void digit_pairs(uint32_t l0, uint32_t h0, uint32_t l1, uint32_t h1, uint32_t (&d)[kXdDigits]) {
  const uint32_t p0 = __byte_perm(l0, l1, 0x5140), p1 = __byte_perm(l0, l1, 0x7362), p2 = __byte_perm(h0, h1, 0x5140),
                 p3 = __byte_perm(h0, h1, 0x7362);
  d[6] = digit_pair<0>(p0);
  d[5] = digit_pair<1>(p0);
  d[4] = digit_pair<0>(p1);
  d[3] = digit_pair<1>(p1);
  d[2] = digit_pair<0>(p2);
  d[1] = digit_pair<1>(p2);
  d[0] = digit_pair<0>(p3);
}

__device__ __forceinline__ uint32_t scale_digits(uint32_t d) {  // / 256, exact
  const __half2 r = __hmul2(*reinterpret_cast<const __half2*>(&d), __float2half2_rn(0.00390625f));
  return *reinterpret_cast<const uint32_t*>(&r);
}

struct OzParams {
  const StreamItem* items;
  const int* cta_begin;
  const int* item_exp;   // per item: the block's ea, and (item_leaf) its column leaf
  const int* item_leaf;
  const char* mat;
  const unsigned char* xd;  // the leaves' digits, xks K steps each
  const float2* x2;         // split x, padded leaf layout: the wide blocks' vectors
  int xks, nv;
  double* y;
  long long ldy;
  const int* vexp;
  int* err;
  long long budget;
  int inject;  // >= 0: CTA 0 withholds the copy of this local item (bounded-wait test)
};

// Producer warp. Stage header (ints): R, C, flags, row, ea, vector stride of a wide block.
template <bool WIDE>
__device__ __forceinline__ void oz_produce(const OzParams& P, const StreamShared& S, int ib, int ie) {
  const int lane = threadIdx.x & 31;
  const uint64_t pol = policy_evict_first();
  const int nh = P.nv > 8 ? 2 : 1;
  StreamParams W{};
  W.err = P.err;
  W.budget = P.budget;
  int issued = 0;
  bool ok = true;
  for (int base = ib; base < ie && ok; base += 32) {
    StreamItem mine{};
    int l_exp = 0, l_leaf = 0;
    if (base + lane < ie) {
      mine = P.items[base + lane];
      l_exp = P.item_exp[base + lane];
      l_leaf = P.item_leaf[base + lane];
    }
    const int cnt = min(32, ie - base);
    for (int t = 0; t < cnt; t++) {
      const int it = base + t - ib, s = it % kOzStages, use = it / kOzStages;
      if (use > 0 && !warp_wait(S.empty + s, (use - 1) & 1, W, S.abort_flag)) {
        ok = false;
        break;
      }
      if (__any_sync(0xFFFFFFFFu, *S.abort_flag != 0)) {
        ok = false;
        break;
      }
      const long long m_off = __shfl_sync(0xFFFFFFFFu, mine.m_off, t);
      const int m_bytes = __shfl_sync(0xFFFFFFFFu, mine.m_bytes, t), row = __shfl_sync(0xFFFFFFFFu, mine.row, t);
      const unsigned shape = __shfl_sync(0xFFFFFFFFu, mine.shape, t);
      const int flags = __shfl_sync(0xFFFFFFFFu, mine.flags, t);
      const long long v_off = __shfl_sync(0xFFFFFFFFu, mine.v_off, t);
      const int ea = __shfl_sync(0xFFFFFFFFu, l_exp, t), leaf = __shfl_sync(0xFFFFFFFFu, l_leaf, t);
      if (lane == 0) {
        unsigned char* stage = S.stage0 + s * kOzStage;
        int* h = reinterpret_cast<int*>(stage);
        const int C = (int)((shape >> 8) & 0xFF), vs = (int)((shape >> 16) & 0xFF);
        const bool wide = WIDE && (flags & kItemFlagWide) != 0;
        h[0] = (int)(shape & 0xFF);
        h[1] = C;
        h[2] = flags;
        h[3] = row;
        h[4] = ea;
        h[5] = vs;
        if (!((P.inject == it) && (blockIdx.x == 0))) {
          const unsigned vbytes = wide ? 8u * (unsigned)(vs * P.nv) : (unsigned)xd_chunk_bytes((C + 15) / 16, nh);
          const void* vsrc = wide ? static_cast<const void*>(P.x2 + v_off * P.nv)
                                  : P.xd + (long long)leaf * xd_chunk_bytes(P.xks, nh);
          mbar_arrive_expect_tx(S.full + s, (unsigned)m_bytes + vbytes);
          bulk_g2s_stream(stage + kStageHeader, P.mat + m_off, (unsigned)m_bytes, S.full + s, pol);
          bulk_g2s(stage + kStageHeader + kStageMat, vsrc, vbytes, S.full + s);
        }
      }
      __syncwarp();
      issued = it + 1;
    }
  }
  if (lane == 0)
    for (int it = max(0, issued - kOzStages); it < issued; it++) {  // copies in flight land before exit
      const int s = it % kOzStages, use = it / kOzStages;
      const long long t0 = clock64();
      while (!mbar_try_wait(S.full + s, use & 1) && clock64() - t0 < P.budget) {
      }
    }
}

// One 16-row quarter of a block: lane (g, t) loads rows r, r + 1 (r = 16 quarter + 2 g) of the columns t, t + 4,
// t + 8, t + 12 of a K step; tile i holds rows r + i. acc[i][w]: weight w's sums for vectors g (0, 1) and g + 8
// (2, 3), rows of the lanes g = 2t and 2t + 1.
__device__ __forceinline__ void oz_block(const double* A, uint32_t X, int R, int C, int r, int E, int nh, float (&acc)[2][6][4]) {
  const int lane = threadIdx.x & 31, t = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int w = 0; w < 6; w++)
#pragma unroll
      for (int e = 0; e < 4; e++) acc[i][w][e] = 0.f;
  const bool pair = (R & 1) == 0;
  const bool in0 = r < R, in1 = r + 1 < R;
  uint32_t xa = X + kXdScale + lane * 8;
  const int half = nh > 1 ? kXdStep : 0, xstep = nh * kXdStep;
  double e[2][4];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int c = k0 + t + 4 * q;
      e[0][q] = e[1][q] = 0.0;
      if (c < C && in0) {
        const double* src = A + r + R * c;
        if (pair) {
          const double2 v = *reinterpret_cast<const double2*>(src);
          e[0][q] = v.x;
          e[1][q] = v.y;
        } else {
          e[0][q] = src[0];
          if (in1) e[1][q] = src[1];
        }
      }
    }
  };
  load(0);
#pragma unroll 1
  for (int k0 = 0; k0 < C; k0 += 16) {
    uint32_t d[2][2][kXdDigits];
#pragma unroll
    for (int i = 0; i < 2; i++) {
      uint32_t l[4], h[4];
#pragma unroll
      for (int q = 0; q < 4; q++) slice_f64(e[i][q], E, l[q], h[q]);
      digit_pairs(l[0], h[0], l[1], h[1], d[i][0]);
      digit_pairs(l[2], h[2], l[3], h[3], d[i][1]);
    }
    if (k0 + 16 < C) load(k0 + 16);
    // the vectors' digits in turn, the next one's fragment loaded ahead (all seven at once do not fit the registers)
    uint32_t a[2][4];
    auto load_digit = [&](int j, uint32_t(&f)[4]) {
      const uint2 u = lds64(xa + 256 * j), v = lds64(xa + 256 * j + half);
      f[0] = u.x;
      f[1] = v.x;
      f[2] = u.y;
      f[3] = v.y;
    };
    load_digit(0, a[0]);
#pragma unroll
    for (int j = 0; j < kXdDigits; j++) {
      if (j + 1 < kXdDigits) load_digit(j + 1, a[(j + 1) & 1]);
#pragma unroll
      for (int p = 0; p < 6 - j; p++)
#pragma unroll
        for (int i = 0; i < 2; i++) mma_m16n8k16(acc[i][p + j], a[j & 1], d[i][0][p], d[i][1][p], false);
      // weight 6, the matrix digit / 256, with weight 5's sums
#pragma unroll
      for (int i = 0; i < 2; i++) mma_m16n8k16(acc[i][5], a[j & 1], scale_digits(d[i][0][6 - j]), scale_digits(d[i][1][6 - j]), false);
    }
    xa += xstep;
  }
}

// (s, c) added to a running pair (fresh: the first)
__device__ __forceinline__ void oz_put(float2* slot, bool fresh, float s, float c) {
  float2 p = fresh ? make_float2(0.f, 0.f) : *slot;
  df_add(p.x, p.y, s, c);
  *slot = p;
}

// The same quarter of a wide block in double-float: the block split with its offset o, the vectors' pairs X ([vector][vs
// points]), the sums added to the warp's running pairs. A lane has rows r, r + 1 (r = 16 quarter + 2 (lane % 8)) and four
// vectors; with up to eight vectors (CS = 2) the half-warps take every second column and join their sums at the end.
// Bound by issue slots like the double-float stream (2D n = 50,001, every block wide: dense phase of 8 / 16 vectors 516 /
// 873 us, the stream's 506 / 820; with four rows and two vectors a lane, whatever the count, 909 / 917). Not inlined: its
// registers would be oz_block's.
template <int CS>
__device__ __noinline__ void oz_wide_block(const double* A, const float2* X, int R, int C, int vs, int quarter, int o, int nv,
                                           float2* mine, bool fresh) {
  __builtin_assume(__isShared(A) && __isShared(X) && __isShared(mine));
  const int lane = threadIdx.x & 31, r = 16 * quarter + 2 * (lane & 7), v0 = 4 * ((lane >> 3) & (CS == 2 ? 1 : 3));
  const int c0 = CS == 2 ? lane >> 4 : 0, Cr = r < R ? C : 0;
  float2 acc[2][4];
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int v = 0; v < 4; v++) acc[i][v] = make_float2(0.f, 0.f);
  const bool pair = (R & 1) == 0;
#pragma unroll 2
  for (int c = c0; c < Cr; c += CS) {
    const double* src = A + r + R * c;
    double a[2];
    if (pair) {
      const double2 d = *reinterpret_cast<const double2*>(src);
      a[0] = d.x;
      a[1] = d.y;
    } else {
      a[0] = src[0];
      a[1] = r + 1 < R ? src[1] : 0.0;
    }
    float h[2], l[2];
#pragma unroll
    for (int i = 0; i < 2; i++) split_f64(a[i], o, h[i], l[i]);
#pragma unroll
    for (int v = 0; v < 4; v++) {
      const float2 x = v0 + v < nv ? X[(v0 + v) * vs + c] : make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 2; i++) df_fma(acc[i][v].x, acc[i][v].y, h[i], l[i], x.x, x.y);
    }
  }
  __syncwarp();  // (a digit block's pairs are other lanes')
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int v = 0; v < 4; v++) {
      if constexpr (CS == 2)
        df_add(acc[i][v].x, acc[i][v].y, __shfl_xor_sync(0xFFFFFFFFu, acc[i][v].x, 16), __shfl_xor_sync(0xFFFFFFFFu, acc[i][v].y, 16));
      if (CS == 1 || i == c0)  // (half-warp i stores row i of the joined sums)
        oz_put(mine + (v0 + v) * kOzRedStride + (r & 15) + i, fresh, acc[i][v].x, acc[i][v].y);
    }
  __syncwarp();
}

// WIDE: the handle has wide blocks (with their code inlined in the only kernel: 407 us at 2D n = 50,001, 375 without it)
template <bool WIDE>
__global__ void __launch_bounds__((kOzWarps + 1) * 32, 1) k_dense_oz(OzParams P) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const StreamShared S = stream_shared<kOzStages, kOzStage>(smem);
  stream_init<kOzStages, kOzWarps>(S);
  const int ib = P.cta_begin[blockIdx.x], ie = P.cta_begin[blockIdx.x + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  if (warp == kOzWarps) {
    oz_produce<WIDE>(P, S, ib, ie);
    return;
  }
  StreamParams W{};
  W.err = P.err;
  W.budget = P.budget;
  const int nv = P.nv, nh = nv > 8 ? 2 : 1;
  float2* mine = S.red + warp * 16 * kOzRedStride;  // the warp's running pairs: [vector][row of its quarter]
  int rows_done = 0, turn = warp;                   // the warp's next quarter, counted from the current item's first
  bool fresh = true;                                // nothing of the current row is in `mine` yet
  auto open_row = [&]() -> bool {                   // the previous row's pairs have been read
    return rows_done == 0 || warp_wait(S.rowfree, (rows_done - 1) & 1, W, S.abort_flag);
  };
  for (int it = 0; it < ie - ib; it++) {
    const int st = it % kOzStages, use = it / kOzStages;
    if (!warp_wait(S.full + st, use & 1, W, S.abort_flag)) break;
    const unsigned char* stage = S.stage0 + st * kOzStage;
    const int* h = reinterpret_cast<const int*>(stage);
    const int R = min(h[0], 64), C = min(h[1], 64), flags = h[2], row = h[3], ea = h[4];
    const int nu = (R + 15) >> 4;
    {
      bool ok = true;
      for (; turn < nu; turn += kOzWarps) {
        const int shift = item_offset(flags);  // the row's output exponent (o of its blocks)
        const double* A = reinterpret_cast<const double*>(stage + kStageHeader);
        const unsigned char* xs = stage + kStageHeader + kStageMat;
        if (WIDE && (flags & kItemFlagWide)) {
          if (fresh && !(ok = open_row())) break;
          const float2* X = reinterpret_cast<const float2*>(xs);
          const int vs = min(h[5], 64);
          if (nh == 1) oz_wide_block<2>(A, X, R, C, vs, turn, shift, nv, mine, fresh);
          else oz_wide_block<1>(A, X, R, C, vs, turn, shift, nv, mine, fresh);
          fresh = false;
          continue;
        }
        float acc[2][6][4];
        oz_block(A, smem_addr(xs), R, C, 16 * turn + 2 * g, ea + 1031, nh, acc);
        if (fresh && !(ok = open_row())) break;
        // the sums below are in units of 2^(96 - 16 + 38) (weight 2 times 2^-38), so that a contribution down to 2^-126 of
        // the row's bound is a float, as in double-float
        const int* ex = reinterpret_cast<const int*>(xs);
        float f[2];
#pragma unroll
        for (int b = 0; b < 2; b++) {
          const int n = ea - shift + ex[g + 8 * b] + 10;
          f[b] = n < -126 ? 0.f : __int_as_float(n > 127 ? 0x7FC00000 : (n + 127) << 23);  // (n > 127: kXdNaN)
        }
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
          for (int e = 0; e < 4; e++) {
            const float tail = fmaf(acc[i][5][e], 0.00390625f, acc[i][4][e]) * 0x1p-54f;
            float s1, e1, s2, e2, s3, e3;
            two_sum(acc[i][0][e] * 0x1p-22f, acc[i][1][e] * 0x1p-30f, s1, e1);
            two_sum(s1, acc[i][2][e] * 0x1p-38f, s2, e2);
            two_sum(s2, acc[i][3][e] * 0x1p-46f, s3, e3);
            const float fb = f[e >> 1];
            // tile i, element e: row 4 t + 2 (e & 1) + i, vector g + 8 (e >> 1)
            oz_put(mine + (g + 8 * (e >> 1)) * kOzRedStride + 4 * t + 2 * (e & 1) + i, fresh, s3 * fb, (((e1 + e2) + e3) + tail) * fb);
          }
        fresh = false;
      }
      if (!ok) break;
      turn -= nu;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(S.empty + st);
    if (!(flags & kItemFlagLast)) continue;
    if (fresh) {  // none of the row's blocks was this warp's
      if (!open_row()) break;
      for (int i = lane; i < 16 * kOzRedStride; i += 32) mine[i] = make_float2(0.f, 0.f);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(S.rowfull);
    if (!warp_wait(S.rowfull, rows_done & 1, W, S.abort_flag)) break;
    const int ey = item_row_exp(flags);
    for (int idx = threadIdx.x; idx < 64 * nv; idx += kOzWarps * 32) {
      const int r = idx & 63, v = idx >> 6;
      if (r >= R) continue;
      float ss = 0.f, cc = 0.f;
      for (int w = r >> 4; w < kOzWarps; w += nu) {  // the warps of this quarter
        const float2 p = S.red[(w * 16 + v) * kOzRedStride + (r & 15)];
        df_add(ss, cc, p.x, p.y);
      }
      double* y = P.y + v * P.ldy + row + r;
      *y += scale2(df_to_f64(ss, cc), ey + P.vexp[v]);  // the row's expansion is there already
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(S.rowfree);
    rows_done++;
    turn = warp;
    fresh = true;
  }
}

}  // namespace h2
