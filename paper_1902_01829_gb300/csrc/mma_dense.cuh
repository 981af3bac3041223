// Dense near field of the scaled forms for passes of more than four vectors, on the tensor cores
// (mma.sync m16n8k16, FP32 accumulators):   y(i) += sum_j D_ij x(j)   (Sec. 2.2), any leaf size, any
// code type, one matrix or a batch.
//
// The product is turned over, Y^T = X^T D^T: the 16 vectors are the M side, eight rows of the leaf the N
// side, 16 columns the K side. The codes then enter as the B operand straight from the registers they are
// loaded into (a lane's four columns of a K step times its four or eight rows, one byte permute per pair),
// and the vectors as the A operand in fragment order, written once per leaf by the upsweep:
//   x_v = 2^(e - 14) (hi + mid + lo), hi, mid, lo fp16 (2^(e-1) <= max |x_v| over the leaf < 2^e: all 24 bits of
//   an FP32 down to 2^-14 of the leaf's largest entry, below that what lies above 2^-38 of it), or for bf16 codes
//   x_v = hi + mid + lo in bf16 (all 24 bits of any FP32).
// A code is a B entry as it is (fp16, bf16); an int16 code q = 256 (h + l) with h = q >> 8 and l = the low
// byte / 256, both exact in fp16, times hi, mid (and lo): l lo is left out, below 2^-23 of its product where |q| >= 256
// (with it 5 MMAs become 6: 2D n = 2^18, 8 vectors, dense phase 261 -> 313 us), and taken in blocks with smaller codes
// (kBlockLow). The leading products h hi and the rest accumulate apart, in FP32, and a block's sums enter the row's
// after sigma 2^(e - 14) is applied, so nothing is rounded to 16 bits and no chain is longer than a block. Blocks with a
// code below 2^-10 of the largest, zeros among them (kBlockWide), are multiplied in FP32 by the same warps
// (mma_wide_block) with the vectors as they are: a row of such a block may see small vector entries alone. In the others
// every row weighs the leaf's largest entry with 2^-10 at least, so what the parts cut off is below 64 2^10 2^-38 of
// sum_j |d_ij| |x_j| for any vector, in most cases below FP32's rounding of the sum. (Small int16 matrices feel a wide
// block's latency: with blocks of codes below 256 wide too, 2D n = 1,000 took 64 us for 16 vectors, 52 so.)
//
// What bounds it: at 16 vectors the FP32 pipes spent 2048 FMAs of a warp on a 64 x 64 block (1360 cycles an
// SM with its loads); 3 (int16: 5) MMAs per tile and K step take 192 (320) and the codes' loads from shared
// memory about as long. tcgen05 would need the codes repacked K-major into shared memory by other warps
// (digits included); mma.sync takes them from registers and is no longer the limit at these sizes.
// Measured, dense phase: 2D n = 2^16 int16, 16 vectors 126 -> 75 us; 32 matrices of 1024 .. 16384 points, 32-point
// leaves, fp16, 1 to 16 vectors 599 -> 203 us; 3D n = 2^16 int16, 8 vectors 393 -> 325 us. The K steps are now
// bound by their chain (loads, permutes, MMAs: about 800 cycles with three warps a scheduler), not by the tensor
// pipe (42% busy).
//
// A CTA per SM, persistent over its items (the dense stream's, h2_mixed.cu): a producer warp copies each
// item's codes and its blocks' vector chunks into a ring of stages; twelve consumer warps take the blocks
// (halves of 64-row blocks) in turn and add up their rows' sums at the row's end.
#pragma once
#include "mixed.cuh"

namespace h2 {

constexpr int kMmaWarps = 12;  // even: a warp keeps to one half of the rows
constexpr int kMmaRedStride = 68;  // floats per vector of a warp's row sums (64 rows, padded against bank conflicts)
constexpr int kMmaRed = kMmaWarps * 16 * kMmaRedStride * 4;
constexpr int kMmaStage = kMixedHeader + kMmaArea;
constexpr int kMmaStages = (kSmemLimit - 256 - kMixedBlkBuf - kMmaRed) / kMmaStage;
constexpr int kMmaSmem = kMmaStages * kMmaStage + 256 + kMmaRed + kMixedBlkBuf;
static_assert(kMmaStages >= 3, "at least three stages");

__device__ __forceinline__ void mma_m16n8k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, bool bf16) {
  if (bf16)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// int16 codes (offset binary c = q + 32768) of two columns, packed: h = (c >> 8) - 128 and l = (c & 255) / 256
// as fp16 pairs (0x6400 | b is the fp16 of 1024 + b)
__device__ __forceinline__ uint32_t int16_high(uint32_t c) {
  const uint32_t v = __byte_perm(c, 0x64646464u, 0x4341);
  const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&v), __float2half2_rn(-1152.f));
  return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ uint32_t int16_low(uint32_t c) {
  const uint32_t v = __byte_perm(c, 0x64646464u, 0x4240);
  const __half2 r = __hfma2(*reinterpret_cast<const __half2*>(&v), __float2half2_rn(0.00390625f), __float2half2_rn(-4.f));
  return *reinterpret_cast<const uint32_t*>(&r);
}

// Producer warp: as mixed_produce, with the blocks' vector chunks in the parts' layout (a wide block's in FP32).
// Stage header (ints): [0] R, [1] nb, [2] row, [3] flags, [4] vector halves (1 or 2); block t at 8 + 4 t:
// columns | panel << 17 | wide << 18 | low << 19 | vector stride << 24, vector offset, matrix offset, scale; [48] nv, [49] xy32, [50..51] y, [52..53] ldy.
// WIDE: the launch's matrices have wide or low blocks.
template <bool WIDE>
__device__ __forceinline__ void mma_produce(const MixedStreamParams& P, const StreamShared& S, int ib, int ie,
                                            MixedBlock* blkbuf) {
  const int lane = threadIdx.x & 31;
  const uint64_t pol = policy_evict_first();
  int issued = 0;
  bool ok = true;
  StreamParams W{};
  W.err = P.err;
  W.budget = P.budget;
  for (int base = ib; base < ie && ok; base += 32) {
    StreamItem mine{};
    if (base + lane < ie) mine = P.items[base + lane];
    const int cnt = min(32, ie - base);
    // the batch's items cover a contiguous range of blocks: stage their records in shared memory
    const long long bfirst = __shfl_sync(0xFFFFFFFFu, mine.v_off, 0);
    const unsigned lshape = __shfl_sync(0xFFFFFFFFu, mine.shape, cnt - 1);
    const long long blast = __shfl_sync(0xFFFFFFFFu, mine.v_off, cnt - 1) + min((int)((lshape >> 8) & 0xFF), kMixedMaxBlocks);
    const int nbatch = (int)min(blast - bfirst, (long long)kMixedBatchBlocks);
    for (int u = lane; u < nbatch; u += 32) blkbuf[u] = P.blk[bfirst + u];
    // each lane fetches the matrix fields of its own item
    unsigned long long l_dmat = 0, l_xp = 0, l_x4 = 0, l_y = 0;
    long long l_ldy = 0;
    int l_nv = 0, l_xy32 = 0, l_xks = 0;
    if (base + lane < ie) {
      const MatDesc& D = P.mats[mine.flags >> 8];
      l_dmat = reinterpret_cast<unsigned long long>(D.dmat);
      l_xp = reinterpret_cast<unsigned long long>(D.xp);
      l_x4 = reinterpret_cast<unsigned long long>(D.x4);
      l_y = reinterpret_cast<unsigned long long>(D.y);
      l_ldy = D.ldy;
      l_nv = D.nv;
      l_xy32 = D.xy32;
      l_xks = D.xks;
    }
    __syncwarp();
    for (int t = 0; t < cnt; t++) {
      const int it = base + t - ib;
      const int s = it % kMmaStages, use = it / kMmaStages;
      const long long m_off = __shfl_sync(0xFFFFFFFFu, mine.m_off, t), b0 = __shfl_sync(0xFFFFFFFFu, mine.v_off, t);
      const int m_bytes = __shfl_sync(0xFFFFFFFFu, mine.m_bytes, t), row = __shfl_sync(0xFFFFFFFFu, mine.row, t);
      const unsigned shape = __shfl_sync(0xFFFFFFFFu, mine.shape, t);
      const int flags = __shfl_sync(0xFFFFFFFFu, mine.flags, t);
      const char* dmat = reinterpret_cast<const char*>(__shfl_sync(0xFFFFFFFFu, l_dmat, t));
      const unsigned char* xp = reinterpret_cast<const unsigned char*>(__shfl_sync(0xFFFFFFFFu, l_xp, t));
      const float* x4 = reinterpret_cast<const float*>(__shfl_sync(0xFFFFFFFFu, l_x4, t));
      const unsigned long long ydst = __shfl_sync(0xFFFFFFFFu, l_y, t);
      const long long ldy = __shfl_sync(0xFFFFFFFFu, l_ldy, t);
      const int nv = __shfl_sync(0xFFFFFFFFu, l_nv, t), xy32 = __shfl_sync(0xFFFFFFFFu, l_xy32, t);
      const int xks = __shfl_sync(0xFFFFFFFFu, l_xks, t);
      const int R = (int)(shape & 0xFF), nb = min((int)((shape >> 8) & 0xFF), kMixedMaxBlocks), nh = nv > 8 ? 2 : 1;
      if (use > 0 && !warp_wait(S.empty + s, (use - 1) & 1, W, S.abort_flag)) {
        ok = false;
        break;
      }
      if (__any_sync(0xFFFFFFFFu, *S.abort_flag != 0)) {
        ok = false;
        break;
      }
      unsigned char* stage = S.stage0 + s * kMmaStage;
      int* hd = reinterpret_cast<int*>(stage);
      MixedBlock mb{};
      const long long bi = b0 - bfirst + lane;
      if (lane < nb && bi >= 0 && bi < nbatch) mb = blkbuf[bi];
      const int codes = (mb.src & 4) ? panel_block_bytes(mb.cols) : (code_stride(R) * (int)mb.cols * 2 + 15) & ~15;
      const bool wide = WIDE && (mb.src & kBlockWide) != 0;  // (the FP32 chunk is no larger than the parts)
      const int vbytes = (lane < nb && nv > 0) ? (wide ? 4 * nv * mb.vs : xp_chunk_bytes((mb.cols + 15) / 16, nh)) : 0;
      int moff = codes, voff = vbytes;  // inclusive prefixes of the blocks' bytes
#pragma unroll
      for (int d = 1; d < kMixedMaxBlocks; d <<= 1) {
        const int o = __shfl_up_sync(0xFFFFFFFFu, moff, d), p = __shfl_up_sync(0xFFFFFFFFu, voff, d);
        if (lane >= d) {
          moff += o;
          voff += p;
        }
      }
      const int vtot = __shfl_sync(0xFFFFFFFFu, voff, kMixedMaxBlocks - 1);
      moff -= codes;
      voff += m_bytes - vbytes;  // the vectors' chunks follow the codes
      if (lane < nb) {
        hd[8 + 4 * lane] = mb.cols | ((mb.src & (4 | kBlockWide | kBlockLow)) << 15) | (mb.vs << 24);
        hd[9 + 4 * lane] = voff;
        hd[10 + 4 * lane] = moff;
        hd[11 + 4 * lane] = __float_as_int(mb.scale);
      }
      if (lane == 0) {
        hd[0] = R;
        hd[1] = nb;
        hd[2] = row;
        hd[3] = flags;
        hd[4] = nh;
        hd[kHdNv] = nv;
        hd[kHdXy32] = xy32;
        *reinterpret_cast<unsigned long long*>(hd + kHdY) = ydst;
        *reinterpret_cast<long long*>(hd + kHdLdy) = ldy;
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_expect_tx(S.full + s, (unsigned)(m_bytes + vtot));
        bulk_g2s_stream(stage + kMixedHeader, dmat + m_off, (unsigned)m_bytes, S.full + s, pol);
      }
      __syncwarp();
      if (vbytes > 0)
        bulk_g2s(stage + kMixedHeader + voff,
                 wide ? static_cast<const void*>(x4 + (long long)mb.voff * nv) : xp + (long long)mb.leaf * xp_chunk_bytes(xks, nh),
                 (unsigned)vbytes, S.full + s);
      __syncwarp();
      issued = it + 1;
    }
  }
  if (lane == 0)
    for (int it = max(0, issued - kMmaStages); it < issued; it++) {  // copies in flight land before exit
      const int s = it % kMmaStages, use = it / kMmaStages;
      const long long t0 = clock64();
      while (!mbar_try_wait(S.full + s, use & 1) && clock64() - t0 < P.budget) {
      }
    }
}

__device__ __forceinline__ uint2 lds64(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
  return v;
}

// Four tiles of one block (C columns): run[i] += sigma sum_c D(row, c) x_v(c), i < 4. Lane (g, t) of the warp
// loads its four rows row .. row + 3 in columns t, t + 4, t + 8, t + 12 of a K step, which stand for k = 2t,
// 2t + 1, 2t + 8, 2t + 9 of the fragments here and in the parts (neighbouring lanes read neighbouring columns:
// with 32 rows half the bank conflicts). Codes at `base`, a column `cb` bytes on (shared-memory addresses); tile i holds row + i. run[i]: vectors g (0, 1) and g + 8
// (2, 3), the rows of lanes g = 2t and 2t + 1. (Four tiles with two accumulators each fit the registers of 13
// warps; the halves of a 64-row block go to two warps.) LOAD 2: C is a multiple of 16 and a column's four
// rows are one aligned 8-byte load; 1: the same with the last K step's columns tested (tested in every case, 64-point
// blocks took 318 us for 301: 2D n = 65,536, 64 vectors); 0: every code is tested and loaded by itself.
template <int F, int LOAD>
__device__ __forceinline__ void mma_block(uint32_t base, int cb, uint32_t X, int C, int rows, float scale, int nh, bool low,
                                          float (&run)[4][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float hi[4][4], lo[4][4];
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int e = 0; e < 4; e++) hi[i][e] = lo[i][e] = 0.f;
  uint32_t col[4];
#pragma unroll
  for (int q = 0; q < 4; q++) col[q] = base + (t + 4 * q) * cb;
  uint32_t xa = X + kXpScale + lane * 8;
  const int half = nh > 1 ? kXpStep : 0, xstep = nh * kXpStep;
  // a K step's codes are loaded before the MMAs of the step before it
  uint32_t w[4][2];
  auto load_codes = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      w[q][0] = w[q][1] = 0u;
      if (LOAD == 2 || k0 + t + 4 * q < C) {
        if constexpr (LOAD > 0) {
          const uint2 u = lds64(col[q]);
          w[q][0] = u.x, w[q][1] = u.y;
        } else {
#pragma unroll
          for (int i = 0; i < 4; i++)
            if (i < rows) w[q][i / 2] |= lds16(col[q] + 2 * i) << (16 * (i & 1));
        }
      }
      col[q] += 16 * cb;
    }
  };
  load_codes(0);
#pragma unroll 1
  for (int k0 = 0; k0 < C; k0 += 16) {
    uint32_t a[3][4];
#pragma unroll
    for (int p = 0; p < 3; p++) {
      const uint2 u = lds64(xa + 256 * p), v = lds64(xa + 256 * p + half);  // (the same again for up to eight vectors)
      a[p][0] = u.x;
      a[p][1] = v.x;
      a[p][2] = u.y;
      a[p][3] = v.y;
    }
    xa += xstep;
    constexpr bool bf = F == kFormBf16, digits = F == kFormInt16;
    uint32_t bh[4][2], bl[4][2];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const uint32_t c = __byte_perm(w[2 * h][i / 2], w[2 * h + 1][i / 2], (i & 1) ? 0x7632u : 0x5410u);
        bh[i][h] = digits ? int16_high(c) : c;
        bl[i][h] = digits ? int16_low(c) : 0u;
      }
    if (k0 + 16 < C) load_codes(k0 + 16);
    // the tiles in turn, so that an MMA does not wait for the one before it
#pragma unroll
    for (int i = 0; i < 4; i++) mma_m16n8k16(hi[i], a[0], bh[i][0], bh[i][1], bf);
#pragma unroll
    for (int p = 1; p < 3; p++)
#pragma unroll
      for (int i = 0; i < 4; i++) mma_m16n8k16(lo[i], a[p], bh[i][0], bh[i][1], bf);
    if constexpr (digits)
#pragma unroll
      for (int p = 0; p < 2; p++)
#pragma unroll
        for (int i = 0; i < 4; i++) mma_m16n8k16(lo[i], a[p], bl[i][0], bl[i][1], bf);
    if (digits && low) {
#pragma unroll
      for (int i = 0; i < 4; i++) mma_m16n8k16(lo[i], a[2], bl[i][0], bl[i][1], bf);
    }
  }
  float sc[2];
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(sc[0]) : "r"(X + 4 * g));
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(sc[1]) : "r"(X + 4 * g + 32));
  const float s0 = F == kFormInt16 ? 256.f * scale : scale;
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int e = 0; e < 4; e++) run[i][e] = fmaf(s0 * sc[e >> 1], hi[i][e] + lo[i][e], run[i][e]);
}

// The same of a wide block, in FP32, for up to 8 NH vectors: codes at `codes`, vectors X ([vector][vs points]); n = 2t +
// (e & 1), its four rows from row rows[e & 1], tile i the i-th of them (rows past R are not stored). Bound by issue slots
// like the streams (2D n = 50,001, int16, every block wide: dense phase of 8 / 16 vectors 105 / 131 us; rows loaded one by
// one and both halves whatever the count: 188 / 190; the stream with as many vectors 166 / 217).
// FOUR: a column's four rows are one aligned load.
template <int F, int NH, bool FOUR>
__device__ __forceinline__ void mma_wide_block(const unsigned char* codes, bool panel, const float* X, int vs, int C, int R,
                                               const int (&rows)[2], float scale, int nv, float (&run)[4][4]) {
  const int g = (threadIdx.x & 31) >> 2;
  float acc[4][2 * NH];
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int e = 0; e < 2 * NH; e++) acc[i][e] = 0.f;
  const uint16_t* A[2];
#pragma unroll
  for (int u = 0; u < 2; u++)
    A[u] = reinterpret_cast<const uint16_t*>(codes) + (panel ? (rows[u] >> 3) * (panel_stride(C) / 2) + (rows[u] & 7) : rows[u]);
  const int cs = panel ? 8 : code_stride(R);
#pragma unroll 4
  for (int c = 0; c < C; c++) {
    float x[NH];
#pragma unroll
    for (int b = 0; b < NH; b++) x[b] = g + 8 * b < nv ? X[(g + 8 * b) * vs + c] : 0.f;
#pragma unroll
    for (int u = 0; u < 2; u++) {
      float a[4];
      if constexpr (FOUR) {
        const uint2 w = *reinterpret_cast<const uint2*>(A[u] + c * cs);
        const float2 lo = codes_to_f2<F>(w.x), hi = codes_to_f2<F>(w.y);
        a[0] = lo.x, a[1] = lo.y, a[2] = hi.x, a[3] = hi.y;
      } else {
#pragma unroll
        for (int i = 0; i < 4; i++) a[i] = rows[u] + i < R ? code_to_f<F>(A[u][c * cs + i]) : 0.f;
      }
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int b = 0; b < NH; b++) acc[i][u + 2 * b] = fmaf(a[i], x[b], acc[i][u + 2 * b]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int e = 0; e < 2 * NH; e++) run[i][e] = fmaf(scale, acc[i][e], run[i][e]);
}

// (WIDE in every launch: 32 matrices of 1024 .. 16384 points, fp16, 667 -> 674 us with no wide block among them)
template <int F, bool WIDE>
__global__ void __launch_bounds__((kMmaWarps + 1) * 32, 1) k_dense_mma(MixedStreamParams P) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const StreamShared S = stream_shared<kMmaStages, kMmaStage>(smem);
  stream_init<kMmaStages, kMmaWarps>(S);
  const int ib = P.cta_begin[blockIdx.x], ie = P.cta_begin[blockIdx.x + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  if (warp == kMmaWarps) {
    mma_produce<WIDE>(P, S, ib, ie, reinterpret_cast<MixedBlock*>(smem + kMmaStages * kMmaStage + 256 + kMmaRed));
    return;
  }
  StreamParams W{};
  W.err = P.err;
  W.budget = P.budget;
  float* red = reinterpret_cast<float*>(S.red);
  float* mine = red + warp * 16 * kMmaRedStride;
  float run[4][4];
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int e = 0; e < 4; e++) run[i][e] = 0.f;
  // the warp's next unit, counted from the current item's first: a block, or (more than 32 rows) half of one
  int rows_done = 0, turn = warp;
  for (int it = 0; it < ie - ib; it++) {
    const int st = it % kMmaStages, use = it / kMmaStages;
    if (!warp_wait(S.full + st, use & 1, W, S.abort_flag)) break;
    const unsigned char* stage = S.stage0 + st * kMmaStage;
    const int* hd = reinterpret_cast<const int*>(stage);
    const int R = min(hd[0], 64), nb = min(hd[1], kMixedMaxBlocks), row = hd[2], flags = hd[3], nh = min(hd[4], 2);
    const int nv = min(hd[kHdNv], 16);
    void* const ydst = reinterpret_cast<void*>(*reinterpret_cast<const unsigned long long*>(hd + kHdY));
    const bool y32 = hd[kHdXy32] != 0;
    const long long ldy = *reinterpret_cast<const long long*>(hd + kHdLdy);
    const int two = R > 32 ? 1 : 0;  // lane g's rows: 8 g + 4 (unit & 1) .., or 4 g ..
    if (nv > 0) {
      for (; turn < nb << two; turn += kMmaWarps) {
        const int4 bh = *reinterpret_cast<const int4*>(hd + 8 + 4 * (turn >> two));
        const int C = min(bh.x & 0xFFFF, 64);
        const bool panel = (bh.x >> 17) & 1;
        const int moff = min(bh.z, kStageMat - 16) & ~15, voff = min(bh.y, kMmaArea - 16) & ~15;
        if (WIDE && ((bh.x >> 18) & 1)) {
          const int n0 = two ? 8 * 2 * t + 4 * (turn & 1) : 4 * 2 * t, rows[2] = {n0, n0 + (two ? 8 : 4)};
          const unsigned char* wc = stage + kMixedHeader + moff;
          const float* wx = reinterpret_cast<const float*>(stage + kMixedHeader + voff);
          const int vs = min((int)((unsigned)bh.x >> 24), 64);
          const bool four = panel || (code_stride(R) & 3) == 0;
          if (four && nh == 1) mma_wide_block<F, 1, true>(wc, panel, wx, vs, C, R, rows, __int_as_float(bh.w), nv, run);
          else if (four) mma_wide_block<F, 2, true>(wc, panel, wx, vs, C, R, rows, __int_as_float(bh.w), nv, run);
          else mma_wide_block<F, 2, false>(wc, panel, wx, vs, C, R, rows, __int_as_float(bh.w), nv, run);
          continue;
        }
        const uint32_t codes = smem_addr(stage + kMixedHeader) + moff, X = smem_addr(stage + kMixedHeader) + voff;
        const int r = two ? 8 * g + 4 * (turn & 1) : 4 * g, cb = panel ? 16 : 2 * code_stride(R);
        // (in the column-major layout the last lanes' rows may lie past R: they read what follows, unused)
        const uint32_t base = codes + (panel ? (r >> 3) * panel_stride(C) + 2 * (r & 7) : 2 * r);
        const bool wide = panel || (code_stride(R) & 3) == 0, low = WIDE && ((bh.x >> 19) & 1);
        if (wide && (C & 15) == 0) mma_block<F, 2>(base, cb, X, C, 4, __int_as_float(bh.w), nh, low, run);
        else if (wide) mma_block<F, 1>(base, cb, X, C, 4, __int_as_float(bh.w), nh, low, run);
        else mma_block<F, 0>(base, cb, X, C, R - r, __int_as_float(bh.w), nh, low, run);
      }
      turn -= nb << two;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(S.empty + st);
    if (!(flags & kItemFlagLast)) continue;
    if (rows_done > 0 && !warp_wait(S.rowfree, (rows_done - 1) & 1, W, S.abort_flag)) break;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const int n = 2 * t + (e & 1);
        mine[(g + 8 * (e >> 1)) * kMmaRedStride + (two ? 8 * n + 4 * (warp & 1) : 4 * n) + i] = run[i][e];
        run[i][e] = 0.f;
      }
    __syncwarp();
    if (lane == 0) mbar_arrive(S.rowfull);
    if (!warp_wait(S.rowfull, rows_done & 1, W, S.abort_flag)) break;
    for (int idx = threadIdx.x; idx < 64 * nv; idx += kMmaWarps * 32) {
      const int r = idx & 63, v = idx >> 6;
      if (r >= R) continue;
      // 64-row leaves: rows 8 n + 4 .. are the odd warps'
      float sum = 0.f;
      if (two) {
#pragma unroll
        for (int w = 0; w < kMmaWarps; w += 2) sum += red[((w + ((r >> 2) & 1)) * 16 + v) * kMmaRedStride + r];
      } else {
#pragma unroll
        for (int w = 0; w < kMmaWarps; w++) sum += red[(w * 16 + v) * kMmaRedStride + r];
      }
      y_store(ydst, y32, v * ldy + row + r, sum, false);  // y was assigned by the expansion
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(S.rowfree);
    rows_done++;
    turn = warp;
  }
}

}  // namespace h2
