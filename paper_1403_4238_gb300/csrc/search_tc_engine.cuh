// Tensor-core search of the persistent engine: the exact BF16 correlation
// form of the masked SSD (Sec. 3, Eq. 3-4) over the tiles of a searching
// CTA.
//
// With b' = byte - 128 (|b'| <= 128, exact in BF16) and m the known flags of
// the target patch Psi_p^ (zero outside the image):
//   SSD(q) = A2 - 2 X(q) + S(q),   A2 = sum_d m(d) sum_c t'_c(d)^2,
//   X(q) = sum_c sum_d m(d) t'_c(d) s'_c(q + d),
//   S(q) = sum_d m(d) sq(q + d),   sq = sum_c s'_c^2 = 256 hi + lo (hi, lo < 256).
// Every product is exact and every partial sum an integer below 2^24
// (|X| <= 17^2 * 3 * 128^2, S <= 17^2 * 49152), so the FP32 accumulation is
// exact and the SSD equals the CUDA-core form's bit for bit.
//
// One MMA (M = 128, N = 16 .. 128, K = 16, BF16 operands in shared memory,
// FP32 accumulators in tensor memory) takes one source row y of a tile
// whose candidate rows are y0 .. y0 + 15 and whose candidate columns start
// at xs + R:
//  * A, the target as a Toeplitz matrix: row m = 8 i + b (candidate row
//    y0 + i, column shift b), K column kk of item (plane p, 8-tap chunk c)
//    holds w_p(k, 8c + kk - b) for target row k = y - y0 - i, where w is
//    m t'_p (p < 3) or m (p = 3, for both square planes), zero outside the
//    patch.  A strip (p, c) stores its 8x8 core matrices for target rows
//    P-1 .. 0 in that order between runs of 15 zero matrices, so the A
//    operand of row y is the 16 consecutive matrices that start at target
//    row y - y0, and an MMA's two K halves are two items of their own (the
//    leading byte offset is the distance between their strips).
//  * B, the source row itself: five plane-row segments side by side (R', G',
//    B', 256 hi -- exact in BF16, as hi < 256 -- and lo); row n of B
//    (candidate columns 8n .. 8n + 7) starts 16 bytes after row n - 1 (rows
//    overlap), chunk c 16 bytes further.
//  * D: accumulator X (the three channel planes, items paired across
//    planes) or S (256 hi and lo of one chunk against the same mask strip:
//    a leading byte offset of 0 in A); lane m, column n is candidate
//    (y0 + m / 8, xs + 8 n + m % 8 + R).
// One producer thread copies the tiles' source rows into a ring of
// shared-memory slots (one bulk copy of two rows, five plane segments each,
// from the planes' tiled layout), two issuer warps issue the X and the S MMAs
// of a slot's rows once they have landed and free the slot with
// tcgen05.commit.  Accumulators are read back (tcgen05.ld), tested against the
// tile's validity bits and reduced to the smallest (SSD << 32 | idx) key: by
// eight warps beside the next tile's MMAs, which fill the other of two
// accumulator buffers, and by all 16 warps after a CTA's last tile.  The
// read-back works in FP32:
// fl(fl(S - 2X) + A2) is exact whenever the SSD is below 2^24 (then |S - 2X|
// < 2^24 too, as A2 < 2^24) and at least 2^24 otherwise (rounding is
// monotone), so a best value below 2^24 is the exact minimum; a warp with a
// thread whose best is not repeats its candidates in integers.
#pragma once
#include "inpaint_engine.h"
#include "ptx.cuh"

namespace inp {

template <int R>
struct TcEngGeom {
  static constexpr int P = 2 * R + 1;
  static constexpr int NC = (P + 14) / 8;              // 8-tap chunks: taps b + dx < P + 7
  static constexpr int NRS = kTcRows + P - 1;          // source rows of a tile
  static constexpr int NSL = NRS / kTcRps;             // ring slots a tile fills
  static constexpr int NSTRIP = 4 * NC;                // (plane, chunk) strips of A: 3 channels, mask
  static constexpr int ZG = 15;                        // zero matrices between strips
  static constexpr int ZERO = ZG + NSTRIP * (P + ZG);  // 16 zero matrices: the empty K half
  static constexpr int NGA = ZERO + 16;                // 8x8 core matrices of the A area
  static constexpr int A_BYTES = NGA * 128;
  static constexpr int NX = 3 * NC;                    // cross-term items of a source row
  static constexpr int NXP = (NX + 1) / 2;             // X MMAs of a source row
  static constexpr int TW = 32;                        // padded target row: taps -8 .. 23
  static constexpr int TPAD_BYTES = (4 * P * TW * 2 + 127) / 128 * 128;
  __host__ __device__ static constexpr int sg(int st) { return ZG + st * (P + ZG); }
  static_assert(NC == (R <= 4 ? 2 : 3), "chunks cover every tap");
  static_assert(NRS % kTcRps == 0, "whole slots per tile");
  static_assert(8 * NC <= TW - 8, "padded target row covers every chunk");
};
// Bytes of one plane-row segment of a tile and of a ring slot (kTcRps rows
// of five segments).
__host__ __device__ inline int tc_lrow(int N, int r) { return 16 * (N + tc_chunks(r) - 1); }
__host__ __device__ inline int tc_slot(int N, int r) { return (kTcRps * 5 * tc_lrow(N, r) + 16 + 127) & ~127; }

// Where a tensor-core search keeps its state: A | padded target | ring.
// The padded target table (written by the searcher's target staging):
// tpad[(p * P + k) * TW + 8 + jj] = w_p(k, jj) for p < 4 (R' G' B', the
// known flag) and jj in [-8, 24), zero outside the patch or where unknown.
struct TcArea {
  uint8_t* a;
  uint16_t* tpad;
  uint8_t* ring;
  int nb;    // ring slots
  int slot;  // bytes per slot
};

// The target patch at (px, py) into the padded table, and per target row its
// share of A2 (whole block; a barrier must follow).  Warp dy reads row dy.
template <int R>
__device__ __forceinline__ void tc_stage_target(const ImgState& s, uint16_t* tpad, int* a2row, int px, int py) {
  using G = TcEngGeom<R>;
  constexpr int P = G::P;
  const int lane = threadIdx.x & 31;
  for (int dy = threadIdx.x >> 5; dy < P; dy += kEngWarps) {
    const int tx = px + lane - R, ty = py + dy - R;
    uint32_t w = 0;
    bool known = false;
    if (lane < P && tx >= 0 && tx < s.W && ty >= 0 && ty < s.H) {
      const uint8_t o = __ldcg(&s.omega[(size_t)ty * s.W + tx]);
      const uint32_t v = __ldcg(&s.img[(size_t)ty * s.pitch + tx]);
      known = o == 0;
      w = known ? v : 0u;
    }
    int sq = 0;
    if (lane < P) {
      const int d0 = known ? (int)(w & 255u) - 128 : 0, d1 = known ? (int)((w >> 8) & 255u) - 128 : 0,
                d2 = known ? (int)((w >> 16) & 255u) - 128 : 0;
      sq = d0 * d0 + d1 * d1 + d2 * d2;
      uint16_t* tp = tpad + dy * G::TW + 8 + lane;
      tp[0] = (uint16_t)bf16_of_int(d0);
      tp[P * G::TW] = (uint16_t)bf16_of_int(d1);
      tp[2 * P * G::TW] = (uint16_t)bf16_of_int(d2);
      tp[3 * P * G::TW] = (uint16_t)bf16_of_int(known ? 1 : 0);
    }
    sq = __reduce_add_sync(0xffffffffu, sq);
    if (lane == 0) a2row[dy] = sq;
  }
}

// The A strips from the padded target (threads [0, nthr)); the zero
// matrices are written only when `pads` (the first round of an image).  The
// writing threads order their stores before the MMAs' reads (proxy fence).
template <int R>
__device__ __forceinline__ void tc_build_a(uint8_t* A, const uint16_t* tpad, bool pads, int nthr) {
  using G = TcEngGeom<R>;
  constexpr int P = G::P, TW = G::TW;
  const int tid = threadIdx.x;
  if (tid >= nthr) return;
  if (pads) {
    for (int e = tid; e < G::NGA * 8; e += nthr) {
      const int rel = (e >> 3) - G::ZG;
      const bool strip = rel >= 0 && rel / (P + G::ZG) < G::NSTRIP && rel % (P + G::ZG) < P;
      if (!strip) reinterpret_cast<uint4*>(A)[e] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  for (int e = tid; e < G::NSTRIP * P * 8; e += nthr) {
    const int b = e & 7, j = (e >> 3) % P, st = (e >> 3) / P;
    const int p = st / G::NC, c = st - p * G::NC, k = P - 1 - j;
    // taps 8c - b .. 8c - b + 7 of target row k, plane p
    const uint16_t* src = tpad + (p * P + k) * TW + 8 + 8 * c - b;
    uint32_t w[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) w[h] = (uint32_t)src[2 * h] | ((uint32_t)src[2 * h + 1] << 16);
    *reinterpret_cast<uint4*>(A + (G::sg(st) + j) * 128 + b * 16) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  fence_proxy_async_smem();
}

// Producer: ring slots [h0, h1) of the tile in tile column tx whose source
// rows start at image row y0 - R (ring sequence numbers g0 + h; slot h holds rows
// 2h, 2h + 1, five plane segments of tc_len elements each).  One thread.
// Returns false if a bounded wait gave up.
template <int R>
__device__ __forceinline__ bool tc_produce(const ImgState& s, const TcArea& ta, EngBars& bars, int tx, int y0,
                                           uint32_t g0, int h0, int h1, unsigned long long limit) {
  const uint32_t bytes = (uint32_t)(kTcRps * 5 * 2 * s.tc_len);
  const int row0 = y0 - s.cy0;  // plane row of image row y0 - R
  for (int h = h0; h < h1; ++h) {
    const uint32_t g = g0 + (uint32_t)h;
    const int slot = (int)(g % (uint32_t)ta.nb);
    if (g >= (uint32_t)ta.nb && !mbar_wait(&bars.tc_empty[slot], ((g / ta.nb) - 1u) & 1u, limit)) return false;
    mbar_expect_tx(&bars.tc_full[slot], bytes);
    const uint16_t* src = s.planes + ((size_t)tx * s.prows + (row0 + kTcRps * h)) * 5 * s.tc_len;
    bulk_load(ta.ring + (size_t)slot * ta.slot, src, bytes, &bars.tc_full[slot]);
  }
  return true;
}

// Issuer of the X MMAs (KIND 0) or the S MMAs (KIND 1) of a tile's NRS source
// rows into the accumulators at `tmem` (X: columns [0, N), S: [128, 128 + N)),
// then a commit to `done`.  One whole warp (the descriptor arithmetic is
// warp-uniform; one elected lane issues).  The parts of a descriptor that
// depend on N are a few registers, the rest are immediates.
template <int R, int KIND>
__device__ __forceinline__ bool tc_issue(const TcArea& ta, EngBars& bars, int N, uint32_t tmem, uint64_t* done,
                                         uint32_t g0, unsigned long long limit) {
  using G = TcEngGeom<R>;
  constexpr int P = G::P, NC = G::NC, NM = KIND == 0 ? G::NXP : NC;
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  const uint32_t hi = (128u >> 4) | (1u << 14);  // stride byte offset 128, descriptor version 1
  const uint32_t d = tmem + (KIND == 0 ? 0u : 128u);
  const uint32_t a_lo0 = smem_addr(ta.a) >> 4, r_lo0 = smem_addr(ta.ring) >> 4;
  const int nb = ta.nb;
  const uint32_t slot_units = (uint32_t)ta.slot >> 4;
  const uint32_t L = (uint32_t)(N + NC - 1);  // 16-byte units of a plane-row segment
  uint32_t boff[NM];                          // B: first item's offset | leading byte offset to the second
#pragma unroll
  for (int q = 0; q < NM; ++q) {
    const int i1 = KIND == 0 ? 2 * q : 3 * NC + q, i2 = KIND == 0 ? 2 * q + 1 : 4 * NC + q;
    const uint32_t o1 = (uint32_t)(i1 / NC) * L + (uint32_t)(i1 % NC);
    // (zero weights take any finite data)
    const uint32_t o2 = KIND == 1 || i2 < G::NX ? (uint32_t)(i2 / NC) * L + (uint32_t)(i2 % NC) : o1 + 1u;
    boff[q] = o1 + ((o2 - o1) << 16);
  }
  int slot = (int)(g0 % (uint32_t)nb);
  uint32_t par = (g0 / (uint32_t)nb) & 1u;
  bool ok = true;
#pragma unroll 1
  for (int h = 0; h < G::NSL; ++h) {
    if (!__all_sync(0xffffffffu, mbar_wait(&bars.tc_full[slot], par, limit))) {
      ok = false;
      break;
    }
    tc_fence_after();
    const uint32_t b_slot = r_lo0 + (uint32_t)slot * slot_units;
#pragma unroll
    for (int rr = 0; rr < kTcRps; ++rr) {
      const int j = kTcRps * h + rr;
      const uint32_t a_row = a_lo0 + (uint32_t)(P - 1 - j) * 8u;
      const uint32_t b_row = b_slot + (rr ? 5u * L : 0u);
#pragma unroll
      for (int q = 0; q < NM; ++q) {
        // A: first item's core matrix for row j, leading byte offset to the second
        // (offsets relative to row j's A base a_lo0 + (P - 1 - j) * 8)
        int a1, a2;
        uint32_t zl = 0u;  // row-dependent part of a leading byte offset
        if (KIND == 0) {
          const int i1 = 2 * q, i2 = 2 * q + 1;
          a1 = G::sg(i1);
          if (i2 < G::NX) {
            a2 = G::sg(i2);
          } else {  // the second K half reads the zero matrices
            a2 = G::ZERO - (P - 1);
            zl = (uint32_t)(j * 8) << 16;
          }
        } else {
          a1 = a2 = G::sg(3 * NC + q);  // both K halves: the mask strip
        }
        const uint32_t alo = a_row + (uint32_t)(a1 * 8 + ((a2 - a1) * 8 << 16)) + zl;
        const uint32_t blo = b_row + boff[q];
        if (q == 0)
          tc_mma_lo_elect(d, alo, hi, blo, hi, idesc, j != 0);
        else
          tc_mma_lo_elect(d, alo, hi, blo, hi, idesc, true);
      }
    }
    tc_commit_elect(&bars.tc_empty[slot]);
    if (++slot == nb) {
      slot = 0;
      par ^= 1u;
    }
  }
  tc_commit_elect(done);  // also when a wait gave up: the MMAs issued so far
  return ok;
}

// The validity bits a warp's read-back needs (its four candidate rows, the
// columns of its group): lane l holds the words of row l / (cols / 8), columns
// 8 (l % (cols / 8)) .. + 7.  One load, issued before the wait for the MMAs.
__device__ __forceinline__ uint2 tc_bits_load(const uint32_t* tbits, int N, int ngroups) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int steps = N / ngroups / 8, r4 = lane / steps;
  if (r4 >= 4) return make_uint2(0u, 0u);
  return __ldcg(reinterpret_cast<const uint2*>(tbits + (4 * (warp & 3) + r4) * (N / 4)) + (warp >> 2) * steps +
                lane - r4 * steps);
}

// Accumulators at `tmem` of tile (y0, xs) -> this thread's best key, after the
// tile's done barrier.  ngroups = warps / 4 column groups: warp w reads the
// tensor-memory lanes of its quarter w % 4 and the columns of group w / 4, 16
// (8 at the end) at a time.  bits: tc_bits_load of the tile.
template <int R>
__device__ __forceinline__ unsigned long long tc_epilogue(const ImgState& s, uint32_t tmem, const TcTiles& tt,
                                                          int ngroups, int a2, uint2 bits, int y0, int tx,
                                                          unsigned long long best) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = warp & 3;
  const int m = 32 * q + lane, i = m >> 3, b = m & 7;
  const int cols = tt.N / ngroups, c0 = (warp >> 2) * cols;
  const int src0 = (lane >> 3) * (cols / 8);  // the lane that holds this row's first words
  // candidate of accumulator column n: n / n1 folds down, 8 (n % n1) columns right
  const int idx0 = (y0 + i) * s.W + tt.xs0 + 8 * tt.N * tx + b + R;
  auto idx_of = [&](int n) {
    const int f = tt.n1 == tt.N ? 0 : n / tt.n1;
    return idx0 + f * tt.h * s.W + 8 * (n - f * tt.n1);
  };
  const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0;
  const float a2f = (float)a2;  // exact: a2 < 2^24
  float bv = __int_as_float(0x7f800000);  // +inf
  int bi = 0;
  bool any = false;
  // eight columns from h: the smallest valid value and its column, kept in a
  // chain of their own (the two halves of a step overlap); candidates in
  // increasing index order (a fold's rows lie below the previous one's), so
  // the strict tests keep the first of equals
  auto test = [&](const uint32_t* X, const uint32_t* S, int h, float& v0, int& n0) {
    const uint32_t wx = __shfl_sync(0xffffffffu, bits.x, src0 + h / 8) >> b;
    const uint32_t wy = __shfl_sync(0xffffffffu, bits.y, src0 + h / 8) >> b;
    any |= ((wx | wy) & 0x01010101u) != 0u;
    v0 = __int_as_float(0x7f800000);
    n0 = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float v = __fadd_rn(__fmaf_rn(-2.0f, __uint_as_float(X[k]), __uint_as_float(S[k])), a2f);
      if (((k < 4 ? wx : wy) & (1u << (8 * (k & 3)))) && v < v0) {
        v0 = v;
        n0 = c0 + h + k;
      }
    }
  };
  auto keep = [&](float v, int n) {
    if (v < bv) {
      bv = v;
      bi = n;
    }
  };
  float v0, v1;
  int n0, n1;
  int h = 0;
#pragma unroll 1
  for (; h + 16 <= cols; h += 16) {
    uint32_t X[16], S[16];
    tc_ld16(ta + (uint32_t)h, X);
    tc_ld16(ta + (uint32_t)(128 + h), S);
    tc_wait_ld();
    test(X, S, h, v0, n0);
    test(X + 8, S + 8, h + 8, v1, n1);
    keep(v0, n0);
    keep(v1, n1);
  }
  if (h < cols) {
    uint32_t X[8], S[8];
    tc_ld8(ta + (uint32_t)h, X);
    tc_ld8(ta + (uint32_t)(128 + h), S);
    tc_wait_ld();
    test(X, S, h, v0, n0);
    keep(v0, n0);
  }
  // tcgen05.ld is a whole warp's instruction, so the warp decides together: it
  // takes the integer pass when any of its threads has no candidate below 2^24
  if (!__any_sync(0xffffffffu, any && !(bv < 16777216.0f))) {
    if (!any) return best;
    const unsigned long long key = ((unsigned long long)(uint32_t)bv << 32) | (unsigned)idx_of(bi);  // exact
    return key < best ? key : best;
  }
  // the exact integer pass over the same accumulators
#pragma unroll 1
  for (int h = 0; h < cols; h += 8) {
    uint32_t X[8], S[8];
    tc_ld8(ta + (uint32_t)h, X);
    tc_ld8(ta + (uint32_t)(128 + h), S);
    const uint2 w = make_uint2(__shfl_sync(0xffffffffu, bits.x, src0 + h / 8),
                               __shfl_sync(0xffffffffu, bits.y, src0 + h / 8));
    tc_wait_ld();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (((k < 4 ? w.x : w.y) >> (8 * (k & 3) + b)) & 1u) {
        const int xv = __float2int_rz(__uint_as_float(X[k]));
        const int sv = __float2int_rz(__uint_as_float(S[k]));
        const uint32_t ssd = (uint32_t)(a2 - 2 * xv + sv);
        const unsigned long long key = ((unsigned long long)ssd << 32) | (unsigned)idx_of(c0 + h + k);
        best = key < best ? key : best;
      }
    }
  }
  return best;
}

}  // namespace inp
