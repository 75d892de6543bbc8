// findBestPatch, plain CUDA-core form (Sec. 3 Eq. 3-4; Algorithm 1 and the
// local-memory staging of Algorithm 2 / Sec. 5.5 as prior art).
//
// For the selected target centre p^ and every valid candidate centre q (patch
// inside the image and fully known: unknown count 0), the SSD over the known
// in-image pixels d of Psi_p^ is
//     SSD(q) = sum_d sum_{c in RGB} (I[p^+d]_c - I[q+d]_c)^2,
// an exact 32-bit integer (at most 65^2 * 3 * 255^2 < 2^31).  Each CTA
// reduces its candidates to one key (SSD << 32 | idx(q)); the smallest key
// over all CTAs is the best patch, ties going to the lowest index.
//
// GB300 design: a CTA stages an (8 + 2r) x (128 + 2r) tile of RGBA words in
// shared memory (every pixel is reused by up to P^2 candidates), each thread
// keeps 4 adjacent candidates in registers, reads one row strip of the tile
// per patch row with 128-bit loads, and per known target pixel issues one
// byte-SIMD absolute difference and one 4-way byte dot product per candidate
// (|a-b| per channel, then sum of squares; alpha is 0 on both sides).
// Unknown target pixels are skipped by a warp-uniform branch on a per-row
// bit mask, so the work is |K| evaluations per candidate, not P^2.
#include "inpaint_internal.cuh"

namespace inp {

// The unknown counts of a thread's S candidates, requested before the SSD work
// that hides them; 1 (not a candidate) outside the search rectangle.
template <int S>
__device__ inline void load_counts(const ImgState& s, int qx0, int qy, int (&cnt)[S]) {
#pragma unroll
  for (int k = 0; k < S; ++k)
    cnt[k] = qx0 + k <= s.cx1 && qy <= s.cy1 ? s.count[(size_t)qy * s.pitch + qx0 + k] : 1;
}

// Smallest key over a thread's S candidates.
template <int S>
__device__ inline unsigned long long best_key(const ImgState& s, const uint32_t (&ssd)[S], const int (&cnt)[S],
                                              int qx0, int qy) {
  unsigned long long best = ~0ull;
#pragma unroll
  for (int k = 0; k < S; ++k) {
    const unsigned long long key = ((unsigned long long)ssd[k] << 32) | (unsigned)(qy * s.W + qx0 + k);
    if (cnt[k] == 0 && key < best) best = key;
  }
  return best;
}

// Stage a ROWS x PITCH window of image words whose top-left is (x0, y0), every
// load of a thread in flight at once (one L2 round trip).  Out-of-image words
// read as 0 (never used by a valid candidate); with AVAIL (partial-overlap
// search) the alpha byte says whether the pixel may be used as a source (0:
// known and in the image; 0xFF, with RGB bytes 0: unknown or outside).
template <int ROWS, int PITCH, bool AVAIL>
__device__ inline void stage_tile(const ImgState& s, uint32_t* dst, int x0, int y0) {
  constexpr int n = ROWS * PITCH, U = (n + kSearchThreads - 1) / kSearchThreads;
  constexpr uint32_t kNone = AVAIL ? 0xff000000u : 0u;
  uint32_t w[U];
  uint8_t o[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = threadIdx.x + u * kSearchThreads;
    const int yy = y0 + i / PITCH, xx = x0 + i % PITCH;
    const bool in = i < n && xx >= 0 && xx < s.W && yy >= 0 && yy < s.H;
    w[u] = in ? s.img[(size_t)yy * s.pitch + xx] : kNone;
    o[u] = AVAIL && in ? s.omega[(size_t)yy * s.W + xx] : 0;
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = threadIdx.x + u * kSearchThreads;
    if (i < n) dst[i] = AVAIL && o[u] ? kNone : w[u];
  }
}

// Target patch: known in-image pixels with their RGBA words (row pitch TP, 0
// elsewhere) and one bit mask per row; unk (may be null): the unknown in-image
// ones.  One warp per row, one lane per column, so the reads of a row are one
// L2 round trip (a thread that walked its row took one per pixel).
template <int P, int TP>
__device__ inline void stage_target(const ImgState& s, int px, int py, uint32_t* tgt, uint32_t* rowmask,
                                    uint32_t* unk) {
  constexpr int R = P / 2;
  static_assert(P <= 32, "one lane per column");
  const int lane = threadIdx.x & 31;
  for (int dy = threadIdx.x >> 5; dy < P; dy += kSearchThreads / 32) {
    const int tx = px + lane - R, ty = py + dy - R;
    const bool in = lane < P && tx >= 0 && tx < s.W && ty >= 0 && ty < s.H;
    uint32_t w = 0;
    bool known = false;
    if (in) {
      const uint8_t o = s.omega[(size_t)ty * s.W + tx];
      const uint32_t v = s.img[(size_t)ty * s.pitch + tx];
      known = o == 0;
      w = known ? v : 0u;
    }
    const unsigned m = __ballot_sync(0xffffffffu, known), u = __ballot_sync(0xffffffffu, in && !known);
    if (lane < TP) tgt[dy * TP + lane] = w;
    if (lane == 0) {
      rowmask[dy] = m;
      if (unk) unk[dy] = u;
    }
  }
}

__device__ inline void write_partial(const ImgState& s, unsigned long long best,
                                     unsigned long long* scratch) {
  best = block_min_u64(best, scratch);
  if (threadIdx.x == 0) s.partial[blockIdx.y * gridDim.x + blockIdx.x] = best;
}

template <int R>
__global__ void __launch_bounds__(kSearchThreads) k_search_plain(ImgState s) {
  constexpr int P = 2 * R + 1;
  constexpr int TW = kSearchTW, TH = kSearchTH, S = kSearchS;
  constexpr int SW = (TW + 2 * R + 3) & ~3;       // tile pitch (words), multiple of 4
  constexpr int SH = TH + 2 * R;
  constexpr int NROW = (S + P - 1 + 3) & ~3;      // words of one row strip
  static_assert(31 * S + NROW <= SW, "row strip must stay inside the tile");
  __shared__ __align__(16) uint32_t src[SH * SW];
  __shared__ uint32_t tgt[P * P];
  __shared__ uint32_t rowmask[P];
  __shared__ unsigned long long red[32];

  const Ctrl* c = s.ctrl;
  if (!loop_active(c)) return;
  const int px = c->px, py = c->py;
  const int ox = s.cx0 + blockIdx.x * TW, oy = s.cy0 + blockIdx.y * TH;
  const int tid = threadIdx.x;

  const int lane = tid & 31, wr = tid >> 5;  // warp = one candidate row of the tile
  int cnt[S];
  load_counts<S>(s, ox + lane * S, oy + wr, cnt);
  stage_target<P, P>(s, px, py, tgt, rowmask, nullptr);
  stage_tile<SH, SW, false>(s, src, ox - R, oy - R);
  __syncthreads();

  uint32_t acc[S];
#pragma unroll
  for (int k = 0; k < S; ++k) acc[k] = 0;

  for (int dy = 0; dy < P; ++dy) {
    const uint32_t m = rowmask[dy];
    if (m == 0) continue;
    uint32_t row[NROW];
    const uint4* sp = reinterpret_cast<const uint4*>(&src[(wr + dy) * SW + lane * S]);
#pragma unroll
    for (int i = 0; i < NROW / 4; ++i) {
      const uint4 v = sp[i];
      row[4 * i] = v.x;
      row[4 * i + 1] = v.y;
      row[4 * i + 2] = v.z;
      row[4 * i + 3] = v.w;
    }
    const uint32_t* trow = &tgt[dy * P];
#pragma unroll
    for (int dx = 0; dx < P; ++dx) {
      if (m & (1u << dx)) {
        const uint32_t a = trow[dx];
#pragma unroll
        for (int k = 0; k < S; ++k) {
          const uint32_t d = __vabsdiffu4(a, row[k + dx]);
          acc[k] = __dp4a(d, d, acc[k]);
        }
      }
    }
  }

  write_partial(s, best_key<S>(s, acc, cnt, ox + lane * S, oy + wr), red);
}

// findBestPatch, partial-overlap variant (Algorithm 1 and Sec. 5.4): every
// centre q of the search rectangle is a candidate, also when Psi_q overlaps
// Omega or crosses the image border.  SSD(q) runs over the offsets whose
// target pixel and source pixel are both known and in the image; q is
// admissible only if a known in-image source pixel lies under every unknown
// in-image target pixel (the copy of Sec. 3 reads those).  Same tiles and
// byte-SIMD arithmetic as k_search_plain, with the source's availability in
// the alpha byte of its staged word: the absolute difference's alpha byte is
// then 0xFF exactly when the source pixel is unavailable, and shifting the
// RGB mask 0x00ffffff right by (difference >> 27) = 31 drops that term.  The
// number of admissible candidates goes to ctrl->n_adm (the update phase's
// work count reads and clears it).
template <int R>
__global__ void __launch_bounds__(kSearchThreads) k_search_overlap(ImgState s) {
  constexpr int P = 2 * R + 1;
  constexpr int TW = kSearchTW, TH = kSearchTH, S = kSearchS;
  constexpr int SW = (TW + 2 * R + 3) & ~3;
  constexpr int SH = TH + 2 * R;
  constexpr int NROW = (S + P - 1 + 3) & ~3;
  static_assert(31 * S + NROW <= SW, "row strip must stay inside the tile");
  __shared__ __align__(16) uint32_t src[SH * SW];
  __shared__ uint32_t tgt[P * P];
  __shared__ uint32_t rowmask[P], unkmask[P];
  __shared__ unsigned long long red[32];
  __shared__ int red32[32];

  Ctrl* c = s.ctrl;
  if (!loop_active(c)) return;
  const int px = c->px, py = c->py;
  const int ox = s.cx0 + blockIdx.x * TW, oy = s.cy0 + blockIdx.y * TH;
  const int tid = threadIdx.x;

  stage_target<P, P>(s, px, py, tgt, rowmask, unkmask);
  stage_tile<SH, SW, true>(s, src, ox - R, oy - R);
  __syncthreads();

  const int lane = tid & 31, wr = tid >> 5;
  uint32_t acc[S], bad[S];
#pragma unroll
  for (int k = 0; k < S; ++k) {
    acc[k] = 0;
    bad[k] = 0;
  }

  for (int dy = 0; dy < P; ++dy) {
    const uint32_t m = rowmask[dy], u = unkmask[dy];
    if ((m | u) == 0) continue;
    uint32_t row[NROW];
    const uint4* sp = reinterpret_cast<const uint4*>(&src[(wr + dy) * SW + lane * S]);
#pragma unroll
    for (int i = 0; i < NROW / 4; ++i) {
      const uint4 v = sp[i];
      row[4 * i] = v.x;
      row[4 * i + 1] = v.y;
      row[4 * i + 2] = v.z;
      row[4 * i + 3] = v.w;
    }
    const uint32_t* trow = &tgt[dy * P];
#pragma unroll
    for (int dx = 0; dx < P; ++dx) {
      if (m & (1u << dx)) {
        const uint32_t a = trow[dx];
#pragma unroll
        for (int k = 0; k < S; ++k) {
          const uint32_t d = __vabsdiffu4(a, row[k + dx]);
          const uint32_t e = d & (0x00ffffffu >> (d >> 27));
          acc[k] = __dp4a(e, e, acc[k]);
        }
      } else if (u & (1u << dx)) {
#pragma unroll
        for (int k = 0; k < S; ++k) bad[k] |= row[k + dx] >> 24;
      }
    }
  }

  unsigned long long best = ~0ull;
  int n_adm = 0;
  const int qy = oy + wr;
#pragma unroll
  for (int k = 0; k < S; ++k) {
    const int qx = ox + lane * S + k;
    if (qx <= s.cx1 && qy <= s.cy1 && bad[k] == 0) {
      const unsigned long long key = ((unsigned long long)acc[k] << 32) | (unsigned)(qy * s.W + qx);
      best = key < best ? key : best;
      ++n_adm;
    }
  }
  n_adm = block_sum_int(n_adm, red32);
  if (tid == 0 && n_adm) atomicAdd(&c->n_adm, n_adm);
  write_partial(s, best, red);
}

// Any radius up to kMaxRadius, same tiles and threads.  A target row is taken
// in chunks of eight columns: a chunk without a known pixel is skipped, one
// that is all known runs without tests, another tests a bit per column; its
// source words and target words arrive by five 128-bit shared loads for up to
// 32 evaluations.  (A compacted list of known pixels, built by one thread and
// read with one source load per evaluation, took 76 us a search at 512x384,
// 25x25.)
struct GenGeom {
  int P, TP, SW, SH;
  __host__ __device__ explicit GenGeom(int R)
      : P(2 * R + 1), TP((2 * R + 1 + 7) & ~7), SW((kSearchTW + 2 * R + 15) & ~3), SH(kSearchTH + 2 * R) {}
  __host__ __device__ size_t bytes() const { return (size_t)(SH * SW + P * TP + 3 * P) * sizeof(uint32_t); }
};

__global__ void __launch_bounds__(kSearchThreads) k_search_generic(ImgState s, int n_sum, int gx) {
  extern __shared__ __align__(16) uint32_t dyn[];
  __shared__ unsigned long long red[32];
  const Ctrl* c = s.ctrl;
  if (!loop_active(c)) return;
  if ((int)blockIdx.x < n_sum) {
    // the first CTAs: confidence sums of the update that follows, one warp each
    // (18 us of ordered additions an iteration at 512x384, 25x25, behind the
    // search before)
    __shared__ __align__(16) double vals[kSumVals];
    if (threadIdx.x < 32)
      for (int k = blockIdx.x; k < c->n_spec; k += n_sum) warp_fill_sum(s, vals, k);
    return;
  }
  const int tile = blockIdx.x - n_sum, tx = tile % gx, ty = tile / gx;
  constexpr int S = kSearchS;
  const int R = s.r;
  const GenGeom g(R);
  uint32_t* src = dyn;                  // SH x SW
  uint32_t* tgt = src + g.SH * g.SW;    // P x TP, 0 where unknown
  uint32_t* rmask = tgt + g.P * g.TP;   // P x 3: bits of the known columns
  const int px = c->px, py = c->py;
  const int ox = s.cx0 + tx * kSearchTW, oy = s.cy0 + ty * kSearchTH;
  const int tid = threadIdx.x, lane = tid & 31, wr = tid >> 5;
  int cnt[S];
  load_counts<S>(s, ox + lane * S, oy + wr, cnt);
  for (int dy = wr; dy < g.P; dy += kSearchThreads / 32) {
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int dx = 32 * b + lane, tx = px + dx - R, ty = py + dy - R;
      uint32_t w = 0;
      bool known = false;
      if (dx < g.P && tx >= 0 && tx < s.W && ty >= 0 && ty < s.H) {
        const uint8_t o = s.omega[(size_t)ty * s.W + tx];
        const uint32_t v = s.img[(size_t)ty * s.pitch + tx];
        known = o == 0;
        w = known ? v : 0u;
      }
      const unsigned m = __ballot_sync(0xffffffffu, known);
      if (dx < g.TP) tgt[dy * g.TP + dx] = w;
      if (lane == 0) rmask[3 * dy + b] = m;
    }
  }
  for (int yy = wr; yy < g.SH; yy += kSearchThreads / 32) {
    const int y = oy - R + yy;
#pragma unroll 4
    for (int xx = lane; xx < g.SW; xx += 32) {
      const int x = ox - R + xx;
      src[yy * g.SW + xx] = x >= 0 && x < s.W && y >= 0 && y < s.H ? s.img[(size_t)y * s.pitch + x] : 0u;
    }
  }
  __syncthreads();
  uint32_t acc[S] = {0u, 0u, 0u, 0u};
  for (int dy = 0; dy < g.P; ++dy) {
    const uint32_t* srow = &src[(wr + dy) * g.SW + lane * S];
    for (int ch = 0; ch < g.TP / 8; ++ch) {
      const uint32_t m = (rmask[3 * dy + (ch >> 2)] >> (8 * (ch & 3))) & 0xffu;
      if (m == 0u) continue;
      uint32_t row[12], t[8];
#pragma unroll
      for (int i = 0; i < 3; ++i) reinterpret_cast<uint4*>(row)[i] = reinterpret_cast<const uint4*>(srow + 8 * ch)[i];
#pragma unroll
      for (int i = 0; i < 2; ++i)
        reinterpret_cast<uint4*>(t)[i] = reinterpret_cast<const uint4*>(&tgt[dy * g.TP + 8 * ch])[i];
      if (m == 0xffu) {
#pragma unroll
        for (int dx = 0; dx < 8; ++dx) {
#pragma unroll
          for (int k = 0; k < S; ++k) {
            const uint32_t d = __vabsdiffu4(t[dx], row[k + dx]);
            acc[k] = __dp4a(d, d, acc[k]);
          }
        }
      } else {
#pragma unroll
        for (int dx = 0; dx < 8; ++dx) {
          if (m & (1u << dx)) {
#pragma unroll
            for (int k = 0; k < S; ++k) {
              const uint32_t d = __vabsdiffu4(t[dx], row[k + dx]);
              acc[k] = __dp4a(d, d, acc[k]);
            }
          }
        }
      }
    }
  }
  const unsigned long long best = block_min_u64(best_key<S>(s, acc, cnt, ox + lane * S, oy + wr), red);
  if (tid == 0) s.partial[tile] = best;
}

// The sums alone (an iteration whose search ran elsewhere).
__global__ void __launch_bounds__(32) k_sums(ImgState s) {
  __shared__ __align__(16) double vals[kSumVals];
  if (!loop_active(s.ctrl)) return;
  for (int k = blockIdx.x; k < s.ctrl->n_spec; k += gridDim.x) warp_fill_sum(s, vals, k);
}

// CTAs for the sums: a window's front is 100-200 pixels (k_prio_list's grid).
constexpr int kSumCtas = 304;

cudaError_t launch_sums(const ImgState& s, cudaStream_t st) {
  k_sums<<<kSumCtas, 32, 0, st>>>(s);
  return cudaGetLastError();
}

cudaError_t prepare_search_plain(int r) {
  if (r <= 8) return cudaSuccess;
  return cudaFuncSetAttribute(k_search_generic, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)GenGeom(r).bytes());
}

dim3 search_plain_grid(const ImgState& s) {
  const int cw = s.cx1 - s.cx0 + 1, ch = s.cy1 - s.cy0 + 1;
  if (cw <= 0 || ch <= 0) return dim3(0, 0, 1);
  return dim3((cw + kSearchTW - 1) / kSearchTW, (ch + kSearchTH - 1) / kSearchTH, 1);
}

cudaError_t launch_search_plain(const ImgState& s, cudaStream_t st, bool sums) {
  const dim3 g = search_plain_grid(s);
  if (g.x == 0) return sums && s.r > 8 ? launch_sums(s, st) : cudaSuccess;
  if (s.overlap) {
    switch (s.r) {
      case 1: k_search_overlap<1><<<g, kSearchThreads, 0, st>>>(s); break;
      case 2: k_search_overlap<2><<<g, kSearchThreads, 0, st>>>(s); break;
      case 3: k_search_overlap<3><<<g, kSearchThreads, 0, st>>>(s); break;
      case 4: k_search_overlap<4><<<g, kSearchThreads, 0, st>>>(s); break;
      case 5: k_search_overlap<5><<<g, kSearchThreads, 0, st>>>(s); break;
      case 6: k_search_overlap<6><<<g, kSearchThreads, 0, st>>>(s); break;
      case 7: k_search_overlap<7><<<g, kSearchThreads, 0, st>>>(s); break;
      case 8: k_search_overlap<8><<<g, kSearchThreads, 0, st>>>(s); break;
      default: return cudaErrorInvalidValue;  // the variant is built for r <= 8
    }
    return cudaGetLastError();
  }
  switch (s.r) {
    case 1: k_search_plain<1><<<g, kSearchThreads, 0, st>>>(s); break;
    case 2: k_search_plain<2><<<g, kSearchThreads, 0, st>>>(s); break;
    case 3: k_search_plain<3><<<g, kSearchThreads, 0, st>>>(s); break;
    case 4: k_search_plain<4><<<g, kSearchThreads, 0, st>>>(s); break;
    case 5: k_search_plain<5><<<g, kSearchThreads, 0, st>>>(s); break;
    case 6: k_search_plain<6><<<g, kSearchThreads, 0, st>>>(s); break;
    case 7: k_search_plain<7><<<g, kSearchThreads, 0, st>>>(s); break;
    case 8: k_search_plain<8><<<g, kSearchThreads, 0, st>>>(s); break;
    default: {
      const int n_sum = sums ? kSumCtas : 0;
      k_search_generic<<<n_sum + (int)(g.x * g.y), kSearchThreads, GenGeom(s.r).bytes(), st>>>(s, n_sum, (int)g.x);
    }
  }
  return cudaGetLastError();
}

}  // namespace inp
