// Persistent fill-loop engine: the whole iterative stage of Sec. 4.2 in one
// cooperative kernel launch.
//
// CTAs form teams; a team runs the fill loop of one image at a time (a list
// of images per team gives the batched form).  One iteration of a team:
//   1. every member CTA searches its share of the candidate centres
//      (findBestPatch, Eq. 3-4).  Resident mode (the leader does not search
//      and the tiles fit): the CTA owns a contiguous range of units of 32
//      candidate rows x 16 columns, or x 4 where it has few, keeps their
//      source window in shared memory for the whole removal and only patches
//      the pixels the previous iteration filled; streaming mode (small teams,
//      whose leader searches too): batches of 32 rows x 64 or 128 columns
//      whose source window and validity counts arrive by TMA, double-buffered.
//      Each lane owns the candidates of one row; the CTA reduces them to one
//      (SSD << 32 | idx) key.  Tensor-core form: search_tc_engine.cuh;
//   2. each member writes its key, tagged with the round, to its slot; the
//      leader polls the slots, runs the copy/update phase and the selection
//      of the next target (update_fast.cuh) and publishes the next epoch;
//   3. the others wait for that epoch (bounded wait, no trap) and go on.
// No host round trip and no kernel boundary per iteration.
#pragma once
#include <cstddef>
#include <type_traits>
#include <cuda.h>

#include "inpaint_engine.h"
#include "ptx.cuh"
#include "search_tc_engine.cuh"
#include "ssd_rows.cuh"
#include "update_fast.cuh"

namespace inp {

// The CTA's dynamic shared memory.  Every function names it itself instead of
// taking a pointer to it, so that the compiler sees shared addresses: through
// a pointer kept in memory each access of the leader's phases was a generic
// load or store with 64-bit address arithmetic.
__device__ __forceinline__ uint8_t* eng_smem() {
  extern __shared__ __align__(128) uint8_t eng_smem_raw[];
  return eng_smem_raw;
}
__device__ __forceinline__ const uint32_t* smem_words(int offset) {
  return reinterpret_cast<const uint32_t*>(eng_smem() + offset);
}

// ---------------------------------------------------------------- search batch

// A search batch is 32 candidate rows x BWC candidate columns.  Lane l of
// warp w owns the NCL adjacent candidates (row l, columns w*NCL ...): every
// lane of a warp uses the same target row at the same time (the row-mask
// branch stays warp-uniform), and the lanes' 128-bit loads of their source
// row strips fall on 32 consecutive tile rows, conflict-free.
template <int R, int SRW>
struct EngGeom {
  static constexpr int P = 2 * R + 1;
  static constexpr int NCL = 4 * SRW;              // candidates per lane (4 or 8)
  static constexpr int BWC = eng_batch_cols(SRW);  // candidate columns per batch (64 or 128)
  static constexpr int B = kEngBatchRows;          // candidate rows per batch (one per lane)
  static constexpr int BW = eng_tile_width(R, SRW);  // staged width (words)
  static constexpr int BH = B + 2 * R;             // staged rows
  static constexpr int SLOT_BYTES = ((BW * BH * 4 + 127) / 128) * 128;
  static constexpr int CW = eng_count_width(SRW);  // count tile width (words), CW / 4 odd
  static constexpr int CNT_BYTES = ((CW * B * 4 + 127) / 128) * 128;
  static constexpr int COFF = R & 3;  // first candidate column within the count tile
  static constexpr int NS = (NCL + P - 1 + 3) & ~3;  // strip words per lane
  static constexpr int TP = (P + 3) & ~3;            // padded target row (words)
  static constexpr unsigned FULL = (1u << P) - 1u;
  static_assert((kEngWarps - 1) * NCL + NS <= BW, "row strip must stay inside the tile");
  static_assert(kEngWarps * NCL + 4 <= CW, "count chunk must stay inside the tile row");
  static_assert(((CW / 4) & 1) == 1, "count rows must start in different bank quadruples");
};

template <int N>
__device__ __forceinline__ void lds_words(uint32_t (&d)[N], const uint32_t* p) {
  const uint4* q = reinterpret_cast<const uint4*>(p);
#pragma unroll
  for (int i = 0; i < N / 4; ++i) {
    const uint4 v = q[i];
    d[4 * i] = v.x;
    d[4 * i + 1] = v.y;
    d[4 * i + 2] = v.z;
    d[4 * i + 3] = v.w;
  }
}

// Row descriptor of a target row (computed once per target): which of its
// P pixels are known.  A row next to the fill front is usually known on one
// contiguous run that touches one end of the row, so the common shapes take
// one jump into a straight run of code instead of a test per column:
//   kRowSkip   nothing known;
//   kRowFrom   known on [s, P) (s = 0: the whole row), s in the low bits;
//   kRowUpTo   known on [0, e), e in the low bits;
//   kRowMask   anything else, the bit mask of known columns in the low bits.
constexpr uint32_t kRowSkip = 0u, kRowFrom = 1u << 30, kRowUpTo = 2u << 30, kRowMask = 3u << 30;

__device__ __forceinline__ uint32_t row_desc(uint32_t m, int P) {
  const uint32_t full = (1u << P) - 1u;
  if (m == 0) return kRowSkip;
  const int s = __ffs(m) - 1;           // lowest known column
  const int e = 32 - __clz(m);          // one past the highest known column
  if (m == ((full >> s) << s)) return kRowFrom | (uint32_t)s;
  if (s == 0 && m == (1u << e) - 1u) return kRowUpTo | (uint32_t)e;
  return kRowMask | m;
}

// SSD of this lane's NCL candidates against the staged target (Eq. 4): for
// every known target pixel one byte-SIMD absolute difference and one 4-way
// byte dot product per candidate (|a-b| per channel, squares summed; alpha
// is 0 on both sides).  `strip` points at the lane's row strip in its tile
// (row pitch `pitch` words), over the target rows [r0, r1); `rowd` holds one
// row descriptor per target row:
// per row one indexed jump into the sequences of ssd_rows.cuh (a run of known
// columns [s, P) enters an ascending sequence at s, a run [0, e) a descending
// one at e - 1); other row shapes test a bit per column.
template <int R, int NCL>
__device__ __forceinline__ void unit_ssd(const uint32_t* __restrict__ strip, int pitch,
                                         const uint32_t* __restrict__ tgt, const uint32_t* __restrict__ rowd,
                                         int r0, int r1, uint32_t (&acc)[NCL]) {
  constexpr int P = 2 * R + 1, NS = (NCL + P - 1 + 3) & ~3, TP = (P + 3) & ~3;
#pragma unroll
  for (int k = 0; k < NCL; ++k) acc[k] = 0;
#pragma unroll 1
  for (int dy = r0; dy < r1; ++dy) {
    const uint32_t desc = rowd[dy];
    if (desc == kRowSkip) continue;
    uint32_t r[NS], t[TP];
    lds_words(r, strip + dy * pitch);
    lds_words(t, tgt + dy * TP);
    const uint32_t kind = desc & (3u << 30);
    if (kind != kRowMask) {
      const uint32_t arg = desc & 0xffffu;
      // entry of the jump table: [0, P) ascending from column s, [P, 2P)
      // descending from column e - 1; clamped so that it stays in the table
      const uint32_t idx = min(kind == kRowFrom ? arg : (uint32_t)P + arg - 1u, (uint32_t)(2 * P - 1));
#define INP_ROW(N, PP) \
  if constexpr (NCL == N && P == PP) INP_SSD_ROW##N##_P##PP(acc, r, t, idx);
#define INP_ROWS(PP) INP_ROW(4, PP) INP_ROW(8, PP) INP_ROW(16, PP)
      INP_ROWS(3) INP_ROWS(5) INP_ROWS(7) INP_ROWS(9) INP_ROWS(11) INP_ROWS(13) INP_ROWS(15) INP_ROWS(17)
#undef INP_ROWS
#undef INP_ROW
    } else {
#pragma unroll
      for (int dx = 0; dx < P; ++dx) {
        if (desc & (1u << dx)) {
#pragma unroll
          for (int k = 0; k < NCL; ++k) {
            const uint32_t d = __vabsdiffu4(t[dx], r[k + dx]);
            acc[k] = __dp4a(d, d, acc[k]);
          }
        }
      }
    }
  }
}

// The partial-overlap form (Algorithm 1, Sec. 5.4) of the same SSD for four
// candidates: the sum runs over the known target pixels whose source pixel is
// available, and a candidate with an unavailable source pixel under a pixel to
// fill is inadmissible (kOvlBad added; the true sum is below it).  The tile's
// words carry the availability in the alpha byte (0xff: unknown or outside the
// image, RGB 0 then).
// Where no lane that has a candidate meets an unavailable word, and where each
// lane's words of the row are all available or all not (rows beyond the image,
// a lane inside the object), a row takes the sequences above, and a lane
// without any takes back what they summed for it (rowsq).  Only the rows at the
// object's sides and the image's left and right border need a mask per word
// (three instructions an evaluation and the masks: 1,200 cycles a row of four
// warps a scheduler at 9x9, against 620; with masks in every row that meets an
// unavailable word a round at 1024x550 took 16.5 us, now 14.2).  Unknown target pixels cost nothing:
// a bit per word tells which candidates have an unavailable source pixel under
// one.
// `flags`: per target pixel 1 known, 2 unknown, 0 outside the image; `rowsq`:
// per target row, the sum over its known pixels of the squared words (alpha
// 0xff).
constexpr uint32_t kOvlBad = 1u << 27;  // (at most P + 1 partial sums of a unit: no overflow)

template <int R>
__device__ __forceinline__ void unit_ssd_overlap(const uint32_t* __restrict__ strip, int pitch,
                                                 const uint32_t* __restrict__ tgt, const uint32_t* __restrict__ rowd,
                                                 const uint8_t* __restrict__ flags, const int* __restrict__ rowsq,
                                                 int r0, int r1, bool live,
                                                 uint32_t (&acc)[4]) {
  constexpr int P = 2 * R + 1, NS = (4 + P - 1 + 3) & ~3, TP = (P + 3) & ~3;
  uint32_t bad[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) acc[k] = bad[k] = 0u;
#pragma unroll 1
  for (int dy = r0; dy < r1; ++dy) {
    uint32_t r[NS], t[TP];
    lds_words(r, strip + dy * pitch);
    uint32_t any = 0u, all = ~0u;
#pragma unroll
    for (int i = 0; i < P + 3; ++i) {
      any |= r[i];
      all &= r[i];
    }
    const uint32_t desc = rowd[dy];
    const bool some = live && (any >> 31), none = all >> 31;
    uint32_t unk = 0u;  // the row's pixels to fill
    bool mixed = false;
    if (__any_sync(0xffffffffu, some)) {
      const int lane = threadIdx.x & 31;
      unk = __ballot_sync(0xffffffffu, flags[dy * P + min(lane, P - 1)] == 2 && lane < P);
      mixed = __any_sync(0xffffffffu, some && !none);
    }
    if (!mixed) {
      if (none && unk) bad[0] = bad[1] = bad[2] = bad[3] = 1u;
      if (desc == kRowSkip) continue;
      lds_words(t, tgt + dy * TP);
      const uint32_t kind = desc & (3u << 30);
      if (kind != kRowMask) {
        const uint32_t arg = desc & 0xffffu;
        const uint32_t idx = min(kind == kRowFrom ? arg : (uint32_t)P + arg - 1u, (uint32_t)(2 * P - 1));
#define INP_ROW(PP) \
  if constexpr (P == PP) INP_SSD_ROW4_P##PP(acc, r, t, idx);
        INP_ROW(3) INP_ROW(5) INP_ROW(7) INP_ROW(9) INP_ROW(11) INP_ROW(13) INP_ROW(15) INP_ROW(17)
#undef INP_ROW
      } else {
#pragma unroll
        for (int dx = 0; dx < P; ++dx) {
          if (desc & (1u << dx)) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t d = __vabsdiffu4(t[dx], r[k + dx]);
              acc[k] = __dp4a(d, d, acc[k]);
            }
          }
        }
      }
      if (none) {
        const uint32_t sq = (uint32_t)rowsq[dy];
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] -= sq;
      }
    } else {
      // av: one bit per unavailable word; m: the RGB mask of an available one
      uint32_t m[NS], av = 0u;
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        m[i] = (int)r[i] < 0 ? 0u : 0x00ffffffu;
        if (i < P + 3) av |= (r[i] >> 31) << i;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) bad[k] |= (av >> k) & unk;
      if (desc == kRowSkip) continue;
      lds_words(t, tgt + dy * TP);
      const uint32_t kind = desc & (3u << 30);
      if (kind != kRowMask) {
        const uint32_t arg = desc & 0xffffu;
        const uint32_t idx = min(kind == kRowFrom ? arg : (uint32_t)P + arg - 1u, (uint32_t)(2 * P - 1));
#define INP_ROW(PP) \
  if constexpr (P == PP) INP_SSD_ROWM_P##PP(acc, r, m, t, idx);
        INP_ROW(3) INP_ROW(5) INP_ROW(7) INP_ROW(9) INP_ROW(11) INP_ROW(13) INP_ROW(15) INP_ROW(17)
#undef INP_ROW
      } else {
#pragma unroll
        for (int dx = 0; dx < P; ++dx) {
          if (desc & (1u << dx)) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t d = __vabsdiffu4(t[dx], r[k + dx]) & m[k + dx];
              acc[k] = __dp4a(d, d, acc[k]);
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) acc[k] += bad[k] ? kOvlBad : 0u;
}

// The compute of a streaming search round, outside the engine body so that its
// registers hold only the row strips, the target row and the accumulators
// (the engine body keeps the leader's state live across the search).  These
// functions take byte offsets into the CTA's shared memory, not pointers: a
// pointer argument is a generic address, whose every access is a generic
// load with 64-bit address arithmetic.

// Smallest key (SSD << 32 | idx) of this lane's NCL candidates in one unit:
// `bits` marks the valid ones, idx0 is the linear index of the first.
template <int R, int NCL>
__device__ __noinline__ unsigned long long unit_best(int strip, int pitch, int tgt, uint32_t bits, unsigned idx0) {
  constexpr int P = 2 * R + 1, TP = (P + 3) & ~3;
  uint32_t acc[NCL];
  unit_ssd<R, NCL>(smem_words(strip), pitch, smem_words(tgt), smem_words(tgt) + P * TP, 0, P, acc);
  unsigned long long best = ~0ull;
#pragma unroll
  for (int k = 0; k < NCL; ++k) {
    const unsigned long long key = ((unsigned long long)acc[k] << 32) | (idx0 + (unsigned)k);
    if ((bits & (1u << k)) && key < best) best = key;
  }
  return best;
}

// ---------------------------------------------------------------- resident search

// Resident mode: the candidate rectangle is cut into units of 32 candidate
// rows (one per lane) x KC candidate columns (one lane's candidates); the
// units, in band-major order, are split into contiguous ranges of equal
// size, one per searching CTA.  A CTA keeps the source window of its units
// in shared memory for the whole removal (one tile per 32-row band its range
// touches) and after each iteration's copy only patches the pixels it filled
// and the validity of the candidates near them.  KC is 16 when that gives a
// CTA 12 units or more (most of its warps one), else 4, with the target rows of the
// CTA's units dealt to its warps in equal shares and the partial SSDs summed
// in shared memory: a small image has few units per CTA (512x384 over 151
// CTAs: 3 of 16 columns, 10 of 4), and a warp alone on its scheduler takes
// about 500 cycles a row, most of it latency.  Only CTAs that do not lead
// search this way (a leader that searches too has a small team and streams).
constexpr int kResRows = 32;   // candidate rows per unit (one per lane)
constexpr int kResMaxSeg = 2;  // bands one CTA's tiles span at most: it has no more units than a band

struct ResSeg {
  int band;      // 32-row band of the search rectangle
  int c_lo;      // first unit column of the band in this CTA's range
  int pitch;     // tile row pitch (words), pitch / 4 odd
  int off;       // byte offset of the tile in the CTA's tile area
};

struct ResPlan {
  int u0, u1;        // this CTA's units [u0, u1), band-major
  int ncu;           // unit columns per band
  int nseg;
  int bits_off;      // byte offset of the validity bits (uint16 per unit and lane)
  ResSeg seg[kResMaxSeg];
};

// Plan of rank `rank`'s units: the tile of each band its range touches.  A range
// has at most ncu units (the condition of the resident mode), so two bands.
template <int R>
__device__ inline void res_plan(ResPlan& pl, int kc, int ncu, int nbands, int rank, int ns) {
  const long long U = (long long)ncu * nbands;
  pl.u0 = (int)(U * rank / ns);
  pl.u1 = (int)(U * (rank + 1) / ns);
  pl.ncu = ncu;
  pl.nseg = 0;
  if (pl.u1 <= pl.u0) {
    pl.bits_off = 0;
    return;
  }
  const int b_lo = pl.u0 / ncu, b_hi = (pl.u1 - 1) / ncu;
  long long off = 0;
  for (int b = b_lo; b <= b_hi; ++b) {
    const int c_lo = b == b_lo ? pl.u0 % ncu : 0;
    const int c_hi = b == b_hi ? (pl.u1 - 1) % ncu + 1 : ncu;
    ResSeg& sg = pl.seg[pl.nseg++];
    sg.band = b;
    sg.c_lo = c_lo;
    sg.pitch = width_odd16((c_hi - c_lo) * kc + 2 * R + 4);  // (+ the strips' rounding)
    sg.off = (int)off;
    off += (((long long)sg.pitch * (kResRows + 2 * R) * 4) + 127) / 128 * 128;
  }
  pl.bits_off = (int)off;
}

// Shared memory that m units of kc columns need at most: two tiles (a range may
// straddle a band boundary), the validity bits and, for kc < 16, the partial
// SSDs.
template <int R>
__host__ __device__ inline int res_need(int kc, int m) {
  return (kResRows + 2 * R) * 4 * (m * kc + 2 * (2 * R + 12)) + 640 + m * 64 + (kc < 16 ? m * kc * 128 : 0);
}

// Partial-overlap search: unit columns and the number of searchers among
// ns_max; returns the most units of one share (0: no candidate).
template <int R>
__host__ __device__ inline int overlap_units(const ImgState& s, int ns_max, int* ncu, int* ns) {
  const int xb = R + ((s.cx0 - R) & ~3);
  const int nbands = s.cy1 >= s.cy0 ? (s.cy1 - s.cy0 + kResRows) / kResRows : 0;
  *ncu = s.cx1 >= s.cx0 ? (s.cx1 - xb + 4) / 4 : 0;
  *ns = ns_max < *ncu * nbands ? ns_max : *ncu * nbands;
  return *ns > 0 ? (*ncu * nbands + *ns - 1) / *ns : 0;
}

// ---------------------------------------------------------------- kernel

// The state of a CTA's tensor-core search that outlives a round: source rows
// through the ring and tiles through the accumulator buffers so far (their
// barriers' phases).
struct TcRun {
  TcArea a;
  uint32_t rows, tiles;
  int k0, n;    // this CTA's turns that are tiles: k0 .. k0 + n - 1 (tc_tile_of)
  int tx0, y0;  // the first one's tile column and candidate row
};

struct EngSmemTail {
  EngBars bars;      // mbarriers (streaming stages, tensor-core ring), tensor-memory base
  ImgState img;      // the image's state block (a leader that does not search reads it here)
  unsigned long long red64[32];
  int red32[32];
  int stop;
  int px, py;
  int a2row[17];  // tensor-core search: per target row, sum of the known pixels' squared shifted values
                  // (partial-overlap search: of their squared values with alpha 0xff)
  int tc_pref;    // tensor-core search: slots the producer prefetched for the next round
  TcRun tc_run;   // a searching leader's tensor-core search between its rounds
  int lim, status, err;  // leader: iteration limit, status and error word (the stop decision)
  uint8_t known[17 * 17];     // round's target: 1 known, 2 (partial-overlap search) unknown in the image, else 0
  ResPlan plan;               // resident mode: this CTA's units and tiles
};

static_assert(offsetof(EngSmemTail, bars) == 0, "the kernel initialises the barriers at the start of shared memory");

constexpr int kTgtOff = (int)((sizeof(EngSmemTail) + 15) & ~size_t(15));
constexpr int kTgtWords = 17 * 20 + 17 + 3;  // padded target rows + row masks (R <= 8)
constexpr size_t kHeadBytes = ((kTgtOff + kTgtWords * 4 + 127) / 128) * 128;

// Shared memory of an engine CTA: head | (the leader only) update state | its
// search's state: resident tiles, validity bits and partial SSDs; or the
// tensor-core form's A strips, target table and ring; or two count tiles and
// two tile slots of the streaming search, used as a double buffer.  The kernel
// is launched with all the shared memory an SM offers.
template <int R>
__host__ __device__ constexpr size_t upd_smem_bytes() {
  return ((sizeof(UpdSmem<R>) + 127) / 128) * 128;
}

// The least shared memory an engine CTA needs: a searching leader with two
// slots (the streaming double buffer).
template <int R, int SRW>
__host__ __device__ constexpr size_t eng_smem_bytes() {
  using G = EngGeom<R, SRW>;
  return kHeadBytes + ((upd_smem_bytes<R>() + 127) / 128) * 128 + (size_t)2 * G::CNT_BYTES +
         (size_t)2 * G::SLOT_BYTES + 128;
}

static_assert(eng_smem_bytes<8, 2>() <= 227 * 1024, "engine CTA must fit in shared memory");
static_assert(eng_smem_bytes<7, 2>() <= 227 * 1024, "engine CTA must fit in shared memory");

// Team publication word: epoch (bits 0-31), next target px (from bit 32, as
// many bits as a column of the image needs), py (the bits above) and the stop
// flag (63).  One acquire load gives a waiting CTA everything it needs to start
// the next search round.  px and py take at most 31 bits together: W H <= 2^30,
// and the bits of two numbers are at most two more than those of their
// product's logarithm.
__device__ inline int pub_bits(int W) { return 32 - __clz(W - 1); }
__device__ inline unsigned long long pub_pack(unsigned epoch, int px, int py, bool stop, int bits) {
  const unsigned hi = (unsigned)px | (unsigned)py << bits | (stop ? 1u << 31 : 0u);
  return (unsigned long long)hi << 32 | epoch;
}
__device__ inline void pub_unpack(unsigned long long v, int bits, int& px, int& py, int& stop) {
  const unsigned hi = (unsigned)(v >> 32);
  px = (int)(hi & ((1u << bits) - 1u));
  py = (int)((hi & 0x7fffffffu) >> bits);
  stop = (int)(hi >> 31);
}

__device__ inline unsigned long long ld_acquire64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ inline void st_release64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ inline void st_relaxed64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ inline unsigned long long ld_relaxed64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// The leader's publishing thread: the last one, which is also update_work's
// fence thread, so the fence it issues after the copy makes its later
// publication of the next round a release.
constexpr int kPubThread = kEngThreads - 1;

// Bounded wait (thread 0) for a publication with an epoch other than `epoch`;
// returns it, or a stop word after setting *err on timeout.
__device__ inline unsigned long long wait_pub(TeamCtl* tc, unsigned epoch, int* err,
                                              unsigned long long limit) {
  unsigned long long v = ld_acquire64(&tc->pub);
  if ((unsigned)v != epoch) return v;
  const unsigned long long t0 = globaltimer();
  while (true) {
    v = ld_acquire64(&tc->pub);
    if ((unsigned)v != epoch) return v;
    if (globaltimer() - t0 > limit) {
      atomicExch(err, INPAINT_ERR_TIMEOUT);
      return pub_pack(epoch + 1u, 0, 0, true, 0);
    }
  }
}

// A searcher's best key of a round travels to the leader tagged with the
// round: (SSD << 38) | (idx << 8) | tag, tag = epoch mod 128 (SSD < 2^26 for
// radius <= 8, idx < 2^30), so the leader polls the keys themselves and no
// separate arrival counter is needed.  Keys of one round carry the same tag,
// so the tagged values order like (SSD, idx).  Slots are set to all ones
// (tag 0xff, never a round's) before every launch.
__device__ inline unsigned long long key_tag(unsigned long long key, unsigned epoch) {
  if (key == ~0ull) return ~0ull & ~0xffull | (epoch & 0x7fu);
  return ((key >> 32) << 38) | ((key & 0x3fffffffull) << 8) | (epoch & 0x7fu);
}

__device__ inline unsigned long long key_untag(unsigned long long t) {
  const unsigned long long ssd = t >> 38, idx = (t >> 8) & 0x3fffffffull;
  if (ssd == 0x3ffffffull && idx == 0x3fffffffull) return ~0ull;
  return (ssd << 32) | idx;
}

// The best key of the round over the tagged slots [0, n) (one warp), each
// polled, bounded, until it carries the round's tag; *late when one did not
// arrive in time.  A key is a message of its own (the leader reads nothing
// else the searchers write), so relaxed loads suffice; a lane polls up to
// five slots at a time (160 slots: every CTA of the chip in one pass).
__device__ inline unsigned long long gather_keys(const unsigned long long* slots, int n, unsigned epoch, int* err,
                                                 unsigned long long limit, bool* late_out) {
  constexpr int U = 5;
  const int lane = threadIdx.x & 31;
  const unsigned tag = epoch & 0x7fu;
  unsigned long long best = ~0ull;
  bool late = false;
  const unsigned long long t0 = globaltimer();
#pragma unroll 1
  for (int b = 0; b < n && !late; b += 32 * U) {
    unsigned pending = 0u;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (b + lane + 32 * u < n) pending |= 1u << u;
#pragma unroll 1
    while (pending) {
      unsigned long long v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = (pending >> u) & 1u ? ld_relaxed64(&slots[b + lane + 32 * u]) : 0ull;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (((pending >> u) & 1u) && (v[u] & 0xffu) == tag) {
          best = v[u] < best ? v[u] : best;  // one tag: tagged values order like their keys
          pending &= ~(1u << u);
        }
      if (pending && globaltimer() - t0 > limit) {
        late = true;
        break;
      }
    }
  }
  late = __any_sync(0xffffffffu, late);
  best = warp_min_u64(best);
  if (late && lane == 0) atomicExch(err, INPAINT_ERR_TIMEOUT);
  *late_out = late;
  return best == ~0ull ? best : key_untag(best);
}

// Partial-overlap search: the number of admissible candidates of round
// `epoch`, from the searchers' tagged counts (epoch << 32 | count) of that
// round's parity, each polled, bounded; one warp.  Read a round later, beside
// the next search, so that the counts need no fence before the keys.
__device__ inline int gather_counts(const unsigned long long* slots, int n, unsigned epoch, int* err,
                                    unsigned long long limit) {
  constexpr int U = 5;
  const int lane = threadIdx.x & 31;
  const unsigned long long t0 = globaltimer();
  int sum = 0;
#pragma unroll 1
  for (int b = lane; b < n; b += 32 * U) {
    unsigned long long v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = b + 32 * u < n ? ld_relaxed64(&slots[b + 32 * u]) : (unsigned long long)epoch << 32;
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll 1
      while ((unsigned)(v[u] >> 32) != epoch) {
        if (globaltimer() - t0 > limit) {
          atomicExch(err, INPAINT_ERR_TIMEOUT);
          break;
        }
        v[u] = ld_relaxed64(&slots[b + 32 * u]);
      }
      sum += (int)(unsigned)v[u];
    }
  }
  __syncwarp();
  return __reduce_add_sync(0xffffffffu, sum);
}

__device__ inline bool ctrl_active(const Ctrl* c) {
  return __ldcg(&c->status) == 0 && __ldcg(&c->remaining) > 0 &&
         __ldcg(&c->iter) < __ldcg(&c->iter_limit);
}

// Roles of a team on one image: CTAs [0, ns) search; the last CTA (the
// leader) runs the speculative phase of each iteration while they search,
// waits for them, applies the update and publishes the next round; any other
// CTA idles until the image is done.  A team of one CTA does all of it in
// sequence.
// Per-image part of the engine: the fill loop of image j for this CTA's
// team (roles below).  Called by k_engine (engine_multi.cu) through
// run_image_r<R>_s<SRW>, once per image of the team's list.
template <int R, int SRW, bool kLeadOnly = false>
__device__ __forceinline__ void run_image(const EngineArgs& ea, int j, EngCtx& x);

// The k-th tile of searching CTA `rank` of ns, or -1.  Tiles go round-robin;
// when the leader (the last of them) searches too, its first turn is its
// speculative phase, which takes about as long as a tile.
__device__ __forceinline__ int tc_tile_of(int k, int rank, int ns, int ntiles, bool lead_searches) {
  const int v = rank + k * ns, t = lead_searches && v >= ns - 1 ? v - 1 : v;
  return (lead_searches && v == ns - 1) || t >= ntiles ? -1 : t;
}

// Where the tensor-core search keeps its state, from byte `off` of the CTA's
// shared memory.  A ring with another slot count than the last image's starts
// its phases over (every slot of an earlier image was consumed, so no barrier
// has a pending phase).  Whole block.
template <int R>
__device__ __forceinline__ void tc_setup(TcRun& t, EngCtx& x, EngBars& bars, const ImgState& s, const TcTiles& tt,
                                         int k0, int ns, bool lead_searches, int off, int nb, int slot) {
  using GT = TcEngGeom<R>;
  uint8_t* area = eng_smem() + off;
  t.a.a = area;
  t.a.tpad = reinterpret_cast<uint16_t*>(area + GT::A_BYTES);
  t.a.ring = area + GT::A_BYTES + GT::TPAD_BYTES;
  t.a.nb = nb;
  t.a.slot = slot;
  t.rows = x.tc_rows;
  t.tiles = x.tc_tiles;
  t.k0 = k0;
  t.n = 0;
  while (tc_tile_of(k0 + t.n, x.rank, ns, tt.ntx * tt.nty, lead_searches) >= 0) ++t.n;
  const int t0 = max(0, tc_tile_of(k0, x.rank, ns, tt.ntx * tt.nty, lead_searches)), ty = t0 / tt.ntx;
  t.tx0 = t0 - ty * tt.ntx;
  t.y0 = s.cy0 + kTcRows * ty;
  if (x.tc_nb != nb) {
    if (x.tc_nb != 0 && threadIdx.x == 0) {
      for (int i = 0; i < kTcRing; ++i) {
        mbar_inval(&bars.tc_full[i]);
        mbar_inval(&bars.tc_empty[i]);
        mbar_init(&bars.tc_full[i], 1);
        mbar_init(&bars.tc_empty[i], 2);
      }
    }
    fence_mbar_init();
    t.rows = 0;
  }
  // the padded target table's columns outside the patch stay zero
  for (int e = threadIdx.x; e < 4 * GT::P * GT::TW; e += kEngThreads) t.a.tpad[e] = 0;
  __syncthreads();
  x.tc_nb = nb;
}

// One round of a CTA's tensor-core search for target (px, py): its tiles;
// `pref` ring slots of the first one are already requested.
// Returns the thread's best key; *bad (of this thread) when a bounded wait
// gave up.  Whole block.
template <int R>
__device__ __forceinline__ unsigned long long tc_round(const ImgState& s, const TcTiles& tt, TcRun& tr,
                                                       EngSmemTail& tl, uint32_t tmem, int px, int py, bool first,
                                                       int pref, int rank, int ns, bool lead_searches,
                                                       unsigned long long limit, int* bad_out) {
  using GT = TcEngGeom<R>;
  constexpr int P = GT::P, NSL = GT::NSL;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int npre = min(tr.a.nb, NSL), n = tr.n;
  auto tile = [&](int k, int& tx, int& y0) {
    if (k == 0) {
      tx = tr.tx0;
      y0 = tr.y0;
      return ((y0 - s.cy0) / kTcRows) * tt.ntx + tx;
    }
    const int t = tc_tile_of(tr.k0 + k, rank, ns, tt.ntx * tt.nty, lead_searches), ty = t / tt.ntx;
    tx = t - ty * tt.ntx;
    y0 = s.cy0 + kTcRows * ty;
    return t;
  };
  int bad = 0, tx, y0;
  // the producer starts the first tile's rows at once, unless it
  // prefetched them while the leader was updating
  if (n > 0 && pref == 0 && warp == kEngWarps - 1 && lane == 0) {
    tile(0, tx, y0);
    if (!tc_produce<R>(s, tr.a, tl.bars, tx, y0, tr.rows, 0, npre, limit)) bad = 1;
  }
  // the last tile's validity bits, requested before a warp's role: by the
  // producer's and the issuers' warps while the others write A (13 warps need
  // as many passes for it as 15), by those when they are done
  const int ng = (tt.N & 31) ? 2 : 4;  // column groups of that tile's read-back
  uint2 bits_last = make_uint2(0u, 0u);
  auto bits_of = [&](int t) { return s.vbits + (size_t)t * kTcRows * (tt.N / 4); };
  auto load_last = [&]() {
    int tx_, y0_;
    if (n > 0 && warp < 4 * ng) bits_last = tc_bits_load(bits_of(tile(n - 1, tx_, y0_)), tt.N, ng);
  };
  tc_stage_target<R>(s, tr.a.tpad, tl.a2row, px, py);
  __syncthreads();
  if (warp >= kEngWarps - 3) load_last();
  else tc_build_a<R>(tr.a.a, tr.a.tpad, first, 32 * (kEngWarps - 3));
  __syncthreads();
  if (warp < kEngWarps - 3) load_last();
  int a2 = 0;
#pragma unroll
  for (int dy = 0; dy < P; ++dy) a2 += tl.a2row[dy];
  unsigned long long best = ~0ull;
  if (warp == kEngWarps - 1) {
    for (int k = 0; k < n && !bad; ++k) {
      tile(k, tx, y0);
      if (lane == 0 && !tc_produce<R>(s, tr.a, tl.bars, tx, y0, tr.rows + (uint32_t)(k * NSL), k == 0 ? npre : 0, NSL, limit))
        bad = 1;
    }
    __syncwarp();
  } else if (warp == kEngWarps - 2 || warp == kEngWarps - 3) {
    for (int k = 0; k < n && !bad; ++k) {
      const uint32_t c = tr.tiles + (uint32_t)k, b = c & 1u, g0 = tr.rows + (uint32_t)(k * NSL);
      // the buffer's previous tile has been read
      if (c >= 2u && !__all_sync(0xffffffffu, mbar_wait(&tl.bars.tc_free[b], ((c >> 1) - 1u) & 1u, limit))) bad = 1;
      tc_fence_after();
      if (warp == kEngWarps - 2 ? !tc_issue<R, 0>(tr.a, tl.bars, tt.N, tmem + 256u * b, &tl.bars.tc_done[b], g0, limit)
                                : !tc_issue<R, 1>(tr.a, tl.bars, tt.N, tmem + 256u * b, &tl.bars.tc_done[b], g0, limit))
        bad = 1;
    }
    // the one warp that waits for the last tile's MMAs (the others sleep at
    // the block barrier: spinning warps would take issue slots from the
    // issuers)
    if (warp == kEngWarps - 2 && n > 0) {
      const uint32_t c = tr.tiles + (uint32_t)(n - 1);
      if (!mbar_wait(&tl.bars.tc_done[c & 1u], (c >> 1) & 1u, limit)) bad = 1;
    }
  } else if (warp < kTcReaders) {
    for (int k = 0; k + 1 < n && !bad; ++k) {
      const int t = tile(k, tx, y0);
      const uint32_t c = tr.tiles + (uint32_t)k, b = c & 1u;
      const uint2 bits = tc_bits_load(bits_of(t), tt.N, kTcReaders / 4);
      if (!__all_sync(0xffffffffu, mbar_wait(&tl.bars.tc_done[b], (c >> 1) & 1u, limit))) {
        bad = 1;
        break;
      }
      tc_fence_after();
      best = tc_epilogue<R>(s, tmem + 256u * b, tt, kTcReaders / 4, a2, bits, y0, tx, best);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tl.bars.tc_free[b]);
    }
  }
  tc_fence_before();
  if (__syncthreads_or(bad)) {
    *bad_out = 1;
    return ~0ull;
  }
  tc_fence_after();
  if (n > 0) {
    const uint32_t b = (tr.tiles + (uint32_t)(n - 1)) & 1u;
    tile(n - 1, tx, y0);
    if (warp < 4 * ng) best = tc_epilogue<R>(s, tmem + 256u * b, tt, ng, a2, bits_last, y0, tx, best);
    tc_fence_before();
    __syncwarp();
    // (all 16 warps read this tile; the block's reduction precedes the next
    // tile's MMAs, so eight arrivals complete the phase)
    if (warp < kTcReaders && lane == 0) mbar_arrive(&tl.bars.tc_free[b]);
  }
  tr.tiles += (uint32_t)n;
  tr.rows += (uint32_t)(n * NSL);
  *bad_out = 0;
  return best;
}

// The loop of a CTA that only searches, in the tensor-core form (the image's
// state block, the stop flag and the first target are in shared memory),
// compiled as a function of its own with every phase inlined: a call would
// save and restore the caller's registers through local memory, which misses
// L1 while shared memory takes nearly all of it.
template <int R>
__device__ __noinline__ void run_tc_search(const EngineArgs& ea, EngCtx& x, const TcTiles tt, int nb, int slot, int ns,
                                           bool lead_searches) {
  using GT = TcEngGeom<R>;
  // working copies of the context (it lives in the kernel's local memory)
  const uint32_t tmem = x.tmem;
  unsigned long long* const tpart = x.tpart;
  EngSmemTail& tl = *reinterpret_cast<EngSmemTail*>(eng_smem());
  const ImgState& s = tl.img;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = x.rank;
  TeamCtl* tc = x.tc;
  const unsigned long long limit = ea.wait_limit_ns;
  const bool withheld = rank + 1 == ea.withhold;  // (the arguments lie in local memory)
  int* const err = ea.err;
  unsigned epoch = x.epoch;
  TcRun tr;
  tc_setup<R>(tr, x, tl.bars, s, tt, 0, ns, lead_searches, (int)kHeadBytes, nb, slot);
  const int npre = min(nb, GT::NSL);
  int pref = 0;
  bool first = true;
  while (!tl.stop) {
    const int px = tl.px, py = tl.py;
    int bad;
    unsigned long long best = tc_round<R>(s, tt, tr, tl, tmem, px, py, first, pref, rank, ns, lead_searches, limit, &bad);
    first = false;
    best = block_min_u64(best, tl.red64);
    if (tid == 0) {
      if (!withheld) st_relaxed64(&tpart[rank], key_tag(best, epoch));
      if (bad) atomicExch(err, INPAINT_ERR_TIMEOUT);
      if (rank == 0) atomicAdd(&s.ctrl->tc_rounds, 1);
    }
    if (bad) break;
    if (warp == kEngWarps - 1 && lane == 0) {
      // once the leader has written this round's fill, the next round's
      // first source rows are final: request them now, while the leader
      // updates (no prefetch if the next publication comes first)
      int n = 0;
      const unsigned long long t0 = globaltimer();
      while (true) {
        if ((int)(ld_acquire(&tc->copied) - (epoch + 1u)) >= 0) {
          asm volatile("fence.proxy.async.global;" ::: "memory");
          n = npre;
          if (!tc_produce<R>(s, tr.a, tl.bars, tr.tx0, tr.y0, tr.rows, 0, n, limit))
            atomicExch(err, INPAINT_ERR_TIMEOUT);
          break;
        }
        if ((unsigned)ld_acquire64(&tc->pub) != epoch || globaltimer() - t0 > limit) break;
      }
      tl.tc_pref = n;
    }
    // wait for the next round
    if (tid == 0) {
      const int bits = pub_bits(s.W);
      pub_unpack(wait_pub(tc, epoch, err, limit), bits, tl.px, tl.py, tl.stop);
    }
    ++epoch;
    __syncthreads();
    pref = tl.tc_pref;
    if (lane == 0) asm volatile("fence.proxy.async.global;" ::: "memory");
  }
  if (pref > 0) {
    // the loop stopped with a prefetch in flight: let it land and release
    // its slots (two arrivals stand for the two issuers' commits)
    if (warp == kEngWarps - 1 && lane == 0) {
      for (int h = 0; h < pref; ++h) {
        const uint32_t g = tr.rows + (uint32_t)h;
        const int sl = (int)(g % (uint32_t)nb);
        if (!mbar_wait(&tl.bars.tc_full[sl], (g / (uint32_t)nb) & 1u, limit)) atomicExch(ea.err, INPAINT_ERR_TIMEOUT);
        mbar_arrive(&tl.bars.tc_empty[sl]);
        mbar_arrive(&tl.bars.tc_empty[sl]);
      }
    }
    tr.rows += (uint32_t)pref;
    __syncthreads();
  }
  x.epoch = epoch;
  x.tc_rows = tr.rows;
  x.tc_tiles = tr.tiles;
}

// A searching leader's share of one tensor-core round (its state at byte `off`
// of shared memory); the block's best key.
template <int R>
__device__ __noinline__ unsigned long long tc_lead_share(const EngineArgs& ea, EngCtx& x, const TcTiles tt, int off,
                                                         int nb, int slot, int ns, int px, int py, bool first) {
  EngSmemTail& tl = *reinterpret_cast<EngSmemTail*>(eng_smem());
  const ImgState& s = tl.img;
  // the run's state stays in shared memory between the rounds (tl.tc_run)
  TcRun tr;
  if (first) tc_setup<R>(tr, x, tl.bars, s, tt, 1, ns, true, off, nb, slot);
  else tr = tl.tc_run;
  int bad;
  unsigned long long best = tc_round<R>(s, tt, tr, tl, x.tmem, px, py, first, 0, x.rank, ns, true, ea.wait_limit_ns, &bad);
  if (bad && threadIdx.x == 0) {
    atomicExch(ea.err, INPAINT_ERR_TIMEOUT);
    tl.err = INPAINT_ERR_TIMEOUT;
  }
  x.tc_rows = tr.rows;
  x.tc_tiles = tr.tiles;
  best = block_min_u64(best, tl.red64);  // (its barriers: every thread has read tl.tc_run)
  if (threadIdx.x == 0) tl.tc_run = tr;
  return best;
}

// The loop of a CTA that searches in resident mode and does not lead (its plan,
// the image's state block, the stop flag and the first target are in shared
// memory), compiled as a function of its own with everything inlined: the
// registers a call saves come back from L2, since L1 is nearly all shared
// memory (two nested calls per unit took 2,000 cycles a round).
// OVL: the partial-overlap form (KC 4): every centre of the rectangle is a
// candidate, the tiles say which source pixels are available, and the number
// of admissible candidates goes to the leader with the key.
template <int R, int KC, bool OVL = false>
__device__ __noinline__ void run_res_search(const EngineArgs& ea, EngCtx& x, int xb, int ncu, int acc_off) {
  static_assert(!OVL || KC == 4, "the partial-overlap search has four candidates per lane");
  constexpr int P = 2 * R + 1, TP = (P + 3) & ~3, TH = kResRows + 2 * R;
  EngSmemTail& tl = *reinterpret_cast<EngSmemTail*>(eng_smem());
  const ImgState& s = tl.img;
  const ResPlan& pl = tl.plan;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = x.rank;
  TeamCtl* const tc = x.tc;
  unsigned long long* const tpart = x.tpart;
  const unsigned long long limit = ea.wait_limit_ns;
  const bool withheld = rank + 1 == ea.withhold;
  int* const err = ea.err;
  unsigned epoch = x.epoch;
  uint8_t* const area = eng_smem() + kHeadBytes;
  uint32_t* const tgt = reinterpret_cast<uint32_t*>(eng_smem() + kTgtOff);
  uint32_t* const rowd = tgt + P * TP;
  uint32_t* const part = reinterpret_cast<uint32_t*>(eng_smem() + acc_off);  // KC < 16: partial SSDs [unit][k][lane]
  const int u0 = pl.u0, n = pl.u1 - pl.u0, b0 = pl.seg[0].band;
  uint16_t* const bits = reinterpret_cast<uint16_t*>(area + pl.bits_off);
  // the source windows of every band segment (plain 16-byte loads; outside
  // the image: zero), then the validity bits of every unit
  for (int g = 0; g < pl.nseg; ++g) {
    const ResSeg sg = pl.seg[g];
    const int x0 = xb - R + sg.c_lo * KC, y0 = s.cy0 + sg.band * kResRows - R;
    const int nq = sg.pitch / 4;
    uint4* dst = reinterpret_cast<uint4*>(area + sg.off);
    if constexpr (OVL) {
      uint32_t* words = reinterpret_cast<uint32_t*>(area + sg.off);
#pragma unroll 4
      for (int i = tid; i < TH * sg.pitch; i += kEngThreads) {
        const int row = i / sg.pitch, y = y0 + row, xw = x0 + i - row * sg.pitch;
        const bool in = y >= 0 && y < s.H && xw >= 0 && xw < s.W;
        const uint32_t w = in ? __ldcg(&s.img[(size_t)y * s.pitch + xw]) : 0u;
        const uint8_t o = in ? __ldcg(&s.omega[(size_t)y * s.W + xw]) : 1;
        words[i] = o ? 0xff000000u : w;
      }
      continue;
    }
    for (int i = tid; i < TH * nq; i += kEngThreads) {
      const int row = i / nq, q = i - row * nq, y = y0 + row, xw = x0 + 4 * q;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (y >= 0 && y < s.H && xw + 3 < s.pitch)
        v = __ldcg(reinterpret_cast<const uint4*>(s.img + (size_t)y * s.pitch + xw));
      dst[i] = v;
    }
  }
  for (int j = warp; j < n; j += kEngWarps) {
    const int u = u0 + j, band = u / ncu, col = u - band * ncu;
    const int qy = s.cy0 + band * kResRows + lane, qx0 = xb + col * KC;
    uint32_t v = 0;
    if (qy <= s.cy1) {
#pragma unroll
      for (int k = 0; k < KC; ++k) {
        const int qx = qx0 + k;
        if (qx >= s.cx0 && qx <= s.cx1 && (OVL || __ldcg(&s.count[(size_t)qy * s.pitch + qx]) == 0)) v |= 1u << k;
      }
    }
    bits[j * 32 + lane] = (uint16_t)v;
  }
  while (!tl.stop) {
    const int px = tl.px, py = tl.py;
    // target patch: warp dy reads row dy (lane = dx); the ballot of the
    // known flags gives the row descriptor
    for (int dy = warp; dy < P; dy += kEngWarps) {
      const int tx = px + lane - R, ty = py + dy - R;
      uint32_t w = 0;
      bool known = false;
      const bool in = lane < P && tx >= 0 && tx < s.W && ty >= 0 && ty < s.H;
      if (in) {
        // both reads in flight together; the pixel is kept only if known
        const uint8_t o = __ldcg(&s.omega[(size_t)ty * s.W + tx]);
        const uint32_t v = __ldcg(&s.img[(size_t)ty * s.pitch + tx]);
        known = o == 0;
        w = known ? v : 0u;
      }
      const unsigned bal = __ballot_sync(0xffffffffu, known);
      if (lane < P) {
        tgt[dy * TP + lane] = w;
        tl.known[dy * P + lane] = (uint8_t)(known ? 1 : OVL && in ? 2 : 0);
      }
      if (lane == 0) rowd[dy] = row_desc(bal & ((1u << P) - 1u), P);
      if constexpr (OVL) {
        const uint32_t wa = known ? w | 0xff000000u : 0u;
        const uint32_t sq = __reduce_add_sync(0xffffffffu, __dp4a(wa, wa, 0u));
        if (lane == 0) tl.a2row[dy] = (int)sq;
      }
    }
    if constexpr (KC < 16)
      for (int i = tid; i < n * KC * 32; i += kEngThreads) part[i] = 0u;
    if (OVL && tid == 0) tl.red32[0] = 0;
    __syncthreads();
    unsigned long long best = ~0ull;
    int n_adm = 0;
    auto take = [&](int j, const uint32_t (&acc)[KC]) {
      const int u = u0 + j, band = u / ncu, col = u - band * ncu;
      const uint32_t vb = bits[j * 32 + lane];
      const unsigned idx0 = (unsigned)((s.cy0 + band * kResRows + lane) * s.W + xb + col * KC);
#pragma unroll
      for (int k = 0; k < KC; ++k) {
        const unsigned long long key = ((unsigned long long)acc[k] << 32) | (idx0 + (unsigned)k);
        const bool adm = (vb & (1u << k)) && (!OVL || acc[k] < kOvlBad);
        if (OVL) n_adm += adm;
        if (adm && key < best) best = key;
      }
    };
    // (KC 16: whole units, warp w takes w, w + 16, ...; else the rows
    // [w T / 16, (w + 1) T / 16) of the T = n P unit rows)
    int t = KC < 16 ? warp * n * P / kEngWarps : warp * P;
    const int t1 = KC < 16 ? (warp + 1) * n * P / kEngWarps : n * P;
#pragma unroll 1
    while (t < t1) {
      const int j = t / P, r0 = t - j * P, r1 = min(P, r0 + t1 - t);
      const int u = u0 + j, band = u / ncu, col = u - band * ncu;
      const ResSeg& sg = pl.seg[band - b0];
      const uint32_t* strip = reinterpret_cast<const uint32_t*>(area + sg.off) + lane * sg.pitch + (col - sg.c_lo) * KC;
      uint32_t acc[KC];
      if constexpr (OVL)
        unit_ssd_overlap<R>(strip, sg.pitch, tgt, rowd, tl.known, tl.a2row, r0, r1, bits[j * 32 + lane] != 0, acc);
      else
        unit_ssd<R, KC>(strip, sg.pitch, tgt, rowd, r0, r1, acc);
      if constexpr (KC < 16) {
#pragma unroll
        for (int k = 0; k < KC; ++k) atomicAdd(&part[(j * KC + k) * 32 + lane], acc[k]);
        t += r1 - r0;
      } else {
        take(j, acc);
        t += kEngWarps * P;
      }
    }
    if constexpr (KC < 16) {
      __syncthreads();
#pragma unroll 1
      for (int j = warp; j < n; j += kEngWarps) {
        uint32_t acc[KC];
#pragma unroll
        for (int k = 0; k < KC; ++k) acc[k] = part[(j * KC + k) * 32 + lane];
        take(j, acc);
      }
    }
    if constexpr (OVL) {
      __syncwarp();
      n_adm = __reduce_add_sync(0xffffffffu, n_adm);
      if (lane == 0 && n_adm) atomicAdd(&tl.red32[0], n_adm);
    }
    best = block_min_u64(best, tl.red64);
    if (tid == 0) {
      if (OVL)
        st_relaxed64(&tpart[x.tsize * (1 + (epoch & 1u)) + rank],
                     (unsigned long long)epoch << 32 | (unsigned)tl.red32[0]);
      if (!withheld) st_relaxed64(&tpart[rank], key_tag(best, epoch));
      // the tiles are brought up to date as soon as the copy is done, while the
      // leader still works on the priorities (after the publication, this and
      // the target's reads were three L2 round trips one after another)
      const unsigned long long t0 = globaltimer();
      while ((int)(ld_acquire(&tc->copied) - (epoch + 1u)) < 0 && (unsigned)ld_acquire64(&tc->pub) == epoch &&
             globaltimer() - t0 <= limit) {
      }
    }
    __syncthreads();
    {
      // the iteration's filled pixels (the target patch's unknown in-image
      // ones) into every tile that holds them, and the candidates within 2R of
      // it that became valid; every load in flight before the first use
      constexpr int NCW = 4 * R + 1, NV = (NCW * NCW + kEngThreads - 1) / kEngThreads;
      const int tx = px + tid % P - R, ty = py + tid / P - R;
      const bool filled = tid < P * P && tx >= 0 && tx < s.W && ty >= 0 && ty < s.H && tl.known[tid < P * P ? tid : 0] != 1;
      uint32_t w = 0u;
      if (filled) w = __ldcg(&s.img[(size_t)ty * s.pitch + tx]);
      int cnt[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int jj = tid + v * kEngThreads, qx = px + jj % NCW - 2 * R, qy = py + jj / NCW - 2 * R;
        const bool in = !OVL && jj < NCW * NCW && qx >= s.cx0 && qx <= s.cx1 && qy >= s.cy0 && qy <= s.cy1;
        cnt[v] = in ? __ldcg(&s.count[(size_t)qy * s.pitch + qx]) : 1;
      }
      if (filled) {
#pragma unroll 1
        for (int g = 0; g < pl.nseg; ++g) {
          const ResSeg& sg = pl.seg[g];
          const int lx = tx - (xb - R + sg.c_lo * KC), ly = ty - (s.cy0 + sg.band * kResRows - R);
          if (lx >= 0 && lx < sg.pitch && ly >= 0 && ly < TH)
            reinterpret_cast<uint32_t*>(area + sg.off)[ly * sg.pitch + lx] = w;
        }
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        if (cnt[v] != 0) continue;
        const int jj = tid + v * kEngThreads, qx = px + jj % NCW - 2 * R, qy = py + jj / NCW - 2 * R;
        const int col = (qx - xb) / KC, j = (qy - s.cy0) / kResRows * ncu + col - u0;
        if (j < 0 || j >= n) continue;
        const int e = j * 32 + (qy - s.cy0) % kResRows;
        atomicOr(reinterpret_cast<unsigned*>(bits) + (e >> 1), (1u << (qx - xb - col * KC)) << (16 * (e & 1)));
      }
    }
    if (tid == 0) {
      const int bits = pub_bits(s.W);
      pub_unpack(wait_pub(tc, epoch, err, limit), bits, tl.px, tl.py, tl.stop);
    }
    ++epoch;
    __syncthreads();
  }
  x.epoch = epoch;
}

// The loop of a leader that does not search, compiled as a function of its
// own: none of the search state is live through its phases, so its
// registers hold the update's working set.
template <int R, int SRW>
__device__ __noinline__ void run_lead_only(const EngineArgs& ea, int j, EngCtx& x) {
  run_image<R, SRW, true>(ea, j, x);
}

template <int R, int SRW, bool kLeadOnly>
__device__ __forceinline__ void run_image(const EngineArgs& ea, int j, EngCtx& x) {
  using G = EngGeom<R, SRW>;
  constexpr int P = G::P, B = G::B;
  uint8_t* const smem = eng_smem();
  EngSmemTail& tl = *reinterpret_cast<EngSmemTail*>(smem);
  uint32_t* tgt = reinterpret_cast<uint32_t*>(smem + kTgtOff);
  uint32_t* rowd = tgt + P * G::TP;  // row descriptors of the target
  uint8_t* upd_base = smem + kHeadBytes;
  UpdSmem<R>& usm = *reinterpret_cast<UpdSmem<R>*>(upd_base);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = x.rank, tsize = x.tsize;
  TeamCtl* const tc = x.tc;
  unsigned long long* const tpart = x.tpart;
  const unsigned long long t_start = x.t_start;  // (the context is in local memory)
  const unsigned long long limit = ea.wait_limit_ns;
  int* const err = ea.err;
  const unsigned long long tick_ns = ea.tick_ns;
  const bool withheld = rank + 1 == ea.withhold;
  uint32_t ph0 = x.ph0, ph1 = x.ph1;
  unsigned epoch = x.epoch;

  // every role reads the image's fields from shared memory, which keeps
  // about forty registers free for its phases.  The barrier before the write is
  // the hand-over from the team's last image: its leader's warps 4-15 may still
  // be in update_drain, with that image's fields and update state, when warps
  // 0-3 come here (with more images than SMs a CTA does several in turn).  The
  // fence orders the last image's accesses to shared memory before this one's
  // bulk copies into it.  Once an image.
  if constexpr (!kLeadOnly) {
    fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) tl.img = ea.imgs[j];
    __syncthreads();
  }
  const ImgState& s = tl.img;
  const CUtensorMap* map = &ea.tmaps[2 * j];
  const CUtensorMap* cmap = &ea.tmaps[2 * j + 1];
  Ctrl* c = s.ctrl;
  const int xb = R + ((s.cx0 - R) & ~3);
  const int ncg = s.cx1 >= s.cx0 ? (s.cx1 - xb + G::BWC) / G::BWC : 0;
  const int nrb = s.cy1 >= s.cy0 ? (s.cy1 - s.cy0 + B) / B : 0;
  const int nbatch = ncg * nrb;
  // Roles: CTAs [0, ns) search, batch b going to CTA b mod ns (batches cost
  // alike).  The last CTA of the team is the leader: it runs the speculative
  // phase of each iteration while the others search, waits for their keys,
  // applies the update and publishes the next round.  When the image has
  // many batches per CTA (small teams in the batched form) the leader also
  // searches its share after the speculative phase, which is short next to
  // a CTA's share of such a search.  A CTA that neither searches nor leads
  // idles until the image is done.
  // Tensor-core form (an image given planes): whole tiles, round-robin, when
  // the A strips and a ring of at least four source-row slots fit beside a
  // searching leader's update state.  The leader searches too when every CTA
  // has three tiles or more.  An image that leaves the choice of the form to
  // the engine (tc_auto) takes the one with the lower estimate for this team.
  const TcTiles tt = s.planes ? tc_tiles(s) : TcTiles{0, 0, 0, 0, 1, 0};
  const int tc_ntiles = tt.ntx * tt.nty;
  const int tc_slot_b = s.planes ? tc_slot(tt.N, R) : 1;
  constexpr int kUpdB = (int)(((upd_smem_bytes<R>() + 127) / 128) * 128);
  const bool tc_lead = tsize == 1 || tc_ntiles >= 3 * tsize;
  const int tc_off = (int)kHeadBytes + (tc_lead && rank == tsize - 1 ? kUpdB : 0);
  int tc_nb = 0;
  bool tcmode = false;
  if (s.planes && ea.tc_cols >= kTcCols && tc_ntiles > 0) {
    const int fixed = (int)kHeadBytes + TcEngGeom<R>::A_BYTES + TcEngGeom<R>::TPAD_BYTES;
    const int tc_ns = tc_lead ? min(tsize, tc_ntiles) : min(tsize - 1, tc_ntiles);
    tcmode = ((int)x.smem_bytes - fixed - (tc_lead ? kUpdB : 0)) / tc_slot_b >= 4 &&
             (!s.tc_auto || tc_round_cycles(s, tc_ns) < plain_round_cycles(s, tsize));
    tc_nb = min(kTcRing, ((int)x.smem_bytes - (tc_off - (int)kHeadBytes) - fixed) / tc_slot_b);
  }
  const bool lead_searches = tcmode ? tc_lead : !s.overlap && (tsize == 1 || nbatch >= 8 * tsize);
  const int nsmax = lead_searches ? tsize : tsize - 1;  // CTAs that may search
  // Plain form, resident mode when the leader does not search and every
  // searching CTA's tiles fit (the same decision in every CTA of the team: it
  // depends only on the image and the team); more than one band of units per
  // CTA streams instead.  A partial-overlap search comes here only when it fits
  // (overlap_fits).
  const int nbands = s.cy1 >= s.cy0 ? (s.cy1 - s.cy0 + kResRows) / kResRows : 0;
  int kc = 16, ncu = 0, ns = 0;
  bool resident = false;
  if (tcmode) {
    ns = min(nsmax, tc_ntiles);
  } else if (s.overlap) {
    kc = 4;
    resident = overlap_units<R>(s, nsmax, &ncu, &ns) > 0;
  } else {
    for (; !lead_searches; kc = 4) {
      ncu = s.cx1 >= s.cx0 ? (s.cx1 - xb + kc) / kc : 0;
      ns = min(nsmax, ncu * nbands);
      const int m = ns > 0 ? (ncu * nbands + ns - 1) / ns : 0;  // most units of one CTA
      resident = m > 0 && m <= ncu && res_need<R>(kc, m) <= (int)x.smem_bytes - (int)kHeadBytes;
      if (m >= 3 * kEngWarps / 4 || kc == 4) break;
    }
    if (!resident) ns = min(nsmax, nbatch);
  }
  const bool leader = rank == tsize - 1;
  const bool searcher = rank < ns;
  if constexpr (!kLeadOnly) {
    if (leader && !searcher) {
      run_lead_only<R, SRW>(ea, j, x);
      return;
    }
  }
  if (tid == 0) {
    tl.stop = !ctrl_active(c) || __ldcg(err) != 0;
    tl.px = __ldcg(&c->px);
    tl.py = __ldcg(&c->py);
    if (resident && searcher) res_plan<R>(tl.plan, kc, ncu, nbands, rank, ns);
  }
  __syncthreads();
  if constexpr (!kLeadOnly) {
    if (tcmode && searcher && !leader) {
      run_tc_search<R>(ea, x, tt, tc_nb, tc_slot_b, ns, tc_lead);
      return;
    }
    if (resident && searcher) {
      const int acc_off = ((int)kHeadBytes + tl.plan.bits_off + (tl.plan.u1 - tl.plan.u0) * 64 + 127) & ~127;
      if (s.overlap) run_res_search<R, 4, true>(ea, x, xb, ncu, acc_off);
      else if (kc == 16) run_res_search<R, 16>(ea, x, xb, ncu, acc_off);
      else run_res_search<R, 4>(ea, x, xb, ncu, acc_off);
      return;
    }
  }
  // the CTA's work area (a searching leader keeps its update state below it)
  uint8_t* area = smem + kHeadBytes + (leader ? ((upd_smem_bytes<R>() + 127) / 128) * 128 : 0);
  // streaming mode: two count tiles and two tile slots (double buffer)
  uint32_t* cnt_t[2] = {reinterpret_cast<uint32_t*>(area),
                        reinterpret_cast<uint32_t*>(area + G::CNT_BYTES)};
  uint8_t* slots = area + 2 * G::CNT_BYTES;
  auto slot_pix = [&](int i) { return reinterpret_cast<uint32_t*>(slots + (size_t)i * G::SLOT_BYTES); };
  int round = 0;        // search rounds of this image in this launch

  // One search round for target (px, py): this CTA's batches; returns its
  // best key.  Whole block.
  auto search_round = [&](int px, int py) -> unsigned long long {
    const int b0 = rank < ns ? rank : nbatch;
    // a batch's stage in streaming mode: its RGBA window and the validity
    // counts of its candidates, on one mbarrier
    auto issue = [&](int b, uint32_t* st, uint32_t* ct, uint64_t* bar) {
      const int gx = b % ncg, gy = b / ncg;
      // (the stage's previous generic reads are ordered before this by the
      // block barrier that ends every batch)
      mbar_expect_tx(bar, (uint32_t)(G::BW * G::BH * 4 + G::CW * B * 4));
      tma_load_2d(st, map, xb - R + G::BWC * gx, s.cy0 + B * gy - R, bar);
      tma_load_2d(ct, cmap, xb - G::COFF + G::BWC * gx, s.cy0 + B * gy, bar);
    };
    const bool first = round == 0;
    if (tcmode) {
      ++round;
      if (tid == 0 && ns == 1) atomicAdd(&c->tc_rounds, 1);  // (else the team's first searcher counts)
      return tc_lead_share<R>(ea, x, tt, tc_off, tc_nb, tc_slot_b, ns, px, py, first);
    }
    if (tid == 0 && b0 < nbatch) issue(b0, slot_pix(0), cnt_t[0], &tl.bars.full[0]);
    // target patch: warp dy reads row dy (lane = dx); the ballot of the
    // known flags gives the row descriptor
    {
      for (int dy = warp; dy < P; dy += kEngWarps) {
        const int tx = px + lane - R, ty = py + dy - R;
        uint32_t w = 0;
        bool known = false;
        if (lane < P && tx >= 0 && tx < s.W && ty >= 0 && ty < s.H) {
          // both reads in flight together; the pixel is kept only if known
          const uint8_t o = __ldcg(&s.omega[(size_t)ty * s.W + tx]);
          const uint32_t v = __ldcg(&s.img[(size_t)ty * s.pitch + tx]);
          known = o == 0;
          w = known ? v : 0u;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, known);
        if (lane < P) {
          tgt[dy * G::TP + lane] = w;
        }
        if (lane == 0) rowd[dy] = row_desc(bal & G::FULL, P);
      }
    }
    __syncthreads();
    unsigned long long best = ~0ull;
    bool ok = true;
    {
      int cur = 0;
      for (int b = b0; b < nbatch; b += ns) {
        const int nb = b + ns;
        if (tid == 0 && nb < nbatch) issue(nb, slot_pix(cur ^ 1), cnt_t[cur ^ 1], &tl.bars.full[cur ^ 1]);
        const int gx = b % ncg, gy = b / ncg;
        const bool got = mbar_wait(&tl.bars.full[cur], cur ? ph1 : ph0, limit);
        if (cur) ph1 ^= 1; else ph0 ^= 1;
        // validity of this lane's candidates from the count tile (16-byte
        // aligned chunk) and the search rectangle
        uint32_t cw[G::NCL + 4];
        lds_words(cw, cnt_t[cur] + lane * G::CW + G::NCL * warp);
        const int qy = s.cy0 + B * gy + lane, qx0 = xb + G::BWC * gx + G::NCL * warp;
        uint32_t bits = 0;
#pragma unroll
        for (int k = 0; k < G::NCL; ++k) {
          const int qx = qx0 + k;
          if (qx >= s.cx0 && qx <= s.cx1 && qy <= s.cy1 && cw[G::COFF + k] == 0) bits |= 1u << k;
        }
        const unsigned long long kb = unit_best<R, G::NCL>(
            (int)(slots - smem) + cur * G::SLOT_BYTES + 4 * (lane * G::BW + G::NCL * warp), G::BW, kTgtOff, bits,
            (unsigned)(qy * s.W + qx0));
        best = kb < best ? kb : best;
        if (__syncthreads_or(!got)) {  // a bounded wait gave up: stop uniformly
          ok = false;
          if (nb < nbatch) {
            mbar_wait(&tl.bars.full[cur ^ 1], cur ? ph0 : ph1, limit);
            if (cur) ph0 ^= 1; else ph1 ^= 1;
          }
          break;
        }
        cur ^= 1;
      }
    }
    ++round;
    if (!ok && tid == 0) {
      atomicExch(err, INPAINT_ERR_TIMEOUT);
      tl.err = INPAINT_ERR_TIMEOUT;  // (a searching leader: its key would be partial)
    }
    return block_min_u64(best, tl.red64);
  };

  // Partial-overlap search: the last round's candidates, for its record (warp 15).
  auto last_counts = [&]() {
    if (!s.overlap || !usm.rec_pending) return;
    const int n = gather_counts(&tpart[tsize * (1 + ((epoch - 1u) & 1u))], ns, epoch - 1u, err, limit);
    if (lane == 0) usm.n_cand = n;
    __syncwarp();
  };

  // One iteration of the leader on the staged target (and its own search
  // share when it searches), up to the publication of the next round and the
  // staging of its target.  Whole block.
  auto lead_round = [&](bool searches) {
    const int px = usm.nx_px, py = usm.nx_py;
    spec_front<R>(usm);
    if (tid < kChainThreads) {
      spec_chains<R>(s, usm);
    } else if (tid < kRecThread) {
      spec_rest<R>(s, usm);
    } else {
      if (tid == kRecThread + 1) {
        // the stop decision's inputs that other CTAs may change
        tl.status = __ldcg(&c->status);
        tl.err = __ldcg(err);
      }
      spec_record<R>(s, usm, false, last_counts);
      __syncwarp();
    }
    if constexpr (!kLeadOnly) {
      if (searches) {
        __syncthreads();
        const unsigned long long best = search_round(px, py);
        if (tid == 0) st_relaxed64(&tpart[rank], key_tag(best, epoch));
      }
    }
    if (tid >= kChainThreads) {
      CopyPlan cpy{};
      if (tid >= kRecThread) {
        bool late;
        const unsigned long long best = gather_keys(tpart, ns, epoch, err, limit, &late);
        if (lane == 0) {
          usm.t_keys = globaltimer();
          set_source<R>(s, usm, best, late || tl.err != 0);
        }
        __syncwarp();
      } else {
        cpy = plan_copy<R>(s, usm);
      }
      work_sync();
      if (usm.ok) update_work<R>(s, usm, cpy, true, tcmode || resident ? &tc->copied : nullptr, epoch + 1u);
    }
    __syncthreads();
    const bool ok = usm.ok != 0;
    bool stop = true;
    unsigned long long wk = 0ull;
    int wi = 0, ny = 0;
    if (ok) {
      update_prio<R>(s, usm, wk, wi, ny);
      stop = usm.remaining <= 0 || wk == 0ull || usm.it + 1 >= tl.lim || tl.status != 0 || tl.err != 0;
    }
    if (tid == kPubThread) {
      // the next round (or the stop) goes out before the bookkeeping; after
      // an update, this thread's fence in update_work ordered every write
      // the searchers read before this store, else the store is a release
      const bool spent = ok && !stop && tick_ns && globaltimer() - t_start > tick_ns;
      if (spent) {
        stop = true;  // the launch's time budget is spent: resume in the next launch
        tc->expired = 1u;
      }
      const unsigned long long v = pub_pack(epoch + 1u, stop ? 0 : wi - ny * s.W, stop ? 0 : ny, stop, pub_bits(s.W));
      if (ok && !spent)
        st_relaxed64(&tc->pub, v);
      else
        st_release64(&tc->pub, v);
      tl.stop = stop;
    }
    if (ok) {
      auto store = [&]() { update_store<R>(s, usm, wk, wi); };
      if (!stop) stage_next<R>(s, wk, wi, ny, usm, store);  // (the time budget is known to the publishing thread only)
      else store();
    }
    ++epoch;
    __syncthreads();
    if (lane == 0) asm volatile("fence.proxy.async.global;" ::: "memory");
  };

  if (leader && !tl.stop) {
    stage_first<R>(s, usm, false);
    if (tid == 0) tl.lim = __ldcg(&c->iter_limit);
    __syncthreads();
  }
  if constexpr (kLeadOnly) {
    if (!tl.stop) {
      do lead_round(false);
      while (!tl.stop);
      if (tid >= kRecThread) last_counts();
      if (tid == kRecThread) update_times<R>(s, usm);
      update_drain<R>(s, usm, false);
    }
    x.epoch = epoch;
    return;
  }
  const bool led = leader && !tl.stop;
  while (!tl.stop) {
    const int px = tl.px, py = tl.py;
    if (leader) {
      lead_round(true);
      continue;
    }
    if (searcher) {
      const unsigned long long best = search_round(px, py);
      if (tid == 0 && !withheld) st_relaxed64(&tpart[rank], key_tag(best, epoch));
    }
    // searchers and idle CTAs: wait for the next round
    if (tid == 0) {
      const int bits = pub_bits(s.W);
      pub_unpack(wait_pub(tc, epoch, err, limit), bits, tl.px, tl.py, tl.stop);
    }
    ++epoch;
    __syncthreads();
    if (lane == 0) asm volatile("fence.proxy.async.global;" ::: "memory");
  }
  if (led) {
    if (tid == kRecThread) update_times<R>(s, usm);
    update_drain<R>(s, usm, false);
  }
  x.ph0 = ph0;
  x.ph1 = ph1;
  x.epoch = epoch;
}

// Shared-memory bytes the engine needs for radius R and SRW rows per warp.
template <int R, int SRW>
constexpr size_t engine_smem_for() {
  return eng_smem_bytes<R, SRW>();
}

// Single-CTA copy/update kernel of the graph-driven loop for R <= 8 (the same
// update phase that the engine runs in a team's leader).
template <int R>
__global__ void __launch_bounds__(kEngThreads) k_update_fast(ImgState s, cudaGraphConditionalHandle cond,
                                                            int use_cond) {
  extern __shared__ __align__(128) uint8_t sm_raw[];
  UpdSmem<R>& usm = *reinterpret_cast<UpdSmem<R>*>(sm_raw);
  if (!loop_active(s.ctrl)) {
    if (use_cond && threadIdx.x == 0) cudaGraphSetConditional(cond, 0);
    return;
  }
  stage_first<R>(s, usm, s.overlap != 0);
  __syncthreads();
  spec_front<R>(usm);
  if (threadIdx.x < kChainThreads) {
    spec_chains<R>(s, usm);
  } else {
    CopyPlan cpy{};
    if (threadIdx.x < kRecThread) {
      spec_rest<R>(s, usm);
      cpy = plan_copy<R>(s, usm);
    } else {
      const int lane = threadIdx.x & 31;
      spec_record<R>(s, usm, false, [] {});
      __syncwarp();
      unsigned long long best = ~0ull;
#pragma unroll 4
      for (int i = lane; i < s.n_partial; i += 32) {
        const unsigned long long v = __ldcg(&s.partial[i]);
        best = v < best ? v : best;
      }
      __syncwarp();
      best = warp_min_u64(best);
      if (lane == 0) set_source<R>(s, usm, best, false);
      __syncwarp();
    }
    work_sync();
    if (usm.ok) update_work<R>(s, usm, cpy, false, nullptr, 0u);
  }
  __syncthreads();
  const bool ok = usm.ok != 0;
  if (ok) {
    unsigned long long wk;
    int wi, ny;
    update_prio<R>(s, usm, wk, wi, ny);
    update_store<R>(s, usm, wk, wi);
    __syncthreads();
    update_drain<R>(s, usm, s.overlap != 0);
    __syncthreads();
  }
  if (use_cond && threadIdx.x == 0) cudaGraphSetConditional(cond, ok && loop_active(s.ctrl) ? 1u : 0u);
}

template <int R>
static cudaError_t upd_fast_t(const ImgState& s, unsigned long long cond, int use_cond, cudaStream_t st) {
  const size_t smem = upd_smem_bytes<R>();
  cudaError_t e = cudaFuncSetAttribute(k_update_fast<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  k_update_fast<R><<<1, kEngThreads, smem, st>>>(s, (cudaGraphConditionalHandle)cond, use_cond);
  return cudaGetLastError();
}

template <int R>
static cudaError_t prio_init_t(const ImgState& s, cudaStream_t st) {
  using G = UpdGeom<R>;
  const size_t smem = sizeof(UpdSmem<R>);
  cudaError_t e = cudaFuncSetAttribute(k_prio_init_fast<R>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((s.W + G::NW - 1) / G::NW, (s.H + G::NW - 1) / G::NW);
  k_prio_init_fast<R><<<grid, 256, smem, st>>>(s);
  return cudaGetLastError();
}

// Host entry points of one radius R, exported through EngineFns.
template <int R>
static size_t eng_smem_r(int srw) {
  return srw == 2 ? engine_smem_for<R, 2>() : engine_smem_for<R, 1>();
}
// Whether the engine runs the image's partial-overlap search with a team of
// tsize CTAs: every searcher's tiles are resident (the streaming search has no
// such form).
template <int R>
static bool overlap_fits_t(const ImgState& s, int tsize, size_t smem) {
  int ncu, ns;
  const int m = overlap_units<R>(s, tsize - 1, &ncu, &ns);
  return m > 0 && m <= ncu && smem > kHeadBytes && res_need<R>(4, m) <= (int)(smem - kHeadBytes);
}
template <int R>
const EngineFns* engine_fns_for() {
  static const EngineFns f = {eng_smem_r<R>, upd_fast_t<R>, prio_init_t<R>, overlap_fits_t<R>};
  return &f;
}

}  // namespace inp
