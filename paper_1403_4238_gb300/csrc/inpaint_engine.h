// Host/device interface of the persistent fill-loop engine (engine.cu).
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>

#include "inpaint_internal.cuh"

namespace inp {

constexpr int kEngThreads = 512;
constexpr int kEngWarps = kEngThreads / 32;
constexpr int kEngBatchRows = 32;  // candidate rows of a search batch (one per lane)

// Smallest staged width >= n words that is a multiple of 4 with an odd
// number of 16-byte chunks: rows of a tile then start in different bank
// quadruples, so 8 lanes reading 16 bytes each from 8 consecutive rows (one
// phase of a 128-bit shared load) touch 32 distinct banks.
__host__ __device__ constexpr int width_odd16(int n) {
  return ((((n + 3) & ~3) / 4) % 2) ? ((n + 3) & ~3) : ((n + 3) & ~3) + 4;
}
// Candidate columns of a search batch: 16 warps side by side, 4 * srw
// candidates per lane.
__host__ __device__ constexpr int eng_batch_cols(int srw) { return kEngWarps * 4 * srw; }
// TMA boxes of a batch: the source window (words) and the validity counts.
__host__ __device__ constexpr int eng_tile_width(int r, int srw) { return width_odd16(eng_batch_cols(srw) + 2 * r); }
__host__ __device__ constexpr int eng_count_width(int srw) { return eng_batch_cols(srw) + 4; }

// Tensor-core search of the engine (Sec. 3, Eq. 3-4 as correlations; the
// exact BF16 form of the tensor-core search).  A tile is kTcRows candidate
// rows x 8N candidate columns (N a multiple of 16, at most 128): the MMA's
// M = 128 rows are 16 candidate rows x 8 column shifts, its N columns blocks
// of 8 candidate columns.  Tiles are numbered row-major; searching CTA k of a
// team takes tiles k, k + ns, ...
constexpr int kTcRows = 16;
constexpr int kTcRing = 8;  // most slots of the shared-memory ring
constexpr int kTcRps = 2;   // source rows per ring slot (one bulk copy)
constexpr int kTcReaders = 8;  // warps that read a tile's accumulators beside the next tile's MMAs
constexpr int kTcCols = 512;   // tensor-memory columns: two buffers of X and S, N <= 128 columns each
struct TcTiles {
  int N;         // MMA N: 8-column candidate blocks per tile
  int ntx, nty;  // tiles per row / per column of the candidate rectangle
  int xs0;       // first source column of tile column 0 (a multiple of 8)
  int n1, h;     // folds: block pitch and row distance of one (n1 = N without folds)
};
__host__ __device__ inline int tc_chunks(int r) { return (2 * r + 1 + 14) / 8; }  // 8-tap chunks of a row
__host__ __device__ inline TcTiles tc_tiles(const ImgState& s) {
  return TcTiles{s.tc_n, s.tc_ntx, s.tc_nty, s.tc_xs0, s.tc_n1, s.tc_h};
}
// Measured cycles of one 128 x N x 16 MMA: 74 at N = 128, 59 at N = 64.
__host__ __device__ inline float tc_mma_cycles(int N) { return 43.5f + 0.24f * (float)N; }

// Tile and plane geometry of an image (the tc_* fields and prows of s); the
// rows every tile reads (y0 - r .. y0 + 15 + r) all exist, and no others: a
// fold's planes begin at the search rectangle's first source row, so that a
// rectangle far down an image takes no more memory than one at the top, and a
// pixel lies in at most two folds.  want > 0: the tiles
// of one image spread over `want` CTAs, so the number of tile columns (narrower
// tiles, cheaper MMAs) is what makes the round shortest; want 0: throughput of
// small teams, so a narrow image is folded until its tiles are close to
// N = 128 wide (an MMA costs 59 cycles at N = 64 and 74 at N = 128: half the
// cycles per candidate for an image 500 wide).  Returns the bytes to allocate
// for the planes and the validity bits behind them (0: no tile).
inline size_t tc_plane_layout(ImgState& s, int want) {
  s.tc_ntx = s.tc_nty = 0;
  if (s.cx1 < s.cx0 || s.cy1 < s.cy0) return 0;
  const int nc = tc_chunks(s.r), rows = s.cy1 - s.cy0 + 1;
  s.tc_xs0 = (s.cx0 - s.r) & ~7;
  const int wneed = s.cx1 - s.r - s.tc_xs0 + 1;  // candidate columns from the first tile's column 0
  const int least = (wneed + 1023) / 1024;
  auto n_of = [&](int ntx) { return ((wneed + 8 * ntx - 1) / (8 * ntx) + 15) & ~15; };
  int ntx = least, folds = 1;
  const int nty1 = (rows + kTcRows - 1) / kTcRows;
  if (want > 0) {
    float best = 0.f;
    for (int t = least; t <= least + 4 && n_of(t) >= 32; ++t) {
      const float c = tc_mma_cycles(n_of(t)) * (float)((t * nty1 + want - 1) / want);
      if (t == least || c < best) {
        best = c;
        ntx = t;
      }
    }
  } else if (least == 1) {
    const int n1 = (wneed + 7) / 8 + nc - 1;
    folds = n1 <= 64 ? 128 / n1 : 1;
    folds = folds < nty1 ? folds : nty1;
  }
  s.tc_f = folds;
  s.tc_ntx = ntx;
  if (folds > 1) {
    s.tc_n1 = (wneed + 7) / 8 + nc - 1;
    s.tc_n = (folds * s.tc_n1 + 15) & ~15;
    s.tc_nty = (nty1 + folds - 1) / folds;
  } else {
    s.tc_n1 = s.tc_n = n_of(ntx);
    s.tc_nty = nty1;
  }
  s.tc_h = kTcRows * s.tc_nty;
  s.tc_len = 8 * (s.tc_n + nc - 1);
  s.prows = s.tc_h + 2 * s.r;
  return (size_t)s.tc_ntx * s.prows * 5 * s.tc_len * 2 + (size_t)s.tc_ntx * s.tc_nty * kTcRows * s.tc_n;
}
// The planes and the bits in a buffer of that size.
inline void tc_bind_planes(ImgState& s, void* p) {
  s.planes = static_cast<uint16_t*>(p);
  s.vbits = reinterpret_cast<uint32_t*>(s.planes + (size_t)s.tc_ntx * s.prows * 5 * s.tc_len);
}

// Estimated cycles of one search round on ns searching CTAs, for the choice
// between the forms and for the batch plan.  Tensor-core form: a tile is
// (rows) x (MMAs a row), after about 4,500 cycles of target staging, A strips
// and read-back.  Plain form: about 0.6 of the patch known, 24 evaluations a
// cycle and CTA (the streaming mode of one- and two-CTA teams measured 20-28 of
// the 64 its two instructions allow), after 2,500 cycles.  The same rate stands
// for larger teams, which are resident and faster (about 40 at 1920x1080, r 6):
// there the estimate leans towards the tensor cores and towards more CTAs.
__host__ __device__ inline float tc_round_cycles(const ImgState& s, int ns) {
  const int P = 2 * s.r + 1, nc = tc_chunks(s.r), tiles = s.tc_ntx * s.tc_nty;
  const float tile = (float)((kTcRows + P - 1) * ((3 * nc + 1) / 2 + nc)) * tc_mma_cycles(s.tc_n) + 300.f;
  return 4500.f + (float)((tiles + ns - 1) / ns) * tile;
}
__host__ __device__ inline float plain_round_cycles(const ImgState& s, int ns) {
  const float P2 = (float)((2 * s.r + 1) * (2 * s.r + 1));
  return 2500.f + (float)(s.cx1 - s.cx0 + 1) * (float)(s.cy1 - s.cy0 + 1) * 0.6f * P2 / (24.f * (float)ns);
}

// The five planes of the search rectangle's current source pixels and the
// validity bits: before every launch of a single image in the tensor-core form
// (the caller may have changed it), after a batch or server image's
// initialisation (its launches keep them up to date).
cudaError_t launch_planes(const ImgState& s, cudaStream_t st);

// Per-team synchronisation words (global memory).
struct TeamCtl {
  unsigned long long pub;  // epoch | next px | next py | stop (pub_pack; release-published)
  unsigned expired;        // the launch's time budget ended this team's work
  unsigned copied;         // e + 1 once round e's fill is in the image and its planes
                           // (release-published; the searchers then bring their
                           // resident tiles up to date or prefetch source rows)
  unsigned pad[28];        // keep teams on separate 128-byte lines
};

struct EngineArgs {
  const ImgState* imgs;        // [n_imgs]
  const CUtensorMap* tmaps;    // [2 * n_imgs]: pixels, counts per image; 64-byte aligned
  const int* cta_team;         // [grid]
  const int* team_first;       // [n_teams + 1] first CTA of each team
  const int* team_img_off;     // [n_teams + 1] offsets into team_img
  const int* team_img;         // images of each team, in processing order
  TeamCtl* teams;              // [n_teams]
  unsigned long long* partials;// [grid] each CTA's best key of the round, tagged with the round
  int* err;                    // INPAINT_ERR_TIMEOUT if a bounded wait gave up
  unsigned long long wait_limit_ns;
  unsigned long long tick_ns;  // > 0: teams stop between iterations once the launch
                               // has run this long (serving ticks); 0: run to the end
  int withhold;                // failure injection: > 0 makes searcher rank withhold - 1
                               // of every team skip its arrival; 0 normally
  int tc_cols;                 // tensor-memory columns every CTA holds for the
                               // tensor-core search (0: no image uses it)
  int overlap;                 // 1: partial-overlap search (one image): behind the keys,
                               // two more slots per CTA with its counts of even and odd rounds
};

// The mbarriers of an engine CTA, at the start of its shared memory (the
// kernel initialises them once per launch).
struct EngBars {
  uint64_t full[2];               // TMA completion of the two streaming stages
  uint64_t tc_full[kTcRing];      // tensor-core search: source rows landed in ring slot
  uint64_t tc_empty[kTcRing];     // their MMAs (both issuers) completed: the slot is free
  uint64_t tc_done[2];            // a tile's MMAs (both issuers) completed, per accumulator buffer
  uint64_t tc_free[2];            // the buffer's accumulators have been read (kTcReaders warps)
  uint32_t tmem;                  // tensor-memory base written by tcgen05.alloc
  uint32_t pad;
};

// Per-CTA engine state carried from one image of a team's list to the next.
struct EngCtx {
  uint32_t smem_bytes;          // dynamic shared memory of the CTA
  int rank, tsize;              // this CTA's rank in its team, team size
  TeamCtl* tc;
  unsigned long long* tpart;    // partial keys of the team's CTAs
  uint32_t ph0, ph1;            // phase parities of the two TMA barriers
  unsigned epoch;               // team publications seen
  unsigned long long t_start;   // global timer at the CTA's start (tick budget)
  uint32_t tmem;                // tensor-memory base address (tensor-core search)
  uint32_t tc_rows;             // ring slots filled so far (their phases)
  uint32_t tc_tiles;            // tiles whose MMAs completed so far (done barrier phases)
  int tc_nb;                    // ring slots tc_rows was counted with (0: none yet)
};

// Per-image engine body for radius R and SRW rows per warp (engine_r<R>.cu),
// called from the one engine kernel (engine_multi.cu) by the image's radius.
#define INP_DECL_RUN_IMAGE(R)                                            \
  __device__ void run_image_r##R##_s1(const EngineArgs& ea, int j, EngCtx& x); \
  __device__ void run_image_r##R##_s2(const EngineArgs& ea, int j, EngCtx& x);
INP_DECL_RUN_IMAGE(1)
INP_DECL_RUN_IMAGE(2)
INP_DECL_RUN_IMAGE(3)
INP_DECL_RUN_IMAGE(4)
INP_DECL_RUN_IMAGE(5)
INP_DECL_RUN_IMAGE(6)
INP_DECL_RUN_IMAGE(7)
INP_DECL_RUN_IMAGE(8)
#undef INP_DECL_RUN_IMAGE

// Host-side entry points of one patch radius (engine_r<R>.cu).
struct EngineFns {
  size_t (*smem_bytes)(int srw);  // least dynamic shared memory the engine needs for this radius
  cudaError_t (*update_fast)(const ImgState& s, unsigned long long cond, int use_cond,
                             cudaStream_t st);
  cudaError_t (*prio_init)(const ImgState& s, cudaStream_t st);
  bool (*overlap_fits)(const ImgState& s, int tsize, size_t smem);
};
const EngineFns* engine_fns_r1();
const EngineFns* engine_fns_r2();
const EngineFns* engine_fns_r3();
const EngineFns* engine_fns_r4();
const EngineFns* engine_fns_r5();
const EngineFns* engine_fns_r6();
const EngineFns* engine_fns_r7();
const EngineFns* engine_fns_r8();

const EngineFns* engine_fns(int r);
// The engine kernel (engine_multi.cu); every launch takes engine_launch_smem()
// bytes, at least the largest engine_fns(r)->smem_bytes(srw) of its images.
cudaError_t engine_occupancy(size_t smem, int* blocks_per_sm);
// Dynamic shared memory of every engine launch: all an SM offers one CTA.
size_t engine_launch_smem();
cudaError_t engine_begin(const EngineArgs& ea, int n_teams, int grid, Ctrl* c, int limit, cudaStream_t st);
cudaError_t engine_end(const EngineArgs& ea, Ctrl* c, cudaStream_t st);
cudaError_t engine_launch(size_t smem, const EngineArgs& ea, int grid, cudaStream_t st);
int make_image_tmap(const ImgState& s, int srw, CUtensorMap* out);  // writes out[0], out[1]
int make_image_tmap_box(const ImgState& s, int box_w, int box_h, CUtensorMap* out);
cudaError_t launch_update_fast(const ImgState& s, unsigned long long cond, int use_cond,
                               cudaStream_t st);

}  // namespace inp
