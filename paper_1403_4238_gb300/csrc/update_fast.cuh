// Copy/update phase of one fill iteration for patch radius R <= 8.
//
// Sec. 3: after findBestPatch the pixels of Psi_q~ are copied into the
// unknown part of Psi_p^, those pixels take the confidence C(p^), and the
// priorities P(p) = C(p) D(p) (Eq. 1-2) that depend on them are recomputed
// before the next target is selected.  Everything involved lies within 3R+2
// pixels of p^, so that neighbourhood is staged in shared memory.
//
// Which pixels are filled (Psi_p^ n Omega) and the confidence they receive
// (C(p^)) are known as soon as p^ is selected; only their colours depend on
// the search result q~.  So an iteration is cut into pieces by what they wait
// for, and by which warps run them (kEngThreads threads, one CTA):
//   all warps      spec_front: post-fill mask, filled set, post-fill front
//                  pixels within 2R+1 of p^ (from the staged neighbourhood);
//   warps 0-3      spec_chains: the confidence terms C(p) of those pixels,
//                  sequential FP64 sums in row-major patch order.  A dependent
//                  FP64 add takes 64 cycles here, so this is the longest piece
//                  (5.2k cycles at R = 4, 10.8k at R = 6, 18.5k at R = 8) and
//                  nothing but the priorities waits for it;
//   warps 4-14     meanwhile spec_rest (tile maxima of the last iteration, the
//                  best priority the fill cannot change, new validity counts,
//                  normals, isophotes the fill cannot change), then, once the
//                  search's key is there, update_work (copy, validity counts,
//                  isophotes of the new pixels, the strongest one of every
//                  front patch);
//   warp 15        meanwhile the last iteration's record, the search's keys
//                  (so that their polling waits for nothing else), and after
//                  the copy the fence that the publication needs;
//   all warps      update_prio: data terms, priorities, and the next target,
//                  which is the better of the window's best and the best
//                  outside it; then update_store and stage_next.
// Before this split the chains, the key gathering and the update ran one
// after another on all warps: 12.6 us an iteration at 512x384, R = 4 (now 6.8).
#pragma once
#include "inpaint_internal.cuh"
#include "ptx.cuh"

namespace inp {

template <int R>
struct UpdGeom {
  static constexpr int P = 2 * R + 1;
  static constexpr int RB = 3 * R + 2;  // staged neighbourhood radius
  static constexpr int NS = 2 * RB + 1;
  static constexpr int R2 = 2 * R + 1;  // priorities that can change
  static constexpr int NW = 2 * R2 + 1;
  static constexpr int NC = 4 * R + 1;  // validity counts that can change
  // level-0 / level-1 priority tiles an NW x NW window can touch (per axis)
  static constexpr int KT0 = (NW + kT0 - 2) / kT0 + 1;
  static constexpr int KT1 = 2;
  static_assert(KT0 * KT0 + KT1 * KT1 + 1 <= 32, "one lane per segment");
};

// The level-0 and level-1 tiles that the window of (px, py) touches.
struct TouchedTiles {
  int tx0, ty0, ntx, nty, ux0, uy0, nux, nuy;
};
template <int R>
__device__ __forceinline__ TouchedTiles touched_tiles(const ImgState& s, int px, int py) {
  static_assert(kT0 == 16 && kT1 == 16, "tile shifts");
  constexpr int R2 = UpdGeom<R>::R2;
  TouchedTiles t;
  t.tx0 = max(0, px - R2) >> 4;
  t.ty0 = max(0, py - R2) >> 4;
  const int tx1 = min(s.W - 1, px + R2) >> 4, ty1 = min(s.H - 1, py + R2) >> 4;
  t.ntx = tx1 - t.tx0 + 1;
  t.nty = ty1 - t.ty0 + 1;
  t.ux0 = t.tx0 >> 4;
  t.uy0 = t.ty0 >> 4;
  t.nux = (tx1 >> 4) - t.ux0 + 1;
  t.nuy = (ty1 >> 4) - t.uy0 + 1;
  return t;
}

constexpr int kChainThreads = 128;  // warps 0-3: the FP64 chains, then the priorities
constexpr int kMidThreads = 352;    // warps 4-14
constexpr int kMidWarps = kMidThreads / 32;
constexpr int kRecThread = kEngThreads - 32;  // first thread of warp 15

// Named barriers: of warps 4-14, of those with warp 15 (the chains join
// neither), of those with the chain warps that had no chains and took
// isophotes instead (which only arrive), and one that warp 15 only arrives at
// when the integral image is there.
__device__ __forceinline__ void mid_sync() { asm volatile("barrier.sync 1, 352;" ::: "memory"); }
__device__ __forceinline__ void work_sync() { asm volatile("barrier.sync 2, 384;" ::: "memory"); }
__device__ __forceinline__ void iso_arrive(int chain_threads) {
  asm volatile("barrier.arrive 3, %0;" ::"r"(kMidThreads + kChainThreads - chain_threads) : "memory");
}
__device__ __forceinline__ void iso_sync(int chain_threads) {
  asm volatile("barrier.sync 3, %0;" ::"r"(kMidThreads + kChainThreads - chain_threads) : "memory");
}
__device__ __forceinline__ void fsat_arrive() { asm volatile("barrier.arrive 4, 384;" ::: "memory"); }
__device__ __forceinline__ void fsat_sync() { asm volatile("barrier.sync 4, 384;" ::: "memory"); }

template <int R>
struct __align__(16) UpdSmem {
  using G = UpdGeom<R>;
  double cf[G::NS * G::NS];   // C of the known pixels, +0.0 elsewhere
  double sC[2][G::NW * G::NW];   // (by iteration parity) post-fill C(p) of the front pixels
                                 // (window index), then the bits of their priority keys
  int snrm[G::NW * G::NW];    // packed normal, or kSpecNotFront / kSpecOutside
  uint32_t ikey[G::NS * G::NS];  // isophote key at a local pixel (isophote_key), 0 if not eligible
  uint32_t dotc[G::NW * G::NW];  // k-th front pixel: |isophote . normal| | normal length code << 12
  int cnt[G::NC * G::NC];        // validity counts after the fill, -1: not changed by it
  int fsat[(G::P + 1) * (G::P + 1)];
  uint8_t om[G::NS * G::NS];  // 0 known, 1 Omega, 2 outside the image
  uint8_t gr[G::NS * G::NS];
  uint8_t filled[G::P * G::P];
  uint16_t list[2][G::NW * G::NW];  // (by parity) front pixels (window index)
  int nlist[2];
  int iso_next;  // next chunk of the isophotes the fill cannot change
  // the staged target: centre, iteration, C(p^), priority key
  int nx_px, nx_py, nx_it;
  double nx_cp;
  unsigned long long nx_key;
  // the iteration being applied, and its record
  int px, py, it, qx, qy, n_filled, n_known, n_cand, newly, remaining;
  uint32_t ssd;
  double pp, cp;
  int ok;           // the key is a source patch and the state is consistent
  int rec_pending;  // the record is not written yet
  // the best front pixel whose priority this iteration's fill cannot change
  // (outside the NW x NW window), and the selected next target
  unsigned long long out_key, next_key;
  int out_idx, out_y, next_idx;
  // per segment of spec_rest (touched level-0 tiles, touched level-1 tiles,
  // the rest) the best priority that the iteration leaves alone; the touched
  // tiles' new maxima are these and the new keys (update_tiles), and are due
  // while tiles_pending
  PrioBest seg[32];
  int tiles_pending, tile_px, tile_py, tile_par;  // the iteration they belong to
  unsigned long long t_start, t_keys;  // global timer: round start, keys gathered
  PrioBest red_pb[4];
  // the data term's divisors: s = sqrt(nn) for the 14 normal lengths, their
  // reciprocals and that of 510 (stage_dterm, once per launch)
  double dsq[kDTabRows], dinv[kDTabRows], dinv510, dinvP;  // dinvP: of P^2
};

// a / b rounded to nearest for a divisor known in advance, from y = RN(1/b):
// q0 = RN(a y), the remainder a - q0 b exact by one FMA, then the corrected
// quotient RN(q0 + r y) (Markstein's division, IBM J. Res. Dev. 34(1), 1990).
// Used only where it is checked to equal RN(a / b) for every input: the data
// term below, for all 14 normal lengths and all 2041 dot products.
__device__ inline double div_known(double a, double b, double y) {
  const double q0 = __dmul_rn(a, y);
  const double r = __fma_rn(-q0, b, a);
  return __fma_rn(r, y, q0);
}

// The data term's divisors into shared memory (threads 0-14; a barrier must
// follow before data_term_known reads them): correctly rounded square roots
// and reciprocals, the same values the host computes.
template <int R>
__device__ inline void stage_dterm(UpdSmem<R>& sm) {
  const int t = threadIdx.x;
  if (t < kDTabRows) {
    const double s = __dsqrt_rn((double)dtab_nn(t));
    sm.dsq[t] = s;
    sm.dinv[t] = __ddiv_rn(1.0, s);
  } else if (t == kDTabRows) {
    sm.dinv510 = __ddiv_rn(1.0, 510.0);
    sm.dinvP = __ddiv_rn(1.0, (double)(UpdGeom<R>::P * UpdGeom<R>::P));
  }
}

// D of Eq. 2 for a normal of length code c, the same bits as
// data_term_direct: fl(fl(dot / s) / 510) (0 for a zero normal, whose dot is
// 0, under any code), both
// quotients by div_known with the staged divisors (no global load on the
// update's path).
template <int R>
__device__ inline double data_term_known(const UpdSmem<R>& sm, int dot, int c) {
  return div_known(div_known((double)dot, sm.dsq[c], sm.dinv[c]), 510.0, sm.dinv510);
}

// Sobel normal of the Omega indicator at local (lx, ly) = image (x, y),
// replicated image borders, packed as the length code << 16 | (nx + 8) << 8 |
// (ny + 8).
template <int R>
__device__ inline int normal_local(const UpdSmem<R>& sm, const ImgState& s, int lx, int ly, int x,
                                   int y) {
  constexpr int NS = UpdGeom<R>::NS;
  const int xl = x > 0 ? -1 : 0, xr = x < s.W - 1 ? 1 : 0;
  const int yu = y > 0 ? -1 : 0, yd = y < s.H - 1 ? 1 : 0;
  auto M = [&](int ox, int oy) { return sm.om[(ly + oy) * NS + lx + ox] == 1 ? 1 : 0; };
  const int m_lu = M(xl, yu), m_cu = M(0, yu), m_ru = M(xr, yu);
  const int m_lc = M(xl, 0), m_rc = M(xr, 0);
  const int m_ld = M(xl, yd), m_cd = M(0, yd), m_rd = M(xr, yd);
  const int nx = (m_ru + 2 * m_rc + m_rd) - (m_lu + 2 * m_lc + m_ld);
  const int ny = (m_ld + 2 * m_cd + m_rd) - (m_lu + 2 * m_cu + m_ru);
  return (dtab_code(nx * nx + ny * ny) << 16) | ((nx + 8) << 8) | (ny + 8);
}

// The sum of C(p) in Eq. 2: the known part of Psi_p in row-major order (dy
// outer, dx inner, one addition at a time).
// Unknown and out-of-image entries hold +0.0 in sm.cf, and adding +0.0 to a
// non-negative double leaves it unchanged, so summing every entry gives
// exactly the sum over the known pixels.
// The next row's entries are loaded, into registers of their own, while a row
// is summed: the chain then runs at the FP64 unit's 64 cycles an addition
// (loading each entry over the one just added: 90).
template <int R>
__device__ inline double conf_local(const UpdSmem<R>& sm, int lx, int ly) {
  constexpr int NS = UpdGeom<R>::NS, P = UpdGeom<R>::P;
  const double* row = &sm.cf[(ly - R) * NS + lx - R];
  double a[P], b[P], sum = 0.0;
#pragma unroll
  for (int i = 0; i < P; ++i) a[i] = row[i];
#pragma unroll 1
  for (int dy = 0; dy < R; ++dy) {  // rows 2 dy and 2 dy + 1
    row += NS;
#pragma unroll
    for (int i = 0; i < P; ++i) b[i] = row[i];
#pragma unroll
    for (int i = 0; i < P; ++i) sum = __dadd_rn(sum, a[i]);
    row += NS;
#pragma unroll
    for (int i = 0; i < P; ++i) a[i] = row[i];
#pragma unroll
    for (int i = 0; i < P; ++i) sum = __dadd_rn(sum, b[i]);
  }
#pragma unroll
  for (int i = 0; i < P; ++i) sum = __dadd_rn(sum, a[i]);
  return sum;
}

// In-image pixels of the patch at (x, y).
template <int R>
__device__ inline int patch_area(const ImgState& s, int x, int y) {
  return (min(x + R, s.W - 1) - max(x - R, 0) + 1) * (min(y + R, s.H - 1) - max(y - R, 0) + 1);
}

__device__ inline int dot_abs(int gx, int gy, int nrm) {
  const int nx = ((nrm >> 8) & 0xff) - 8, ny = (nrm & 0xff) - 8;
  const int d = (-gy) * nx + gx * ny;
  return d < 0 ? -d : d;
}

__device__ inline int nn_of(int nrm) {
  const int nx = ((nrm >> 8) & 0xff) - 8, ny = (nrm & 0xff) - 8;
  return nx * nx + ny * ny;
}

// D of Eq. 2 evaluated directly (initialisation).
__device__ inline double data_term_direct(int dot, int nn) {
  if (nn == 0) return 0.0;
  return __ddiv_rn(__ddiv_rn((double)dot, __dsqrt_rn((double)nn)), 510.0);
}


// Stages the NS x NS neighbourhood of (cx, cy): mask (2 outside the image),
// grey levels and confidences (+0.0 under Omega and outside).  NT threads;
// each has up to U entries' loads in flight together, and `meanwhile` runs
// before the first use of them.  FILL: the state after the fill of Psi at
// (cx, cy), whose unknown pixels take the confidence *cp, and the filled
// flags.
template <int R, int NT, bool FILL, class F>
__device__ inline void stage_nbhd(const ImgState& s, int cx, int cy, UpdSmem<R>& sm, const double* cp, F&& meanwhile) {
  using G = UpdGeom<R>;
  constexpr int RB = G::RB, NS = G::NS, P = G::P;
  constexpr int U = (NS * NS + NT - 1) / NT < 6 ? (NS * NS + NT - 1) / NT : 6;
  double cfill = 0.0;
  if (FILL) cfill = __ldcg(cp);
  if ((int)threadIdx.x >= NS * NS) meanwhile();  // (more threads than entries)
#pragma unroll 1
  for (int i0 = threadIdx.x; i0 < NS * NS; i0 += U * NT) {
    uint8_t o[U], g[U];
    double cf[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * NT;
      const int x = cx - RB + i % NS, y = cy - RB + i / NS;
      o[u] = 2;
      g[u] = 0;
      cf[u] = 0.0;
      if (i < NS * NS && x >= 0 && x < s.W && y >= 0 && y < s.H) {
        const int q = y * s.W + x;
        o[u] = __ldcg(&s.omega[q]);
        g[u] = __ldcg(&s.gray[q]);
        cf[u] = __ldcg(&s.conf[q]);  // read unconditionally, kept for known pixels
      }
    }
    if (i0 == (int)threadIdx.x) meanwhile();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * NT;
      if (i >= NS * NS) break;
      const int dx = i % NS - RB, dy = i / NS - RB;
      double c = o[u] ? 0.0 : cf[u];
      if (FILL && abs(dx) <= R && abs(dy) <= R) {
        const bool f = o[u] == 1;
        sm.filled[(dy + R) * P + dx + R] = f;
        if (f) {
          o[u] = 0;
          c = cfill;
        }
      }
      sm.om[i] = o[u];
      sm.gr[i] = g[u];
      sm.cf[i] = c;
    }
  }
}

// Isophote candidate at local pixel (lx, ly): eligible when it and its four
// neighbours are known.  The key orders candidates by |grad|^2 of the
// central-difference grey gradient, then by the lowest local index (the first
// in row-major order of any patch): (|grad|^2 + 1) << 12 | (4095 - index).
template <int R>
__device__ inline uint32_t isophote_key(const UpdSmem<R>& sm, int lx, int ly) {
  constexpr int NS = UpdGeom<R>::NS;
  static_assert(NS * NS <= 4096, "local index fits in 12 bits");
  const int i = ly * NS + lx;
  if (lx < 1 || lx >= NS - 1 || ly < 1 || ly >= NS - 1) return 0u;
  // all nine reads issued together (no short-circuit chain of loads)
  const int o = sm.om[i] | sm.om[i - 1] | sm.om[i + 1] | sm.om[i - NS] | sm.om[i + NS];
  const int gx = (int)sm.gr[i + 1] - (int)sm.gr[i - 1];
  const int gy = (int)sm.gr[i + NS] - (int)sm.gr[i - NS];
  return o == 0 ? ((uint32_t)(gx * gx + gy * gy + 1) << 12) | (uint32_t)(4095 - i) : 0u;
}

// |grad . normal| (the data term's numerator) of the isophote with key `ik`.
template <int R>
__device__ inline int isophote_dot(const UpdSmem<R>& sm, uint32_t ik, int nrm) {
  constexpr int NS = UpdGeom<R>::NS;
  if (ik == 0u) return 0;
  const int l = 4095 - (int)(ik & 4095u);
  return dot_abs((int)sm.gr[l + 1] - (int)sm.gr[l - 1], (int)sm.gr[l + NS] - (int)sm.gr[l - NS], nrm);
}

__device__ inline bool front_local(const uint8_t* om, int l, int NS) {
  // the five reads are independent (no short-circuit chain of loads)
  const int c = om[l], a = om[l - 1], b = om[l + 1], u = om[l - NS], d = om[l + NS];
  return c == 1 && (a == 0 || b == 0 || u == 0 || d == 0);
}

// The isophotes the fill cannot change: it changes grey levels and the mask
// only inside Psi_p^, so a candidate can change only in the box of Chebyshev
// radius R + 1 around p^.  Handed out in chunks of 64 from sm.iso_next: the
// chain warps without chains, then the others as they get to it.  Whole warps.
template <int R>
__device__ inline void static_isophotes(UpdSmem<R>& sm) {
  constexpr int NS = UpdGeom<R>::NS, RB = UpdGeom<R>::RB, RR = R + 1;
  const int lane = threadIdx.x & 31;
  while (true) {
    int base = 0;
    if (lane == 0) base = atomicAdd(&sm.iso_next, 64);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= NS * NS) break;
#pragma unroll
    for (int h = 0; h < 64; h += 32) {
      const int i = base + h + lane, lx = i % NS, ly = i / NS;
      if (i < NS * NS && (abs(lx - RB) > RR || abs(ly - RB) > RR)) sm.ikey[i] = isophote_key<R>(sm, lx, ly);
    }
    __syncwarp();
  }
}

// Initial priorities of the front pixels (every key is 0 before), one CTA per
// NW x NW window of the image; direct evaluation of every term.  Most windows
// hold no front pixel, which a look at their Omega bits shows; in the others
// the front pixels go to the threads one by one, so that their chains of
// additions run side by side (evaluated where they lay, every window staged:
// 23 us at 512x384 r 4, 93 us at 1920x1080 r 6).
template <int R>
__global__ void __launch_bounds__(256, 2) k_prio_init_fast(ImgState s) {
  using G = UpdGeom<R>;
  constexpr int RB = G::RB, NS = G::NS, R2 = G::R2, NW = G::NW;
  extern __shared__ __align__(128) uint8_t sm_raw[];
  UpdSmem<R>& sm = *reinterpret_cast<UpdSmem<R>*>(sm_raw);
  const int cx = R2 + blockIdx.x * NW, cy = R2 + blockIdx.y * NW;
  constexpr int NWD = (NW + 62) / 32;  // words that hold a window row, at most
  bool any = false;
  if ((int)threadIdx.x < NW * NWD) {
    const int y = cy - R2 + (int)threadIdx.x / NWD, w = ((cx - R2) >> 5) + (int)threadIdx.x % NWD, ow = obits_pitch(s.W);
    if (y < s.H && w < ow && 32 * w <= cx + R2) {
      const uint32_t* row = s.obits + (size_t)y * ow + w;
      const uint32_t o = row[0];
      const uint32_t up = y > 0 ? row[-ow] : ~0u, down = y + 1 < s.H ? row[ow] : ~0u;
      const uint32_t left = o << 1 | (w > 0 ? row[-1] >> 31 : 1u), right = o >> 1 | (w + 1 < ow ? row[1] << 31 : 1u << 31);
      // the pixels of the window: columns [cx - R2, min(cx + R2, W - 1)]
      const int lo = max(cx - R2 - 32 * w, 0), hi = min(min(cx + R2, s.W - 1) - 32 * w, 31);
      const uint32_t in = (~0u << lo) & (~0u >> (31 - hi));
      any = (o & ~(up & down & left & right) & in) != 0u;
    }
  }
  if (threadIdx.x == 0) sm.nlist[0] = 0;
  if (!__syncthreads_or(any)) return;
  stage_nbhd<R, 256, false>(s, cx, cy, sm, nullptr, [] {});
  __syncthreads();
#pragma unroll 1
  for (int i = threadIdx.x; i < NS * NS; i += 256) sm.ikey[i] = isophote_key<R>(sm, i % NS, i / NS);
#pragma unroll 1
  for (int i = threadIdx.x; i < NW * NW; i += 256) {
    const int l = (RB + i / NW - R2) * NS + RB + i % NW - R2;
    if (front_local(sm.om, l, NS)) sm.list[0][atomicAdd(&sm.nlist[0], 1)] = (uint16_t)i;
  }
  __syncthreads();
  const int n = sm.nlist[0];
#pragma unroll 1
  for (int k = threadIdx.x; k < n; k += 256) {
    const int i = sm.list[0][k], wx = i % NW - R2, wy = i / NW - R2;
    const int lx = RB + wx, ly = RB + wy, l = ly * NS + lx, x = cx + wx, y = cy + wy;
    const double c = __ddiv_rn(conf_local<R>(sm, lx, ly), (double)patch_area<R>(s, x, y));
    const int nrm = normal_local<R>(sm, s, lx, ly, x, y);
    uint32_t ik = 0u;
#pragma unroll 1
    for (int dy = -R; dy <= R; ++dy) {
#pragma unroll
      for (int dx = -R; dx <= R; ++dx) ik = max(ik, sm.ikey[l + dy * NS + dx]);
    }
    const double d = data_term_direct(isophote_dot<R>(sm, ik, nrm), nn_of(nrm));
    const size_t p = (size_t)y * s.W + x;
    s.prio[p] = (unsigned long long)__double_as_longlong(__dmul_rn(c, d)) + 1ull;
    s.pconf[p] = c;
  }
}

// The iteration state from the control block and the neighbourhood of its
// target, for the first iteration of a launch.  Whole block; the caller's
// barrier makes it visible.  `overlap_counts`: the partial-overlap search
// counted its admissible candidates in ctrl->n_adm.
template <int R>
__device__ inline void stage_first(const ImgState& s, UpdSmem<R>& sm, bool overlap_counts) {
  const Ctrl* c = s.ctrl;
  const int px = __ldcg(&c->px), py = __ldcg(&c->py);
  stage_dterm<R>(sm);
  if (threadIdx.x == kEngThreads - 1) {
    sm.nx_px = px;
    sm.nx_py = py;
    sm.nx_it = __ldcg(&c->iter);
    sm.nx_cp = __ldcg(&c->conf);
    sm.nx_key = (unsigned long long)__double_as_longlong(__ldcg(&c->prio)) + 1ull;
    sm.n_cand = overlap_counts ? __ldcg(&c->n_adm) : __ldcg(&c->n_valid);
    sm.remaining = __ldcg(&c->remaining);
    sm.newly = 0;
    sm.nlist[0] = sm.nlist[1] = 0;
    sm.rec_pending = 0;
    sm.tiles_pending = 0;
    sm.iso_next = 0;
  }
  stage_nbhd<R, kEngThreads, true>(s, px, py, sm, &c->conf, [] {});
}

// The next iteration's input, once the next target idx (in row npy) has been
// selected: its neighbourhood after its fill, and in sm.nx_* its centre,
// iteration number and confidence.  `meanwhile` runs while the loads are in
// flight.  Whole block; the caller's barrier makes it visible.
template <int R, class F>
__device__ inline void stage_next(const ImgState& s, unsigned long long key, int idx, int npy, UpdSmem<R>& sm,
                                  F&& meanwhile) {
  const int npx = idx - npy * s.W;
  const bool mine = threadIdx.x == kEngThreads - 1;  // a thread with the fewest staging entries
  double ncp = 0.0;
  if (mine) ncp = __ldcg(&s.pconf[idx]);
  stage_nbhd<R, kEngThreads, true>(s, npx, npy, sm, &s.pconf[idx], meanwhile);
  if (mine) {
    sm.nx_px = npx;
    sm.nx_py = npy;
    sm.nx_it = sm.it + 1;
    sm.nx_cp = ncp;
    sm.nx_key = key;
    sm.nlist[(sm.it + 1) & 1] = 0;
    sm.iso_next = 0;
  }
}

// The post-fill front of the window from the staged neighbourhood.  Whole
// block; ends with a __syncthreads.
template <int R>
__device__ inline void spec_front(UpdSmem<R>& sm) {
  using G = UpdGeom<R>;
  constexpr int RB = G::RB, NS = G::NS, R2 = G::R2, NW = G::NW;
  const int tid = threadIdx.x, lane = tid & 31, par = sm.nx_it & 1;
#pragma unroll 1
  for (int i0 = 0; i0 < NW * NW; i0 += kEngThreads) {
    const int i = i0 + tid;
    bool fr = false;
    if (i < NW * NW) {
      const int l = (RB + i / NW - R2) * NS + RB + i % NW - R2;
      fr = front_local(sm.om, l, NS);
      sm.snrm[i] = sm.om[l] != 2 ? kSpecNotFront : kSpecOutside;  // front pixels: overwritten by spec_rest
    }
    const unsigned bal = __ballot_sync(0xffffffffu, fr);
    if (bal != 0u) {
      int base = 0;
      if (lane == 0) base = atomicAdd(&sm.nlist[par], __popc(bal));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (fr) sm.list[par][base + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)i;
    }
  }
  __syncthreads();
}

// Confidence terms of the front pixels (warps 0-3): one dependent row-major
// chain per pixel, packed into as few warps as the front needs: up to three
// warps of chains still run at the 64 cycles of one dependent add, four at 76
// (the unit takes a warp instruction about every 19 cycles whatever the
// active lanes).
__device__ __forceinline__ int chain_threads(int nfront) { return nfront <= 96 ? (nfront + 31) & ~31 : kChainThreads; }

template <int R>
__device__ inline void spec_chains(const ImgState& s, UpdSmem<R>& sm) {
  using G = UpdGeom<R>;
  constexpr int RB = G::RB, R2 = G::R2, NW = G::NW, P2 = G::P * G::P;
  const int par = sm.nx_it & 1, nfront = sm.nlist[par], nt = chain_threads(nfront);
  if ((int)threadIdx.x >= nt) {
    static_isophotes<R>(sm);
    iso_arrive(nt);
    return;
  }
#pragma unroll 1
  for (int k = threadIdx.x; k < nfront; k += nt) {
    const int i = sm.list[par][k];
    const int wx = i % NW - R2, wy = i / NW - R2;
    const int n_in = patch_area<R>(s, sm.nx_px + wx, sm.nx_py + wy);
    const double sum = conf_local<R>(sm, RB + wx, RB + wy), q = div_known(sum, (double)P2, sm.dinvP);
    // a second correction by the same reciprocal: after the first the
    // quotient is within an ulp, so this one rounds it correctly (Markstein),
    // unless the remainder underflows or is inf - inf: sums outside
    // [2^-830, inf) (an imported state's) and clipped patches divide.  (The range
    // by the sum's high word: an FP64 compare is a turn of the busy unit.)
    const double c = __fma_rn(__fma_rn(-q, (double)P2, sum), sm.dinvP, q);
    constexpr unsigned kLo = (1023u - 830u) << 20, kInf = 2047u << 20;
    const bool in_range = (unsigned)__double2hiint(sum) - kLo < kInf - kLo;
    sm.sC[par][i] = n_in == P2 && in_range ? c : __ddiv_rn(sum, (double)n_in);
  }
}

// Integral image of the filled flags of Psi_p^ (validity-count
// decrements); one warp.
template <int R>
__device__ inline void warp_fsat(UpdSmem<R>& sm) {
  constexpr int P = UpdGeom<R>::P, P1 = P + 1;
  const int lane = threadIdx.x & 31;
  if (lane <= P) {
    sm.fsat[lane] = 0;
    sm.fsat[lane * P1] = 0;
  }
  __syncwarp();
  if (lane < P) {
    int run = 0;
#pragma unroll 1
    for (int u = 0; u < P; ++u) {
      run += sm.filled[lane * P + u];
      sm.fsat[(lane + 1) * P1 + u + 1] = run;
    }
  }
  __syncwarp();
  if (lane < P) {
    int run = 0;
#pragma unroll 1
    for (int v = 1; v <= P; ++v) {
      run += sm.fsat[v * P1 + lane + 1];
      sm.fsat[v * P1 + lane + 1] = run;
    }
  }
}

// The engine's phase clocks of the iteration applied last (round start to
// keys, keys to the next round's start), by the thread that also writes the
// records.
template <int R>
__device__ inline void update_times(const ImgState& s, UpdSmem<R>& sm) {
  const unsigned long long now = globaltimer();
  if (sm.rec_pending) {
    atomicAdd(&s.ctrl->t_search, sm.t_keys - sm.t_start);
    atomicAdd(&s.ctrl->t_update, now - sm.t_keys);
    atomicAdd(&s.ctrl->timed_iters, 1);
  }
  sm.t_start = now;
}

// Writes the record of the iteration applied last (trace, counters) and the
// next target in the control block; one thread.  Nothing else reads these
// while a launch runs, so the persistent engine writes them during the next
// iteration's search.
template <int R>
__device__ inline void write_record(const ImgState& s, UpdSmem<R>& sm, bool overlap_counts) {
  Ctrl* c = s.ctrl;
  inpaint_step_info e;
  e.iter = sm.it;
  e.px = sm.px;
  e.py = sm.py;
  e.qx = sm.qx;
  e.qy = sm.qy;
  e.ssd = sm.ssd;
  e.priority = sm.pp;
  e.confidence = sm.cp;
  e.filled = sm.n_filled;
  e.remaining = sm.remaining;
  e.n_known = sm.n_known;
  e.n_cand = sm.n_cand;
  c->last = e;
  if (sm.it < s.trace_cap) s.trace[sm.it] = e;
  c->remaining = sm.remaining;
  c->iter = sm.it + 1;
  atomicAdd(&c->evals, (unsigned long long)sm.n_cand * (unsigned long long)sm.n_known);
  sm.n_cand += sm.newly;
  sm.newly = 0;
  c->n_valid = sm.n_cand;
  if (overlap_counts) c->n_adm = 0;  // the next search counts afresh
  if (sm.remaining > 0 && sm.next_key != 0ull) {
    c->px = sm.next_idx % s.W;
    c->py = sm.next_idx / s.W;
    c->prio = __longlong_as_double((long long)(sm.next_key - 1ull));
    c->conf = __ldcg(&s.pconf[sm.next_idx]);
  } else {
    c->px = -1;
    c->py = -1;
    if (sm.remaining > 0) c->status = INPAINT_ERR_INTERNAL;  // Omega non-empty but no front
  }
  sm.rec_pending = 0;
}

// The tile maxima of the last update: for a level-0 tile its window touched,
// the best of the pixels outside the window (seg, kept from spec_rest) and of
// the new keys; for a level-1 tile, the best of its other level-0 tiles (seg)
// and of those.  Warps 4-14; a barrier of theirs follows the writes.
template <int R>
__device__ inline void update_tiles(const ImgState& s, UpdSmem<R>& sm) {
  constexpr int R2 = UpdGeom<R>::R2, NW = UpdGeom<R>::NW;
  const int lane = threadIdx.x & 31, wid = ((int)threadIdx.x - kChainThreads) >> 5;
  const int par = sm.tile_par, x0 = sm.tile_px - R2, y0 = sm.tile_py - R2, W = s.W;
  const TouchedTiles g = touched_tiles<R>(s, sm.tile_px, sm.tile_py);
  const int n0 = g.ntx * g.nty, nfront = sm.nlist[par];
#pragma unroll 1
  for (int t = wid; t < n0; t += kMidWarps) {
    const int v = t / g.ntx, tx = g.tx0 + t - v * g.ntx, ty = g.ty0 + v;
    unsigned long long k = sm.seg[t].key;
    int idx = sm.seg[t].idx;
#pragma unroll 1
    for (int e = lane; e < nfront; e += 32) {
      const int i = sm.list[par][e], x = x0 + i % NW, y = y0 + i / NW;
      if ((x >> 4) == tx && (y >> 4) == ty)
        prio_take(k, idx, (unsigned long long)__double_as_longlong(sm.sC[par][i]), y * W + x);
    }
    __syncwarp();
    warp_best_prio(k, idx);
    if (lane == 0) {
      PrioBest& e = s.tiles0[ty * s.t0x + tx];
      sm.seg[t].key = e.key = k;
      sm.seg[t].idx = e.idx = idx;
    }
  }
  mid_sync();
  if (wid == 0) {
    // lane t: the new maximum of level-0 tile t, and the level-1 tile it is in
    const int v = lane / g.ntx, tx = g.tx0 + lane - v * g.ntx, ty = g.ty0 + v;
    const bool in = lane < n0;
    const int mine = in ? ((ty >> 4) - g.uy0) * g.nux + (tx >> 4) - g.ux0 : -1;
    const unsigned long long k0 = in ? sm.seg[lane].key : 0ull;
    const int i0 = in ? sm.seg[lane].idx : 0x7fffffff;
#pragma unroll 1
    for (int u = 0; u < g.nux * g.nuy; ++u) {
      unsigned long long k = mine == u ? k0 : 0ull;
      int idx = mine == u ? i0 : 0x7fffffff;
      if (lane == 31) {  // (n0 <= 16) the level-1 tile's other level-0 tiles
        k = sm.seg[n0 + u].key;
        idx = sm.seg[n0 + u].idx;
      }
      warp_best_prio(k, idx);
      if (lane == 0) {
        const int uy = g.uy0 + (u >= g.nux ? 1 : 0), ux = g.ux0 + u - (u >= g.nux ? g.nux : 0);
        s.tiles1[uy * s.t1x + ux].key = k;
        s.tiles1[uy * s.t1x + ux].idx = idx;
      }
    }
  }
  __syncwarp();
  mid_sync();
}

// The best priority that the fill of (px, py) leaves alone, by segments: the
// pixels outside the window of each level-0 tile it touches, the untouched
// level-0 tiles of each level-1 tile it touches, and the untouched level-1
// tiles; one warp per segment.  Warps 4-14.  (A warp's lanes are brought
// together after the predicated loads and at the end of each branch: left to
// drift apart they took the keys one lane set after the other, 2.5k cycles
// of the round.)
template <int R>
__device__ inline void scan_segments(const ImgState& s, UpdSmem<R>& sm, const TouchedTiles& g, int px, int py) {
  constexpr int R2 = UpdGeom<R>::R2;
  const int lane = threadIdx.x & 31, W = s.W, H = s.H;
  const int n0 = g.ntx * g.nty, nseg = n0 + g.nux * g.nuy + 1;
#pragma unroll 1
  for (int e = ((int)threadIdx.x - kChainThreads) >> 5; e < nseg; e += kMidWarps) {
    unsigned long long k = 0ull;
    int idx = 0x7fffffff;
    if (e < n0) {
      const int v = e / g.ntx, xt = (g.tx0 + e - v * g.ntx) * kT0 + (lane & 15), yt = (g.ty0 + v) * kT0 + (lane >> 4);
      unsigned long long kk[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int y = yt + 2 * j;
        const bool use = xt < W && y < H && (abs(xt - px) > R2 || abs(y - py) > R2);
        kk[j] = use ? __ldcg(&s.prio[y * W + xt]) : 0ull;
      }
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 8; ++j) prio_take(k, idx, kk[j], (yt + 2 * j) * W + xt);
      __syncwarp();
    } else if (e < nseg - 1) {
      const int u = e - n0, v = u >= g.nux ? 1 : 0;
      const int tx = (g.ux0 + u - v * g.nux) * kT1 + (lane & 15);
      const int ty = (g.uy0 + v) * kT1 + (lane >> 4);
      const bool in_x = tx >= g.tx0 && tx < g.tx0 + g.ntx;
      uint4 b[8];  // all eight loads in flight (one after the other: 4.3k cycles)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int yy = ty + 2 * j;
        const bool touched = in_x && yy >= g.ty0 && yy < g.ty0 + g.nty;
        b[j] = tx < s.t0x && yy < s.t0y && !touched
                   ? __ldcg(reinterpret_cast<const uint4*>(&s.tiles0[yy * s.t0x + tx]))
                   : make_uint4(0u, 0u, 0x7fffffffu, 0u);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        prio_take(k, idx, ((unsigned long long)b[j].y << 32) | b[j].x, (int)b[j].z);
      __syncwarp();
    } else {
      const int n1 = s.t1x * s.t1y;
#pragma unroll 1
      for (int j = lane; j < n1; j += 32) {
        const int uy = j / s.t1x, ux = j - uy * s.t1x;
        if (ux >= g.ux0 && ux < g.ux0 + g.nux && uy >= g.uy0 && uy < g.uy0 + g.nuy) continue;
        prio_take(k, idx, __ldcg(&s.tiles1[j].key), __ldcg(&s.tiles1[j].idx));
      }
    }
    __syncwarp();
    warp_best_prio(k, idx);
    if (lane == 0) {
      sm.seg[e].key = k;
      sm.seg[e].idx = idx;
    }
  }
}

// What warps 4-14 do while the search and the chains run.
template <int R>
__device__ inline void spec_rest(const ImgState& s, UpdSmem<R>& sm) {
  using G = UpdGeom<R>;
  constexpr int P = G::P, RB = G::RB, R2 = G::R2, NW = G::NW, NC = G::NC, P1 = P + 1;
  const int px = sm.nx_px, py = sm.nx_py, t0 = (int)threadIdx.x - kChainThreads, W = s.W, H = s.H;
#pragma unroll 1
  for (int j = t0; j < NC * NC; j += kMidThreads) {
    const int x = px + j % NC - 2 * R, y = py + j / NC - 2 * R;
    const bool ok = x >= 0 && x < W && y >= 0 && y < H;
    cp_async4(&sm.cnt[j], ok ? &s.count[y * s.pitch + x] : s.count, ok);
  }
  // (every thread reads the flag before update_tiles' barriers, which precede its reset)
  if (sm.tiles_pending) update_tiles<R>(s, sm);
  const TouchedTiles g = touched_tiles<R>(s, px, py);
  scan_segments<R>(s, sm, g, px, py);
  // normals of the front pixels
  const int par = sm.nx_it & 1, nfront = sm.nlist[par];
#pragma unroll 1
  for (int k = t0; k < nfront; k += kMidThreads) {
    const int i = sm.list[par][k];
    const int wx = i % NW - R2, wy = i / NW - R2;
    sm.snrm[i] = normal_local<R>(sm, s, RB + wx, RB + wy, px + wx, py + wy);
  }
  __syncwarp();
  static_isophotes<R>(sm);
  cp_async_wait_all();
  __syncwarp();
  iso_sync(chain_threads(nfront));
  if (t0 < 32) {
    const int nseg = g.ntx * g.nty + g.nux * g.nuy + 1;
    unsigned long long k = t0 < nseg ? sm.seg[t0].key : 0ull;
    int idx = t0 < nseg ? sm.seg[t0].idx : 0x7fffffff;
    warp_best_prio(k, idx);
    if (t0 == 0) {
      sm.out_key = k;
      sm.out_idx = idx;
      sm.out_y = idx / W;
      sm.tiles_pending = 0;
    }
  }
  // validity counts after the fill: the centre at (wx, wy) from p^ loses the
  // filled pixels of its patch (their integral image is warp 15's)
  __syncwarp();
  fsat_sync();
#pragma unroll 1
  for (int j = t0; j < NC * NC; j += kMidThreads) {
    const int jy = j / NC, wy = jy - 2 * R, wx = j - jy * NC - 2 * R;
    const int u0 = max(0, wx), u1 = min(P, wx + 2 * R + 1), v0 = max(0, wy), v1 = min(P, wy + 2 * R + 1);
    const int dec = sm.fsat[v1 * P1 + u1] - sm.fsat[v0 * P1 + u1] - sm.fsat[v1 * P1 + u0] + sm.fsat[v0 * P1 + u0];
    const int x = px + wx, y = py + wy;
    sm.cnt[j] = dec != 0 && x >= 0 && x < W && y >= 0 && y < H ? sm.cnt[j] - dec : -1;
  }
}

// Warp 15 meanwhile: the integral image of the filled flags, then (one thread)
// the last iteration's record and the scalars of the iteration on the staged
// target.  `before` (whole warp) runs before the record.
template <int R, class F>
__device__ inline void spec_record(const ImgState& s, UpdSmem<R>& sm, bool overlap_counts, F&& before) {
  constexpr int P = UpdGeom<R>::P;
  warp_fsat<R>(sm);
  __syncwarp();
  fsat_arrive();
  before();
  if (threadIdx.x != kRecThread) return;
  update_times<R>(s, sm);
  if (sm.rec_pending) write_record<R>(s, sm, overlap_counts);
  const int filled = sm.fsat[P * (P + 1) + P], W = s.W, H = s.H, px = sm.nx_px, py = sm.nx_py;
  sm.px = px;
  sm.py = py;
  sm.it = sm.nx_it;
  sm.cp = sm.nx_cp;
  sm.pp = __longlong_as_double((long long)(sm.nx_key - 1ull));
  sm.n_filled = filled;
  sm.remaining -= filled;
  sm.n_known = (min(px + R, W - 1) - max(px - R, 0) + 1) * (min(py + R, H - 1) - max(py - R, 0) + 1) - filled;
}

// The search's result (one thread): q~ and its SSD, or why there is none.
template <int R>
__device__ inline void set_source(const ImgState& s, UpdSmem<R>& sm, unsigned long long best, bool late) {
  int ok = 0;
  if (!late) {
    if (best == ~0ull) {
      s.ctrl->status = INPAINT_ERR_NO_SOURCE;
    } else if (sm.n_filled == 0) {
      s.ctrl->status = INPAINT_ERR_INTERNAL;  // p^ not in Omega
    } else {
      const int q = (int)(best & 0xffffffffull);
      sm.qy = q / s.W;
      sm.qx = q - sm.qy * s.W;
      sm.ssd = (uint32_t)(best >> 32);
      ok = 1;
    }
  }
  sm.ok = ok;
}

// What a thread of warps 4-14 copies, worked out before the search's key is
// there: one thread copies a pixel of Psi_p^ n Omega; when there are two
// threads per pixel, the second one writes its planes (they take as long as
// all the rest).
struct CopyPlan {
  bool mine, second;
  int src;           // words from the source centre
  int q, qi, l;      // the target pixel: linear index, word index, local index
  uint16_t *p0, *p1; // its places in the planes
};

template <int R>
__device__ inline CopyPlan plan_copy(const ImgState& s, const UpdSmem<R>& sm) {
  using G = UpdGeom<R>;
  constexpr int P = G::P;
  constexpr bool kTwo = 2 * P * P <= kMidThreads;
  const int t0 = (int)threadIdx.x - kChainThreads;
  CopyPlan c;
  c.second = kTwo && t0 >= P * P;
  const int tp = c.second ? t0 - P * P : t0;
  const bool planes = s.planes != nullptr;
  c.mine = tp < P * P && (!c.second || planes) && sm.filled[tp < P * P ? tp : 0];
  const int dy = tp / P - R, dx = tp % P - R, tx = sm.nx_px + dx, ty = sm.nx_py + dy;
  c.src = dy * s.pitch + dx;
  c.q = ty * s.W + tx;
  c.qi = ty * s.pitch + tx;
  c.l = (G::RB + dy) * G::NS + G::RB + dx;
  c.p0 = c.p1 = nullptr;
  if (c.mine && planes && (c.second || !kTwo)) plane_places(s, tx, ty, c.p0, c.p1);
  return c;
}

// Applies the iteration whose source set_source has stored (warps 4-15, after
// a barrier of theirs): the copy of the unknown in-image part of Psi_p^ from
// Psi_q~, the validity counts of the candidates it touches, the isophotes of
// the new grey levels and, for every front pixel, the strongest isophote of
// its patch and its product with the normal.  The block's barrier must follow.
// The last thread issues a gpu-scope fence once the writes the next search
// reads (pixels, planes, mask, counts, validity bits) are issued, and then, if `copied` is
// given, tells the searchers so; its warp has no later work, so the fence
// waits off the path, and the same fence makes its later publication of the
// next round a release.
template <int R>
__device__ inline void update_work(const ImgState& s, UpdSmem<R>& sm, const CopyPlan& cpy, bool fence,
                                   unsigned* copied, unsigned copied_val) {
  using G = UpdGeom<R>;
  constexpr int P = G::P, RB = G::RB, NS = G::NS, R2 = G::R2, NW = G::NW, NC = G::NC;
  static_assert(P * P <= kMidThreads, "one thread per patch pixel");
  const int t0 = (int)threadIdx.x - kChainThreads, lane = threadIdx.x & 31;
  if (t0 >= kMidThreads) {
    work_sync();
    if (fence && lane == 31) {
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      if (copied) asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(copied), "r"(copied_val) : "memory");
    }
    return;
  }
  const int px = sm.px, py = sm.py;
  {
    uint32_t w = 0u;
    if (cpy.mine) w = __ldcg(&s.img[sm.qy * s.pitch + sm.qx + cpy.src]);  // in flight during the counts
    int newly = 0;
#pragma unroll 1
    for (int j = t0; j < NC * NC; j += kMidThreads) {
      const int nv = sm.cnt[j];
      if (nv < 0) continue;
      const int jy = j / NC, y = py + jy - 2 * R, x = px + j - jy * NC - 2 * R;
      s.count[y * s.pitch + x] = nv;
      if (nv == 0 && x >= s.cx0 && x <= s.cx1 && y >= s.cy0 && y <= s.cy1) {
        ++newly;
        if (s.planes) vbit_set(s, x, y);
      }
    }
    if (cpy.mine) {
      if (!cpy.second) {
        const uint8_t g = (uint8_t)luma_word(w);
        s.img[cpy.qi] = w;
        s.gray[cpy.q] = g;
        s.conf[cpy.q] = sm.cp;
        s.omega[cpy.q] = 0;
        sm.gr[cpy.l] = g;
      }
      if (cpy.p0) plane_write(cpy.p0, s.tc_len, w);
      if (cpy.p1) plane_write(cpy.p1, s.tc_len, w);
    }
    if (newly) atomicAdd(&sm.newly, newly);
  }
  __syncwarp();
  work_sync();
  constexpr int NB = 2 * (R + 1) + 1;  // the box the fill can change
#pragma unroll 1
  for (int j = t0; j < NB * NB; j += kMidThreads) {
    const int lx = RB - R - 1 + j % NB, ly = RB - R - 1 + j / NB;
    sm.ikey[ly * NS + lx] = isophote_key<R>(sm, lx, ly);
  }
  // strongest isophote of a front pixel's patch: one warp per pixel, each
  // lane with a fixed set of patch offsets (a separable windowed maximum over
  // the whole window took 1.8k + 0.5k cycles at R = 6)
  constexpr int NL = (P * P + 31) / 32;
  int off[NL];
#pragma unroll
  for (int j = 0; j < NL; ++j) {
    const int e = lane + 32 * j;
    off[j] = e < P * P ? (e / P - R) * NS + e % P - R : 0;  // past the end: the centre once more
  }
  const int par = sm.it & 1, nfront = sm.nlist[par];
  __syncwarp();
  mid_sync();
#pragma unroll 1
  for (int b = t0 >> 5; b < nfront; b += 32 * kMidWarps) {
    uint32_t mine = 0u;  // lane j: the key of the warp's j-th pixel
    int j = 0;
#pragma unroll 1
    for (int k = b; k < nfront && j < 32; k += kMidWarps, ++j) {
      const int i = sm.list[par][k], l = (RB + i / NW - R2) * NS + RB + i % NW - R2;
      uint32_t best = 0u;
#pragma unroll
      for (int q = 0; q < NL; ++q) best = max(best, sm.ikey[l + off[q]]);
      best = __reduce_max_sync(0xffffffffu, best);
      if (lane == j) mine = best;
    }
    if (lane < j) {
      const int k = b + kMidWarps * lane, nrm = sm.snrm[sm.list[par][k]];
      sm.dotc[k] = (uint32_t)isophote_dot<R>(sm, mine, nrm) | ((uint32_t)(nrm >> 16) << 12);
    }
  }
}

// Priorities of the new front (warps 0-3) and the next target: the better of
// the window's best and the best outside it.  Whole block, after a barrier;
// has one barrier, after which every thread holds the target (key 0: none).
// (*ny: its row, found where a division by W is off the path.)
template <int R>
__device__ inline void update_prio(const ImgState& s, UpdSmem<R>& sm, unsigned long long& wk, int& wi, int& ny) {
  using G = UpdGeom<R>;
  constexpr int R2 = G::R2, NW = G::NW;
  const int tid = threadIdx.x;
  wk = 0ull;
  wi = 0x7fffffff;
  if (tid < kChainThreads) {
    int mine_i = 0x7fffffff, mine_y = 0;
    const int par = sm.it & 1, nfront = sm.nlist[par], nt = chain_threads(nfront), W = s.W;
    if (tid < nt) {
#pragma unroll 1
      for (int k = tid; k < nfront; k += nt) {
        const int i = sm.list[par][k];
        const uint32_t dc = sm.dotc[k];
        const double cc = sm.sC[par][i];
        const double d = data_term_known(sm, (int)(dc & 0xfffu), (int)(dc >> 12));
        const int py = sm.py + i / NW - R2, p = py * W + sm.px + i % NW - R2;
        const unsigned long long key = (unsigned long long)__double_as_longlong(__dmul_rn(cc, d)) + 1ull;
        s.prio[p] = key;
        s.pconf[p] = cc;
        sm.sC[par][i] = __longlong_as_double((long long)key);
        if (prio_better(key, p, wk, mine_i)) {
          wk = key;
          mine_i = p;
          mine_y = py;
        }
      }
    }
    __syncwarp();
    wi = mine_i;
    warp_best_prio(wk, wi);
    if (wk != 0ull && mine_i == wi) sm.red_pb[tid >> 5] = PrioBest{wk, wi, mine_y};
    else if ((tid & 31) == 0 && wk == 0ull) sm.red_pb[tid >> 5] = PrioBest{0ull, 0x7fffffff, 0};
  }
  __syncthreads();
  // every warp reduces the five candidates (lanes 0-3: the warps', 4: outside)
  const int lane = tid & 31;
  PrioBest b = {0ull, 0x7fffffff, 0};
  if (lane < kChainThreads / 32) b = sm.red_pb[lane];
  else if (lane == kChainThreads / 32) b = PrioBest{sm.out_key, sm.out_idx, sm.out_y};
  wk = b.key;
  wi = b.idx;
  warp_best_prio(wk, wi);
  const unsigned at = __ballot_sync(0xffffffffu, b.key == wk && b.idx == wi);
  ny = __shfl_sync(0xffffffffu, b.pad, __ffs(at) - 1);
}

// After the selection (whole block, no barrier inside): key 0 for the
// window's pixels that are not on the front, and the state of the deferred
// record and tile maxima.
template <int R>
__device__ inline void update_store(const ImgState& s, UpdSmem<R>& sm, unsigned long long wk, int wi) {
  using G = UpdGeom<R>;
  constexpr int R2 = G::R2, NW = G::NW;
#pragma unroll 1
  for (int i = threadIdx.x; i < NW * NW; i += kEngThreads)
    if (sm.snrm[i] == kSpecNotFront) s.prio[(sm.py + i / NW - R2) * s.W + sm.px + i % NW - R2] = 0ull;
  if (threadIdx.x == 0) {
    sm.next_key = sm.remaining > 0 ? wk : 0ull;
    sm.next_idx = wi;
    sm.tile_px = sm.px;
    sm.tile_py = sm.py;
    sm.tile_par = sm.it & 1;
    sm.tiles_pending = 1;
    sm.rec_pending = 1;
  }
}

// The deferred record and tile maxima of the last iteration, before a launch
// leaves the image.  Whole block, after a barrier.
template <int R>
__device__ inline void update_drain(const ImgState& s, UpdSmem<R>& sm, bool overlap_counts) {
  if (threadIdx.x == kRecThread && sm.rec_pending) write_record<R>(s, sm, overlap_counts);
  if ((int)threadIdx.x >= kChainThreads && (int)threadIdx.x < kRecThread && sm.tiles_pending) update_tiles<R>(s, sm);
}

}  // namespace inp
