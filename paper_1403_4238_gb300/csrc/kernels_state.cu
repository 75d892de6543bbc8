// Initialisation, priority and copy/update kernels of the fill loop.
//
// Sec. 3 of the paper: the fill front dOmega, the priority P(p) = C(p) D(p)
// (Eq. 1-2), the copy of the best source patch into the unknown part of the
// target patch, and the confidence update.  Table 2 lists these as the grey
// conversion, border update, source marking, priority and confidence updates
// and the RGB/grey update; here they are: one init pass per image, then, for
// patch radii above 8, three small kernels per iteration that touch only the
// neighbourhood of the filled patch (radii to 8: update_fast.cuh).
//
// Bit-exactness of the FP64 priority: the library is compiled with
// --fmad=false, the confidence sum runs in row-major patch order (dy outer,
// dx inner) in one thread, and division/sqrt use the IEEE round-to-nearest
// intrinsics, so each value equals the single-threaded CPU evaluation of the
// same expression.
#include "inpaint_internal.cuh"

namespace inp {

// ---------------------------------------------------------------- priority

__device__ inline int omega_clamped(const ImgState& s, int x, int y) {
  x = x < 0 ? 0 : (x >= s.W ? s.W - 1 : x);
  y = y < 0 ? 0 : (y >= s.H ? s.H - 1 : y);
  return s.omega[(size_t)y * s.W + x] ? 1 : 0;
}

// Fill front membership: p in Omega with an in-image 4-neighbour in Phi.  The
// five reads are independent (a chain of them, one L2 round trip each, took half
// of k_fill_big).
__device__ inline bool on_front(const ImgState& s, int x, int y) {
  const uint8_t* o = s.omega + (size_t)y * s.W + x;
  const uint8_t c = o[0], l = x > 0 ? o[-1] : 1, r = x + 1 < s.W ? o[1] : 1;
  const uint8_t u = y > 0 ? o[-s.W] : 1, d = y + 1 < s.H ? o[s.W] : 1;
  return (c != 0) & ((l == 0) | (r == 0) | (u == 0) | (d == 0));
}

// D(p) of Eq. 2 from the isophote's gradient; normal to the front: Sobel of
// the Omega indicator (replicated borders).
__device__ inline double data_term_at(const ImgState& s, int x, int y, int gx, int gy) {
  const int m_lu = omega_clamped(s, x - 1, y - 1), m_cu = omega_clamped(s, x, y - 1);
  const int m_ru = omega_clamped(s, x + 1, y - 1), m_lc = omega_clamped(s, x - 1, y);
  const int m_rc = omega_clamped(s, x + 1, y), m_ld = omega_clamped(s, x - 1, y + 1);
  const int m_cd = omega_clamped(s, x, y + 1), m_rd = omega_clamped(s, x + 1, y + 1);
  const int nx = (m_ru + 2 * m_rc + m_rd) - (m_lu + 2 * m_lc + m_ld);
  const int ny = (m_ld + 2 * m_cd + m_rd) - (m_lu + 2 * m_cu + m_ru);
  int dot = (-gy) * nx + gx * ny;
  dot = dot < 0 ? -dot : dot;
  const int nn = nx * nx + ny * ny;
  return nn != 0 ? __ddiv_rn(__ddiv_rn((double)dot, __dsqrt_rn((double)nn)), 510.0) : 0.0;
}

// P(p) of Eq. 1 with C(p), D(p) of Eq. 2; writes C(p) to *c_out (debug check).
__device__ double priority_at(const ImgState& s, int x, int y, double* c_out) {
  const int W = s.W, H = s.H, r = s.r;
  // Confidence term: known part of Psi_p over its in-image area, summed in
  // row-major order.
  double sum = 0.0;
  int n_in = 0;
  for (int dy = -r; dy <= r; ++dy) {
    const int qy = y + dy;
    if (qy < 0 || qy >= H) continue;
    for (int dx = -r; dx <= r; ++dx) {
      const int qx = x + dx;
      if (qx < 0 || qx >= W) continue;
      ++n_in;
      const size_t q = (size_t)qy * W + qx;
      if (s.omega[q] == 0) sum = __dadd_rn(sum, s.conf[q]);
    }
  }
  const double c = __ddiv_rn(sum, (double)n_in);

  // Isophote: strongest central-difference grey gradient among pixels of
  // Psi_p whose four neighbours are known (first in row-major order on ties).
  int best = -1, gx = 0, gy = 0;
  for (int dy = -r; dy <= r; ++dy) {
    const int qy = y + dy;
    if (qy < 1 || qy >= H - 1) continue;
    for (int dx = -r; dx <= r; ++dx) {
      const int qx = x + dx;
      if (qx < 1 || qx >= W - 1) continue;
      const size_t q = (size_t)qy * W + qx;
      if (s.omega[q] | s.omega[q - 1] | s.omega[q + 1] | s.omega[q - W] | s.omega[q + W]) continue;
      const int tx = (int)s.gray[q + 1] - (int)s.gray[q - 1];
      const int ty = (int)s.gray[q + W] - (int)s.gray[q - W];
      const int mag = tx * tx + ty * ty;
      if (mag > best) {
        best = mag;
        gx = tx;
        gy = ty;
      }
    }
  }
  const double d = data_term_at(s, x, y, gx, gy);
  *c_out = c;
  return __dmul_rn(c, d);
}

// Appends pixel i to the list of front pixels to evaluate when `mine`; whole
// warps (one counter update per warp).
__device__ inline void append_front(const ImgState& s, bool mine, int i) {
  const unsigned bal = __ballot_sync(0xffffffffu, mine);
  if (bal == 0u) return;
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == 0) base = atomicAdd(&s.ctrl->n_front, __popc(bal));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (mine) s.front[base + __popc(bal & ((1u << lane) - 1u))] = i;
}

// Priorities of the listed front pixels for patch radii above the engine's:
// one CTA per pixel.  kSum (initialisation): warp 0 sums the confidences while
// warp 1 finds the strongest isophote; else the sums are in fsum already.  (One
// thread per pixel reading the patch from global memory, in the update's one
// CTA, took 390 us an iteration at 512x384, 25x25.)
template <bool kSum>
__global__ void __launch_bounds__(kSum ? 64 : 32) k_prio_list(ImgState s) {
  __shared__ unsigned long long iso_s;
  __shared__ __align__(16) double vals[kSum ? kSumVals : 2];
  const int n = s.ctrl->n_front;
  const int W = s.W, H = s.H, r = s.r, P = 2 * r + 1;
  const int lane = threadIdx.x & 31;
  for (int k = blockIdx.x; k < n; k += gridDim.x) {
    const int p = s.front[k], y = p / W, x = p - y * W;
    const int x0 = max(x - r, 0), x1 = min(x + r, W - 1), y0 = max(y - r, 0), y1 = min(y + r, H - 1);
    double sum = kSum ? 0.0 : s.fsum[k];
    if (kSum && threadIdx.x < 32) {
      sum = warp_ordered_sum(s, vals, x0, x1, y0, y1, [&](int, int, size_t q, double& c) {
        c = s.conf[q];
        return s.omega[q] == 0;
      });
    } else {
      // key: (|grad|^2 + 1) << 32 | ~(row-major index in the patch), 0: none
      unsigned long long best = 0ull;
      const int ya = max(y - r, 1), yb = min(y + r, H - 2), xa = max(x - r, 1), xb = min(x + r, W - 2);
      for (int xx = xa + lane; xx <= xb; xx += 32) {
#pragma unroll 4
        for (int yy = ya; yy <= yb; ++yy) {
          const size_t q = (size_t)yy * W + xx;
          const int o = s.omega[q] | s.omega[q - 1] | s.omega[q + 1] | s.omega[q - W] | s.omega[q + W];
          const int gx = (int)s.gray[q + 1] - (int)s.gray[q - 1], gy = (int)s.gray[q + W] - (int)s.gray[q - W];
          const unsigned long long key = ((unsigned long long)(gx * gx + gy * gy + 1) << 32) |
                                         (0xffffffffu - (unsigned)((yy - ya) * P + xx - xa));
          if (o == 0 && key > best) best = key;
        }
      }
      __syncwarp();
      const unsigned mh = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32));
      const unsigned ml = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32) == mh ? (unsigned)best : 0u);
      if (lane == 0) iso_s = ((unsigned long long)mh << 32) | ml;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      const double cc = __ddiv_rn(sum, (double)((x1 - x0 + 1) * (y1 - y0 + 1)));
      const unsigned long long iso = iso_s;
      int gx = 0, gy = 0;
      if (iso >> 32) {
        const int l = (int)(0xffffffffu - (unsigned)iso);
        const size_t q = (size_t)(max(y - r, 1) + l / P) * W + max(x - r, 1) + l % P;
        gx = (int)s.gray[q + 1] - (int)s.gray[q - 1];
        gy = (int)s.gray[q + W] - (int)s.gray[q - W];
      }
      s.prio[p] = (unsigned long long)__double_as_longlong(__dmul_rn(cc, data_term_at(s, x, y, gx, gy))) + 1ull;
      s.pconf[p] = cc;
    }
    __syncthreads();
  }
}

// The front of the window of the current target as it is after the coming fill
// (the patch's unknown pixels known then), listed in front.  It does not depend
// on the search's result, so its confidence sums run beside the search, as CTAs
// of the same launch (search_plain.cu; 512x384, 25x25: 70 us an iteration with the
// sums behind the fill, 64 so).  Whole block of kUpdThreads.
__device__ inline void block_spec_list(const ImgState& s, int* n) {
  const Ctrl* c = s.ctrl;
  const int px = __ldcg(&c->px), py = __ldcg(&c->py), r = s.r, R2 = 2 * r + 1, side = 2 * R2 + 1, lane = threadIdx.x & 31;
  auto known = [&](int x, int y) {
    if (x < 0 || x >= s.W || y < 0 || y >= s.H) return false;
    const bool k = s.omega[(size_t)y * s.W + x] == 0;
    return k || (abs(x - px) <= r && abs(y - py) <= r);
  };
  if (threadIdx.x == 0) *n = 0;
  __syncthreads();
  constexpr int V = 3;
  for (int j0 = threadIdx.x; j0 - (int)threadIdx.x < side * side; j0 += V * kUpdThreads) {
    bool fr[V];
#pragma unroll
    for (int u = 0; u < V; ++u) {
      const int j = j0 + u * kUpdThreads, x = px - R2 + j % side, y = py - R2 + j / side;
      const bool in = j < side * side && x >= 0 && x < s.W && y >= 0 && y < s.H;
      const bool k0 = known(x, y), kl = known(x - 1, y), kr = known(x + 1, y), ku = known(x, y - 1), kd = known(x, y + 1);
      fr[u] = in & !k0 & (kl | kr | ku | kd);
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < V; ++u) {
      const int j = j0 + u * kUpdThreads;
      const unsigned bal = __ballot_sync(0xffffffffu, fr[u]);
      int base = 0;
      if (lane == 0 && bal) base = atomicAdd(n, __popc(bal));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (fr[u])
        s.front[base + __popc(bal & ((1u << lane) - 1u))] = (py - R2 + j / side) * s.W + px - R2 + j % side;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) s.ctrl->n_spec = *n;
}

// The first target's list (initialisation).  Single CTA.
__global__ void __launch_bounds__(kUpdThreads) k_spec_first(ImgState s) {
  __shared__ int n;
  if (s.ctrl->px >= 0) block_spec_list(s, &n);
}

// CTAs of k_prio_list (a grid-stride loop): a window's front is 100-200 pixels.
constexpr int kPrioCtas = 608;

// ---------------------------------------------------------------- init

// RGB + mask -> packed state, with key 0 everywhere, the bits of Omega
// (ImgState::obits; columns past the image read as Omega) and the control
// block of a fresh loop.
__global__ void k_unpack(ImgState s, const uint8_t* rgb, int rgb_stride, const uint8_t* mask,
                         int mask_stride, const double* conf_in) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  if (x == 0 && y == 0) {
    Ctrl* c = s.ctrl;
    c->iter = 0;
    c->remaining = 0;
    c->status = 0;
    c->px = -1;
    c->py = -1;
    c->n_valid = 0;
    c->iter_limit = 0x7fffffff;
    c->n_adm = 0;
    c->prio = 0.0;
    c->conf = 0.0;
    c->evals = 0ull;
    c->t_search = 0ull;
    c->t_update = 0ull;
    c->timed_iters = 0;
    c->tc_rounds = 0;
    c->n_front = 0;
    c->tiles_done = 0;
    c->engine_err = 0;
  }
  int om = 1;
  if (x < s.W) {
    const uint8_t* p = rgb + (size_t)y * rgb_stride + 3 * (size_t)x;
    const uint32_t w = pack_rgb(p[0], p[1], p[2]);
    const size_t i = (size_t)y * s.W + x;
    om = mask[(size_t)y * mask_stride + x] != 0;
    s.img[(size_t)y * s.pitch + x] = w;
    s.omega[i] = (uint8_t)om;
    s.gray[i] = om ? 0 : (uint8_t)luma_word(w);
    s.conf[i] = om ? 0.0 : (conf_in ? conf_in[i] : 1.0);
    s.prio[i] = 0ull;
    s.pconf[i] = 0.0;
  } else if (x < s.pitch) {
    s.count[(size_t)y * s.pitch + x] = kCountInvalid;  // row padding
  }
  const unsigned bal = __ballot_sync(0xffffffffu, om != 0);
  if ((threadIdx.x & 31) == 0 && x < s.W) s.obits[(size_t)y * obits_pitch(s.W) + (x >> 5)] = bal;
}

__device__ inline bool in_rect(const ImgState& s, int x, int y) {
  return x >= s.cx0 && x <= s.cx1 && y >= s.cy0 && y <= s.cy1;
}

// Unknown pixels per candidate centre, |Omega| and the number of valid
// centres: one CTA per kCountCols x kCountRows tile, one thread per column.
// A patch row's count is the population of at most 65 bits of a row of
// Omega bits; the thread slides the sum of 2 r + 1 rows down its column.  (An
// integral image took four passes over 4 bytes a pixel, whose column pass
// alone was 31 us at 512x384 and 33 us at 1920x1080: one thread walks 64
// dependent rows.)
constexpr int kCountCols = 128, kCountRows = 16;

__global__ void __launch_bounds__(kCountCols) k_count(ImgState s) {
  constexpr int WW = kCountCols / 32 + 3;  // a word of halo on either side, one for the funnel shifts
  __shared__ uint32_t rows[(kCountRows + 2 * kMaxRadius) * WW];
  __shared__ int scratch[32];
  const int r = s.r, P = 2 * r + 1, tid = threadIdx.x;
  const int x0 = blockIdx.x * kCountCols, y0 = blockIdx.y * kCountRows, ow = obits_pitch(s.W);
  for (int e = tid; e < (kCountRows + 2 * r) * WW; e += kCountCols) {
    const int v = e / WW, y = y0 - r + v, w = (x0 >> 5) - 1 + e - v * WW;
    rows[e] = y >= 0 && y < s.H && w >= 0 && w < ow ? s.obits[(size_t)y * ow + w] : 0u;
  }
  __syncthreads();
  const int x = x0 + tid, a = 32 + tid - r, w0 = a >> 5, sh = a & 31;
  const uint32_t m0 = P >= 32 ? 0xffffffffu : (1u << P) - 1u;
  const uint32_t m1 = P < 32 ? 0u : P >= 64 ? 0xffffffffu : (1u << (P - 32)) - 1u;
  auto patch_row = [&](int v) {
    const uint32_t* b = rows + v * WW + w0;
    int n = __popc(__funnelshift_r(b[0], b[1], sh) & m0);
    if (P > 32) n += __popc(__funnelshift_r(b[1], b[2], sh) & m1);
    if (P > 64) n += (b[2] >> sh) & 1u;
    return n;
  };
  int valid = 0, om = 0;
  if (x < s.W) {
    const bool xin = x - r >= 0 && x + r < s.W;
    int cnt = 0;
    for (int v = 0; v < 2 * r; ++v) cnt += patch_row(v);
#pragma unroll 4
    for (int v = 0; v < kCountRows; ++v) {
      const int y = y0 + v;
      if (y >= s.H) break;
      cnt += patch_row(v + 2 * r);
      const bool in = xin && y - r >= 0 && y + r < s.H;
      s.count[(size_t)y * s.pitch + x] = in ? cnt : kCountInvalid;
      valid += in && cnt == 0 && in_rect(s, x, y) ? 1 : 0;
      om += (rows[(v + r) * WW + 1 + (tid >> 5)] >> (tid & 31)) & 1u;
      cnt -= patch_row(v);
    }
  }
  __syncwarp();
  om = block_sum_int(om, scratch);
  valid = block_sum_int(valid, scratch);
  if (tid == 0) {
    if (om) atomicAdd(&s.ctrl->remaining, om);
    if (valid) atomicAdd(&s.ctrl->n_valid, valid);
  }
}

// The list of the front pixels (patch radius > 8).
__global__ void k_front_all(ImgState s) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  append_front(s, x < s.W && on_front(s, x, y), y * s.W + x);
}

// All tiles and the first target: one CTA per level-1 tile, one warp per
// level-0 tile in turn; the last CTA to finish selects.
__global__ void __launch_bounds__(1024) k_tiles_all(ImgState s) {
  __shared__ int last;
  const int ux = blockIdx.x, uy = blockIdx.y, warp = threadIdx.x >> 5;
  for (int t = warp; t < kT1 * kT1; t += 32) {
    const int tx = ux * kT1 + t % kT1, ty = uy * kT1 + t / kT1;
    if (tx < s.t0x && ty < s.t0y) warp_rescan_t0(s, tx, ty);
  }
  __syncthreads();
  if (warp != 0) return;
  warp_rescan_t1(s, ux, uy);
  __syncwarp();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&s.ctrl->tiles_done, 1) == (int)(gridDim.x * gridDim.y) - 1;
    __threadfence();
  }
  __syncwarp();
  if (last && loop_active(s.ctrl)) warp_select(s);
}

// ---------------------------------------------------------------- update

struct UpdSmem {
  uint8_t filled[(2 * kMaxRadius + 1) * (2 * kMaxRadius + 1)];
  int32_t fsat[(2 * kMaxRadius + 2) * (2 * kMaxRadius + 2)];
  unsigned long long u64s[32];
  int ints[32];
};

// One iteration's copy and validity update for patch radii above the
// engine's.  Single CTA; k_prio_list (the front pixels listed before the search,
// with the sums taken beside it) and k_select_big follow.  Every round trip here
// is a serial one, so a thread's reads go out together (17 us cold with a chain
// of reads per window pixel and the list counted in global memory, now 13).
__global__ void __launch_bounds__(kUpdThreads) k_fill_big(ImgState s) {
  __shared__ UpdSmem sm;
  Ctrl* c = s.ctrl;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int W = s.W, H = s.H, r = s.r, P = 2 * r + 1;
  if (!loop_active(c)) {
    if (tid == 0) c->n_front = -1;
    return;
  }
  {
    // findBestPatch result: lowest (SSD << 32 | idx) over all search CTAs.
    unsigned long long best = ~0ull;
    for (int i = tid; i < s.n_partial; i += nt) {
      const unsigned long long v = s.partial[i];
      best = v < best ? v : best;
    }
    best = block_min_u64(best, sm.u64s);
    if (best == ~0ull) {  // no fully-known source patch: leave the state as is
      if (tid == 0) {
        c->status = INPAINT_ERR_NO_SOURCE;
        c->n_front = -1;
      }
      return;
    }
    const uint32_t ssd = (uint32_t)(best >> 32);
    const int q = (int)(best & 0xffffffffull);
    const int qx = q % W, qy = q / W;
    const int px = c->px, py = c->py;
    const double cp = c->conf, pp = c->prio;
    const int n_cand = c->n_valid;

    // Copy Psi_q~ into the unknown in-image part of Psi_p^; those pixels
    // take confidence C(p^) and leave Omega.  Sources are known pixels, so
    // they are never written here.
    int my_filled = 0;
    for (int i = tid; i < P * P; i += nt) {
      const int dy = i / P - r, dx = i % P - r;
      const int tx = px + dx, ty = py + dy;
      uint8_t f = 0;
      if (tx >= 0 && tx < W && ty >= 0 && ty < H) {
        const size_t t = (size_t)ty * W + tx;
        if (s.omega[t]) {
          const uint32_t w = s.img[(size_t)(qy + dy) * s.pitch + qx + dx];
          s.img[(size_t)ty * s.pitch + tx] = w;
          s.gray[t] = (uint8_t)luma_word(w);
          s.conf[t] = cp;
          s.omega[t] = 0;
          f = 1;
          ++my_filled;
        }
      }
      sm.filled[i] = f;
    }
    const int filled = block_sum_int(my_filled, sm.ints);  // has __syncthreads
    const int nx_in = min(px + r, W - 1) - max(px - r, 0) + 1;
    const int ny_in = min(py + r, H - 1) - max(py - r, 0) + 1;
    const int n_known = nx_in * ny_in - filled;

    // Integral image of the filled flags over the patch, in shared memory.
    const int P1 = P + 1;
    for (int v = tid; v <= P; v += nt) {
      sm.fsat[v] = 0;           // row 0
      sm.fsat[v * P1] = 0;      // column 0
    }
    __syncthreads();
    for (int v = tid; v < P; v += nt) {
      int run = 0;
      for (int u = 0; u < P; ++u) {
        run += sm.filled[v * P + u];
        sm.fsat[(v + 1) * P1 + u + 1] = run;
      }
    }
    __syncthreads();
    for (int u = tid + 1; u <= P; u += nt) {
      int run = 0;
#pragma unroll 5
      for (int v = 1; v <= P; ++v) {
        run += sm.fsat[v * P1 + u];
        sm.fsat[v * P1 + u] = run;
      }
    }
    __syncthreads();

    // Validity map: every centre within 2r of p^ loses the filled pixels of
    // its patch from its unknown count.
    const int side = 4 * r + 1;
    int newly = 0;
    constexpr int U = 5;  // counts of a thread in flight together
    for (int j0 = tid; j0 < side * side; j0 += U * nt) {
      int cnt[U], dec[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + u * nt, wy = j / side - 2 * r, wx = j % side - 2 * r;
        const int x = px + wx, y = py + wy;
        cnt[u] = dec[u] = 0;
        if (j < side * side && x >= 0 && x < W && y >= 0 && y < H) {
          // (a patch at most 2 r away overlaps the target's)
          const int u0 = max(0, wx), u1 = min(P - 1, wx + 2 * r);
          const int v0 = max(0, wy), v1 = min(P - 1, wy + 2 * r);
          dec[u] = sm.fsat[(v1 + 1) * P1 + u1 + 1] - sm.fsat[v0 * P1 + u1 + 1] -
                   sm.fsat[(v1 + 1) * P1 + u0] + sm.fsat[v0 * P1 + u0];
          cnt[u] = s.count[(size_t)y * s.pitch + x];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (dec[u] == 0) continue;
        const int j = j0 + u * nt, y = py + j / side - 2 * r, x = px + j % side - 2 * r;
        s.count[(size_t)y * s.pitch + x] = cnt[u] - dec[u];
        if (cnt[u] == dec[u] && in_rect(s, x, y)) ++newly;
      }
    }
    newly = block_sum_int(newly, sm.ints);  // also orders the global writes above

    // Priorities that can change are those of the front pixels within 2r+1 of
    // p^ (listed before the search); the window's others have none.
    const int R2 = 2 * r + 1, side2 = 2 * R2 + 1;
    __syncthreads();
    constexpr int V = 3;
    for (int j0 = tid; j0 < side2 * side2; j0 += V * nt) {
      bool off[V];
#pragma unroll
      for (int u = 0; u < V; ++u) {
        const int j = j0 + u * nt, x = px - R2 + j % side2, y = py - R2 + j / side2;
        off[u] = j < side2 * side2 && x >= 0 && x < W && y >= 0 && y < H && !on_front(s, x, y);
      }
#pragma unroll
      for (int u = 0; u < V; ++u) {
        const int j = j0 + u * nt, i = (py - R2 + j / side2) * W + px - R2 + j % side2;
        if (off[u]) {
          s.prio[i] = 0ull;
          s.pconf[i] = 0.0;
        }
      }
    }
    __syncthreads();
    if (tid == 0) {
      c->n_front = c->n_spec;
      if (filled == 0) {  // p^ must lie in Omega; stop rather than loop without progress
        c->status = INPAINT_ERR_INTERNAL;
        c->n_front = -1;
        return;
      }
      const int it = c->iter, remaining = c->remaining - filled;
      inpaint_step_info e;
      e.iter = it;
      e.px = px;
      e.py = py;
      e.qx = qx;
      e.qy = qy;
      e.ssd = ssd;
      e.priority = pp;
      e.confidence = cp;
      e.filled = filled;
      e.remaining = remaining;
      e.n_known = n_known;
      e.n_cand = n_cand;
      c->last = e;
      if (it < s.trace_cap) s.trace[it] = e;
      c->remaining = remaining;
      c->iter = it + 1;
      c->n_valid = n_cand + newly;
      c->evals += (unsigned long long)n_cand * (unsigned long long)n_known;
    }
  }
}

// After k_prio_list: the tiles over the window of the target just filled, the
// selection of the next one and its list.  Single CTA.
__global__ void __launch_bounds__(kUpdThreads) k_select_big(ImgState s, cudaGraphConditionalHandle cond,
                                                            int use_cond) {
  __shared__ int n_list;
  Ctrl* c = s.ctrl;
  const int tid = threadIdx.x;
  if (c->n_front >= 0) {
    const int px = c->px, py = c->py, R2 = 2 * s.r + 1;
    block_refresh_tiles(s, max(0, px - R2), min(s.W - 1, px + R2), max(0, py - R2), min(s.H - 1, py + R2));
    if (tid < 32) {
      if (c->remaining > 0) {
        warp_select(s);
      } else if (tid == 0) {
        c->px = -1;
        c->py = -1;
      }
    }
    __syncthreads();
    // (the next iteration's list; the selection above is visible after the barrier)
    if (c->remaining > 0 && c->status == 0) block_spec_list(s, &n_list);
    __syncthreads();
  }
  if (use_cond && tid == 0) cudaGraphSetConditional(cond, c->n_front >= 0 && loop_active(c) ? 1u : 0u);
}

// Debug self-check: recount every candidate's unknown pixels and re-evaluate
// every priority key from scratch; any difference sets INPAINT_ERR_INTERNAL.
__global__ void k_verify(ImgState s) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= s.W || s.ctrl->status != 0) return;
  const int r = s.r;
  const size_t i = (size_t)y * s.W + x, ic = (size_t)y * s.pitch + x;
  bool bad = false;
  if (x - r >= 0 && x + r < s.W && y - r >= 0 && y + r < s.H) {
    int cnt = 0;
    for (int dy = -r; dy <= r; ++dy)
      for (int dx = -r; dx <= r; ++dx) cnt += s.omega[(size_t)(y + dy) * s.W + x + dx];
    bad |= cnt != s.count[ic];
  } else {
    bad |= s.count[ic] < kCountInvalid - (2 * r + 1) * (2 * r + 1);
  }
  unsigned long long key = 0ull;
  if (on_front(s, x, y)) {
    double c;
    key = (unsigned long long)__double_as_longlong(priority_at(s, x, y, &c)) + 1ull;
  }
  bad |= key != s.prio[i];
  if (bad) atomicCAS(&s.ctrl->status, 0, (int)INPAINT_ERR_INTERNAL);
}

__global__ void k_export(ImgState s, uint8_t* rgb) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)s.W * s.H) return;
  const uint32_t w = s.img[(i / s.W) * s.pitch + i % s.W];
  rgb[3 * i] = (uint8_t)(w & 255u);
  rgb[3 * i + 1] = (uint8_t)((w >> 8) & 255u);
  rgb[3 * i + 2] = (uint8_t)((w >> 16) & 255u);
}

__global__ void k_set_limit(Ctrl* c, int limit) { c->iter_limit = limit; }

// ---------------------------------------------------------------- launchers

static cudaError_t init_state(const ImgState& s, const uint8_t* rgb, int rgb_stride, const uint8_t* mask,
                              int mask_stride, const double* conf, cudaStream_t st) {
  const int W = s.W, H = s.H;
  k_unpack<<<dim3((s.pitch + 255) / 256, H), 256, 0, st>>>(s, rgb, rgb_stride, mask, mask_stride, conf);
  k_count<<<dim3((W + kCountCols - 1) / kCountCols, (H + kCountRows - 1) / kCountRows), kCountCols, 0, st>>>(s);
  if (s.r <= 8) {
    const cudaError_t e = launch_prio_init_fast(s, st);
    if (e != cudaSuccess) return e;
  } else {
    k_front_all<<<dim3((W + 255) / 256, H), 256, 0, st>>>(s);
    k_prio_list<true><<<kPrioCtas, 64, 0, st>>>(s);
  }
  k_tiles_all<<<dim3(s.t1x, s.t1y), 1024, 0, st>>>(s);
  if (s.r > 8) k_spec_first<<<1, kUpdThreads, 0, st>>>(s);
  return cudaGetLastError();
}

cudaError_t launch_init(const ImgState& s, const uint8_t* rgb, int rgb_stride, const uint8_t* mask,
                        int mask_stride, cudaStream_t st) {
  return init_state(s, rgb, rgb_stride, mask, mask_stride, nullptr, st);
}

cudaError_t launch_import(const ImgState& s, const uint8_t* rgb, const uint8_t* omega,
                          const double* conf, cudaStream_t st) {
  return init_state(s, rgb, 3 * s.W, omega, s.W, conf, st);
}

cudaError_t launch_update(const ImgState& s, unsigned long long cond_handle, int use_cond, cudaStream_t st) {
  k_fill_big<<<1, kUpdThreads, 0, st>>>(s);
  k_prio_list<false><<<kPrioCtas, 32, 0, st>>>(s);
  k_select_big<<<1, kUpdThreads, 0, st>>>(s, (cudaGraphConditionalHandle)cond_handle, use_cond);
  return cudaGetLastError();
}

cudaError_t launch_set_limit(const ImgState& s, int limit, cudaStream_t st) {
  k_set_limit<<<1, 1, 0, st>>>(s.ctrl, limit);
  return cudaGetLastError();
}

cudaError_t launch_verify_count(const ImgState& s, cudaStream_t st) {
  k_verify<<<dim3((s.W + 127) / 128, s.H), 128, 0, st>>>(s);
  return cudaGetLastError();
}

cudaError_t launch_export(const ImgState& s, uint8_t* rgb_dense, cudaStream_t st) {
  const size_t n = (size_t)s.W * s.H;
  k_export<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(s, rgb_dense);
  return cudaGetLastError();
}

}  // namespace inp
