// The persistent engine kernel: one cooperative launch runs the fill loops
// of every image of every team to completion (single image: one team of all
// CTAs; batch: many teams, each with a list of images).  The per-image body
// for the image's patch radius is selected at run time.
#include "inpaint_engine.h"
#include "ptx.cuh"

namespace inp {

__device__ inline unsigned long long ld_acquire64_pub(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Dispatch on the image's patch radius and search rows per warp.
__device__ inline void run_by_radius(const EngineArgs& ea, int j, EngCtx& x) {
  const bool two = ea.imgs[j].srw == 2;
  switch (ea.imgs[j].r) {
#define INP_CASE(R)                                  \
  case R:                                            \
    if (two) run_image_r##R##_s2(ea, j, x);          \
    else run_image_r##R##_s1(ea, j, x);              \
    break;
    INP_CASE(1) INP_CASE(2) INP_CASE(3) INP_CASE(4) INP_CASE(5) INP_CASE(6) INP_CASE(7)
    INP_CASE(8)
#undef INP_CASE
    default:
      break;
  }
}

__global__ void __launch_bounds__(kEngThreads, 1) k_engine(EngineArgs ea) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  EngCtx x;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(x.smem_bytes));
  const int team = ea.cta_team[blockIdx.x];
  const int first = ea.team_first[team];
  x.rank = blockIdx.x - first;
  x.tsize = ea.team_first[team + 1] - first;
  x.tc = &ea.teams[team];
  x.tpart = ea.partials + first;
  // the barriers sit at the start of shared memory
  EngBars* bars = reinterpret_cast<EngBars*>(smem_raw);
  if (threadIdx.x == 0) {
    mbar_init(&bars->full[0], 1);
    mbar_init(&bars->full[1], 1);
    if (ea.tc_cols > 0) {
      for (int i = 0; i < kTcRing; ++i) {
        mbar_init(&bars->tc_full[i], 1);
        mbar_init(&bars->tc_empty[i], 2);  // one commit from each issuer
      }
      for (int b = 0; b < 2; ++b) {
        mbar_init(&bars->tc_done[b], 2);
        mbar_init(&bars->tc_free[b], kTcReaders);
      }
    }
  }
  fence_mbar_init();
  // tensor memory of the tensor-core search: held for the whole launch (one
  // CTA per SM, so the allocation never waits on another engine CTA)
  if (ea.tc_cols > 0 && threadIdx.x < 32) tc_alloc(&bars->tmem, (uint32_t)ea.tc_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  x.tmem = ea.tc_cols > 0 ? bars->tmem : 0u;
  x.tc_rows = 0;
  x.tc_tiles = 0;
  x.tc_nb = 0;
  x.ph0 = 0;
  x.ph1 = 0;
  x.epoch = (unsigned)ld_acquire64_pub(&x.tc->pub);
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(x.t_start));
  for (int li = ea.team_img_off[team]; li < ea.team_img_off[team + 1]; ++li) {
    run_by_radius(ea, ea.team_img[li], x);
    // the leader's last publication of the image was acquired by every CTA
    // of the team, so all of them see the same flag here
    unsigned expired;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(expired) : "l"(&x.tc->expired) : "memory");
    if (expired) break;
  }
  // every tile's MMAs were waited for before its accumulators were read
  if (ea.tc_cols > 0) {
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
      tc_fence_after();
      tc_dealloc(x.tmem, (uint32_t)ea.tc_cols);
    }
  }
}

// What a launch starts from: fresh teams, no error, key (and count) slots of
// all ones (a tag no round carries), and of a single image its iteration limit.
__global__ void __launch_bounds__(256) k_engine_begin(TeamCtl* teams, int n_teams, int* err, unsigned long long* slots,
                                                      int n_slots, Ctrl* c, int limit) {
  for (int i = threadIdx.x; i < n_slots; i += 256) slots[i] = ~0ull;
  for (int i = threadIdx.x; i < n_teams; i += 256) {
    teams[i].pub = 0ull;
    teams[i].expired = 0u;
    teams[i].copied = 0u;
  }
  if (threadIdx.x == 0) {
    *err = 0;
    if (c) c->iter_limit = limit;
  }
}

// After a launch of a single image: no limit again, and the launch's error
// beside the state, so that one copy brings both to the host.
__global__ void k_engine_end(Ctrl* c, const int* err) {
  c->iter_limit = 0x7fffffff;
  c->engine_err = *err;
}

// (One launch each; as memory operations, three before and two behind a
// launch, they were 15 us of a 175 us removal at 128x96.)
cudaError_t engine_begin(const EngineArgs& ea, int n_teams, int grid, Ctrl* c, int limit, cudaStream_t st) {
  k_engine_begin<<<1, 256, 0, st>>>(ea.teams, n_teams, ea.err, ea.partials, grid * (ea.overlap ? 3 : 1), c, limit);
  return cudaGetLastError();
}

cudaError_t engine_end(const EngineArgs& ea, Ctrl* c, cudaStream_t st) {
  k_engine_end<<<1, 1, 0, st>>>(c, ea.err);
  return cudaGetLastError();
}

cudaError_t engine_occupancy(size_t smem, int* blocks_per_sm) {
  cudaError_t e = cudaFuncSetAttribute(k_engine, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_engine, kEngThreads, smem);
}

size_t engine_launch_smem() {
  static size_t cached = 0;
  if (cached) return cached;
  int dev = 0, optin = 0;
  cudaFuncAttributes fa;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, k_engine) != cudaSuccess)
    return 0;
  cached = (size_t)optin - fa.sharedSizeBytes;
  return cached;
}

cudaError_t engine_launch(size_t smem, const EngineArgs& ea, int grid, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_engine, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<EngineArgs*>(&ea)};
  return cudaLaunchCooperativeKernel((const void*)k_engine, dim3(grid), dim3(kEngThreads), args, smem, st);
}

}  // namespace inp
