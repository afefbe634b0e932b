// Fused selection kernels of libm3e: the whole per-frame method of the paper
// (Algorithm 1: load, selection cuts, track reconstruction, vertex fit, store)
// run by one group of threads per frame:
//   k_select_warp  persistent, one warp per frame, frames from a device work
//                  queue (lowest latency per frame; frames too large for a warp's
//                  shared-memory stage go to the deferred list);
//   k_select_cta   one CTA per frame: the deferred frames, and the plain
//                  per-frame form over a whole batch.
#include "m3e_device.cuh"

namespace m3e {
namespace {

// Persistent warp-per-frame kernel: each warp takes `grab` frames at a time from
// the device work queue; a frame that outgrows the warp's shared-memory stage is
// appended to the deferred list for the CTA kernel.
template <bool DEBUG>
__global__ void __launch_bounds__(WARPS_PER_CTA * 32, 5)  // as many CTAs per SM as its shared memory allows
    k_select_warp(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmWarp& sm = reinterpret_cast<SmWarp*>(smem_raw)[threadIdx.x >> 5];
  const WarpGroup g;
  clear_stats(g, sm);
  const int nf = (int)P.n_frames;
  for (;;) {
    int f0 = 0;
    if (g.leader()) f0 = atomicAdd(&P.work[0], P.grab);
    f0 = __shfl_sync(FULL, f0, 0);
    if (f0 >= nf) break;
    const int f1 = min(f0 + P.grab, nf);
    for (int f = f0; f < f1; ++f) {
      int r = frame_front<WarpGroup, SmWarp, W_HITS, W_TRIP, true, DEBUG>(g, sm, C, P, f);
      if (r == PENDING) r = frame_back<WarpGroup, SmWarp, W_TRIP, W_TRK, W_COMBO, true, DEBUG>(g, sm, C, P, f);
      if (r == DEFERRED) {
        if (g.leader()) {
          const int k = atomicAdd(P.defer_count, 1);
          P.defer_list[k] = f;
          if (P.stats) sm.acc[ST_DEFER] += 1;
        }
      } else {
        finish_frame(g, sm, P, f, r);
      }
      g.sync();
    }
  }
  flush_stats(g, sm, P.stats);
}

// CTA-per-frame kernel.  LIST: frames from the deferred list written by the warp
// kernel earlier on the same stream; otherwise frames 0..n-1, one CTA each
// (grid-stride when the grid is smaller).
template <int NT, bool DEBUG, bool LIST>
__global__ void __launch_bounds__(NT) k_select_cta(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmCta& sm = *reinterpret_cast<SmCta*>(smem_raw);
  const CtaGroup<NT> g;
  clear_stats(g, sm);
  if (LIST) pdl_wait();
  const int count = LIST ? *P.in_count : (int)P.n_frames;
  for (int i = blockIdx.x; i < count; i += gridDim.x) {
    const int f = LIST ? P.in_list[i] : i;
    int r = frame_front<CtaGroup<NT>, SmCta, C_HITS, C_TRIP, false, DEBUG>(g, sm, C, P, f);
    if (r == PENDING) r = frame_back<CtaGroup<NT>, SmCta, C_TRIP, C_TRK, C_COMBO, false, DEBUG>(g, sm, C, P, f);
    finish_frame(g, sm, P, f, r);
    g.sync();
  }
  flush_stats(g, sm, P.stats);
}

// Small batches: a CTA per frame with a stage of 512 hits, so that a whole small batch is
// resident at once and the call takes one frame's latency.  A frame beyond the stage is
// marked in its reason for k_select_marked.
using SmSmall = FrameSm<SMALL_HITS, SMALL_TRIP, C_TRK, C_COMBO, false, false>;
static_assert(8 * (sizeof(SmSmall) + 1024) <= 228 * 1024, "eight CTAs per SM");
constexpr uint8_t MARK = 0xff;

// NT: threads of a CTA, CTAS: of them per SM.  Measured (us, batches of nominal / throughput /
// 32-track frames): 64 frames 14 / 19 / 23 with 256 threads, 14 / 23 / 32 with 128; 2048
// frames 35 / 54 / 72 against 24 / 47 / 70.  The wide CTAs serve batches that they hold
// resident at once.
template <int NT, int CTAS>
__global__ void __launch_bounds__(NT, CTAS)
    k_select_small(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmSmall& sm = *reinterpret_cast<SmSmall*>(smem_raw);
  const CtaGroup<NT> g;
  pdl_trigger();
  const int f = blockIdx.x;
  int r = frame_front<CtaGroup<NT>, SmSmall, SMALL_HITS, SMALL_TRIP, true, false, false, true>(g, sm, C, P, f);
  if (r == PENDING)
    r = frame_back<CtaGroup<NT>, SmSmall, SMALL_TRIP, C_TRK, C_COMBO, true, false, true>(g, sm, C, P, f);
  if (r != DEFERRED) finish_frame<CtaGroup<NT>, SmSmall, true>(g, sm, P, f, r);
  else if (g.leader()) P.reason[f] = MARK;
}

// The frames that k_select_small marked, with the stage of the configuration limits; one
// look at the marks per thread (the grid has a thread for every frame of a small batch).
__global__ void __launch_bounds__(CTA_THREADS)
    k_select_marked(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmCta& sm = *reinterpret_cast<SmCta*>(smem_raw);
  __shared__ int list[CTA_THREADS];
  __shared__ int count;
  const CtaGroup<CTA_THREADS> g;
  if (g.leader()) count = 0;
  pdl_wait();
  __syncthreads();
  const int64_t mine = blockIdx.x + (int64_t)gridDim.x * threadIdx.x;
  if (mine < P.n_frames && P.reason[mine] == MARK) list[atomicAdd(&count, 1)] = (int)mine;
  __syncthreads();
  const int n = count;
  for (int i = 0; i < n; ++i) {
    const int f = list[i];
    int r = frame_front<CtaGroup<CTA_THREADS>, SmCta, C_HITS, C_TRIP, false, false, false, true>(g, sm, C, P, f);
    if (r == PENDING)
      r = frame_back<CtaGroup<CTA_THREADS>, SmCta, C_TRIP, C_TRK, C_COMBO, false, false, true>(g, sm, C, P, f);
    finish_frame<CtaGroup<CTA_THREADS>, SmCta, true>(g, sm, P, f, r);
    g.sync();
  }
}

template <class K>
cudaError_t set_smem(K k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

size_t fused_smem_bytes() { return sizeof(SmWarp) * WARPS_PER_CTA; }
size_t cta_smem_bytes() { return sizeof(SmCta); }

int fused_blocks_per_sm() {
  int nb = 0;
  set_smem(k_select_warp<false>, fused_smem_bytes());
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_select_warp<false>, WARPS_PER_CTA * 32,
                                                    fused_smem_bytes()) != cudaSuccess)
    return 1;
  return nb > 0 ? nb : 1;
}

cudaError_t launch_fused(const DevCfg& c, const KParams& p, int grid, bool debug, cudaStream_t s) {
  const size_t sm = fused_smem_bytes();
  if (debug) {
    cudaError_t e = set_smem(k_select_warp<true>, sm);
    if (e != cudaSuccess) return e;
    k_select_warp<true><<<grid, WARPS_PER_CTA * 32, sm, s>>>(c, p);
  } else {
    cudaError_t e = set_smem(k_select_warp<false>, sm);
    if (e != cudaSuccess) return e;
    k_select_warp<false><<<grid, WARPS_PER_CTA * 32, sm, s>>>(c, p);
  }
  return cudaGetLastError();
}

// pdl: the kernel before it on the stream is the one that wrote the list.
cudaError_t launch_deferred(const DevCfg& c, const KParams& p, int grid, bool debug, cudaStream_t s, bool pdl) {
  const size_t sm = cta_smem_bytes();
  if (debug) {
    cudaError_t e = set_smem(k_select_cta<CTA_THREADS, true, true>, sm);
    if (e != cudaSuccess) return e;
    e = launch_kernel(pdl, k_select_cta<CTA_THREADS, true, true>, grid, CTA_THREADS, sm, s, c, p);
    if (e != cudaSuccess) return e;
  } else {
    cudaError_t e = set_smem(k_select_cta<CTA_THREADS, false, true>, sm);
    if (e != cudaSuccess) return e;
    e = launch_kernel(pdl, k_select_cta<CTA_THREADS, false, true>, grid, CTA_THREADS, sm, s, c, p);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

// A batch of at most SMALL_FRAMES frames (no scratch, no counters to clear).
cudaError_t launch_small(const DevCfg& c, KParams p, int sms, cudaStream_t s) {
  p.defer_hits = SMALL_HITS;
  const bool wide = p.n_frames <= 4 * sms;
  cudaError_t e = wide ? set_smem(k_select_small<256, 4>, sizeof(SmSmall)) : set_smem(k_select_small<128, 8>, sizeof(SmSmall));
  if (e == cudaSuccess) e = set_smem(k_select_marked, sizeof(SmCta));
  if (e != cudaSuccess) return e;
  if (wide) k_select_small<256, 4><<<(int)p.n_frames, 256, sizeof(SmSmall), s>>>(c, p);
  else k_select_small<128, 8><<<(int)p.n_frames, 128, sizeof(SmSmall), s>>>(c, p);
  const int grid = (int)(p.n_frames < 2 * sms ? p.n_frames : 2 * sms);
  return launch_kernel(true, k_select_marked, grid, CTA_THREADS, sizeof(SmCta), s, c, p);
}

cudaError_t launch_plain(const DevCfg& c, const KParams& p, bool debug, cudaStream_t s) {
  const size_t sm = cta_smem_bytes();
  const int grid = (int)(p.n_frames < 0x7fffffff ? p.n_frames : 0x7fffffff);
  if (grid == 0) return cudaSuccess;
  if (debug) {
    cudaError_t e = set_smem(k_select_cta<PLAIN_THREADS, true, false>, sm);
    if (e != cudaSuccess) return e;
    k_select_cta<PLAIN_THREADS, true, false><<<grid, PLAIN_THREADS, sm, s>>>(c, p);
  } else {
    cudaError_t e = set_smem(k_select_cta<PLAIN_THREADS, false, false>, sm);
    if (e != cudaSuccess) return e;
    k_select_cta<PLAIN_THREADS, false, false><<<grid, PLAIN_THREADS, sm, s>>>(c, p);
  }
  return cudaGetLastError();
}

}  // namespace m3e
