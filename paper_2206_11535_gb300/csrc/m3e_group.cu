// Group form of the selection: one persistent kernel without global intermediates, for
// calls that must not use scratch and for batches too small to pay for the staged form's
// eight launches.  A CTA takes G_FRAMES frames at a time through the method together:
//   warp per frame       load, sort and selection cuts, in shared memory
//   thread per triplet   track reconstruction over the triplets of all the CTA's frames
//   warp per frame       track and combination caps, energy test
//   thread per combination   vertex over the combinations of all the CTA's frames
// so that the fits, the largest part, run with full warps even when a frame has only a few
// triplets (8.6 at the nominal muon rate), and the warps of a CTA share their instructions.
// Frames beyond a frame's stage go to the deferred list for the CTA-per-frame kernel.
#include "m3e_device.cuh"

namespace m3e {
namespace {

// Frames and CTAs per SM, 15,625 nominal frames without allocation: 8 and 4 63 us, 4 and 8
// 65 us, 16 and 2 62 us, 8 and 3 (80 registers, no spills) 68 us; the warp-per-frame kernel
// that this one replaces there took 121 us (no_instruction stalls 5.1 per issue, 14.7 of 32
// lanes; here 1.3 and 24.2).  Bound by the barriers behind the cuts (7.0 per issue): a group
// waits for its largest frame.
constexpr int G_FRAMES = 8;
constexpr int G_THREADS = 32 * G_FRAMES;
constexpr int G_CTAS = 4;        // resident CTAs per SM
constexpr int G_TRK = 48;         // kept tracks of a frame
constexpr int NO_TRACK = 255;

// One frame's stage.  What the cuts need beyond the hits and the triplets makes room for
// the tracks once they are done, phi for the e- list once the fits are done, the triplets
// for the combinations.
struct GroupFrame {
  static constexpr bool kIdx = false, kStats = false, kPackB = true;
  using TripT = uchar4;
  alignas(16) float2 xy[W_HITS];
  float z[W_HITS];
  union {
    alignas(16) float phi[W_HITS];
    alignas(16) float4 nEP[G_TRK / 2];
  };
  union {
    struct {                      // selection cuts (FrameSm has their description)
      alignas(16) float ox[W_L0];
      alignas(16) float oy[W_L0];
      alignas(16) float zx[W_L2];
      alignas(16) float zy[W_L2];
      float2 zzi[W_L2];
      uint16_t p01[W_P01];
      alignas(16) uint16_t cand[W_CAND];
      uint8_t zbs[NZB + 1];
    };
    struct {                      // kept tracks, in the order in which they were fitted
      float2 pEP[G_TRK];          // e+ tracks as energy_test reads them
      float2 ep[G_TRK];           // (eps E, P_z)
      float cx[G_TRK], cy[G_TRK], R[G_TRK], ct[G_TRK], st[G_TRK], ah0[G_TRK];
      uint8_t i0[G_TRK];          // layer-0 hit
      uint8_t slot[W_TRIP];       // the track of each triplet, or NO_TRACK
      uint8_t pidx[G_TRK], nidx[G_TRK];  // the track of each entry of the e+ / e- list
    };
  };
  union {
    TripT trip[W_TRIP];
    uint32_t combo[W_TRIP];       // combinations to fit: tracks a | b << 8 | e- << 16
  } u;
  uint32_t bcur[NBK / 4];
  uint16_t bstart[NBK + 1], inidx[1];
  int ntrip, npos, nneg, ncombo, nstore, flag, bad;
  unsigned long long acc[1], facc[1];
};
static_assert(W_HITS <= 256 && G_TRK < NO_TRACK, "8-bit indices");

__device__ __forceinline__ TrackR load_track(const GroupFrame& s, int k, const DevCfg& C) {
  TrackR t;
  const int h = s.i0[k];
  const float2 ep = s.ep[k];
  t.cx = s.cx[k];
  t.cy = s.cy[k];
  t.R = s.R[k];
  t.ct = s.ct[k];
  t.st = s.st[k];
  t.rt = __fmul_rn(t.R, t.st);  // as the track record's, whatever the compiler contracts
  t.p = __fmul_rn(C.kB, t.R);
  t.E = fabsf(ep.x);
  t.sms = C.hl[0] / t.p;
  const float2 h0 = s.xy[h];
  t.h0x = h0.x;
  t.h0y = h0.y;
  t.h0z = s.z[h];
  t.ah0 = s.ah0[k];
  t.eps = ep.x > 0.f ? 1.f : -1.f;
  return t;
}

// This CTA's item i of the frames' item counts (inc: their inclusive prefix, lane w has
// frame w's): the frame, and the item's number in it.
__device__ __forceinline__ int frame_of(int inc, int i, int& k) {
  int w = 0;
#pragma unroll
  for (int st = G_FRAMES / 2; st; st >>= 1) {
    const int pv = __shfl_sync(FULL, inc, w + st - 1);
    if (pv <= i) w += st;
  }
  const int before = __shfl_sync(FULL, inc, w ? w - 1 : 0);
  k = i - (w ? before : 0);
  return w;
}

__device__ __forceinline__ int prefix8(int v) {  // inclusive prefix over the first G_FRAMES lanes
#pragma unroll
  for (int o = 1; o < G_FRAMES; o <<= 1) {
    const int t = __shfl_up_sync(FULL, v, o);
    if ((int)(threadIdx.x & 31) >= o) v += t;
  }
  return v;
}

__global__ void __launch_bounds__(G_THREADS, G_CTAS)
    k_select_group(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  GroupFrame* const fr = reinterpret_cast<GroupFrame*>(smem_raw);
  __shared__ int s_base, s_n[G_FRAMES], s_found[G_FRAMES];
  const WarpGroup g;
  const int w0 = threadIdx.x >> 5, lane = threadIdx.x & 31;
  GroupFrame& sm = fr[w0];
  const int nf = (int)P.n_frames;
  pdl_trigger();
  for (;;) {
    if (threadIdx.x == 0) s_base = atomicAdd(&P.work[0], G_FRAMES);
    __syncthreads();
    const int f = s_base + w0;
    if (s_base >= nf) break;
    // ---- cuts, warp per frame
    int r = M3E_DROP;
    if (f < nf) r = frame_front<WarpGroup, GroupFrame, W_HITS, W_TRIP, true, false, false, true, true>(g, sm, C, P, f);
    if (r == PENDING && sm.ntrip == 0) r = M3E_DROP;
    if (lane == 0) {
      s_n[w0] = r == PENDING ? sm.ntrip : 0;
      s_found[w0] = 0;
    }
    __syncthreads();
    // ---- fits, thread per triplet
    int inc = prefix8(lane < G_FRAMES ? s_n[lane] : 0);
    int total = __shfl_sync(FULL, inc, G_FRAMES - 1);
    for (int i0 = 32 * w0; i0 < total; i0 += G_THREADS) {
      const int i = i0 + lane;
      int t;
      const int w = frame_of(inc, min(i, total - 1), t);
      if (i < total) {
        GroupFrame& s = fr[w];
        const uchar4 q = s.u.trip[t];
        const SmHits<GroupFrame> v{s};
        const TrackOut o = build_track(v, C, q.x, q.y, q.z);
        int slot = NO_TRACK;
        if (o.status == 5) {
          slot = atomicAdd(&s.nstore, 1);
          if (slot < G_TRK) {
            float tk[14];
            track_record(v.pos(q.x), v.pos(q.y), o, C, tk);
            s.cx[slot] = tk[0];
            s.cy[slot] = tk[1];
            s.R[slot] = tk[3];
            s.ct[slot] = tk[4];
            s.st[slot] = tk[5];
            s.ah0[slot] = tk[12];
            s.ep[slot] = make_float2(tk[13] * tk[7], pz_track(tk[6], tk[4]));
            s.i0[slot] = q.x;
          }
        }
        s.slot[t] = (uint8_t)min(slot, NO_TRACK);
      }
    }
    __syncthreads();
    // ---- energy test, warp per frame
    int nwrite = 0;
    if (r == PENDING) {
      const int nt = sm.ntrip;
      if (sm.nstore > G_TRK) {
        r = DEFERRED;
      } else {
        int npos = 0, nneg = 0, ncombo = 0, nopen = 0;
        for (int t0 = 0; t0 < nt; t0 += 32) {
          const int k = t0 + lane < nt ? sm.slot[t0 + lane] : NO_TRACK;
          const float2 te = k != NO_TRACK ? sm.ep[k] : make_float2(0.f, 0.f);
          list_tracks(te, sm.pEP, sm.nEP, G_TRK, npos, nneg,
                      [&](int j, bool pos) { (pos ? sm.pidx : sm.nidx)[j] = (uint8_t)k; });
        }
        close_lists(sm.nEP, G_TRK, nneg);
        if (npos + nneg > C.max_trk) r = M3E_TRACK_OVERFLOW;
        if (r == PENDING) {
          energy_test(C, sm.pEP, sm.nEP, npos, nneg, true, false, C.max_combo, ncombo, nwrite, nopen, [&](int k, int a, int b, int c) {
            if (k < W_TRIP) sm.u.combo[k] = (uint32_t)sm.pidx[a] | (uint32_t)sm.pidx[b] << 8 | (uint32_t)sm.nidx[c] << 16;
          });
          if (ncombo > C.max_combo) r = M3E_COMBO_OVERFLOW;
          else if (nwrite == 0) r = M3E_DROP;
          else if (nwrite > W_TRIP) r = DEFERRED;
        }
      }
    }
    if (lane == 0) s_n[w0] = r == PENDING ? nwrite : 0;
    __syncthreads();
    // ---- vertices, thread per combination
    inc = prefix8(lane < G_FRAMES ? s_n[lane] : 0);
    total = __shfl_sync(FULL, inc, G_FRAMES - 1);
    for (int i0 = 32 * w0; i0 < total; i0 += G_THREADS) {
      const int i = i0 + lane;
      int k;
      const int w = frame_of(inc, min(i, total - 1), k);
      if (i < total && !*(volatile int*)&s_found[w]) {
        const GroupFrame& s = fr[w];
        const uint32_t code = s.u.combo[k];
        const int a = code & 255, b = (code >> 8) & 255, e = code >> 16;
        const float ca[3] = {s.cx[a], s.cy[a], __fmul_rn(s.R[a], s.st[a])}, cb[3] = {s.cx[b], s.cy[b], __fmul_rn(s.R[b], s.st[b])},
                    ce[3] = {s.cx[e], s.cy[e], __fmul_rn(s.R[e], s.st[e])};
        if (vertex_prefilter(ca, cb, ce, C.isect_lim) == 2 &&
            vertex(load_track(s, a, C), load_track(s, b, C), load_track(s, e, C), C).pass)
          s_found[w] = 1;
      }
    }
    __syncthreads();
    // ---- decision
    if (f < nf && lane == 0) {
      if (r == DEFERRED) {
        P.defer_list[atomicAdd(P.defer_count, 1)] = f;
      } else {
        if (r == PENDING) r = s_found[w0] ? M3E_VERTEX : M3E_DROP;
        P.keep[f] = (uint8_t)(r != M3E_DROP);
        P.reason[f] = (uint8_t)r;
      }
    }
  }
}

}  // namespace

size_t group_smem_bytes() { return sizeof(GroupFrame) * G_FRAMES; }

// Resident CTAs per SM (and the shared-memory limit of the kernel, once per context).
int group_blocks_per_sm() {
  int nb = 0;
  cudaFuncSetAttribute(k_select_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)group_smem_bytes());
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_select_group, G_THREADS, group_smem_bytes()) != cudaSuccess)
    return 1;
  return nb > 0 ? nb : 1;
}

cudaError_t launch_group(const DevCfg& c, const KParams& p, int resident, cudaStream_t s) {
  const int64_t want = (p.n_frames + G_FRAMES - 1) / G_FRAMES;
  k_select_group<<<(int)(want < resident ? want : resident), G_THREADS, group_smem_bytes(), s>>>(c, p);
  return cudaGetLastError();
}

}  // namespace m3e
