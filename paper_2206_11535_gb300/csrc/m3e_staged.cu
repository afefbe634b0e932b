// Staged selection kernels of libm3e: the same method as the fused kernels,
// with the work of a batch regrouped by candidate instead of by frame.
//   stage 1  warp per frame: decode, phi-bin sort, selection cuts (Algorithm 2);
//            the sorted hits and the selected triplets go to global memory
//   stage 2  thread per triplet of the whole batch: track reconstruction (Algorithm 3)
//   stage 3  warp per frame: track cap, energy test (Algorithm 4, part 1);
//            combinations go to global memory
//   stage 4  thread per combination of the whole batch: vertex (Algorithm 4, part 2)
//   stage 5  thread per frame: decision (store_frame of Algorithm 1)
// Every kernel is small and runs one kind of work, so warps share their
// instructions and lanes; a frame's candidates stay contiguous, so its hits and
// tracks are read from L2 by neighbouring threads.  Frames that exceed a stage's
// capacity are deferred to the CTA-per-frame kernel with identical decisions.
#include <algorithm>

#include "m3e_device.cuh"

namespace m3e {
namespace {

constexpr int NL3 = NB + 2;                        // layer-3 bin starts per frame (NB + 1, in whole words)
constexpr int FILTERED = INT32_MIN;                // bit of a combination's first triplet: prefilter passed
constexpr int S1_TRIP = 160;                       // stage-1 warp-tier triplet capacity
// input indices only for the candidate record; the instance without statistics code has
// no room for them
using SmFrontN = FrameSm<W_HITS, S1_TRIP, 1, 1, false, false>;
using SmFront = FrameSm<W_HITS, S1_TRIP, 1, 1, false>;
using SmFrontD = FrameSm<W_HITS, S1_TRIP, 1, 1>;
constexpr int M_HITS = 1024;                       // stage-1 middle tier (CTA per frame)
using SmFrontMid = FrameSm<M_HITS, C_TRIP, 1, 1>;
using SmFrontCta = FrameSm<C_HITS, C_TRIP, 1, 1>;
constexpr int S3_WARPS = 4;
constexpr int S3_BUF = 96;   // combinations a warp of stage 3 collects before writing
constexpr int S3_CHUNK = 4;  // frames a warp of stage 3 takes at a time, at most

template <bool STATS>
struct S3Sm {                                      // stage 3, per warp
  float4 nEP[C_TRK / 2];                           // tracks as energy_test reads them
  float2 pEP[C_TRK];
  uint16_t pidx[C_TRK], nidx[C_TRK];               // triplet of each, counted in its frame
  int4 buf[S3_BUF];                                // combinations to write
  unsigned long long acc[STATS ? ST_REASON0 + 8 : 1];
};

// ---- stage 1: write-out of a frame whose cuts selected triplets
// The sorted hits of frame f take the places of its input hits (off[f] - off_base
// onwards, so no allocator is needed); its triplets go to a range taken from the
// triplet allocator, whose atomic is issued first and waited for only after the
// hits are written.  A frame that does not fit is deferred (returns false).
template <class G, class Sm, bool DEBUG>
__device__ __forceinline__ bool emit_frame(const G& g, Sm& sm, const DevCfg& C, const KParams& P, const SParams& S,
                                           int f, int n, int ntrip, long long* bcast) {
  long long tb = 0;
  if (g.leader()) tb = (long long)atomicAdd(&S.counters[0], (unsigned long long)ntrip);
  const long long hb = P.off[f] - P.off_base;
  const bool hits_fit = hb + n <= S.hits_cap;
  const int l3s = sm.bstart[3 * NB];  // phi of a sorted hit serves only the layer-3 search of stage 2
#pragma unroll 1
  for (int i = g.rank(); hits_fit && i < n; i += G::N) {
    const float2 p = sm.xy[i];
    S.hp[hb + i] = make_float4(p.x, p.y, sm.z[i], i >= l3s ? sm.phi[i] : 0.f);
    if constexpr (DEBUG) {
      static_assert(Sm::kIdx, "the candidate record needs the input indices");
      S.hidx[hb + i] = sm.inidx[i];
    }
  }
  if constexpr (G::N == 32) {
    tb = __shfl_sync(FULL, tb, 0);
  } else {
    if (g.leader()) bcast[1] = tb;
    g.sync();
    tb = bcast[1];
    g.sync();
  }
  if (!hits_fit || tb + ntrip > S.trip_cap) {
    // out of space: mark the triplet slots this frame owns below the cap as unused
    for (int64_t t = tb + g.rank(); t < S.trip_cap && t < tb + ntrip; t += G::N) S.trip[t] = make_int4(-1, 0, 0, 0);
    return false;
  }
  if (g.rank() < NL3 / 2)
    reinterpret_cast<uint32_t*>(S.l3 + (int64_t)f * NL3)[g.rank()] =
        (uint32_t)sm.bstart[3 * NB + 2 * g.rank()] | (uint32_t)sm.bstart[3 * NB + 2 * g.rank() + 1] << 16;
#pragma unroll 1
  for (int t = g.rank(); t < ntrip; t += G::N) {
    const auto q = sm.u.trip[t];
    S.trip[tb + t] = make_int4(f, (int)hb, (int)q.x | ((int)q.y << 16), (int)q.z);
  }
  if (g.leader()) {
    S.fstate[f] = PENDING;
    S.ftbase[f] = (int)tb;
    S.fntrip[f] = ntrip;
    S.ffound[f] = 0;
  }
  return true;
}

// After frame_front: decide, emit, or defer one frame (stage-1 tiers).
template <class G, class Sm, bool DEBUG, bool NOST = false>
__device__ __forceinline__ void stage1_finish(const G& g, Sm& sm, const DevCfg& C, const KParams& P, const SParams& S,
                                              int f, int r, long long* bcast) {
  const int ntrip = sm.ntrip;
  if (r == PENDING && ntrip == 0) r = M3E_DROP;  // no triplet: no track, no vertex
  if (r == PENDING) {
    const int n = (int)(P.off[f + 1] - P.off[f]);
    if (emit_frame<G, Sm, DEBUG>(g, sm, C, P, S, f, n, ntrip, bcast)) {
      if (!NOST && g.leader() && P.stats)
        for (int k = 0; k < ST_REASON0; ++k) sm.acc[k] += sm.facc[k];
    } else {
      r = DEFERRED;
    }
  }
  if (r == DEFERRED) {
    if (g.leader()) {
      S.fstate[f] = DEFERRED;
      const int k = atomicAdd(P.defer_count, 1);
      P.defer_list[k] = f;
      if (!NOST && P.stats) sm.acc[ST_DEFER] += 1;
    }
  } else if (r != PENDING) {
    if (g.leader()) S.fstate[f] = r;
    finish_frame<G, Sm, NOST>(g, sm, P, f, r);
  }
  g.sync();
}

__device__ __forceinline__ unsigned ld_acquire_sys_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Host entry point: wait until the copy engine has flagged chunk k as arrived.
// The wait is bounded by P.gate_ms; it also ends once another warp has given up.
// Returns false when it gave up (ERR_GATE latched).
__device__ bool gate_wait(const KParams& P, int k) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) {
    const unsigned long long t_end = global_ns() + (unsigned long long)P.gate_ms * 1000000ull;
    unsigned ns = 64;
    while (ld_acquire_sys_u32(P.gate + k) == 0u) {
      if ((*(volatile int*)P.err & ERR_GATE) || global_ns() > t_end) {
        atomicOr(P.err, ERR_GATE);
        ok = 0;
        break;
      }
      __nanosleep(ns);
      if (ns < 2048) ns *= 2;
    }
  }
  __syncwarp();
  return __shfl_sync(FULL, ok, 0) != 0;
}

// ---- stage 1, warp tier: one warp per frame, frames from the device queue.
// GATED (host entry point): the hits arrive while the kernel runs; a frame is
// taken only after its chunk's arrival flag, and the hits are read past L1.
// NOST: the instance for runs without statistics (no statistics code at all).
// Bound by instruction issue and shared-memory latency (1,857 warp instructions per
// throughput frame at 66% issue active; shared-memory loads are the largest stall): 1e6
// throughput frames 2.36 -> 2.15 ms with the packed partner masks, one decode per hit and no
// address list, at 64 registers and 8 CTAs per SM (2.20 ms at 56 registers and 9 CTAs),
// 2.09 ms with x and y in one copy per hit, and 2.02 ms with its loops rolled: a warp is
// seldom where another one is, so every instruction fetched less counts (the masks unrolled
// by 4 instead of 1: 2.27 ms).  2.01 ms with the layer-3 bin starts written two by two.
template <bool DEBUG, bool GATED = false, bool NOST = false>
__global__ void __launch_bounds__(WARPS_PER_CTA * 32)
    k_stage1(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P, const __grid_constant__ SParams S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using Sm = typename std::conditional<DEBUG, SmFrontD, typename std::conditional<NOST, SmFrontN, SmFront>::type>::type;
  Sm& sm = reinterpret_cast<Sm*>(smem_raw)[threadIdx.x >> 5];
  __shared__ long long bcast[WARPS_PER_CTA][2];
  const WarpGroup g;
  if (!NOST) clear_stats(g, sm);
  pdl_trigger();
  const int nf = (int)P.n_frames;
  int arrived = -1;  // chunks up to this one are known to have arrived
  bool stop = false;
  while (!stop) {
    int f0 = 0;
    if (g.leader()) f0 = atomicAdd(&P.work[0], P.grab);
    f0 = __shfl_sync(FULL, f0, 0);
    if (f0 >= nf) break;
    const int f1 = min(f0 + P.grab, nf);
    for (int f = f0; f < f1; ++f) {
      if constexpr (GATED) {
        const int k = f / P.gate_frames;
        if (k > arrived) {
          if (!gate_wait(P, k)) {
            stop = true;
            break;
          }
          arrived = k;
        }
      }
      const int r = frame_front<WarpGroup, Sm, W_HITS, S1_TRIP, true, DEBUG, GATED, NOST, true>(g, sm, C, P, f, f + 1 < f1);
      stage1_finish<WarpGroup, Sm, DEBUG, NOST>(g, sm, C, P, S, f, r, bcast[threadIdx.x >> 5]);
    }
  }
  if (!NOST) flush_stats(g, sm, P.stats);
}

// ---- stage 1, CTA tiers: one CTA per frame deferred by the tier below (large
// frames); the middle tier stages up to M_HITS hits, the top tier C_HITS.
// NT: threads of a CTA (the middle tier's is a tuning parameter).
template <class Sm, int CH, bool DEBUG, int NT = CTA_THREADS, bool NOST = false>
__global__ void __launch_bounds__(NT)
    k_stage1c(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P, const __grid_constant__ SParams S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Sm& sm = *reinterpret_cast<Sm*>(smem_raw);
  __shared__ long long bcast[2];
  const CtaGroup<NT> g;
  clear_stats(g, sm);
  pdl_trigger();
  pdl_wait();
  const int count = *P.in_count;
  for (int i = blockIdx.x; i < count; i += gridDim.x) {
    const int f = P.in_list[i];
    int r;
    if (CH < C_HITS && P.off[f + 1] - P.off[f] > CH) r = DEFERRED;  // for the next tier
    else r = frame_front<CtaGroup<NT>, Sm, CH, C_TRIP, false, DEBUG, false, NOST>(g, sm, C, P, f);
    stage1_finish<CtaGroup<NT>, Sm, DEBUG, NOST>(g, sm, C, P, S, f, r, bcast);
  }
  if (!NOST) flush_stats(g, sm, P.stats);
}

// ---- stage 2: one thread per selected triplet
// Bound by issue and the latency of the hit loads (2,060 warp instructions per throughput frame
// at 73% issue active, 27 of 32 lanes, 27 warps per SM).  What it holds across the fits counts
// twice, as a spill and as a load issued late: with the next record fetched into L1 instead of
// into four registers, 32-bit indices, the layer-3 range loaded beside the triplet's hits and
// the layer-3 scan unrolled by 6, 1e6 throughput frames take 2.26 ms instead of 2.32, without
// spills.  The next triplet's hits fetched ahead too: 2.29 ms; 9 CTAs per SM at 56 registers:
// 2.31 ms; the record by cp.async: 2.27 ms.
template <bool DEBUG>
__global__ void __launch_bounds__(128, 8)  // 8 CTAs per SM (64 registers: the first fit parked in shared memory)
    k_stage2(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P, const __grid_constant__ SParams S) {
  static_assert(sizeof(FitPark) == 11 * 128 * sizeof(float), "one slot per thread of a 128-thread CTA");
  __shared__ FitPark park;
  pdl_trigger();
  pdl_wait();
  // below 2^31 (scratch_entries), so i + stride does not wrap
  const unsigned n = (unsigned)min((int64_t)S.counters[0], S.trip_cap);
  const unsigned stride = gridDim.x * blockDim.x;
  unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  for (; i < n; i += stride) {
    // the record carries the frame, its first sorted hit and the three frame-relative
    // indices; the next record is fetched into L1 while this triplet is fitted
    const int4 r = S.trip[i];
    if (i + stride < n) asm volatile("prefetch.global.L1 [%0];" ::"l"(S.trip + i + stride));
    const int f = r.x;
    if (f < 0) continue;
    const int64_t base = (int64_t)(unsigned)r.y;
    const int i0 = r.z & 0xffff, i1 = (int)((unsigned)r.z >> 16), i2 = r.w;
    const uint16_t* l3 = S.l3 + (int64_t)f * NL3;
    // (the candidate record's instance keeps the order of loads in which its values were rounded)
    const GHits<!DEBUG> v{S.hp + base, l3, &park, DEBUG ? 0u : (unsigned)__ldg(l3) | (unsigned)__ldg(l3 + NB) << 16};
    const TrackOut o = build_track(v, C, i0, i1, i2);
    float2 te = make_float2(0.f, 0.f);
    if (o.status == 5) {
      float tk[14];
      track_record(v.pos(i0), v.pos(i1), o, C, tk);
      te = make_float2(tk[13] * tk[7], pz_track(tk[6], tk[4]));  // what the energy test reads
      store_record(S.trec, i, tk, r.y + i0);
    }
    S.tek[i] = te;
    if (DEBUG) {
      const int t = (int)(i - S.ftbase[f]);
      if (t < P.dump.cap_trip) {
        const int64_t d = (int64_t)f * P.dump.cap_trip + t;
        P.dump.trip[4 * d + 0] = S.hidx[base + i0];
        P.dump.trip[4 * d + 1] = S.hidx[base + i1];
        P.dump.trip[4 * d + 2] = S.hidx[base + i2];
        P.dump.trip[4 * d + 3] = o.i3 >= 0 ? (int)S.hidx[base + o.i3] : -1;
        P.dump.trk_status[d] = o.status;
        P.dump.trk_val[4 * d + 0] = o.kbar;
        P.dump.trk_val[4 * d + 1] = o.th01;
        P.dump.trk_val[4 * d + 2] = o.chi2;
        P.dump.trk_val[4 * d + 3] = o.mbest;
      }
    }
  }
}

__device__ __forceinline__ void load_circle(const float4* __restrict__ rec, int64_t k, float& cx, float& cy,
                                            float& rt) {
  const float4 a = __ldg(rec + 2 * k);
  cx = a.x;
  cy = a.y;
  rt = a.z;
}

// ---- stage 3: warp per frame, track cap and energy test (NOST: the instance for
// runs without statistics).
// A warp takes P.grab frames at a time: their states are read together, a lane each, the
// tracks of the next frame are fetched into L1 while one is tested, and the combinations of all of
// them are written behind one allocation, a fourth of the atomics on the one counter.
// Bound by issue (850 warp instructions per throughput frame, 71% issue active, 10 CTAs per
// SM at 48 registers; 9 CTAs at 56 take 2% longer, 12 CTAs 13%): 1e6 throughput frames 854 -> 719 us,
// 200,000 uneven frames 541 -> 283 us, most of that from frames that stop at the combination
// cap.  Taking 16 frames at a time cost 745 and 535 us (heavy frames queue in one warp).
// Before they are written the combinations go through the vertex's first two steps, which
// three in four do not survive: their gathers of track circles from DRAM bounded stage 4 and
// fit beside the arithmetic here (this stage 719 -> 817 us, stage 4 399 -> 225 us).  The next
// frame's tracks went into four registers at first, and the kernel spilled 148 bytes a thread;
// fetched into L1 instead, nothing and 793 us.
template <bool DEBUG, bool NOST = false>
__global__ void __launch_bounds__(S3_WARPS * 32, 10)
    k_stage3(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P, const __grid_constant__ SParams S) {
  __shared__ S3Sm<!NOST> smem[S3_WARPS];
  S3Sm<!NOST>& sm = smem[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  if (!NOST)
    for (int k = lane; k < ST_REASON0 + 8; k += 32) sm.acc[k] = 0;
  __syncwarp();
  pdl_trigger();
  pdl_wait();
  const int nf = (int)P.n_frames;
  const bool stats = !NOST && P.stats != nullptr;
  // all energy-test survivors count towards the cap; a decision-only run writes only those
  // whose P_z leaves the momentum cut open (pz_fails_ptot)
  const bool prune = !DEBUG && !stats;
  for (;;) {
    int f0 = 0;
    if (lane == 0) f0 = (int)atomicAdd(&S.counters[2], (unsigned long long)P.grab);
    f0 = __shfl_sync(FULL, f0, 0);
    if (f0 >= nf) break;
    // this lane's frame: state, triplet range, decision taken here, combinations collected
    const int f = f0 + lane;
    const bool mine = lane < P.grab && f < nf;
    int tbase = 0, ntrip = 0, r = PENDING, at = -1, stat_combo = 0, stat_open = 0;
    bool pending = false;
    if (mine) {
      pending = S.fstate[f] == PENDING;
      tbase = S.ftbase[f];
      ntrip = S.fntrip[f];
    }
    unsigned todo = __ballot_sync(FULL, pending);
    int fill = 0;  // combinations in the buffer
    auto load = [&](int j, int t) {  // (eps E, P_z) of triplet t + lane of lane j's frame, (0, 0) beyond them
      const int tb = __shfl_sync(FULL, tbase, j), nt = __shfl_sync(FULL, ntrip, j);
      return t + lane < nt ? __ldg(S.tek + tb + t + lane) : make_float2(0.f, 0.f);
    };
    // n combinations get a range of the scratch: its start, or -1 when it is full
    auto allocate = [&](int n) -> long long {
      long long cb = 0;
      if (lane == 0) cb = (long long)atomicAdd(&S.counters[1], (unsigned long long)n);
      cb = __shfl_sync(FULL, cb, 0);
      if (cb + n <= S.combo_cap) return cb;
      for (int64_t t = cb + lane; t < S.combo_cap; t += 32) S.combo[t] = make_int4(-1, 0, 0, 0);
      return -1;
    };
    // frames whose combinations went to the range at cb (at: this lane's place in it), or found no room
    auto placed = [&](long long cb) {
      if (at < 0) return;
      if (cb < 0) {
        r = DEFERRED;
      } else {
        if (DEBUG) S.fcbase[f] = cb + at;
        if (stats) {
          atomicAdd(&sm.acc[ST_COMBO], (unsigned long long)stat_combo);
          atomicAdd(&sm.acc[ST_PZOPEN], (unsigned long long)stat_open);
        }
      }
      at = -1;
    };
    auto flush = [&]() {
      if (fill == 0) return;
      __syncwarp();
      if (!DEBUG) {
        // only the combinations that the vertex's first two steps leave go on; the others
        // decide nothing (the candidate record wants them all)
        int kept = 0;
        for (int t0 = 0; t0 < fill; t0 += 32) {
          const int t = t0 + lane;
          bool keep = t < fill;
          int4 q = make_int4(0, 0, 0, 0);
          if (keep) {
            q = sm.buf[t];
            float c[9];
            load_circle(S.trec, q.y, c[0], c[1], c[2]);
            load_circle(S.trec, q.z, c[3], c[4], c[5]);
            load_circle(S.trec, q.w, c[6], c[7], c[8]);
            keep = vertex_prefilter(c, c + 3, c + 6, C.isect_lim) == 2;
          }
          const unsigned m = __ballot_sync(FULL, keep);
          __syncwarp();
          q.y |= FILTERED;
          if (keep) sm.buf[kept + __popc(m & below)] = q;  // never beyond the entries read
          kept += __popc(m);
          __syncwarp();
        }
        fill = kept;
      }
      const long long cb = fill ? allocate(fill) : 0;
      for (int t = lane; cb >= 0 && t < fill; t += 32) S.combo[cb + t] = sm.buf[t];
      placed(cb);
      fill = 0;
      __syncwarp();
    };
    while (todo) {
      const int j = __ffs(todo) - 1;
      todo &= todo - 1u;
      const int tb = __shfl_sync(FULL, tbase, j), nt = __shfl_sync(FULL, ntrip, j), fj = f0 + j;
      const float2 te0 = load(j, 0), te1 = load(j, 32);
      if (todo) {
        const int tn = __shfl_sync(FULL, tbase, __ffs(todo) - 1), nn = __shfl_sync(FULL, ntrip, __ffs(todo) - 1);
        if (4 * lane < nn && lane < 16) asm volatile("prefetch.global.L1 [%0];" ::"l"(S.tek + tn + 4 * lane));
      }
      // kept tracks of the frame's triplets, split by charge
      int npos = 0, nneg = 0;
      auto list = [&](const float2& te, int t0) {
        list_tracks(te, sm.pEP, sm.nEP, C_TRK, npos, nneg,
                    [&](int k, bool pos) { (pos ? sm.pidx : sm.nidx)[k] = (uint16_t)(t0 + lane); });
      };
      list(te0, 0);
      if (nt > 32) list(te1, 32);
      for (int t0 = 64; t0 < nt; t0 += 32) list(load(j, t0), t0);
      close_lists(sm.nEP, C_TRK, nneg);
      int rj = PENDING, ncombo = 0, nopen = 0, nw = fill;
      if (npos + nneg > C.max_trk) rj = M3E_TRACK_OVERFLOW;
      if (rj == PENDING) {
        if (stats && lane == 0) {
          sm.acc[ST_TRK] += npos + nneg;
          sm.acc[ST_ETEST] += (unsigned long long)(npos * (npos - 1) / 2) * nneg;
        }
        auto record = [&](int a, int b, int c) {
          return make_int4(fj, tb + sm.pidx[a], tb + sm.pidx[b], tb + sm.nidx[c]);
        };
        energy_test(C, sm.pEP, sm.nEP, npos, nneg, prune, stats, DEBUG ? 1 << 30 : C.max_combo, ncombo, nw, nopen,
                    [&](int k, int a, int b, int c) {
                      if (k < S3_BUF) sm.buf[k] = record(a, b, c);
                    });
        if (DEBUG && lane == 0) P.dump.n_combo[fj] = ncombo;
        if (ncombo > C.max_combo) rj = M3E_COMBO_OVERFLOW;
        else if (nw == fill) rj = M3E_DROP;  // no combination, or none that can pass
        else {
          const int own = nw - fill;
          const bool fits = nw <= S3_BUF;
          if (!fits) flush();
          if (lane == j) {
            at = fill;
            stat_combo = ncombo;
            stat_open = nopen;
          }
          if (fits) {
            fill = nw;
          } else {
            // not beside the earlier ones: a second pass writes this frame's, in the same order
            const long long cb = allocate(own);
            int again = 0, c1 = 0, c2 = 0;
            if (cb >= 0)
              energy_test(C, sm.pEP, sm.nEP, npos, nneg, prune, false, 1 << 30, c1, again, c2,
                          [&](int k, int a, int b, int c) { S.combo[cb + k] = record(a, b, c); });
            placed(cb);
          }
        }
      }
      if (lane == j) r = rj == PENDING ? r : rj;
      __syncwarp();
    }
    flush();
    if (pending && r == DEFERRED) {
      S.fstate[f] = DEFERRED;
      P.defer_list[atomicAdd(P.defer_count, 1)] = f;
      if (stats) atomicAdd(&sm.acc[ST_DEFER], 1ull);
    } else if (pending && r != PENDING) {
      S.fstate[f] = r;
      P.keep[f] = (uint8_t)(r != M3E_DROP);
      P.reason[f] = (uint8_t)r;
      if (stats) atomicAdd(&sm.acc[ST_REASON0 + r], 1ull);
    }
  }
  __syncwarp();
  if (stats)
    for (int k = lane; k < ST_REASON0 + 8; k += 32)
      if (sm.acc[k]) atomicAdd(P.stats + k, sm.acc[k]);
}

// ---- stage 4: vertex of every combination, compacted per warp
// Most combinations stop at the first two steps (a pair of track circles that
// does not intersect, or no intersection inside the target filter).  Each warp
// therefore runs those steps on 32 combinations at a time, appends the survivors
// to a queue in shared memory, and runs the full vertex on 32 queued survivors at
// a time, so that all lanes do the expensive part together.  In a decision-only run stage 3
// has already dropped the others and marked these (FILTERED), except in frames with more
// combinations than its buffer.
// Bound by the latency of the track records and by spills: 1e6 throughput frames 229 us at 64
// registers (8 CTAs per SM) with every combination filtered again, 217 without that, 213 at 80
// registers, 191 at 96, 200 at 128 (no spills, 4 CTAs per SM); 200,000 uneven frames 68 -> 59.
// 205 with the e+ tracks ordered by value (vertex), which waits for both tracks' circles.
constexpr int S4_WARPS = 4;

template <bool DEBUG>
__device__ __forceinline__ void stage4_dump(const DevCfg& C, const KParams& P, const SParams& S, int64_t i,
                                            const int4& r, const VtxOut& v, const TrackR& A, const TrackR& B,
                                            const TrackR& E) {
  const float esum = fabsf(S.tek[r.y].x) + fabsf(S.tek[r.z].x) + fabsf(S.tek[r.w].x);
  const int f = r.x;
  const int c = (int)(i - S.fcbase[f]);
  if (c < P.dump.cap_combo) {
    const int64_t d = (int64_t)f * P.dump.cap_combo + c;
    const int tb = S.ftbase[f];
    P.dump.combo[4 * d + 0] = r.y - tb;
    P.dump.combo[4 * d + 1] = r.z - tb;
    P.dump.combo[4 * d + 2] = r.w - tb;
    P.dump.combo[4 * d + 3] = v.status | (v.pass << 8);
    P.dump.combo_val[4 * d + 0] = esum - C.m_mu;
    P.dump.combo_val[4 * d + 1] = v.chi2;
    P.dump.combo_val[4 * d + 2] = v.tdist;
    P.dump.combo_val[4 * d + 3] = v.ptot;
    if (P.dump.combo_aux) {
      float dm, fm;
      vertex_soft(A, B, E, C.isect_lim, dm, fm);
      P.dump.combo_aux[4 * d + 0] = dm;
      P.dump.combo_aux[4 * d + 1] = fm;
      P.dump.combo_aux[4 * d + 2] = v.chi2_second;
      P.dump.combo_aux[4 * d + 3] = 0.f;
    }
  }
}

template <bool DEBUG, bool NOST = false>
__global__ void __launch_bounds__(S4_WARPS * 32, 5)  // 96 registers
    k_stage4(const __grid_constant__ DevCfg C, const __grid_constant__ KParams P, const __grid_constant__ SParams S) {
  __shared__ long long queue[S4_WARPS][64];
  long long* q = queue[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  pdl_trigger();
  pdl_wait();
  const int64_t n = min((int64_t)S.counters[1], S.combo_cap);
  const int64_t stride = (int64_t)gridDim.x * S4_WARPS * 32;
  int qn = 0;
  unsigned nv = 0, nvo = 0;
  int64_t base = ((int64_t)blockIdx.x * S4_WARPS + (threadIdx.x >> 5)) * 32;
  // the combination records are fetched into L1 one step ahead; the three circles are
  // read together with the frame's state, before it is known whether they are needed
  for (;; base += stride) {
    const bool more = base < n;  // uniform in the warp
    if (more) {
      const int64_t i = base + lane;
      const int4 r = i < n ? S.combo[i] : make_int4(-1, 0, 0, 0);
      if (i + stride < n) asm volatile("prefetch.global.L1 [%0];" ::"l"(S.combo + i + stride));
      bool cand = false;
      if (i < n && r.x >= 0) {
        const int f = r.x;
        float ca[3], cb[3], ce[3];
        if (DEBUG || r.y >= 0) {
          load_circle(S.trec, r.y, ca[0], ca[1], ca[2]);
          load_circle(S.trec, r.z, cb[0], cb[1], cb[2]);
          load_circle(S.trec, r.w, ce[0], ce[1], ce[2]);
        }
        const bool open = DEBUG || !*((volatile int*)S.ffound + f);
        if (!DEBUG && r.y < 0) {
          cand = open;
        } else if (open) {
          const int st = vertex_prefilter(ca, cb, ce, C.isect_lim);
          cand = st == 2;
          if (DEBUG && !cand) {  // record the combination with its early status (the same geometry)
            const TrackR A = load_track(S.trec, S.hp, r.y, C), B = load_track(S.trec, S.hp, r.z, C), E = load_track(S.trec, S.hp, r.w, C);
            stage4_dump<DEBUG>(C, P, S, i, r, vertex(A, B, E, C), A, B, E);
          }
        }
      }
      const unsigned m = __ballot_sync(FULL, cand);
      if (cand) q[qn + __popc(m & ((1u << lane) - 1u))] = i;
      qn += __popc(m);
    }
    __syncwarp();
    while (qn >= 32 || (!more && qn > 0)) {
      const int take = qn < 32 ? qn : 32;
      if (lane < take) {
        const int64_t i = q[qn - take + lane];
        int4 r = S.combo[i];
        r.y &= ~FILTERED;
        const TrackR A = load_track(S.trec, S.hp, r.y, C), B = load_track(S.trec, S.hp, r.z, C), E = load_track(S.trec, S.hp, r.w, C);
        const VtxOut v = vertex(A, B, E, C);
        nv += v.status == 2;
        if (!NOST && P.stats && v.status == 2)
          nvo += !pz_fails_ptot(pz_sum(pz_track(A.p, A.ct), pz_track(B.p, B.ct), pz_track(E.p, E.ct)), C.ptot_max);
        if (v.pass) S.ffound[r.x] = 1;
        if (DEBUG) stage4_dump<DEBUG>(C, P, S, i, r, v, A, B, E);
      }
      qn -= take;
      __syncwarp();
    }
    if (!more) break;
  }
  if (!NOST && P.stats) {
    const unsigned s = __reduce_add_sync(FULL, nv), so = __reduce_add_sync(FULL, nvo);
    if (lane == 0 && s) atomicAdd(P.stats + ST_VTX, (unsigned long long)s);
    if (lane == 0 && so) atomicAdd(P.stats + ST_VTXOPEN, (unsigned long long)so);
  }
}

// ---- stage 5: decision of the frames still pending
__global__ void __launch_bounds__(256)
    k_stage5(const __grid_constant__ KParams P, const __grid_constant__ SParams S) {
  __shared__ unsigned cnt[2];
  if (threadIdx.x < 2) cnt[threadIdx.x] = 0;
  pdl_trigger();
  pdl_wait();
  __syncthreads();
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f < P.n_frames && S.fstate[f] == PENDING) {
    const int r = S.ffound[f] ? M3E_VERTEX : M3E_DROP;
    P.keep[f] = (uint8_t)(r != M3E_DROP);
    P.reason[f] = (uint8_t)r;
    if (P.stats) atomicAdd(&cnt[r], 1u);
  }
  __syncthreads();
  if (P.stats && threadIdx.x < 2 && cnt[threadIdx.x])
    atomicAdd(P.stats + ST_REASON0 + threadIdx.x, (unsigned long long)cnt[threadIdx.x]);
}

template <class K>
cudaError_t set_smem(K k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

size_t stage1_smem_bytes(bool debug, bool nost) {
  return (debug ? sizeof(SmFrontD) : nost ? sizeof(SmFrontN) : sizeof(SmFront)) * WARPS_PER_CTA;
}
size_t stage1c_smem_bytes() { return sizeof(SmFrontCta); }
size_t stage1m_smem_bytes() { return sizeof(SmFrontMid); }

int stage_blocks_per_sm(int stage) {
  int nb = 0;
  cudaError_t e = cudaSuccess;
  if (stage == 1) {
    set_smem(k_stage1<false, false, true>, stage1_smem_bytes(false, true));
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_stage1<false, false, true>, WARPS_PER_CTA * 32,
                                                      stage1_smem_bytes(false, true));
  } else if (stage == 2) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_stage2<false>, 128, 0);
  } else if (stage == 3) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_stage3<false, true>, S3_WARPS * 32, 0);
  } else if (stage == 4) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_stage4<false, true>, S4_WARPS * 32, 0);
  } else if (stage == 5) {
    set_smem(k_stage1c<SmFrontCta, C_HITS, false, CTA_THREADS, true>, stage1c_smem_bytes());
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_stage1c<SmFrontCta, C_HITS, false, CTA_THREADS, true>, CTA_THREADS,
                                                      stage1c_smem_bytes());
  } else {
    set_smem(k_stage1c<SmFrontMid, M_HITS, false, CTA_THREADS, true>, stage1m_smem_bytes());
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_stage1c<SmFrontMid, M_HITS, false, CTA_THREADS, true>, CTA_THREADS,
                                                      stage1m_smem_bytes());
  }
  return e == cudaSuccess && nb > 0 ? nb : 1;
}

template <int NT>
int mid_blocks_per_sm_t() {
  int nb = 0;
  set_smem(k_stage1c<SmFrontMid, M_HITS, false, NT, true>, stage1m_smem_bytes());
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &nb, k_stage1c<SmFrontMid, M_HITS, false, NT, true>, NT, stage1m_smem_bytes());
  return e == cudaSuccess && nb > 0 ? nb : 1;
}

int stage1_mid_blocks_per_sm(int threads) {
  return threads == 128 ? mid_blocks_per_sm_t<128>() : (threads == 512 ? mid_blocks_per_sm_t<512>() : mid_blocks_per_sm_t<256>());
}

// Stage 1 (warp tier; middle CTA tier over the warp tier's deferred frames; top
// CTA tier over the middle tier's), stages 2-5.  grids: stage 1 warp tier, 2, 3,
// 4, stage 1 top tier, stage 1 middle tier.  Frames deferred by the top tier or by
// stage 3 end up in S.list2 for the caller's CTA-per-frame kernel.  ev (9 events or
// null): before stage 1 and after each kernel.
// One launch of a CTA tier of stage 1 (the instance without statistics code when nost).
template <class Sm, int CH, bool DEBUG, int NT>
cudaError_t launch_tier(bool pdl, const DevCfg& c, const KParams& p, const SParams& s, int grid, size_t smem,
                        cudaStream_t st, bool nost) {
  if constexpr (!DEBUG) {
    if (nost) {
      const cudaError_t e = set_smem(k_stage1c<Sm, CH, false, NT, true>, smem);
      return e != cudaSuccess ? e : launch_kernel(pdl, k_stage1c<Sm, CH, false, NT, true>, grid, NT, smem, st, c, p, s);
    }
  }
  const cudaError_t e = set_smem(k_stage1c<Sm, CH, DEBUG, NT>, smem);
  return e != cudaSuccess ? e : launch_kernel(pdl, k_stage1c<Sm, CH, DEBUG, NT>, grid, NT, smem, st, c, p, s);
}

cudaError_t launch_staged(const DevCfg& c, const KParams& p, const SParams& s, const int grids[6], bool debug,
                          cudaStream_t st, cudaEvent_t* ev, cudaEvent_t after_s1, int mid_threads) {
  const bool gated = p.gate != nullptr && !debug;
  const bool nost = p.stats == nullptr;
  // every kernel after the first a programmatic dependent of the one before it, unless each
  // is timed apart or a copy stream's event comes between
  const bool pdl = ev == nullptr && p.n_frames <= DEPENDENT_FRAMES;
  const size_t sm1 = stage1_smem_bytes(debug, nost), smc = stage1c_smem_bytes(), smm = stage1m_smem_bytes();
  cudaError_t e = debug ? set_smem(k_stage1<true>, sm1)
                  : gated ? (nost ? set_smem(k_stage1<false, true, true>, sm1) : set_smem(k_stage1<false, true>, sm1))
                          : (nost ? set_smem(k_stage1<false, false, true>, sm1) : set_smem(k_stage1<false>, sm1));
  if (e != cudaSuccess) return e;
  KParams p1 = p, pm = p, pc = p, p3 = p;
  p1.defer_list = s.list1;
  p1.defer_count = s.lcount;
  pm.in_list = s.list1;
  pm.in_count = s.lcount;
  pm.defer_list = s.list1b;
  pm.defer_count = s.lcount + 2;
  pc.in_list = s.list1b;
  pc.in_count = s.lcount + 2;
  pc.defer_list = s.list2;
  pc.defer_count = s.lcount + 1;
  p3.defer_list = s.list2;
  p3.defer_count = s.lcount + 1;
  // frames a warp of stage 3 takes at a time: two takes for every resident warp
  p3.grab = (int)std::max<int64_t>(1, std::min<int64_t>(S3_CHUNK, p.n_frames / (2 * (int64_t)grids[2] * S3_WARPS)));
  if (ev) cudaEventRecord(ev[0], st);
  if (debug) k_stage1<true><<<grids[0], WARPS_PER_CTA * 32, sm1, st>>>(c, p1, s);
  else if (gated && nost) k_stage1<false, true, true><<<grids[0], WARPS_PER_CTA * 32, sm1, st>>>(c, p1, s);
  else if (gated) k_stage1<false, true><<<grids[0], WARPS_PER_CTA * 32, sm1, st>>>(c, p1, s);
  else if (nost) k_stage1<false, false, true><<<grids[0], WARPS_PER_CTA * 32, sm1, st>>>(c, p1, s);
  else k_stage1<false><<<grids[0], WARPS_PER_CTA * 32, sm1, st>>>(c, p1, s);
  // the later kernels read the hits too: order them after every copy of the host entry
  if (after_s1) cudaStreamWaitEvent(st, after_s1, 0);
  if (ev) cudaEventRecord(ev[1], st);
  e = debug ? launch_tier<SmFrontMid, M_HITS, true, CTA_THREADS>(pdl && !after_s1, c, pm, s, grids[5], smm, st, false)
            : mid_threads == 128 ? launch_tier<SmFrontMid, M_HITS, false, 128>(pdl && !after_s1, c, pm, s, grids[5], smm, st, nost)
            : mid_threads == 512 ? launch_tier<SmFrontMid, M_HITS, false, 512>(pdl && !after_s1, c, pm, s, grids[5], smm, st, nost)
                                 : launch_tier<SmFrontMid, M_HITS, false, CTA_THREADS>(pdl && !after_s1, c, pm, s, grids[5], smm, st, nost);
  if (e != cudaSuccess) return e;
  if (ev) cudaEventRecord(ev[2], st);
  e = debug ? launch_tier<SmFrontCta, C_HITS, true, CTA_THREADS>(pdl, c, pc, s, grids[4], smc, st, false)
            : launch_tier<SmFrontCta, C_HITS, false, CTA_THREADS>(pdl, c, pc, s, grids[4], smc, st, nost);
  if (e != cudaSuccess) return e;
  if (ev) cudaEventRecord(ev[3], st);
  const auto go = [&](auto k, int grid, int threads, const auto&... args) {
    if (e == cudaSuccess) e = launch_kernel(pdl, k, grid, threads, 0, st, args...);
  };
  if (debug) go(k_stage2<true>, grids[1], 128, c, p, s);
  else go(k_stage2<false>, grids[1], 128, c, p, s);
  if (ev) cudaEventRecord(ev[4], st);
  if (debug) go(k_stage3<true>, grids[2], S3_WARPS * 32, c, p3, s);
  else if (nost) go(k_stage3<false, true>, grids[2], S3_WARPS * 32, c, p3, s);
  else go(k_stage3<false>, grids[2], S3_WARPS * 32, c, p3, s);
  if (ev) cudaEventRecord(ev[5], st);
  if (debug) go(k_stage4<true>, grids[3], S4_WARPS * 32, c, p, s);
  else if (nost) go(k_stage4<false, true>, grids[3], S4_WARPS * 32, c, p, s);
  else go(k_stage4<false>, grids[3], S4_WARPS * 32, c, p, s);
  if (ev) cudaEventRecord(ev[6], st);
  go(k_stage5, (int)((p.n_frames + 255) / 256), 256, p, s);
  if (e != cudaSuccess) return e;
  if (ev) cudaEventRecord(ev[7], st);
  return cudaGetLastError();
}

}  // namespace m3e
