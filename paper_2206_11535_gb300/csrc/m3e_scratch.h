// Device scratch of the selection: its arrays, their capacities and how they grow.  No kernel
// code, and the memory calls are passed in, so that a host program can let one of them fail.
#pragma once
#include <algorithm>
#include <cstdint>
#include <initializer_list>

#include "m3e_internal.cuh"

namespace m3e {

// Device scratch of one launch sequence: work queue, deferred-frame list and the
// global candidate arrays of the staged form.  The context holds one set for the
// device entry points and two for the double-buffered host entry point.
struct Scratch {
  int* work = nullptr;                      // [0] work-queue head, [1] list-1 count, [2] list-2 count
  unsigned long long* counters = nullptr;   // staged: [0] triplets, [1] combinations, [2] stage-3 queue, [3] hits
  int* defer = nullptr;                     // list 1: deferred frames
  int* defer2 = nullptr;                    // list 2 (staged form)
  int* defer1b = nullptr;                   // list 1b (staged form)
  int64_t defer_cap = 0;
  float* hf = nullptr;                      // hx, hy, hz, hphi
  uint16_t* hidx = nullptr;
  int64_t hits_cap = 0;
  uint16_t* l3 = nullptr;
  int* fint = nullptr;                      // fstate, ftbase, fntrip, ffound
  long long* fcbase = nullptr;              // per frame: first combination
  int64_t frames_cap = 0;
  int4* trip = nullptr;
  float2* tek = nullptr;
  float4* trec = nullptr;
  int64_t trip_cap = 0;
  int4* combo = nullptr;
  int64_t combo_cap = 0;
  int64_t lean_frames = 0;                  // batches up to this one have the first figures per frame only
};

// The memory calls: M3E_OK, or the code that the entry point returns (get: the array is null then).
struct ScratchMemory {
  int (*get)(void** array, size_t bytes);
  int (*put)(void* array);  // takes null
};

struct ScratchArray {
  void** array;
  size_t elem;
  template <class T>
  ScratchArray(T*& a, size_t bytes) : array(reinterpret_cast<void**>(&a)), elem(bytes) {}
};

// Arrays that share the capacity cap hold at least `need` entries afterwards.  The capacity is
// 0 while one of them is missing: after a failure the group is empty and counts as empty, so
// that a later, smaller batch allocates it instead of running on a null array.
inline int resize(const ScratchMemory& m, int64_t& cap, int64_t need, std::initializer_list<ScratchArray> group) {
  if (need <= cap) return M3E_OK;
  cap = 0;
  int rc = M3E_OK;
  for (const ScratchArray& a : group) {
    const int r = m.put(*a.array);
    rc = rc ? rc : r;
    *a.array = nullptr;
  }
  for (const ScratchArray& a : group) rc = rc ? rc : m.get(a.array, a.elem * (size_t)need);
  if (rc) {
    for (const ScratchArray& a : group) {
      m.put(*a.array);
      *a.array = nullptr;
    }
    return rc;
  }
  cap = need;
  return M3E_OK;
}

// Scratch for a batch of nf frames (staged arrays only when staged).  The sorted hits,
// triplets and combinations of a batch share its scratch, and frames that find it full go
// to the CTA-per-frame kernel, which runs them many times slower.  The sizes per frame are
// those of the throughput mix (85 hits, 44 triplets) with a margin; a batch of denser
// frames needs more, so up to the scratch of ROOMY_FRAMES frames a batch gets the second,
// roomier figure (20,001 frames of 32 tracks, 137 hits and 108 triplets each: 7,000 frames
// deferred and 855 us with the first figures alone, 348 us with these; more costs a
// millisecond of allocation per GB when a context is prepared).  That is 27.5 KB a frame
// instead of 9.1; where it does not fit, the first figures do, and only cost speed.
constexpr int64_t ROOMY_FRAMES = 1 << 20;
constexpr int64_t HITS_PER_FRAME[2] = {128, 384};
constexpr int64_t TRIPLETS_PER_FRAME[2] = {64, 256};
constexpr int64_t COMBOS_PER_FRAME[2] = {192, 384};

inline int64_t scratch_entries(const int64_t (&per_frame)[2], int64_t nf, bool roomy) {
  // indices travel as int32 in the records: at most 2^31 - 2^16 entries
  const int64_t lim = ((int64_t)1 << 31) - (1 << 16);
  const int64_t more = roomy ? std::min(per_frame[1] * nf, per_frame[0] * ROOMY_FRAMES) : 0;
  return std::min(std::max({per_frame[0] * nf, more, (int64_t)1 << 16}), lim);
}

inline int resize_staged(const ScratchMemory& m, Scratch& sc, int64_t nf, bool roomy) {
  int rc = resize(m, sc.hits_cap, scratch_entries(HITS_PER_FRAME, nf, roomy),
                  {{sc.hf, 4 * sizeof(float)}, {sc.hidx, sizeof(uint16_t)}});
  if (!rc)
    rc = resize(m, sc.frames_cap, nf,
                {{sc.l3, (NB + 2) * sizeof(uint16_t)}, {sc.fint, 4 * sizeof(int)}, {sc.fcbase, sizeof(long long)}});
  if (!rc)
    rc = resize(m, sc.trip_cap, scratch_entries(TRIPLETS_PER_FRAME, nf, roomy),
                {{sc.trip, sizeof(int4)}, {sc.tek, sizeof(float2)}, {sc.trec, 2 * sizeof(float4)}});
  if (!rc) rc = resize(m, sc.combo_cap, scratch_entries(COMBOS_PER_FRAME, nf, roomy), {{sc.combo, sizeof(int4)}});
  return rc;
}

inline void free_staged(const ScratchMemory& m, Scratch& sc) {
  for (const ScratchArray& a : {ScratchArray(sc.hf, 0), ScratchArray(sc.hidx, 0), ScratchArray(sc.l3, 0),
                                ScratchArray(sc.fint, 0), ScratchArray(sc.fcbase, 0), ScratchArray(sc.trip, 0),
                                ScratchArray(sc.tek, 0), ScratchArray(sc.trec, 0), ScratchArray(sc.combo, 0)}) {
    m.put(*a.array);
    *a.array = nullptr;
  }
  sc.hits_cap = sc.frames_cap = sc.trip_cap = sc.combo_cap = 0;
}

inline int ensure_scratch(const ScratchMemory& m, Scratch& sc, int64_t nf, bool staged) {
  int64_t one = sc.work ? 1 : 0, one2 = sc.counters ? 1 : 0;
  int rc = resize(m, one, 1, {{sc.work, 4 * sizeof(int)}});
  if (!rc) rc = resize(m, one2, 1, {{sc.counters, 4 * sizeof(unsigned long long)}});
  if (!rc)
    rc = resize(m, sc.defer_cap, std::max<int64_t>(nf, 4096),
                {{sc.defer, sizeof(int)}, {sc.defer2, sizeof(int)}, {sc.defer1b, sizeof(int)}});
  if (rc || !staged) return rc;
  // batches that are known not to fit with the roomy figures are not tried with them again:
  // the arrays that serve them would be freed for it
  const bool roomy = nf > sc.lean_frames;
  rc = resize_staged(m, sc, nf, roomy);
  if (rc == M3E_ENOMEM && roomy) {
    free_staged(m, sc);
    rc = resize_staged(m, sc, nf, false);
    if (!rc) sc.lean_frames = nf;
  }
  return rc;
}

inline void free_scratch(const ScratchMemory& m, Scratch& sc) {
  free_staged(m, sc);
  for (void* a : {(void*)sc.work, (void*)sc.counters, (void*)sc.defer, (void*)sc.defer2, (void*)sc.defer1b}) m.put(a);
  sc = Scratch();
}

}  // namespace m3e
