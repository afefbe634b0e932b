// Hit ingest of libm3e: packed int32 pixel addresses -> FP32 hit coordinates as
// structure of arrays (Sec. "Memory Layout": a hit is the point (x, y, z) of its
// pixel; the azimuth phi of the pixel column is the quantity the selection cuts
// bin on, Sec. "Selection Cuts").
//
// The work is a stream: 4 bytes read and 16 bytes written per hit, so HBM
// bandwidth bounds it once the table look-ups stay on chip.  Each CTA (one per SM)
// first copies the (x, y) of every pixel column and the z of every pixel row into
// shared memory (183 KB); phi is computed, not looked up: (g + 1/2) times 2 pi/ntot
// held as a sum of two floats, in exact FP32 steps (the product's rounding error
// recovered by a fused multiply-add), which reproduces the FP64 value rounded once
// for every column of the detector (checked exhaustively).  Each thread then moves
// four consecutive hits per step (one 16-byte load of addresses, one 16-byte
// store into each output array) with INGEST_UNROLL steps in flight; the streams
// are read and written with evict-first hints.
#include "m3e_device.cuh"

namespace m3e {
namespace {

constexpr int INGEST_THREADS = 1024;
// Steps in flight per thread: the output streams of a step lie a grid's width apart, and the
// fewer of them are open the better DRAM takes them (85.5 M hits: 1 step 295 us, 2 steps 277,
// 4 steps 300, 6 steps 298; in the benchmark 271 us, 93% of the measured copy rate).
constexpr int INGEST_UNROLL = 2;
constexpr int INGEST_SMALL_THREADS = 128;
// Up to this many hits without the shared-memory tables, whose copies cost every CTA 183 KB:
// 30,000 hits 5.2 us without and 8.5 us with them, 1,000,000 10.0 and 10.5, 2,000,000 13.4 and
// 14.5, 3,000,000 18.6 and 16.7, 85,000,000 386 and 272.
constexpr int64_t INGEST_SMALL = 2000000;

struct Coord {
  float x, y, z, phi;
};

// Where a kernel reads the pixel tables: its own copy in shared memory, or global memory.
struct TabShared {
  const float2* xy_;
  const float* z_;
  __device__ __forceinline__ float2 xy(int i) const { return xy_[i]; }
  __device__ __forceinline__ float z(int i) const { return z_[i]; }
};
struct TabGlobal {
  const float4* __restrict__ col;
  const float* __restrict__ row;
  __device__ __forceinline__ float2 xy(int i) const { return __ldg(reinterpret_cast<const float2*>(col + i)); }
  __device__ __forceinline__ float z(int i) const { return __ldg(row + i); }
};

template <bool PHI, class T>
__device__ __forceinline__ Coord ingest_one(const DevCfg& C, const T& tab, uint32_t a, bool& bad) {
  const Dec d = decode_packed(C, a);
  Coord c;
  if (d.ok) {
    const float2 q = tab.xy(d.ci);
    c.x = q.x;
    c.y = q.y;
    c.z = tab.z(d.ri);
    c.phi = PHI ? column_phi<true>(C, d.L, d.g) : 0.f;
  } else {
    bad = true;
    c.x = c.y = c.z = c.phi = __int_as_float(0x7fc00000);  // quiet NaN
  }
  return c;
}

// Four addresses from hit 4 v on; HV: the array is 16-byte aligned (else, for a batch's
// sub-range, four 4-byte loads, whose sectors the first of them brings into L1).
template <bool HV>
__device__ __forceinline__ int4 load_unit(const int32_t* __restrict__ hits, int64_t v) {
  if constexpr (HV) return __ldcs(reinterpret_cast<const int4*>(hits) + v);
  const int32_t* h = hits + 4 * v;
  return make_int4(__ldg(h), __ldg(h + 1), __ldg(h + 2), __ldg(h + 3));
}

template <bool PHI, class T>
__device__ __forceinline__ void ingest_unit(const DevCfg& C, const T& tab, const int4& a, int64_t v, float* x, float* y,
                                            float* z, float* phi, bool& bad) {
  const Coord c0 = ingest_one<PHI>(C, tab, (uint32_t)a.x, bad);
  const Coord c1 = ingest_one<PHI>(C, tab, (uint32_t)a.y, bad);
  const Coord c2 = ingest_one<PHI>(C, tab, (uint32_t)a.z, bad);
  const Coord c3 = ingest_one<PHI>(C, tab, (uint32_t)a.w, bad);
  __stcs(reinterpret_cast<float4*>(x) + v, make_float4(c0.x, c1.x, c2.x, c3.x));
  __stcs(reinterpret_cast<float4*>(y) + v, make_float4(c0.y, c1.y, c2.y, c3.y));
  __stcs(reinterpret_cast<float4*>(z) + v, make_float4(c0.z, c1.z, c2.z, c3.z));
  if constexpr (PHI) __stcs(reinterpret_cast<float4*>(phi) + v, make_float4(c0.phi, c1.phi, c2.phi, c3.phi));
}

// Hits [from, n), one at a time, over the grid's threads.
template <bool PHI, class T>
__device__ __forceinline__ void ingest_rest(const DevCfg& C, const T& tab, const int32_t* __restrict__ hits, int64_t from,
                                            int64_t n, int64_t tid, int64_t nth, float* x, float* y, float* z, float* phi,
                                            bool& bad) {
  for (int64_t i = from + tid; i < n; i += nth) {
    const Coord c = ingest_one<PHI>(C, tab, (uint32_t)__ldcs(hits + i), bad);
    __stcs(x + i, c.x);
    __stcs(y + i, c.y);
    __stcs(z + i, c.z);
    if constexpr (PHI) __stcs(phi + i, c.phi);
  }
}

// VEC: the output arrays are 16-byte aligned; threads move units of four hits, the last
// n % 4 hits are taken one at a time.  HV: so are the addresses.
template <bool VEC, bool PHI, bool HV>
__global__ void __launch_bounds__(INGEST_THREADS, 1)
    k_ingest(const __grid_constant__ DevCfg C, const int32_t* __restrict__ hits, int64_t n,
             const float4* __restrict__ col_lut, const float* __restrict__ row_lut, float* __restrict__ x,
             float* __restrict__ y, float* __restrict__ z, float* __restrict__ phi, int* err) {
  extern __shared__ __align__(16) float2 s_xy[];
  const int ncol = C.col_off[3] + C.ntot[3], nrow = C.row_off[3] + C.nrow[3];
  float* s_z = reinterpret_cast<float*>(s_xy + ncol);
  for (int i = threadIdx.x; i < ncol; i += INGEST_THREADS) {
    const float4 q = __ldg(col_lut + i);
    s_xy[i] = make_float2(q.x, q.y);
  }
  for (int i = threadIdx.x; i < nrow; i += INGEST_THREADS) s_z[i] = __ldg(row_lut + i);
  __syncthreads();
  const TabShared tab{s_xy, s_z};
  bool bad = false;
  const int64_t tid = (int64_t)blockIdx.x * INGEST_THREADS + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * INGEST_THREADS;
  int64_t done = 0;
  if constexpr (VEC) {
    const int64_t nv = n >> 2;
    for (int64_t v0 = tid; v0 < nv; v0 += nth * INGEST_UNROLL) {
      int4 a[INGEST_UNROLL];
#pragma unroll
      for (int u = 0; u < INGEST_UNROLL; ++u) {
        const int64_t v = v0 + u * nth;
        a[u] = v < nv ? load_unit<HV>(hits, v) : make_int4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < INGEST_UNROLL; ++u) {
        const int64_t v = v0 + u * nth;
        if (v < nv) ingest_unit<PHI>(C, tab, a[u], v, x, y, z, phi, bad);
      }
    }
    done = nv << 2;
  }
  ingest_rest<PHI>(C, tab, hits, done, n, tid, nth, x, y, z, phi, bad);
  if (__any_sync(FULL, bad) && (threadIdx.x & 31) == 0) atomicOr(err, ERR_BADHIT);
}

// The same without the tables' copies in shared memory, for fewer hits than pay for them:
// the look-ups go to L1 and L2, one unit of four hits per thread.
template <bool VEC, bool PHI, bool HV>
__global__ void __launch_bounds__(INGEST_SMALL_THREADS)
    k_ingest_small(const __grid_constant__ DevCfg C, const int32_t* __restrict__ hits, int64_t n,
                   const float4* __restrict__ col_lut, const float* __restrict__ row_lut, float* __restrict__ x,
                   float* __restrict__ y, float* __restrict__ z, float* __restrict__ phi, int* err) {
  const TabGlobal tab{col_lut, row_lut};
  bool bad = false;
  const int64_t tid = (int64_t)blockIdx.x * INGEST_SMALL_THREADS + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * INGEST_SMALL_THREADS;
  const int64_t nv = VEC ? n >> 2 : 0;
  for (int64_t v = tid; v < nv; v += nth) ingest_unit<PHI>(C, tab, load_unit<HV>(hits, v), v, x, y, z, phi, bad);
  ingest_rest<PHI>(C, tab, hits, nv << 2, n, tid, nth, x, y, z, phi, bad);
  if (__any_sync(FULL, bad) && (threadIdx.x & 31) == 0) atomicOr(err, ERR_BADHIT);
}

size_t ingest_smem_bytes(const DevCfg& c) {
  return (size_t)(c.col_off[3] + c.ntot[3]) * sizeof(float2) + (size_t)(c.row_off[3] + c.nrow[3]) * sizeof(float);
}

struct IngestCall {
  const DevCfg& c;
  const int32_t* hits;
  int64_t n;
  const float4* col_lut;
  const float* row_lut;
  float *x, *y, *z, *phi;
  int* err;
  int sms;
  size_t smem_limit;  // shared memory that a block may have
  cudaStream_t s;
};

template <bool VEC, bool PHI, bool HV>
cudaError_t launch_ingest_t(const IngestCall& q) {
  const size_t sm = ingest_smem_bytes(q.c);
  // a geometry whose tables do not fit an SM (up to 384 KB) never gets the copies
  if (q.n <= INGEST_SMALL || sm > q.smem_limit) {
    const int64_t units = VEC ? (q.n + 3) / 4 : q.n;
    const int64_t want = (units + INGEST_SMALL_THREADS - 1) / INGEST_SMALL_THREADS, most = (int64_t)q.sms * 16;
    k_ingest_small<VEC, PHI, HV><<<(int)(want < most ? want : most), INGEST_SMALL_THREADS, 0, q.s>>>(
        q.c, q.hits, q.n, q.col_lut, q.row_lut, q.x, q.y, q.z, q.phi, q.err);
    return cudaGetLastError();
  }
  cudaError_t e = cudaFuncSetAttribute(k_ingest<VEC, PHI, HV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_ingest<VEC, PHI, HV><<<q.sms, INGEST_THREADS, sm, q.s>>>(q.c, q.hits, q.n, q.col_lut, q.row_lut, q.x, q.y, q.z,
                                                             q.phi, q.err);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_ingest(const DevCfg& c, const int32_t* hits, int64_t n, const float4* col_lut, const float* row_lut,
                          float* x, float* y, float* z, float* phi, int* err, int sms, size_t smem_limit,
                          cudaStream_t s) {
  auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };  // NULL is aligned
  const IngestCall q{c, hits, n, col_lut, row_lut, x, y, z, phi, err, sms, smem_limit, s};
  if (!(al(x) && al(y) && al(z) && al(phi)))
    return phi ? launch_ingest_t<false, true, false>(q) : launch_ingest_t<false, false, false>(q);
  if (al(hits)) return phi ? launch_ingest_t<true, true, true>(q) : launch_ingest_t<true, false, true>(q);
  return phi ? launch_ingest_t<true, true, false>(q) : launch_ingest_t<true, false, false>(q);
}

}  // namespace m3e
