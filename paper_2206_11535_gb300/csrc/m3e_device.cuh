// Device code shared by the fused and the staged selection kernels: thread
// groups, the shared-memory frame stage, decode, the triplet fit, track
// reconstruction and the vertex, all in FP32 (the build uses the approximate
// division and square root, a few ulp; exact comparisons that decide an integer
// use explicitly rounded intrinsics).
#pragma once

#include <cfloat>
#include <type_traits>

#include "m3e_internal.cuh"

namespace m3e {
namespace {

constexpr float PI_F = 3.14159265358979323846f;
constexpr float TWO_PI_F = 6.28318530717958647692f;
constexpr unsigned FULL = 0xffffffffu;

// ------------------------------------------------------------------ thread groups

struct WarpGroup {
  static constexpr int N = 32;
  __device__ __forceinline__ int rank() const { return threadIdx.x & 31; }
  __device__ __forceinline__ void sync() const { __syncwarp(); }
  __device__ __forceinline__ bool any(bool p) const { return __any_sync(FULL, p) != 0; }
  __device__ __forceinline__ bool leader() const { return (threadIdx.x & 31) == 0; }
};

template <int NT>
struct CtaGroup {
  static constexpr int N = NT;
  __device__ __forceinline__ int rank() const { return threadIdx.x; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
  __device__ __forceinline__ bool any(bool p) const { return __syncthreads_or(p) != 0; }
  __device__ __forceinline__ bool leader() const { return threadIdx.x == 0; }
};

// ------------------------------------------------------------------ shared-memory stage

// Kept tracks as structure of arrays: the energy test reads E[] with one index for
// all lanes (broadcast) and the vertex stage gathers by track index without the
// bank conflicts of a 64-byte record stride.
template <int CK>
struct TrkSoA {
  float cx[CK], cy[CK], rt[CK];     // transverse circle through the layer-0 and layer-1 hits
  float R[CK], ct[CK], st[CK];      // 3D radius and cos/sin of the first segment's polar angle
  float p[CK], E[CK], sms[CK];      // momentum, energy, MS width at layer 0
  float h0x[CK], h0y[CK], h0z[CK];  // layer-0 hit
  float ah0[CK];                    // angle of the layer-0 hit seen from the circle centre
  float eps[CK];                    // turning sense, +1 clockwise (positive charge)
  int tid[CK];                      // index of the triplet it came from
};

// IDX: whether the stage keeps each hit's input index (candidate record only); STATS:
// whether it has room for statistics.  A stage without them holds more frames in flight
// per SM.  Triplets of a stage of at most 256 hits are kept as 8-bit indices.
template <int CH, int CT, int CK, int CC, bool IDX = true, bool STATS = true, int CH32 = (CH <= W_HITS ? CH : 1)>
struct FrameSm {
  static constexpr bool kIdx = IDX, kStats = STATS;
  static constexpr bool kPackB = CH < 256;  // bucket cursors as bytes, four to a word
  using TripT = typename std::conditional<(CH <= 256), uchar4, ushort4>::type;
  alignas(16) float2 xy[CH];
  float z[CH], phi[CH];         // phi: layer-3 hits only (the 4th-hit search)
  uint16_t inidx[IDX ? CH : 1];
  uint16_t bstart[NBK + 2];       // one more than needed: read in pairs
  uint32_t bcur[kPackB ? NBK / 4 : NBK];  // bucket counts, then cursors
  // warp stage, selection cuts (warp_cuts): x and y of the layer-0 hits apart, the layer-2
  // hits in z-bin order (bin starts zbs; z and sorted index in zzi), the (layer-1 hit, Phi01 partner) pairs of a
  // chunk of 32 layer-1 hits (layer-0 hit, lane of the layer-1 hit) and the candidate
  // triplets of one round of pairs
  alignas(16) float ox[CH32 == 1 ? 4 : W_L0];
  alignas(16) float oy[CH32 == 1 ? 4 : W_L0];
  alignas(16) float zx[CH32 == 1 ? 4 : W_L2];
  alignas(16) float zy[CH32 == 1 ? 4 : W_L2];
  float2 zzi[CH32 == 1 ? 1 : W_L2];
  uint16_t p01[CH32 == 1 ? 1 : W_P01];
  uint8_t zbs[CH32 == 1 ? 1 : NZB + 1];
  alignas(16) uint16_t cand[CH32 == 1 ? 1 : W_CAND];  // also the z-bin counters (32-bit words)
  // CTA stage, selection cuts: the layer-2 hits in z-bin order (sorted-hit indices),
  // the bin starts of that order and the bin cursors of its counting sort
  uint16_t zidx[CH32 == 1 ? CH : 1];
  uint16_t zbs2[CH32 == 1 ? NZB + 1 : 1];
  uint32_t zcur[CH32 == 1 ? NZB : 1];
  uint8_t own[CH32 == 1 ? 16 : 1][2][32];  // per warp: the lanes that have window entries / candidates, in order
  TrkSoA<CK> t;                 // positives from the front, negatives from the back
  union {
    TripT trip[CT];             // selected triplets (sorted-hit indices)
    uint32_t combo[CC];         // e+ e+ e- combinations (track indices), after the fits
  } u;
  int ntrip, npos, nneg, ncombo, nstore, flag, bad;
  unsigned long long acc[STATS ? ST_REASON0 + 8 : 1];  // statistics of this group's frames
  unsigned long long facc[STATS ? ST_REASON0 : 1];     // statistics of the current frame
};

using SmWarp = FrameSm<W_HITS, W_TRIP, W_TRK, W_COMBO>;
using SmCta = FrameSm<C_HITS, C_TRIP, C_TRK, C_COMBO>;

// ------------------------------------------------------------------ small helpers

// Two FP32 operations in one instruction, each rounded as the scalar one.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// The bits below bit k of a word, all 32 for k of 32 and more (k >= 0).
__device__ __forceinline__ uint32_t bits_below(int k) { return __funnelshift_lc(0xffffffffu, 0u, (unsigned)k); }

// Asynchronous 4- and 8-byte copies from global to shared memory (no register holds the
// value), and the wait for all of this thread's copies.
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
// Programmatic dependent launch.  pdl_wait: wait until the preceding kernel of the stream
// has finished and its writes are visible (nothing to wait for in an ordinary launch);
// every block of a kernel launched as a dependent calls it before it reads or writes
// memory.  pdl_trigger: the following kernel's blocks may be placed once every block of
// this one has got here or ended.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

template <class T>
__device__ __forceinline__ T make_trip(int i0, int i1, int i2) {  // a triplet of sorted-hit indices
  T t;
  t.x = (decltype(t.x))i0;
  t.y = (decltype(t.y))i1;
  t.z = (decltype(t.z))i2;
  t.w = 0;
  return t;
}

struct Dec {
  int L, g, row, b;
  int ci, ri;  // indices of the hit's column and row in the look-up tables
  bool ok;
};

// A per-layer constant selected by the (data-dependent) layer: selects over the
// four values instead of an indexed load, which the constant cache would serialise
// over the distinct layers of a warp.
template <class T>
__device__ __forceinline__ T by_layer(const T (&v)[4], int L) {
  return L == 0 ? v[0] : (L == 1 ? v[1] : (L == 2 ? v[2] : v[3]));
}
// a 16-bit field of a packed per-layer word
__device__ __forceinline__ int field16(unsigned long long w, int L) { return (int)((w >> (16 * L)) & 0xffffull); }

__device__ __forceinline__ Dec decode(const DevCfg& C, uint32_t a) {
  Dec d;
  d.L = (a >> 26) & 3;
  const int lad = (a >> 21) & 31, col = (a >> 13) & 255;
  d.row = a & 8191;
  d.ok = (a >> 28) == 0 && lad < C.nlad[d.L] && col < C.ncol[d.L] && d.row < C.nrow[d.L];
  d.g = lad * C.ncol[d.L] + col;
  d.ci = C.col_off[d.L] + d.g;
  d.ri = C.row_off[d.L] + d.row;
  // phi bin floor(g NB / ntot) without an integer division: g NB < 2^24 is exact in
  // FP32, and (g NB + 1/2) / ntot lies at least 1/(2 ntot) >= 6e-5 from an integer,
  // far more than the two roundings (< 4e-6 at values below NB)
  d.b = d.ok ? (int)__fmul_rn(__fadd_rn((float)(d.g * NB), 0.5f), C.intot[d.L]) : 0;
  return d;
}

// decode() with the per-layer constants from the 16-byte entries of a table in shared
// memory (DevCfg::ltab): one load per hit, where the constant cache would serialise
// the loads of a warp's several layers.  The same values as decode().
__device__ __forceinline__ Dec decode_s(const uint4* tab, uint32_t a) {
  Dec d;
  d.L = (a >> 26) & 3;
  const uint4 t = tab[d.L];
  const int lad = (a >> 21) & 31, col = (a >> 13) & 255;
  d.row = a & 8191;
  const int nlad = (int)(t.x & 63u), ncol = (int)((t.x >> 6) & 511u), nrow = (int)(t.x >> 15);
  d.ok = (a >> 28) == 0 && lad < nlad && col < ncol && d.row < nrow;
  d.g = lad * ncol + col;
  d.ci = (int)t.y + d.g;
  d.ri = (int)t.z + d.row;
  d.b = d.ok ? (int)__fmul_rn(__fadd_rn((float)(d.g * NB), 0.5f), __uint_as_float(t.w)) : 0;
  return d;
}

// decode without the phi bin and without loads indexed by the hit's layer: the
// per-layer integers come from packed 16-bit fields.  For a kernel that does little
// else per hit (the ingest), where loads of per-layer constants at the warp's
// several layers would serialise in the constant cache and bound the kernel.
__device__ __forceinline__ Dec decode_packed(const DevCfg& C, uint32_t a) {
  Dec d;
  d.L = (a >> 26) & 3;
  const int lad = (a >> 21) & 31, col = (a >> 13) & 255;
  d.row = a & 8191;
  const int nlad = field16(C.pk_nlad, d.L), ncol = field16(C.pk_ncol, d.L);
  d.ok = (a >> 28) == 0 && lad < nlad && col < ncol && d.row < field16(C.pk_nrow, d.L);
  d.g = lad * ncol + col;
  d.ci = field16(C.pk_coloff, d.L) + d.g;
  d.ri = field16(C.pk_rowoff, d.L) + d.row;
  d.b = 0;
  return d;
}

// Azimuth of the centre of global column g of layer L, (g + 1/2) 2 pi / ntot: the
// step 2 pi / ntot is held as a sum of two floats and the product's rounding error
// is recovered by a fused multiply-add, which gives the FP64 value rounded once to
// FP32 for every column of the detector (the look-up table's value, checked
// exhaustively by the tests).
template <bool SEL = false>
__device__ __forceinline__ float column_phi(const DevCfg& C, int L, int g) {
  const float p = (float)g + 0.5f;  // exact: g < 2^23
  const float sh = SEL ? by_layer(C.phs_hi, L) : C.phs_hi[L], sl = SEL ? by_layer(C.phs_lo, L) : C.phs_lo[L];
  const float hi = __fmul_rn(p, sh);
  const float lo = __fmaf_rn(p, sh, -hi);
  return __fadd_rn(hi, __fmaf_rn(p, sl, lo));
}

__device__ __forceinline__ float wrap_2pi(float a) {  // (-2 pi, 2 pi) -> [0, 2 pi)
  if (a < 0.f) a += TWO_PI_F;
  if (a >= TWO_PI_F) a -= TWO_PI_F;
  return a;
}

__device__ __forceinline__ float wrap_pi(float a) {  // (-2 pi, 2 pi) -> [-pi, pi]
  if (a > PI_F) a -= TWO_PI_F;
  if (a < -PI_F) a += TWO_PI_F;
  return a;
}

// sin(x) - x cos(x) for x in (0, pi], given s = sin x and c = cos x.  For small x
// the two terms cancel to x^3/3, so the Taylor series
// sum_k (-1)^(k+1) 2k x^(2k+1) / (2k+1)! is used below 0.5 (five terms:
// truncation below FP32 rounding).
__device__ __forceinline__ float sin_minus_xcos(float x, float s, float c) {
  if (x < 0.5f) {
    const float x2 = x * x;
    float t = 1.f / 3991680.f;
    t = t * x2 - 1.f / 45360.f;
    t = t * x2 + 1.f / 840.f;
    t = t * x2 - 1.f / 30.f;
    t = t * x2 + 1.f / 3.f;
    return t * x2 * x;
  }
  return s - x * c;
}

// ------------------------------------------------------------------ triplet fit

struct SegF {
  float phi, RC, th, dphi, dth, zp;
};

// One segment of the circle solution: chord d, axial length z, transverse radius
// Rct of the circle through the triplet, and the arc angle Phi travelled along the
// segment with sh = sin(Phi/2) and ch = cos(Phi/2).  Helix relations
// d = 2 R_t sin(Phi/2), z = R_t Phi cot(theta), R_t = R sin(theta) give the 3D
// radius R_C, the polar angle theta_C and the derivatives dPhi/dR, dtheta/dR at
// the circle solution.  The divisions share the reciprocals of Phi and of
// sin(Phi/2): dPhi/dR = -R_C / (d^2 cos(Phi/2) / (8 sin^3(Phi/2)) + zp^2 / Phi).
__device__ __forceinline__ SegF segment_core(float d, float z, float Rct, float sh, float ch, float ph) {
  SegF s;
  const float iph = 1.f / ph, ish = 1.f / sh;
  const float zp = z * iph;
  s.RC = sqrtf(Rct * Rct + zp * zp);
  s.th = 0.f;  // the polar angle atan2(Rct, zp) itself: computed where it is needed
  const float ish2 = ish * ish;
  s.dphi = -s.RC / (0.125f * d * d * ch * ish2 * ish + zp * zp * iph);
  const float g = 0.5f * ph * ish;
  const float gp = 0.5f * sin_minus_xcos(0.5f * ph, sh, ch) * ish2;
  const float dg = d * g;
  s.dth = z * d * gp * s.dphi / (z * z + dg * dg);
  s.phi = ph;
  s.zp = zp;
  return s;
}

struct TFitF {
  float eps, Rct, ccx, ccy;
  float Rref;                  // expansion point of the kink model: R_C of segment 0
  float alpha, a0p, beta, b0p; // Phi_MS ~ alpha u + a0p, Theta_MS ~ beta u + b0p, u = R - Rref
  float s2;                    // sin^2 of the mean polar angle
  float kappa, skappa;
  float zp0, RC0, dth0;         // segment 0: z / Phi (theta_C0 = atan2(Rct, zp0)), R_C, dtheta/dR
  float zp1;                   // z / Phi of segment 1 = R_t cot(theta_C1)
  float ph0, ph1;              // arc angles of the segments (alignment gradient)
  int valid;
};

// Single triplet fit, hits a -> b -> c, scattering at b (Sec. "Single Triplet
// Fit"): linear kink model around the circle solution and its closed-form
// minimum in the 3D radius.  The model is written in u = R - R_C0 so that the
// small offsets (R_C0 - R_C1, theta_C1 - theta_C0) enter directly instead of as
// differences of large products; the algebra equals the minimum of
// [Phi_MS^2 sin^2(theta) + Theta_MS^2] / sigma_MS^2.  Inlined at both calls of a
// track: as a call, its 18-float result and the caller's live values went through
// local memory.
__device__ __forceinline__ TFitF fit_triplet(float ax, float ay, float az, float bx, float by, float bz, float cx,
                                          float cy, float cz, float hl, float kB) {
  TFitF f;
  f.valid = 0;
  const float ux = ax - bx, uy = ay - by, vx = cx - bx, vy = cy - by;
  const float cross = ux * vy - uy * vx;
  const float u2 = ux * ux + uy * uy, v2 = vx * vx + vy * vy;
  const float wx = cx - ax, wy = cy - ay;
  const float d01 = sqrtf(u2), d12 = sqrtf(v2), d20 = sqrtf(wx * wx + wy * wy);
  if (!(cross != 0.f)) return f;
  const float i2c = 0.5f / cross;
  const float rtc = d01 * d12 * d20 * i2c;
  if (!isfinite(rtc) || rtc == 0.f) return f;
  f.Rct = fabsf(rtc);
  f.eps = rtc > 0.f ? 1.f : -1.f;
  f.ccx = bx + (vy * u2 - uy * v2) * i2c;
  f.ccy = by + (ux * v2 - vx * u2) * i2c;
  // Arc angle of each segment from the triangle: the track's arc from a to b is
  // the one that does not hold c, so it turns by twice the inscribed angle at c,
  // Phi01 = 2 atan2(|cross|, (a - c).(b - c)) (more than pi when that angle is
  // obtuse), and Phi12 likewise by twice the angle at a.  sin(Phi/2) and
  // cos(Phi/2) are that angle's sine and cosine, |cross| / (lengths) and
  // dot / (lengths): full precision up to a half turn and beyond, where the arc
  // sine of d / 2R_t would lose half its digits.
  const float acr = fabsf(cross);
  const float dotc = (ax - cx) * (bx - cx) + (ay - cy) * (by - cy);
  const float dota = (bx - ax) * (cx - ax) + (by - ay) * (cy - ay);
  const float il0 = 1.f / (d20 * d12), il1 = 1.f / (d01 * d20);
  f.ph0 = 2.f * atan2f(acr, dotc);
  f.ph1 = 2.f * atan2f(acr, dota);
  const SegF s0 = segment_core(d01, bz - az, f.Rct, acr * il0, dotc * il0, f.ph0);
  const SegF s1 = segment_core(d12, cz - bz, f.Rct, acr * il1, dota * il1, f.ph1);
  const float dR = s0.RC - s1.RC;
  f.Rref = s0.RC;
  f.alpha = 0.5f * (s0.dphi + s1.dphi);
  f.a0p = 0.5f * s1.dphi * dR;
  f.beta = s1.dth - s0.dth;
  // polar angles from cos = zp / R_C, sin = R_t / R_C of each segment: their difference
  // as one well-conditioned atan2, and sin^2 of their mean from cos(theta0 + theta1)
  // (the common factor 1 / (R_C0 R_C1) drops out of the atan2)
  const float R2 = f.Rct * f.Rct;
  f.b0p = atan2f(f.Rct * (s0.zp - s1.zp), fmaf(s0.zp, s1.zp, R2)) + s1.dth * dR;
  f.s2 = 0.5f * (1.f - (s0.zp * s1.zp - R2) / (s0.RC * s1.RC));
  const float den = f.alpha * f.alpha * f.s2 + f.beta * f.beta;
  const float u = -(f.alpha * f.a0p * f.s2 + f.beta * f.b0p) / den;
  const float Rs = f.Rref + u;
  if (!(Rs > 0.f) || !isfinite(Rs)) return f;
  const float iRs = 1.f / Rs;
  f.kappa = f.eps * iRs;
  f.skappa = hl * iRs * iRs * iRs / (kB * sqrtf(den));  // sigma_MS(p*) / sqrt(den) / R*^2
  if (!isfinite(f.kappa) || !isfinite(f.skappa) || !(f.skappa > 0.f)) return f;
  f.zp0 = s0.zp;
  f.RC0 = s0.RC;
  f.dth0 = s0.dth;
  f.zp1 = s1.zp;
  f.valid = 1;
  return f;
}

// [Phi_MS^2 sin^2(theta) + Theta_MS^2] / sigma_MS^2 of the kink model at R, with
// isg = 1 / sigma_MS.
__device__ __forceinline__ float kink_chi2(const TFitF& f, float R, float isg) {
  const float u = R - f.Rref;
  const float kp = f.alpha * u + f.a0p, kt = f.beta * u + f.b0p;
  return (kp * kp * f.s2 + kt * kt) * (isg * isg);
}

// ------------------------------------------------------------------ hit views

// Hits of one frame, sorted by (layer, phi bin), as build_track reads them: from
// the shared-memory stage of a fused kernel, or from global memory in the staged
// form (pointers already offset to the frame).
// pos(i) = (x, y, z, phi) of sorted hit i.
template <class S>
struct SmHits {
  static constexpr bool kPark = false;
  const S& s;
  __device__ __forceinline__ float4 pos(int i) const { const float2 p = s.xy[i]; return make_float4(p.x, p.y, s.z[i], s.phi[i]); }
  __device__ __forceinline__ int l3(int b) const { return s.bstart[3 * NB + b]; }  // layer-3 bin starts
  __device__ __forceinline__ int l3_first() const { return l3(0); }
  __device__ __forceinline__ int l3_end() const { return l3(NB); }
};

// The first triplet fit's values that the global fit and the track record need,
// parked in shared memory across the layer-3 search and the second fit (staged form,
// one slot per thread of a 128-thread CTA): fewer live registers in the track stage.
struct FitPark {
  float v[11][128];
};

__device__ __forceinline__ void park_fit(FitPark& pk, const TFitF& f) {
  volatile float* q = &pk.v[0][threadIdx.x & 127];
  q[0 * 128] = f.skappa;
  q[1 * 128] = f.kappa;
  q[2 * 128] = f.alpha;
  q[3 * 128] = f.a0p;
  q[4 * 128] = f.beta;
  q[5 * 128] = f.b0p;
  q[6 * 128] = f.s2;
  q[7 * 128] = f.Rref;
  q[8 * 128] = f.Rct;
  q[9 * 128] = f.zp0;
  q[10 * 128] = f.dth0;
}

__device__ __forceinline__ TFitF unpark_fit(const FitPark& pk) {
  const volatile float* q = &pk.v[0][threadIdx.x & 127];
  TFitF f;
  f.skappa = q[0 * 128];
  f.kappa = q[1 * 128];
  f.alpha = q[2 * 128];
  f.a0p = q[3 * 128];
  f.beta = q[4 * 128];
  f.b0p = q[5 * 128];
  f.s2 = q[6 * 128];
  f.Rref = q[7 * 128];
  f.Rct = q[8 * 128];
  f.zp0 = q[9 * 128];
  f.dth0 = q[10 * 128];
  f.RC0 = f.Rref;  // R_C of segment 0 is the expansion point
  f.eps = f.ccx = f.ccy = f.zp1 = f.ph0 = f.ph1 = 0.f;
  f.valid = 1;
  return f;
}

template <bool EARLY>                // EARLY: the layer-3 range is loaded with the triplet's hits
struct GHits {                       // one 16-byte load per hit
  static constexpr bool kPark = true;
  const float4* __restrict__ ps;
  const uint16_t* __restrict__ l3s;  // NB + 1 layer-3 bin starts, frame-relative
  FitPark* park;
  unsigned range;                    // EARLY: layer-3 hits, first | end << 16
  __device__ __forceinline__ float4 pos(int i) const { return __ldg(ps + i); }
  __device__ __forceinline__ int l3(int b) const { return __ldg(l3s + b); }
  __device__ __forceinline__ int l3_first() const { return EARLY ? (int)(range & 0xffff) : l3(0); }
  __device__ __forceinline__ int l3_end() const { return EARLY ? (int)(range >> 16) : l3(NB); }
};

// ------------------------------------------------------------------ track reconstruction

constexpr int SCAN3_MAX = 96;

struct TrackOut {
  int status, i3;
  float kbar, th01, chi2, mbest;
  float Rct, zp0, dth0, RC0;  // of the first triplet's fit: what the track record needs besides kbar
};

// Global fit of a track from its two triplet fits (weighted mean curvature, chi2 of
// both kink models at it, chi2 cut) and what the track record needs.
__device__ __forceinline__ TrackOut global_fit(TrackOut o, const TFitF& f1, const TFitF& f2, const DevCfg& C) {
  const float w1 = 1.f / (f1.skappa * f1.skappa), w2 = 1.f / (f2.skappa * f2.skappa);
  const float kb = (f1.kappa * w1 + f2.kappa * w2) / (w1 + w2);
  o.kbar = kb;
  if (!(kb != 0.f) || !isfinite(kb)) return o;
  const float Rb = 1.f / fabsf(kb);
  const float pb = C.kB * Rb;
  const float chi2 = kink_chi2(f1, Rb, pb * C.ihl[1]) + kink_chi2(f2, Rb, pb * C.ihl[2]);
  o.chi2 = chi2;
  if (!isfinite(chi2)) return o;
  o.status = 4;
  if (!(chi2 < C.chi2_trk)) return o;
  o.status = 5;
  o.th01 = atan2f(f1.Rct, f1.zp0) + f1.dth0 * (Rb - f1.RC0);  // theta01 (candidate record)
  o.Rct = f1.Rct;
  o.zp0 = f1.zp0;
  o.dth0 = f1.dth0;
  o.RC0 = f1.RC0;
  return o;
}

// Algorithm 3 for one selected triplet (sorted-hit indices i0, i1, i2): fit,
// estimate the layer-3 point from the first triplet's circle and the second
// segment's polar angle, take the closest layer-3 hit ((r3 dphi)^2 + dz^2, ties
// to the smaller address), fit (h1, h2, h3), weighted mean curvature and chi2 of
// both triplets at it, chi2 cut.  The caller turns a kept track (status 5) into
// its record with track_record.
//
// Closest hit: a frame with at most SCAN3_MAX layer-3 hits scans them all (the
// loads are independent, so their latencies overlap); a larger one visits them
// by phi bin in rings around the bin of the estimated point.  Every hit of ring m >= 3 lies at least (m - 2) bin widths
// minus one column from the estimated phi (one ring of slack covers a bin index
// rounded across an edge), so once (r3 * that)^2 exceeds the best metric no
// farther hit can win: the search returns the same hit as a scan of all hits.
template <class V>
__device__ __forceinline__ TrackOut build_track(const V& v, const DevCfg& C, int i0, int i1, int i2) {
  TrackOut o;
  o.status = 0;
  o.i3 = -1;
  o.kbar = o.th01 = o.chi2 = o.mbest = 0.f;
  o.Rct = o.zp0 = o.dth0 = o.RC0 = 0.f;
  const float4 p0 = v.pos(i0), p1 = v.pos(i1), p2 = v.pos(i2);
  const float x0 = p0.x, y0 = p0.y, z0 = p0.z;
  const float x1 = p1.x, y1 = p1.y, z1 = p1.z;
  const float x2 = p2.x, y2 = p2.y, z2 = p2.z;
  const TFitF f1 = fit_triplet(x0, y0, z0, x1, y1, z1, x2, y2, z2, C.hl[1], C.kB);
  if (!f1.valid) return o;
  if constexpr (V::kPark) park_fit(*v.park, f1);
  const float r3 = C.r3;
  const float D = sqrtf(f1.ccx * f1.ccx + f1.ccy * f1.ccy);
  o.status = 1;
  if (!(D > 0.f) || D > f1.Rct + r3 || D < fabsf(f1.Rct - r3)) return o;
  const float iD = 1.f / D;
  const float a = (r3 * r3 - (f1.Rct - D) * (f1.Rct + D)) * (0.5f * iD);
  const float hh = sqrtf(fmaxf((r3 - a) * (r3 + a), 0.f));
  const float ux = f1.ccx * iD, uy = f1.ccy * iD;
  const float qx0 = a * ux - hh * uy, qy0 = a * uy + hh * ux;
  const float qx1 = a * ux + hh * uy, qy1 = a * uy - hh * ux;
  // turning angle from h2 to each crossing q in the turning sense: the angle from
  // (h2 - c) to (q - c) is atan2(cross, dot); clockwise turning decreases it.  The
  // crossing reached first is found without the angles: with (dot, -eps cross) as
  // the direction of the turn, a turn of less than a half (-eps cross >= 0) comes
  // before one of more, and within a half the turn of q1 is the smaller one when
  // the direction of q1 lies clockwise of that of q0 (negative 2D cross product).
  // Only the chosen turn is evaluated.
  const float wx = x2 - f1.ccx, wy = y2 - f1.ccy;
  const float vx0 = qx0 - f1.ccx, vy0 = qy0 - f1.ccy, vx1 = qx1 - f1.ccx, vy1 = qy1 - f1.ccy;
  const float cr0 = wx * vy0 - wy * vx0, dt0 = wx * vx0 + wy * vy0;
  const float cr1 = wx * vy1 - wy * vx1, dt1 = wx * vx1 + wy * vy1;
  const float t0 = -f1.eps * cr0, t1 = -f1.eps * cr1;
  const bool lo0 = !(t0 < 0.f), lo1 = !(t1 < 0.f);
  const bool take1 = (lo1 && !lo0) || (lo1 == lo0 && dt0 * t1 - t0 * dt1 < 0.f);
  const float al = wrap_2pi(-f1.eps * atan2f(take1 ? cr1 : cr0, take1 ? dt1 : dt0));
  const float qx = take1 ? qx1 : qx0, qy = take1 ? qy1 : qy0;
  const float z3 = z2 + al * f1.zp1;  // R_t * dPhi * cot(theta_C12)
  float phi3 = atan2f(qy, qx);
  if (phi3 < 0.f) phi3 += TWO_PI_F;
  int b3 = (int)(phi3 * (NB / TWO_PI_F));
  b3 = b3 < 0 ? 0 : (b3 >= NB ? NB - 1 : b3);
  int best = -1;
  float mb = FLT_MAX;
  // (r3 dphi)^2 + dz^2, rounded in one fixed order wherever it is inlined; both differences
  // in one instruction, and dphi (of azimuths in [0, 2 pi)) wrapped by taking the smaller of
  // |d| and 2 pi - |d| (track stage of 1e6 throughput frames 2357 -> 2341 us against a
  // rounding to the nearest multiple of 2 pi)
  const unsigned long long from = pack2(-z3, -phi3);
  auto metric = [&](const float4& q) {
    const unsigned long long dd = add2(pack2(q.z, q.w), from);
    const float dz = __uint_as_float((unsigned)dd), d = fabsf(__uint_as_float((unsigned)(dd >> 32)));
    const float rd = __fmul_rn(r3, fminf(d, __fsub_rn(TWO_PI_F, d)));
    return __fmaf_rn(rd, rd, __fmul_rn(dz, dz));
  };
  // the full rule: an equal metric goes to the smaller address.  The address orders the
  // layer's hits by column, then row, and the coordinates grow with these (a column's phi,
  // a row's z), so the comparison needs no address
  auto visit = [&](int j) {
    const float4 q = v.pos(j);
    const float mm = metric(q);
    bool take = best < 0 || mm < mb;
    if (mm == mb && !take) {
      const float4 o = v.pos(best);
      take = q.w < o.w || (q.w == o.w && q.z < o.z);
    }
    if (take) {
      best = j;
      mb = mm;
    }
  };
  const int l3a = v.l3_first(), l3e = v.l3_end();
  if (l3e - l3a <= SCAN3_MAX) {
    // few layer-3 hits: a straight scan, whose loads do not depend on each other.
    // It reads no addresses: it notes whether another hit has the same metric as
    // the best so far, and only then (rarely) repeats the scan with the full rule.
    bool tie = false;
    if (l3a < l3e) {
      best = l3a;
      mb = metric(v.pos(l3a));
    }
#pragma unroll 6
    for (int j = l3a + 1; j < l3e; ++j) {
      const float mm = metric(v.pos(j));
      if (mm < mb) {
        best = j;
        mb = mm;
        tie = false;
      } else if (mm == mb) {
        tie = true;
      }
    }
    if (tie) {
      best = -1;
      mb = FLT_MAX;
      for (int j = l3a; j < l3e; ++j) visit(j);
    }
  } else {
    for (int m = 0; m <= NB / 2; ++m) {
      if (m >= 3) {
        const float dmin = (float)(m - 2) * (TWO_PI_F / NB) - C.colw3;
        if (dmin > 0.f && (r3 * dmin) * (r3 * dmin) > mb) break;
      }
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (side == 1 && (m == 0 || m == NB / 2)) continue;
        const int bb = (b3 + (side ? -m : m)) & (NB - 1);
        const int e = v.l3(bb + 1);
        for (int j = v.l3(bb); j < e; ++j) visit(j);
      }
    }
  }
  o.status = 2;
  if (best < 0) return o;
  o.i3 = best;
  o.mbest = mb;
  const float4 p3 = v.pos(best);
  const TFitF f2 = fit_triplet(x1, y1, z1, x2, y2, z2, p3.x, p3.y, p3.z, C.hl[2], C.kB);
  o.status = 3;
  if (!f2.valid) return o;
  if constexpr (V::kPark) return global_fit(o, unpark_fit(*v.park), f2, C);
  else return global_fit(o, f1, f2, C);
}


// Record of a kept track for the vertex stage (layout below), from the layer-0 and
// layer-1 hits p0, p1 and the reconstruction o: transverse circle of radius
// R sin(theta01) through the two hits, centre on the side the track turns to.
// theta01 = theta_C0 + dtheta/dR (R - R_C0) enters through its cosine and sine,
// the rotation of (cos, sin) theta_C0 = (zp0, R_t) / R_C0 by the small correction.
__device__ __forceinline__ void track_record(const float4& p0, const float4& p1, const TrackOut& o, const DevCfg& C,
                                             float* tr) {
  const float x0 = p0.x, y0 = p0.y, x1 = p1.x, y1 = p1.y;
  const float Rb = 1.f / fabsf(o.kbar);
  const float pb = C.kB * Rb;
  float sd, cd;
  __sincosf(o.dth0 * (Rb - o.RC0), &sd, &cd);
  const float iRC = 1.f / o.RC0;
  const float ct = (o.zp0 * cd - o.Rct * sd) * iRC, st = (o.Rct * cd + o.zp0 * sd) * iRC;
  const float eps = o.kbar > 0.f ? 1.f : -1.f;
  const float rt = Rb * st;
  const float dx = x1 - x0, dy = y1 - y0;
  const float d = sqrtf(dx * dx + dy * dy);
  const float ex = dx / d, ey = dy / d;
  const float hd = 0.5f * d;
  const float off = sqrtf(fmaxf((rt - hd) * (rt + hd), 0.f));
  const float cx = 0.5f * (x0 + x1) + eps * ey * off;
  const float cy = 0.5f * (y0 + y1) - eps * ex * off;
  tr[0] = cx;
  tr[1] = cy;
  tr[2] = rt;
  tr[3] = Rb;
  tr[4] = ct;
  tr[5] = st;
  tr[6] = pb;
  tr[7] = sqrtf(pb * pb + C.me2);
  tr[8] = C.hl[0] / pb;
  tr[9] = x0;
  tr[10] = y0;
  tr[11] = p0.z;
  tr[12] = atan2f(y0 - cy, x0 - cx);
  tr[13] = eps;
}

// Track record layout (14 floats): cx cy rt R ct st p E sms h0x h0y h0z ah0 eps
template <int CK>
__device__ __forceinline__ void store_track(TrkSoA<CK>& T, int k, const float* tr, int tid) {
  T.cx[k] = tr[0];
  T.cy[k] = tr[1];
  T.rt[k] = tr[2];
  T.R[k] = tr[3];
  T.ct[k] = tr[4];
  T.st[k] = tr[5];
  T.p[k] = tr[6];
  T.E[k] = tr[7];
  T.sms[k] = tr[8];
  T.h0x[k] = tr[9];
  T.h0y[k] = tr[10];
  T.h0z[k] = tr[11];
  T.ah0[k] = tr[12];
  T.eps[k] = tr[13];
  T.tid[k] = tid;
}

// ------------------------------------------------------------------ vertex

struct TrackR {  // one kept track in registers (record layout above)
  float cx, cy, rt, R, ct, st, p, E, sms, h0x, h0y, h0z, ah0, eps;
};

template <int CK>
__device__ __forceinline__ TrackR load_track(const TrkSoA<CK>& T, int k) {
  TrackR t;
  t.cx = T.cx[k]; t.cy = T.cy[k]; t.rt = T.rt[k]; t.R = T.R[k]; t.ct = T.ct[k]; t.st = T.st[k];
  t.p = T.p[k]; t.E = T.E[k]; t.sms = T.sms[k]; t.h0x = T.h0x[k]; t.h0y = T.h0y[k]; t.h0z = T.h0z[k];
  t.ah0 = T.ah0[k]; t.eps = T.eps[k];
  return t;
}

// The global record of the staged form, one 32-byte sector: cx cy rt R, ct st ah0 and the
// layer-0 hit's place among the sorted hits, complemented for a negative charge.  Momentum
// and scattering width follow from R by the operations of track_record (E is not filled).
// With 64 bytes the track stage of 1e6 throughput frames took 2334 us instead of 2317, and
// the scratch a third more.
__device__ __forceinline__ void store_record(float4* rec, int64_t k, const float* tr, int hit) {
  rec[2 * k] = make_float4(tr[0], tr[1], tr[2], tr[3]);
  rec[2 * k + 1] = make_float4(tr[4], tr[5], tr[12], __int_as_float(tr[13] > 0.f ? hit : ~hit));
}
__device__ __forceinline__ TrackR load_track(const float4* __restrict__ rec, const float4* __restrict__ hits, int64_t k,
                                             const DevCfg& C) {
  const float4 a = __ldg(rec + 2 * k), b = __ldg(rec + 2 * k + 1);
  const int h = __float_as_int(b.w);
  const float4 q = __ldg(hits + (h < 0 ? ~h : h));
  TrackR t;
  t.cx = a.x; t.cy = a.y; t.rt = a.z; t.R = a.w;
  t.ct = b.x; t.st = b.y; t.ah0 = b.z;
  t.p = __fmul_rn(C.kB, t.R);
  t.E = 0.f;
  t.sms = C.hl[0] / t.p;
  t.h0x = q.x; t.h0y = q.y; t.h0z = q.z;
  t.eps = h < 0 ? -1.f : 1.f;
  return t;
}

// Turning angle travelled from point (x, y) forward to the track's layer-0 hit.
__device__ __forceinline__ float arc_to_h0(const TrackR& t, float x, float y) {
  return wrap_2pi(t.eps * (atan2f(y - t.cy, x - t.cx) - t.ah0));
}

__device__ __forceinline__ float point_var(const TrackR& t, float x, float y, float sp2) {
  const float s = t.rt * arc_to_h0(t, x, y);
  return t.sms * t.sms * s * s + sp2;
}

__device__ __forceinline__ float target_distance(const DevCfg& C, float x, float y, float z) {
  const float px = sqrtf(x * x + y * y), pz = fabsf(z);
  const float ex = -C.tgt_r, ez = C.tgt_h;
  float t = ((px - C.tgt_r) * ex + pz * ez) / (ex * ex + ez * ez);
  t = fminf(1.f, fmaxf(0.f, t));
  const float dx = px - (C.tgt_r + t * ex), dz = pz - t * ez;
  return sqrtf(dx * dx + dz * dz);
}

// Longitudinal momentum sum of a combination (the z part of |sum p|, Sec. "Vertex
// Fit"), rounded in one fixed order, so that the vertex and the early test below
// see the same value.  It does not depend on the vertex position.
__device__ __forceinline__ float pz_track(float p, float ct) { return __fmul_rn(p, ct); }
__device__ __forceinline__ float pz_sum(float pa, float pb, float pe) { return __fadd_rn(__fadd_rn(pa, pb), pe); }

// |sum p| >= |P_z|: the vertex's sum of squares only adds non-negative terms and
// rounding is monotone, so its |sum p| is at least sqrt(fl(P_z^2)).  When P_z^2
// exceeds the squared momentum cut by a relative 1e-4 (far more than any rounding
// of the cut or the square root), the combination fails the cut whatever its
// vertex, and the decision-only runs skip its vertex.  Runs that report each
// combination's status (debug records, statistics) still fit it.
__device__ __forceinline__ bool pz_fails_ptot(float Pz, float ptot_max) {
  return __fmul_rn(Pz, Pz) > ptot_max * ptot_max * 1.0001f;
}

struct VtxOut {
  int status, pass;
  float chi2, tdist, ptot;
  float chi2_second;  // second-smallest chi2 over the choices (candidate record only)
};

// Whether the transverse circles (centre, radius) of two tracks intersect, with
// the distance D of the centres, the foot aa of the chord on the centre line and
// the squared half chord h2.
__device__ __forceinline__ bool circles_meet(float acx, float acy, float ar, float bcx, float bcy, float br, float& D,
                                             float& aa, float& h2) {
  const float ex = bcx - acx, ey = bcy - acy;
  D = sqrtf(ex * ex + ey * ey);
  if (!(D > 0.f)) return false;
  aa = ((ar - br) * (ar + br) + D * D) / (2.f * D);
  h2 = (ar - aa) * (ar + aa);
  return !(h2 < 0.f);
}

// Intersection points of the circles of tracks a and b, in two fixed slots (q0
// first, as the oracle orders them), each with its target-filter flag.  Returns
// false when the circles do not intersect.  One routine for the prefilter of the
// vertex stage and for the vertex itself, so both take the same decisions.
__device__ __forceinline__ bool pair_geometry(float acx, float acy, float ar, float bcx, float bcy, float br,
                                              float lim, float& x0, float& y0, bool& k0, float& x1, float& y1,
                                              bool& k1) {
  k0 = k1 = false;
  float D, aa, h2;
  if (!circles_meet(acx, acy, ar, bcx, bcy, br, D, aa, h2)) return false;
  const float ex = (bcx - acx) / D, ey = (bcy - acy) / D;
  const float bx = acx + aa * ex, by = acy + aa * ey;
  const float h = sqrtf(h2);
  x0 = bx - h * ey;
  y0 = by + h * ex;
  x1 = bx + h * ey;
  y1 = by - h * ex;
  k0 = sqrtf(x0 * x0 + y0 * y0) <= lim;
  k1 = h2 != 0.f && sqrtf(x1 * x1 + y1 * y1) <= lim;
  return true;
}

// The quantities that decide the geometric steps of the vertex, over all three
// pairs whatever the status (candidate record only, for the boundary bands of a
// parity check): the smallest squared half chord relative to the product of the
// two radii, and the smallest distance of an intersection point from the filter
// radius.  Symmetric in the tracks, so independent of their order.
__device__ __forceinline__ void vertex_soft(const TrackR& A, const TrackR& B, const TrackR& E, float lim, float& disc,
                                            float& margin) {
  disc = margin = FLT_MAX;
  const TrackR* V[3] = {&A, &B, &E};
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    const TrackR& a = *V[k == 2 ? 1 : 0];
    const TrackR& b = *V[k == 0 ? 1 : 2];
    float D, aa, h2;
    const bool meet = circles_meet(a.cx, a.cy, a.rt, b.cx, b.cy, b.rt, D, aa, h2);
    if (!(D > 0.f)) continue;
    disc = fminf(disc, fabsf(h2) / (a.rt * b.rt));
    if (!meet) continue;
    float x0, y0, x1, y1;
    bool k0, k1;
    pair_geometry(a.cx, a.cy, a.rt, b.cx, b.cy, b.rt, lim, x0, y0, k0, x1, y1, k1);
    margin = fminf(margin, fabsf(sqrtf(x0 * x0 + y0 * y0) - lim));
    if (h2 != 0.f) margin = fminf(margin, fabsf(sqrtf(x1 * x1 + y1 * y1) - lim));
  }
}

// The two e+ tracks of a combination enter the vertex ordered by their circle centres.  The
// roundings of the vertex depend on the order, and the numbers of the tracks depend on the form
// and, where the threads of a CTA number them by arrival, on the run: with an order by value
// every form and every run takes the same decision, whatever the order of a frame's hits.  (With
// equal centres the circles do not meet, either way.)  1e6 throughput frames 5264 -> 5283 us.
__device__ __forceinline__ bool swapped(float acx, float acy, float bcx, float bcy) {
  return acx != bcx ? acx > bcx : acy > bcy;
}

// Status of a combination after the first two vertex steps: 0 a pair of circles
// does not intersect, 1 the target filter leaves a pair without points, 2 go on.
__device__ __forceinline__ int vertex_prefilter(const float* ta, const float* tb, const float* e, float lim) {
  const bool sw = swapped(ta[0], ta[1], tb[0], tb[1]);
  const float a[3] = {sw ? tb[0] : ta[0], sw ? tb[1] : ta[1], sw ? tb[2] : ta[2]};
  const float b[3] = {sw ? ta[0] : tb[0], sw ? ta[1] : tb[1], sw ? ta[2] : tb[2]};
  float x0, y0, x1, y1;
  bool k0, k1, k2, k3, k4, k5;
  if (!pair_geometry(a[0], a[1], a[2], b[0], b[1], b[2], lim, x0, y0, k0, x1, y1, k1)) return 0;
  if (!pair_geometry(a[0], a[1], a[2], e[0], e[1], e[2], lim, x0, y0, k2, x1, y1, k3)) return 0;
  if (!pair_geometry(b[0], b[1], b[2], e[0], e[1], e[2], lim, x0, y0, k4, x1, y1, k5)) return 0;
  return (k0 || k1) && (k2 || k3) && (k4 || k5) ? 2 : 1;
}

// pair_geometry plus the error of each surviving point (sum of both tracks' errors).
__device__ __forceinline__ int pair_points(const TrackR& a, const TrackR& b, const DevCfg& C, float& x0, float& y0,
                                           float& v0, bool& k0, float& x1, float& y1, float& v1, bool& k1) {
  v0 = v1 = 1.f;
  if (!pair_geometry(a.cx, a.cy, a.rt, b.cx, b.cy, b.rt, C.isect_lim, x0, y0, k0, x1, y1, k1)) return 0;
  if (k0) v0 = point_var(a, x0, y0, C.sig_pix2) + point_var(b, x0, y0, C.sig_pix2);
  if (k1) v1 = point_var(a, x1, y1, C.sig_pix2) + point_var(b, x1, y1, C.sig_pix2);
  return 1;
}

// Closest point of track t to (mx, my), its z on the helix and its error.  The
// closest point lies on the ray from the centre through (mx, my), so its angle
// seen from the centre is that of (mx - cx, my - cy).
__device__ __forceinline__ void closest(const TrackR& t, float mx, float my, float sp2, float& px, float& py,
                                        float& z, float& var, bool& bad) {
  const float dx = mx - t.cx, dy = my - t.cy;
  const float dn = sqrtf(dx * dx + dy * dy);
  if (!(dn > 0.f)) bad = true;
  const float sc = t.rt / dn;
  px = t.cx + sc * dx;
  py = t.cy + sc * dy;
  const float dphi = wrap_2pi(t.eps * (atan2f(dy, dx) - t.ah0));
  z = t.h0z - dphi * t.R * t.ct;
  const float s = t.rt * dphi;
  var = t.sms * t.sms * s * s + sp2;
}

// Vertex of one e+ e+ e- combination (Sec. "Vertex Fit", "Signal Estimation"):
// pairwise circle intersections, target-disk filter, error-weighted transverse
// mean for each choice of one point per pair, closest points, z projection, chi2;
// the smallest-chi2 choice is cut on chi2, target distance and |sum p|.  The loop
// over the (at most 8) choices stays rolled: its body is large, and one copy keeps
// the kernel's instruction footprint small.
__device__ __forceinline__ VtxOut vertex(const TrackR& Ta, const TrackR& Tb, const TrackR& E, const DevCfg& C) {
  const bool sw = swapped(Ta.cx, Ta.cy, Tb.cx, Tb.cy);
  const TrackR A = sw ? Tb : Ta, B = sw ? Ta : Tb;
  VtxOut o;
  o.status = 0;
  o.pass = 0;
  o.chi2 = o.tdist = o.ptot = FLT_MAX;
  o.chi2_second = FLT_MAX;
  float x00, y00, v00, x01, y01, v01, x10, y10, v10, x11, y11, v11, x20, y20, v20, x21, y21, v21;
  bool k00, k01, k10, k11, k20, k21;
  if (!pair_points(A, B, C, x00, y00, v00, k00, x01, y01, v01, k01)) return o;
  if (!pair_points(A, E, C, x10, y10, v10, k10, x11, y11, v11, k11)) return o;
  if (!pair_points(B, E, C, x20, y20, v20, k20, x21, y21, v21, k21)) return o;
  o.status = 1;
  if (!(k00 || k01) || !(k10 || k11) || !(k20 || k21)) return o;
  float best = FLT_MAX, bmx = 0.f, bmy = 0.f, bmz = 0.f;
  bool have = false;
  // the valid choices as a bit set, visited in increasing order (s2 fastest, as the
  // oracle's loops), so each lane runs only its own choices
  unsigned valid = 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const bool s0 = (c >> 2) & 1, s1 = (c >> 1) & 1, s2 = c & 1;
    if ((s0 ? k01 : k00) && (s1 ? k11 : k10) && (s2 ? k21 : k20)) valid |= 1u << c;
  }
#pragma unroll 1
  while (valid) {
    const int c = __ffs(valid) - 1;
    valid &= valid - 1;
    const bool s0 = (c >> 2) & 1, s1 = (c >> 1) & 1, s2 = c & 1;
    const float w0 = 1.f / (s0 ? v01 : v00), w1 = 1.f / (s1 ? v11 : v10), w2 = 1.f / (s2 ? v21 : v20);
    const float iws = 1.f / (w0 + w1 + w2);
    const float mx = ((s0 ? x01 : x00) * w0 + (s1 ? x11 : x10) * w1 + (s2 ? x21 : x20) * w2) * iws;
    const float my = ((s0 ? y01 : y00) * w0 + (s1 ? y11 : y10) * w1 + (s2 ? y21 : y20) * w2) * iws;
    float pa, qa, za, va, pb, qb, zb, vb, pe, qe, ze, ve;
    bool bad = false;
    closest(A, mx, my, C.sig_pix2, pa, qa, za, va, bad);
    closest(B, mx, my, C.sig_pix2, pb, qb, zb, vb, bad);
    closest(E, mx, my, C.sig_pix2, pe, qe, ze, ve, bad);
    if (bad) continue;
    const float ia = 1.f / va, ib = 1.f / vb, ie = 1.f / ve;
    const float mz = (za * ia + zb * ib + ze * ie) / (ia + ib + ie);
    const float chi2 = ((pa - mx) * (pa - mx) + (qa - my) * (qa - my) + (za - mz) * (za - mz)) * ia +
                       ((pb - mx) * (pb - mx) + (qb - my) * (qb - my) + (zb - mz) * (zb - mz)) * ib +
                       ((pe - mx) * (pe - mx) + (qe - my) * (qe - my) + (ze - mz) * (ze - mz)) * ie;
    if (!have || chi2 < best) {
      if (have) o.chi2_second = best;
      have = true;
      best = chi2;
      bmx = mx;
      bmy = my;
      bmz = mz;
    } else if (chi2 < o.chi2_second) {
      o.chi2_second = chi2;
    }
  }
  if (!have || !isfinite(best)) return o;
  o.status = 2;
  o.chi2 = best;
  o.tdist = target_distance(C, bmx, bmy, bmz);
  float Px = 0.f, Py = 0.f;
  const TrackR* V[3] = {&A, &B, &E};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const TrackR& t = *V[i];
    const float dx = bmx - t.cx, dy = bmy - t.cy;
    const float idn = 1.f / sqrtf(dx * dx + dy * dy);
    const float ux = dx * idn, uy = dy * idn;  // direction of the closest point from the centre
    const float pt = t.p * t.st;
    Px += pt * t.eps * uy;
    Py -= pt * t.eps * ux;
  }
  const float Pz = pz_sum(pz_track(A.p, A.ct), pz_track(B.p, B.ct), pz_track(E.p, E.ct));
  o.ptot = sqrtf(Px * Px + Py * Py + Pz * Pz);
  o.pass = o.chi2 <= C.vtx_chi2 && o.tdist <= C.tgt_dist && o.ptot <= C.ptot_max;
  return o;
}

// ------------------------------------------------------------------ energy test

// The pr-th pair (a, b), a < b, of the order (0,1), (0,2), (1,2), (0,3), ...: the root is
// exact to one unit for every pair of C_TRK tracks, and each side is corrected once.
__device__ __forceinline__ void pair_of(int pr, int& a, int& b) {
  b = (int)((1.f + sqrtf(1.f + 8.f * (float)pr)) * 0.5f);
  if (b * (b - 1) / 2 > pr) --b;
  if ((b + 1) * b / 2 <= pr) ++b;
  a = pr - b * (b - 1) / 2;
}

// Energy test of every (e+ pair, e-) combination of a frame by one warp (Algorithm 4,
// part 1), a pair per lane and two e- at a time (two sums per instruction).  pEP: E and
// p cos(theta) of each e+ track; nEP: the e- tracks two by two, E of c and c + 1, then
// p cos(theta) of c and c + 1, an odd last track paired with a NaN energy, which passes no
// window.  Counts the combinations passing (ncombo) and, with stats, those whose P_z leaves
// the momentum cut open (nopen); put(k, a, b, c) gets the k-th combination to fit, in
// (pair, e-) order: all that pass, or with prune the open ones.  Once more than `enough`
// passed the frame overflows whatever follows, and the rest is not looked at.
template <class Put>
__device__ __forceinline__ void energy_test(const DevCfg& C, const float2* pEP, const float4* nEP, int npos, int nneg,
                                            bool prune, bool stats, int enough, int& ncombo, int& nwrite, int& nopen, const Put& put) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const int npair = npos * (npos - 1) / 2;
  const unsigned long long mmu = pack2(-C.m_mu, -C.m_mu);
  for (int p0 = 0; p0 < npair && ncombo <= enough; p0 += 32) {
    const int pr = p0 + lane;
    int a = 0, b = 0;
    float eab = __int_as_float(0x7fc00000), pzab = 0.f;  // NaN: a lane without a pair passes no window
    if (pr < npair) {
      pair_of(pr, a, b);
      const float2 ta = pEP[a], tb = pEP[b];
      eab = ta.x + tb.x;
      pzab = __fadd_rn(ta.y, tb.y);
    }
    const unsigned long long e2 = pack2(eab, eab), z2 = pack2(pzab, pzab);
    int cnt = 0, co = 0;
    for (int c = 0; c < nneg; c += 2) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(nEP + (c >> 1));
      const unsigned long long d = add2(add2(e2, v.x), mmu), z = add2(z2, v.y);
      const bool ok0 = fabsf(__uint_as_float((unsigned)d)) <= C.e_win;
      const bool ok1 = fabsf(__uint_as_float((unsigned)(d >> 32))) <= C.e_win;
      cnt += ok0;
      cnt += ok1;
      const bool open0 = ok0 && !pz_fails_ptot(__uint_as_float((unsigned)z), C.ptot_max);
      const bool open1 = ok1 && !pz_fails_ptot(__uint_as_float((unsigned)(z >> 32)), C.ptot_max);
      const bool wr0 = prune ? open0 : ok0, wr1 = prune ? open1 : ok1;
      if (__any_sync(FULL, wr0 || wr1)) {
        co += open0;
        co += open1;
        const unsigned m0 = __ballot_sync(FULL, wr0), m1 = __ballot_sync(FULL, wr1);
        if (wr0) put(nwrite + __popc(m0 & below), a, b, c);
        if (wr1) put(nwrite + __popc(m0) + __popc(m1 & below), a, b, c + 1);
        nwrite += __popc(m0) + __popc(m1);
      }
    }
    ncombo += __reduce_add_sync(FULL, cnt);
    if (stats) nopen += __reduce_add_sync(FULL, co);
  }
}

// Kept tracks of 32 triplets into the lists of energy_test (te: (eps E, P_z) of this lane's
// triplet, E > 0, or (0, 0)); put(k, positive) gets the place of this lane's track.
template <class Put>
__device__ __forceinline__ void list_tracks(const float2& te, float2* pEP, float4* nEP, int cap, int& npos, int& nneg,
                                            const Put& put) {
  const unsigned below = (1u << (threadIdx.x & 31)) - 1u;
  const bool pos = te.x > 0.f, neg = te.x < 0.f;
  const unsigned mp = __ballot_sync(FULL, pos), mn = __ballot_sync(FULL, neg);
  const int kp = npos + __popc(mp & below), kn = nneg + __popc(mn & below);
  npos += __popc(mp);
  nneg += __popc(mn);
  if (pos && kp < cap) {
    pEP[kp] = te;
    put(kp, true);
  }
  if (neg && kn < cap) {
    float* q = reinterpret_cast<float*>(nEP + (kn >> 1)) + (kn & 1);
    q[0] = -te.x;
    q[2] = te.y;
    put(kn, false);
  }
}
// The NaN beside an odd last e- track; then the lists are complete.
__device__ __forceinline__ void close_lists(float4* nEP, int cap, int nneg) {
  if ((threadIdx.x & 31) == 0 && (nneg & 1) && nneg < cap)
    reinterpret_cast<float*>(nEP + (nneg >> 1))[1] = __int_as_float(0x7fc00000);
  __syncwarp();
}

// ------------------------------------------------------------------ one frame


// The exact cut tests, written with explicitly rounded operations so that every
// stage and tier takes the same decision whatever the compiler contracts:
// Phi cut between two hits: h_a . h_b >= cos(phi_max) r_a r_b.
__device__ __forceinline__ bool phi_pass(float xa, float ya, float xb, float yb, float c) {
  return fmaf(xa, xb, __fmul_rn(ya, yb)) >= c;
}
// Delta lambda: |tan(lambda12) - tan(lambda01)| <= dl_max, with tan(lambda01) given.
__device__ __forceinline__ bool dl_pass(float z1, float z2, float tl01, const DevCfg& C) {
  return fabsf(fmaf(__fsub_rn(z2, z1), C.inv_dr12, -tl01)) <= C.dl_max;
}
__device__ __forceinline__ float tan_l01(float z0, float z1, const DevCfg& C) {
  return __fmul_rn(__fsub_rn(z1, z0), C.inv_dr01);
}
// r_tc window without division or root: (d01 d12 d20)^2 against (2 r cross)^2.
__device__ __forceinline__ bool rtc_pass(float x0, float y0, float x1, float y1, float x2, float y2,
                                         const DevCfg& C) {
  const float ax = __fsub_rn(x0, x1), ay = __fsub_rn(y0, y1), bx = __fsub_rn(x2, x1), by = __fsub_rn(y2, y1);
  const float cr = fmaf(ax, by, -__fmul_rn(ay, bx));
  const float ex = __fsub_rn(x2, x0), ey = __fsub_rn(y2, y0);
  const float Pq = __fmul_rn(__fmul_rn(fmaf(ax, ax, __fmul_rn(ay, ay)), fmaf(bx, bx, __fmul_rn(by, by))),
                             fmaf(ex, ex, __fmul_rn(ey, ey)));
  const float Qq = __fmul_rn(cr, cr);
  return cr != 0.f && Pq >= __fmul_rn(C.rtc_lo2, Qq) && Pq <= __fmul_rn(C.rtc_hi2, Qq);
}
// z bin of a layer-2 point in the warp stage: monotone in z, so every hit with z in
// [zlo, zhi] lies in bins zbin(zlo) .. zbin(zhi).
__device__ __forceinline__ int zbin2(float z, const DevCfg& C) {
  const int b = (int)__fmul_rn(__fadd_rn(z, C.zoff2), C.izw2);
  return b < 0 ? 0 : (b > NZB - 1 ? NZB - 1 : b);
}

// The phi bin of sorted layer-1 hit i: the last bin whose start is at most i (bins
// are in order; an empty bin shares its start with the next one).
__device__ __forceinline__ int layer1_bin(const uint16_t* bstart, int i) {
  int lo = 0, hi = NB - 1;
#pragma unroll
  for (int step = 0; step < 5; ++step) {  // NB = 32
    const int mid = (lo + hi + 1) >> 1;
    if ((int)bstart[NB + mid] <= i) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Add one hit to bucket key; returns the bucket's count (cursor) before it.  With
// packed cursors a bucket is one byte of a word: counts and starts stay below the
// 256 hits such a frame can hold, so no byte carries into the next.
template <class S>
__device__ __forceinline__ int bucket_add(S& sm, int key) {
  if constexpr (S::kPackB) {
    const int sh = 8 * (key & 3);
    return (int)((atomicAdd(&sm.bcur[key >> 2], 1u << sh) >> sh) & 255u);
  } else {
    return (int)atomicAdd(&sm.bcur[key], 1u);
  }
}

// Exclusive prefix of the bucket counts: bucket starts into bstart and, as the
// placement cursors, back into bcur.
template <class G, class S>
__device__ __forceinline__ void bucket_scan(const G& g, S& sm) {
  static_assert(NBK == 4 * 32, "one word of four packed buckets per lane");
  if (g.rank() < 32) {
    const int lane = g.rank();
    int v[NBK / 32];
    int s = 0;
#pragma unroll
    for (int k = 0; k < NBK / 32; ++k) {
      if constexpr (S::kPackB) v[k] = (int)((sm.bcur[lane] >> (8 * k)) & 255u);
      else v[k] = (int)sm.bcur[lane * (NBK / 32) + k];
      s += v[k];
    }
    int inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += t;
    }
    int ex = inc - s;
    uint32_t w = 0;
#pragma unroll
    for (int k = 0; k < NBK / 32; ++k) {
      sm.bstart[lane * (NBK / 32) + k] = (uint16_t)ex;
      if constexpr (S::kPackB) w |= (uint32_t)ex << (8 * k);
      else sm.bcur[lane * (NBK / 32) + k] = (uint32_t)ex;
      ex += v[k];
    }
    if constexpr (S::kPackB) sm.bcur[lane] = w;
    if (lane == 31) sm.bstart[NBK] = (uint16_t)inc;
  }
  g.sync();
}

// Which of n <= 32 hits (xs, ys: 16-byte aligned, readable to the next multiple of four)
// pass the Phi cut with the hit whose coordinates xx, yy hold twice: bit q for hit q.  The
// test is phi_pass, two hits per instruction; the sign of (product - c), which its rounding
// leaves as it is, is shifted into the mask, the last hit first.
__device__ __forceinline__ uint32_t phi_mask(const float* xs, const float* ys, int n, unsigned long long xx,
                                             unsigned long long yy, float c) {
  const unsigned long long mc = pack2(-c, -c);
  uint32_t m = 0u;
#pragma unroll 1
  for (int q = ((n + 3) & ~3) - 4; q >= 0; q -= 4) {
    const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(xs + q);
    const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(ys + q);
    const unsigned long long t1 = add2(fma2(X.y, xx, mul2(Y.y, yy)), mc);
    const unsigned long long t0 = add2(fma2(X.x, xx, mul2(Y.x, yy)), mc);
    m = __funnelshift_l((uint32_t)(t1 >> 32), m, 1);
    m = __funnelshift_l((uint32_t)t1, m, 1);
    m = __funnelshift_l((uint32_t)(t0 >> 32), m, 1);
    m = __funnelshift_l((uint32_t)t0, m, 1);
  }
  return ~m & bits_below(n);
}

// Selection cuts of a warp-stage frame (Algorithm 2), on the hits sorted by (layer,
// phi bin).  The layer-2 hits are also put in z-bin order (x, y, z and index packed
// in one record), so that for a (layer-1 hit, Phi01 partner) pair the Delta lambda
// cut, seen as a z window on the layer-2 hit, becomes a contiguous range of that
// order.  Per chunk of 32 layer-1 hits (a lane each):
//   1. the Phi01 partners as a bit mask over the layer-0 hits and the Phi12
//      partners as a bit mask over the z-ordered layer-2 hits, from passes over
//      those hits that all lanes take together (one broadcast load per hit);
//   2. the pairs of layer-1 hits that have Phi12 partners, numbered by a prefix sum
//      and listed with their layer-0 hit;
//   3. the pairs, 32 at a time: each lane takes its pair's layer-1 hit from the lane
//      that the list names, forms the z window (widened by 1e-3 mm against
//      rounding) and its bin range, and keeps the Phi12 partners inside it: the
//      candidate triplets, numbered by a prefix sum and listed;
//   4. the candidates, 32 at a time, through the exact Delta lambda and r_tc tests,
//      the survivors appended in a fixed order by ballot.
// The exact tests are the expressions every other stage uses (phi_pass, dl_pass,
// rtc_pass), and the z window contains every hit that passes Delta lambda, so the
// selected set equals the brute-force one.  sm.bad = 2 when a capacity is exceeded
// (the frame goes to a larger stage).  npair / ntt: this lane's share of the pair
// tests within the reachable phi bins (counted, with stats, as the other stages
// count them) and of the candidate triplets (Phi01 partners times Phi12 partners).
template <class S, int CT>
__device__ __forceinline__ void warp_cuts(S& sm, const DevCfg& C, bool stats, unsigned& npair, unsigned& ntt) {
  const int lane = threadIdx.x & 31;
  const int n0 = sm.bstart[NB], l1a = n0, l1b = sm.bstart[2 * NB], l2b = sm.bstart[3 * NB];
  const int n1 = l1b - l1a, n2 = l2b - l1b;
  bool over = n0 > W_L0 || n2 > W_L2;
  int nt = 0;
  if (!over) {
    // layer-2 hits in z-bin order: counting sort with byte counters packed four to a
    // word (in the candidate buffer, free until step 3), two hits per lane
    uint32_t* zc = reinterpret_cast<uint32_t*>(sm.cand);
    if (lane < NZB / 4) zc[lane] = 0u;
    __syncwarp();
    const int bq0 = lane < n2 ? zbin2(sm.z[l1b + lane], C) : -1;
    const int bq1 = lane + 32 < n2 ? zbin2(sm.z[l1b + lane + 32], C) : -1;
    if (bq0 >= 0) atomicAdd(&zc[bq0 >> 2], 1u << (8 * (bq0 & 3)));
    if (bq1 >= 0) atomicAdd(&zc[bq1 >> 2], 1u << (8 * (bq1 & 3)));
    __syncwarp();
    const uint32_t w = zc[lane >> 1];  // bins 2 lane, 2 lane + 1
    const int ca = (int)((w >> (16 * (lane & 1))) & 255u), cb = (int)((w >> (16 * (lane & 1) + 8)) & 255u);
    int inc = ca + cb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += t;
    }
    const int ex = inc - ca - cb;
    sm.zbs[2 * lane] = (uint8_t)ex;
    sm.zbs[2 * lane + 1] = (uint8_t)(ex + ca);
    if (lane == 31) sm.zbs[NZB] = (uint8_t)inc;
    __syncwarp();
    if (lane < NZB / 4) {
      uint32_t cw = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) cw |= (uint32_t)sm.zbs[4 * lane + k] << (8 * k);
      zc[lane] = cw;  // placement cursors
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int bq = h ? bq1 : bq0;
      if (lane + 32 * h < n0) {
        const float2 p0 = sm.xy[lane + 32 * h];
        sm.ox[lane + 32 * h] = p0.x;
        sm.oy[lane + 32 * h] = p0.y;
      }
      if (bq >= 0) {
        const int i2 = l1b + lane + 32 * h;
        const int pos = (int)((atomicAdd(&zc[bq >> 2], 1u << (8 * (bq & 3))) >> (8 * (bq & 3))) & 255u);
        const float2 p2 = sm.xy[i2];
        sm.zx[pos] = p2.x;
        sm.zy[pos] = p2.y;
        sm.zzi[pos] = make_float2(sm.z[i2], __int_as_float(i2));
      }
    }
    __syncwarp();
  }
  for (int j0 = 0; j0 < n1 && !over; j0 += 32) {
    const int j = j0 + lane;
    const bool has = j < n1;
    const int i1 = l1a + j;
    float x1 = 0.f, y1 = 0.f, z1 = 0.f;
    if (has) {
      const float2 p1 = sm.xy[i1];
      x1 = p1.x;
      y1 = p1.y;
      z1 = sm.z[i1];
      if (stats) {  // the pair tests within the reachable phi bins, as the other stages count them
        const int nb0 = min(2 * C.k01 + 1, NB), nb2 = min(2 * C.k12 + 1, NB);
        const int b1 = layer1_bin(sm.bstart, i1);
        const int s0 = nb0 == NB ? 0 : (b1 - C.k01 + NB) & (NB - 1);
        const int s2 = nb2 == NB ? 0 : (b1 - C.k12 + NB) & (NB - 1);
        npair += sm.bstart[min(s0 + nb0, NB)] - sm.bstart[s0] + (s0 + nb0 > NB ? sm.bstart[s0 + nb0 - NB] : 0);
        npair += sm.bstart[2 * NB + min(s2 + nb2, NB)] - sm.bstart[2 * NB + s2] +
                 (s2 + nb2 > NB ? sm.bstart[2 * NB + s2 + nb2 - NB] - sm.bstart[2 * NB] : 0);
      }
    }
    // 1. Phi01 and Phi12 partners as bit masks (a lane without a layer-1 hit has none: its
    // (0, 0) would pass a cut above pi/2)
    const unsigned long long xx = pack2(x1, x1), yy = pack2(y1, y1);
    const uint32_t a0 = phi_mask(sm.ox, sm.oy, min(n0, 32), xx, yy, C.c01);
    const uint32_t a1 = n0 > 32 ? phi_mask(sm.ox + 32, sm.oy + 32, n0 - 32, xx, yy, C.c01) : 0u;
    const uint32_t b0 = phi_mask(sm.zx, sm.zy, min(n2, 32), xx, yy, C.c12);
    const uint32_t b1 = n2 > 32 ? phi_mask(sm.zx + 32, sm.zy + 32, n2 - 32, xx, yy, C.c12) : 0u;
    const int c01 = has ? __popc(a0) + __popc(a1) : 0, c12all = __popc(b0) + __popc(b1);
    ntt += (unsigned)(c01 * c12all);
    // 2. the pairs whose layer-1 hit has Phi12 partners, listed by their layer-0 hit
    const int pc = c12all ? c01 : 0;
    int pe = pc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, pe, o);
      if (lane >= o) pe += t;
    }
    const int pre = pe - pc;
    const int T = __shfl_sync(FULL, pe, 31);
    if (T > W_P01) {
      over = true;
      break;
    }
    if (pc) {
      int wpos = pre;
#pragma unroll 1
      for (uint32_t m = a0; m; m &= m - 1u) sm.p01[wpos++] = (uint16_t)((__ffs(m) - 1) | (lane << 8));
#pragma unroll 1
      for (uint32_t m = a1; m; m &= m - 1u) sm.p01[wpos++] = (uint16_t)((__ffs(m) + 31) | (lane << 8));
    }
    __syncwarp();
    // 3. the pairs, 32 at a time
#pragma unroll 1
    for (int k0 = 0; k0 < T; k0 += 32) {
      const int k = k0 + lane;
      const int pair = k < T ? sm.p01[k] : 0;
      const int i0 = pair & 255, ow = pair >> 8;  // layer-0 hit, lane of the layer-1 hit
      const float px1 = __shfl_sync(FULL, x1, ow), py1 = __shfl_sync(FULL, y1, ow), pz1 = __shfl_sync(FULL, z1, ow);
      uint32_t cl = __shfl_sync(FULL, b0, ow), ch = 0u;
      if (n2 > 32) ch = __shfl_sync(FULL, b1, ow);
      const float2 h0 = sm.xy[i0];
      const float x0 = h0.x, y0 = h0.y, tl01 = tan_l01(sm.z[i0], pz1, C);
      int lo = 0, hi = 0;
      if (k < T) {
        const float zlo = pz1 + (tl01 - C.dl_max) * C.dr12 - 1e-3f;
        const float zhi = pz1 + (tl01 + C.dl_max) * C.dr12 + 1e-3f;
        lo = sm.zbs[zbin2(zlo, C)];
        hi = sm.zbs[zbin2(zhi, C) + 1];
      }
      cl &= bits_below(hi) & ~bits_below(lo);
      if (n2 > 32) ch &= bits_below(max(hi - 32, 0)) & ~bits_below(max(lo - 32, 0));
      const int tri01 = i0 | ((l1a + j0 + ow) << 8);  // the pair's layer-0 and layer-1 sorted indices
      const int cnt = __popc(cl) + __popc(ch);
      int ce = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, ce, o);
        if (lane >= o) ce += t;
      }
      const int cpre = ce - cnt, ctot = __shfl_sync(FULL, ce, 31);
      for (int c0 = 0; c0 < ctot; c0 += W_CAND) {
        // each lane lists its candidates numbered c0 .. c0 + W_CAND - 1: pair lane, z-order position
        int idx = cpre - c0;
#pragma unroll 1
        for (uint32_t m = cl; m; m &= m - 1u, ++idx)
          if ((unsigned)idx < (unsigned)W_CAND) sm.cand[idx] = (uint16_t)((lane << 6) | (__ffs(m) - 1));
#pragma unroll 1
        for (uint32_t m = ch; m; m &= m - 1u, ++idx)
          if ((unsigned)idx < (unsigned)W_CAND) sm.cand[idx] = (uint16_t)((lane << 6) | (__ffs(m) + 31));
        __syncwarp();
        // 4. the exact tests, 32 candidates at a time
        const int ne = min(ctot - c0, W_CAND);
#pragma unroll 1
        for (int e0 = 0; e0 < ne; e0 += 32) {
          const int e = e0 + lane;
          const int ent = e < ne ? sm.cand[e] : 0;
          const int pl = ent >> 6;
          const float cx0 = __shfl_sync(FULL, x0, pl), cy0 = __shfl_sync(FULL, y0, pl);
          const float cx1 = __shfl_sync(FULL, px1, pl), cy1 = __shfl_sync(FULL, py1, pl);
          const float cz1 = __shfl_sync(FULL, pz1, pl), ctl = __shfl_sync(FULL, tl01, pl);
          const int ct = __shfl_sync(FULL, tri01, pl);
          const float2 h = sm.zzi[ent & 63];
          const bool pass = e < ne && dl_pass(cz1, h.x, ctl, C) &&
                            rtc_pass(cx0, cy0, cx1, cy1, sm.zx[ent & 63], sm.zy[ent & 63], C);
          const unsigned bm = __ballot_sync(FULL, pass);
          const int kk = nt + __popc(bm & ((1u << lane) - 1u));
          if (pass && kk < CT) sm.u.trip[kk] = make_trip<typename S::TripT>(ct & 255, ct >> 8, __float_as_int(h.y));
          nt += __popc(bm);
        }
        __syncwarp();
        if (nt > C.max_trip) break;  // the frame overflows: its decision is known
      }
      if (nt > C.max_trip) break;
    }
    if (nt > C.max_trip) break;
  }
  if (over) npair = ntt = 0;  // the frame is counted by the stage that takes it over
  if (lane == 0) {
    sm.ntrip = nt;
    sm.bad = over ? 2 : 0;
  }
  __syncwarp();
}

constexpr int PENDING = -2;  // frame_front result: triplets selected, later stages to run

// Stages A-C of one frame (load, sort, selection cuts).  Returns a final reason,
// DEFERRED (frame too large for this stage), or PENDING with the selected
// triplets in sm.u.trip and their count in sm.ntrip.
// LIVE: the hits sit in a ring that the host rewrites while the kernel runs
// (streaming), so they are read with loads that bypass the caches instead of
// the read-only path.
// prefetch_next: the group takes frame f + 1 next; its addresses are fetched into
// L1 while this frame is processed.
// NOST: compiled for runs without statistics (P.stats is null).  TAB: the warp stage
// decodes with the per-layer constants from a shared-memory table (decode_s) instead of
// the constant cache (the staged form's stage 1 measured faster so, the fused kernels
// slower).
template <class G, class S, int CH, int CT, bool DEFER, bool DEBUG, bool LIVE = false, bool NOST = false,
          bool TAB = false>
__device__ int frame_front(const G& g, S& sm, const DevCfg& C, const KParams& P, int f, bool prefetch_next = false) {
  const bool stats = !NOST && P.stats != nullptr;
  const int64_t base = P.off[f] - P.off_base;
  const int64_t n64 = P.off[f + 1] - P.off[f];
  if constexpr (G::N == 32 && !LIVE) {
    if (prefetch_next) {
      const int64_t nb = P.off[f + 1] - P.off_base, ne = P.off[f + 2] - P.off_base;
      const int64_t a = nb + 32 * g.rank();
      if (g.rank() < 8 && a < ne) prefetch_l1(P.hits + a);
    }
  }
  if (DEBUG && g.leader()) {
    P.dump.n_trip[f] = 0;
    P.dump.n_combo[f] = 0;
  }
  if (n64 < 0) {
    if (g.leader()) atomicOr(P.err, ERR_NEGSIZE);
    return M3E_ERR_BADHIT;
  }
  if (DEFER && n64 > (CH < P.defer_hits ? CH : P.defer_hits)) return DEFERRED;
  const int n = (int)(n64 > 0x7fffffff ? 0x7fffffff : n64);
  const int32_t* hp = P.hits + base;

  // ---- A: decode and histogram
  for (int k = g.rank(); k < (S::kPackB ? NBK / 4 : NBK); k += G::N) sm.bcur[k] = 0;
  // warp stage: the per-layer decode table (DevCfg::ltab) for parts A and B, in the
  // space of the layer-2 z order, which part C fills later
  uint4* const ltab = reinterpret_cast<uint4*>(sm.zx);
  if constexpr (G::N == 32 && DEFER && TAB) {
    static_assert(sizeof(sm.zx) >= 4 * sizeof(uint4), "room for the decode table");
    if (g.rank() < 4) ltab[g.rank()] = C.ltab[g.rank()];
  }
  if (g.leader()) {
    sm.bad = 0;
    sm.ntrip = 0;
    sm.npos = 0;
    sm.nneg = 0;
    sm.ncombo = 0;
    sm.nstore = 0;
    sm.flag = 0;
    if (stats)
      for (int k = 0; k < ST_REASON0; ++k) sm.facc[k] = 0;
  }
  g.sync();
  if constexpr (G::N == 32 && DEFER) {
    // warp stage (n <= CH): each lane holds its hits' addresses in registers, so the
    // loads of a frame (addresses, then the table entries) are all in flight at once
    constexpr int K = (CH + 31) / 32;
    const int lane = g.rank();
    uint32_t av[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int i = lane + 32 * k;
      av[k] = i < n ? (uint32_t)(LIVE ? __ldcv(hp + i) : __ldg(hp + i)) : 0u;
    }
    // the bucket and the table indices (15 bits each) of a hit stay in registers
    bool bad = false;
    int key[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (lane + 32 * k < n) {
        const Dec d = TAB ? decode_s(ltab, av[k]) : decode(C, av[k]);
        key[k] = d.L * NB + d.b;
        av[k] = (uint32_t)d.ci | (uint32_t)d.ri << 15;
        if (!d.ok) bad = true;
        else bucket_add(sm, key[k]);
      }
    }
    if (__any_sync(FULL, bad)) {
      if (g.leader()) atomicOr(P.err, ERR_BADHIT);
      return M3E_ERR_BADHIT;
    }
    if (n > C.max_hits) return M3E_HIT_OVERFLOW;
    if (stats && g.leader()) {
      sm.facc[ST_FRAMES] += 1;
      sm.facc[ST_HITS] += n;
    }
    // ---- B: counting sort by (layer, phi bin); the table entries go straight from
    // global to shared memory (asynchronous 4-byte copies, all of the lane's in flight)
    bucket_scan(g, sm);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int i = lane + 32 * k;
      if (i < n) {
        const int pos = bucket_add(sm, key[k]);
        const float* cl = reinterpret_cast<const float*>(P.col_lut + (av[k] & 0x7fffu));
        cp_async8(&sm.xy[pos], cl);
        if (key[k] >= 3 * NB) cp_async4(&sm.phi[pos], cl + 2);
        cp_async4(&sm.z[pos], P.row_lut + (av[k] >> 15));
        if constexpr (S::kIdx) sm.inidx[pos] = (uint16_t)i;
      }
    }
    cp_async_wait_all();
  } else {
    for (int i = g.rank(); i < n; i += G::N) {
      const Dec d = decode(C, (uint32_t)(LIVE ? __ldcv(hp + i) : __ldg(hp + i)));
      if (!d.ok) sm.bad = 1;
      else if (n <= CH) bucket_add(sm, d.L * NB + d.b);
    }
    g.sync();
    if (sm.bad) {
      if (g.leader()) atomicOr(P.err, ERR_BADHIT);
      return M3E_ERR_BADHIT;
    }
    if (n > C.max_hits || n > CH) return M3E_HIT_OVERFLOW;
    if (stats && g.leader()) {
      sm.facc[ST_FRAMES] += 1;
      sm.facc[ST_HITS] += n;
    }

    // ---- B: counting sort by (layer, phi bin)
    bucket_scan(g, sm);
    for (int i = g.rank(); i < n; i += G::N) {
      const uint32_t a = (uint32_t)(LIVE ? __ldcv(hp + i) : __ldg(hp + i));
      const Dec d = decode(C, a);
      const int key = d.L * NB + d.b;
      const int pos = bucket_add(sm, key);
      const float4 c4 = __ldg(P.col_lut + d.ci);
      sm.xy[pos] = make_float2(c4.x, c4.y);
      sm.phi[pos] = c4.z;
      sm.z[pos] = __ldg(P.row_lut + d.ri);
      if constexpr (S::kIdx) sm.inidx[pos] = (uint16_t)i;
    }
  }
  g.sync();

  // ---- C: selection cuts (Algorithm 2), pairs restricted to reachable phi bins.
  // The bins of a window are contiguous in the sorted order, so a window is one
  // index range, or two when it wraps past phi = 2 pi.
  {
    unsigned npair = 0, ntt = 0;
    const int l1a = sm.bstart[NB], l1b = sm.bstart[2 * NB];
    const int nb0 = min(2 * C.k01 + 1, NB), nb2 = min(2 * C.k12 + 1, NB);
    if constexpr (G::N == 32) {
      warp_cuts<S, CT>(sm, C, stats, npair, ntt);
    } else {
      // CTA stage.  The layer-2 hits are first put in z-bin order, so that the Delta
      // lambda cut of a (layer-0, layer-1) pair, seen as a z window on the layer-2 hit
      // (widened by 1e-3 mm against rounding), is one contiguous range of that order.
      // Each warp holds 32 layer-1 hits at a time and tests the entries of their Phi01
      // windows 32 at a time; the z ranges of the pairs that pass are numbered by a
      // prefix sum, and their candidates are tested 32 at a time with the exact Phi12, Delta lambda and r_tc expressions of the warp stage.  The z window holds every hit that
      // passes Delta lambda, so the selected set equals the brute-force one.  A frame
      // whose triplet count passed max_trip overflows whatever follows: the warps stop.
      constexpr int NW = G::N / 32;
      const int lane = g.rank() & 31, wid = g.rank() >> 5;
      const int l2b = sm.bstart[3 * NB];
      static_assert(NZB == 64, "two z bins per lane in the prefix sum");
      for (int k = g.rank(); k < NZB; k += G::N) sm.zcur[k] = 0u;
      g.sync();
      for (int i = l1b + g.rank(); i < l2b; i += G::N) atomicAdd(&sm.zcur[zbin2(sm.z[i], C)], 1u);
      g.sync();
      if (g.rank() < 32) {
        const int ca = (int)sm.zcur[2 * lane], cb = (int)sm.zcur[2 * lane + 1];
        int inc = ca + cb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(FULL, inc, o);
          if (lane >= o) inc += t;
        }
        const int ex = inc - ca - cb;
        sm.zbs2[2 * lane] = (uint16_t)ex;
        sm.zbs2[2 * lane + 1] = (uint16_t)(ex + ca);
        sm.zcur[2 * lane] = (uint32_t)ex;
        sm.zcur[2 * lane + 1] = (uint32_t)(ex + ca);
        if (lane == 31) sm.zbs2[NZB] = (uint16_t)inc;
      }
      g.sync();
      for (int i = l1b + g.rank(); i < l2b; i += G::N) sm.zidx[atomicAdd(&sm.zcur[zbin2(sm.z[i], C)], 1u)] = (uint16_t)i;
      g.sync();
      auto overflowed = [&]() {
        int ov = 0;
        if (lane == 0) ov = *(volatile int*)&sm.ntrip > C.max_trip;
        return __shfl_sync(FULL, ov, 0) != 0;
      };
      // a warp takes every NW-th layer-1 hit, 32 of them at a time (a lane each);
      // the Phi01 windows of those hits are tested 32 entries at a time
      const int nh = l1b - l1a > wid ? (l1b - l1a - wid + NW - 1) / NW : 0;
      bool stop = false;
      for (int mb = 0; mb < nh && !stop; mb += 32) {
        const bool has = mb + lane < nh;
        const int i1 = l1a + wid + NW * (mb + lane);
        float x1 = 0.f, y1 = 0.f, z1 = 0.f;
        int a0 = 0, n0a = 0, n0w = 0, c12 = 0;
        if (has) {
          const float2 p1 = sm.xy[i1];
          x1 = p1.x;
          y1 = p1.y;
          z1 = sm.z[i1];
          const int b1 = layer1_bin(sm.bstart, i1);
          const int s0 = nb0 == NB ? 0 : (b1 - C.k01 + NB) & (NB - 1);
          a0 = sm.bstart[s0];
          n0a = sm.bstart[min(s0 + nb0, NB)] - a0;
          n0w = n0a + (s0 + nb0 > NB ? sm.bstart[s0 + nb0 - NB] : 0);
          if (stats) {  // the pair tests within the reachable phi bins, and the Phi12 partners
            const int s2 = nb2 == NB ? 0 : (b1 - C.k12 + NB) & (NB - 1);
            const int a2 = sm.bstart[2 * NB + s2], n2a = sm.bstart[2 * NB + min(s2 + nb2, NB)] - a2;
            const int w2 = sm.bstart[2 * NB];
            npair += n0w + n2a + (s2 + nb2 > NB ? sm.bstart[2 * NB + s2 + nb2 - NB] - w2 : 0);
            for (int k = l1b; k < l2b; ++k) c12 += phi_pass(x1, y1, sm.xy[k].x, sm.xy[k].y, C.c12);
          }
        }
        int pe = n0w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(FULL, pe, o);
          if (lane >= o) pe += t;
        }
        const int pre1 = pe - n0w, T1 = __shfl_sync(FULL, pe, 31);
        // Which lane owns entry e: the lanes with entries are listed in order; the starts that
        // fall on these 32 entries are or-ed into a word, and the starts up to e counted.
        const unsigned upto = 0xffffffffu >> (31 - lane);
        uint8_t* const own1 = sm.own[wid][0];
        uint8_t* const own2 = sm.own[wid][1];
        const unsigned ne1 = __ballot_sync(FULL, n0w > 0);
        __syncwarp();
        if (n0w > 0) own1[__popc(ne1 & upto) - 1] = (uint8_t)lane;
        __syncwarp();
        int before1 = -1;  // starts before these entries, less one
        for (int e0 = 0; e0 < T1 && !stop; e0 += 32) {
          const int e = e0 + lane;
          const unsigned s1 = __reduce_or_sync(FULL, n0w > 0 && (unsigned)(pre1 - e0) < 32u ? 1u << (pre1 - e0) : 0u);
          const int ow = own1[before1 + __popc(s1 & upto)];
          before1 += __popc(s1);
          const int oa0 = __shfl_sync(FULL, a0, ow), on0a = __shfl_sync(FULL, n0a, ow);
          const int opre = __shfl_sync(FULL, pre1, ow), oi1 = __shfl_sync(FULL, i1, ow);
          const float ox1 = __shfl_sync(FULL, x1, ow), oy1 = __shfl_sync(FULL, y1, ow), oz1 = __shfl_sync(FULL, z1, ow);
          const int oc12 = __shfl_sync(FULL, c12, ow);
          int i0 = 0;
          bool p01 = false;
          if (e < T1) {
            const int k = e - opre;
            i0 = k < on0a ? oa0 + k : k - on0a;
            const float2 h0 = sm.xy[i0];
            p01 = phi_pass(h0.x, h0.y, ox1, oy1, C.c01);
          }
          if (p01) ntt += oc12;
          // the Phi01 pairs' z ranges in the z order of layer 2, then their candidates
          float tl01 = 0.f;
          int lo = 0, cnt = 0;
          if (p01) {
            tl01 = tan_l01(sm.z[i0], oz1, C);
            const float zlo = oz1 + (tl01 - C.dl_max) * C.dr12 - 1e-3f;
            const float zhi = oz1 + (tl01 + C.dl_max) * C.dr12 + 1e-3f;
            lo = sm.zbs2[zbin2(zlo, C)];
            cnt = sm.zbs2[zbin2(zhi, C) + 1] - lo;
          }
          int ce = cnt;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL, ce, o);
            if (lane >= o) ce += t;
          }
          const int pre2 = ce - cnt, T2 = __shfl_sync(FULL, ce, 31);
          const unsigned ne2 = __ballot_sync(FULL, cnt > 0);
          __syncwarp();
          if (cnt > 0) own2[__popc(ne2 & upto) - 1] = (uint8_t)lane;
          __syncwarp();
          int before2 = -1;
          for (int c0 = 0; c0 < T2 && !stop; c0 += 32) {
            const int c = c0 + lane;
            const unsigned s2 = __reduce_or_sync(FULL, cnt > 0 && (unsigned)(pre2 - c0) < 32u ? 1u << (pre2 - c0) : 0u);
            const int pw = own2[before2 + __popc(s2 & upto)];  // the lane whose candidate c is
            before2 += __popc(s2);
            const int pi0 = __shfl_sync(FULL, i0, pw), pi1 = __shfl_sync(FULL, oi1, pw);
            const int plo = __shfl_sync(FULL, lo, pw), ppre = __shfl_sync(FULL, pre2, pw);
            const float ptl = __shfl_sync(FULL, tl01, pw);
            const float px1 = __shfl_sync(FULL, ox1, pw), py1 = __shfl_sync(FULL, oy1, pw), pz1 = __shfl_sync(FULL, oz1, pw);
            if (c < T2) {
              const int i2 = sm.zidx[plo + c - ppre];
              const float2 h2 = sm.xy[i2], h0 = sm.xy[pi0];
              const float x2 = h2.x, y2 = h2.y, z2 = sm.z[i2];
              if (phi_pass(px1, py1, x2, y2, C.c12) && dl_pass(pz1, z2, ptl, C) &&
                  rtc_pass(h0.x, h0.y, px1, py1, x2, y2, C)) {
                const int kk = atomicAdd(&sm.ntrip, 1);
                if (kk < CT) sm.u.trip[kk] = make_trip<typename S::TripT>(pi0, pi1, i2);
              }
            }
            stop = overflowed();
          }
        }
      }
    }
    if (stats) {
      atomicAdd(&sm.facc[ST_PAIRS], (unsigned long long)npair);
      atomicAdd(&sm.facc[ST_TTESTS], (unsigned long long)ntt);
    }
  }
  g.sync();
  if (DEFER && sm.bad == 2) return DEFERRED;  // partner lists beyond the warp stage's capacity
  const int ntrip = sm.ntrip;
  if (DEBUG && g.leader()) P.dump.n_trip[f] = ntrip;
  if (ntrip > C.max_trip) return M3E_TRIPLET_OVERFLOW;
  if (DEFER && ntrip > CT) return DEFERRED;
  if (stats && g.leader()) sm.facc[ST_TRIP] += ntrip;
  return PENDING;
}

// Stages D-F of one frame after frame_front returned PENDING: track
// reconstruction, energy test and vertex.  Returns a final reason or DEFERRED.
template <class G, class S, int CT, int CK, int CC, bool DEFER, bool DEBUG, bool NOST = false>
__device__ int frame_back(const G& g, S& sm, const DevCfg& C, const KParams& P, int f) {
  const bool stats = !NOST && P.stats != nullptr;
  const int ntrip = sm.ntrip;
  const SmHits<S> view{sm};
  // ---- D: track reconstruction (Algorithm 3), one thread per triplet
  for (int t = g.rank(); t < ntrip; t += G::N) {
    const auto tr = sm.u.trip[t];
    const TrackOut o = build_track(view, C, tr.x, tr.y, tr.z);
    if (o.status == 5) {
      float tk[14];
      track_record(view.pos(tr.x), view.pos(tr.y), o, C, tk);
      int slot = -1;
      if (tk[13] > 0.f) {
        const int k = atomicAdd(&sm.npos, 1);
        if (k < CK) slot = k;
      } else {
        const int k = atomicAdd(&sm.nneg, 1);
        if (k < CK) slot = CK - 1 - k;
      }
      if (slot >= 0) store_track(sm.t, slot, tk, t);
    }
    if (DEBUG && t < P.dump.cap_trip) {
      const int64_t r = (int64_t)f * P.dump.cap_trip + t;
      P.dump.trip[4 * r + 0] = sm.inidx[tr.x];
      P.dump.trip[4 * r + 1] = sm.inidx[tr.y];
      P.dump.trip[4 * r + 2] = sm.inidx[tr.z];
      P.dump.trip[4 * r + 3] = o.i3 >= 0 ? (int)sm.inidx[o.i3] : -1;
      P.dump.trk_status[r] = o.status;
      P.dump.trk_val[4 * r + 0] = o.kbar;
      P.dump.trk_val[4 * r + 1] = o.th01;
      P.dump.trk_val[4 * r + 2] = o.chi2;
      P.dump.trk_val[4 * r + 3] = o.mbest;
    }
  }
  g.sync();
  const int npos = sm.npos, nneg = sm.nneg;
  const int ntrk = npos + nneg;
  if (ntrk > C.max_trk) return M3E_TRACK_OVERFLOW;
  if (DEFER && ntrk > CK) return DEFERRED;
  if (stats && g.leader()) sm.facc[ST_TRK] += ntrk;

  // ---- E: energy test of every (e+ pair, e-) combination (Algorithm 4, part 1):
  // one e+ pair per thread, the e- loop uniform across the group (broadcast reads).
  // All passing combinations count towards the cap; a decision-only run stores only
  // those whose P_z leaves the momentum cut open (pz_fails_ptot).
  const bool prune = !DEBUG && !stats;
  {
    const int npair = npos * (npos - 1) / 2;
    for (int pr = g.rank(); pr < npair; pr += G::N) {
      // past the cap the decision is known (the candidate record wants the full count)
      if (!DEBUG && *(volatile int*)&sm.ncombo > C.max_combo) break;
      int a, b;
      pair_of(pr, a, b);
      const float eab = sm.t.E[a] + sm.t.E[b];
      const float pzab = __fadd_rn(pz_track(sm.t.p[a], sm.t.ct[a]), pz_track(sm.t.p[b], sm.t.ct[b]));
      for (int c = 0; c < nneg; ++c) {
        const int ci = CK - 1 - c;
        const float e = (eab + sm.t.E[ci]) - C.m_mu;
        if (fabsf(e) <= C.e_win) {
          const int k = atomicAdd(&sm.ncombo, 1);
          const uint32_t code = (uint32_t)a | ((uint32_t)b << 8) | ((uint32_t)ci << 16);
          const bool open = !pz_fails_ptot(__fadd_rn(pzab, pz_track(sm.t.p[ci], sm.t.ct[ci])), C.ptot_max);
          if (!prune) {
            if (k < CC) sm.u.combo[k] = code;
            if (stats && open) atomicAdd(&sm.facc[ST_PZOPEN], 1ull);
          } else if (open) {
            const int k2 = atomicAdd(&sm.nstore, 1);
            if (k2 < CC) sm.u.combo[k2] = code;
          }
        }
      }
    }
    if (stats && g.leader()) sm.facc[ST_ETEST] += (unsigned long long)npair * nneg;
  }
  g.sync();
  const int ncombo = sm.ncombo;
  const int nvtx = prune ? sm.nstore : ncombo;  // combinations to fit
  if (DEBUG && g.leader()) P.dump.n_combo[f] = ncombo;
  if (ncombo > C.max_combo) {
    if (stats && g.leader()) sm.facc[ST_PZOPEN] = 0;  // counted, as the combinations, only when fitted
    return M3E_COMBO_OVERFLOW;
  }
  if (DEFER && nvtx > CC) return DEFERRED;
  if (stats && g.leader()) sm.facc[ST_COMBO] += ncombo;

  // ---- F: vertex of each combination (Algorithm 4, part 2), early exit
  bool found = false;
  unsigned nv = 0, nvo = 0;
  for (int c0 = 0; c0 < nvtx; c0 += G::N) {
    const int c = c0 + g.rank();
    bool pass = false;
    if (c < nvtx) {
      const uint32_t cb = sm.u.combo[c];
      const int a = cb & 255, b = (cb >> 8) & 255, e = (cb >> 16) & 255;
      const VtxOut v = vertex(load_track(sm.t, a), load_track(sm.t, b), load_track(sm.t, e), C);
      pass = v.pass != 0;
      nv += v.status == 2;
      if (stats && v.status == 2)
        nvo += !pz_fails_ptot(pz_sum(pz_track(sm.t.p[a], sm.t.ct[a]), pz_track(sm.t.p[b], sm.t.ct[b]),
                                     pz_track(sm.t.p[e], sm.t.ct[e])), C.ptot_max);
      if (DEBUG && c < P.dump.cap_combo) {
        const int64_t r = (int64_t)f * P.dump.cap_combo + c;
        P.dump.combo[4 * r + 0] = sm.t.tid[a];
        P.dump.combo[4 * r + 1] = sm.t.tid[b];
        P.dump.combo[4 * r + 2] = sm.t.tid[e];
        P.dump.combo[4 * r + 3] = v.status | (v.pass << 8);
        P.dump.combo_val[4 * r + 0] = (sm.t.E[a] + sm.t.E[b] + sm.t.E[e]) - C.m_mu;
        P.dump.combo_val[4 * r + 1] = v.chi2;
        P.dump.combo_val[4 * r + 2] = v.tdist;
        P.dump.combo_val[4 * r + 3] = v.ptot;
        if (P.dump.combo_aux) {
          float dm, fm;
          vertex_soft(load_track(sm.t, a), load_track(sm.t, b), load_track(sm.t, e), C.isect_lim, dm, fm);
          P.dump.combo_aux[4 * r + 0] = dm;
          P.dump.combo_aux[4 * r + 1] = fm;
          P.dump.combo_aux[4 * r + 2] = v.chi2_second;
          P.dump.combo_aux[4 * r + 3] = 0.f;
        }
      }
    }
    found = g.any(pass) || found;
    if (found && !DEBUG) break;
  }
  if (stats && nv) atomicAdd(&sm.facc[ST_VTX], (unsigned long long)nv);
  if (stats && nvo) atomicAdd(&sm.facc[ST_VTXOPEN], (unsigned long long)nvo);
  return found ? M3E_VERTEX : M3E_DROP;
}

template <class G, class S, bool NOST = false>
__device__ __forceinline__ void finish_frame(const G& g, S& sm, const KParams& P, int f, int r) {
  g.sync();
  if (g.leader()) {
    P.keep[f] = (uint8_t)(r != M3E_DROP);
    P.reason[f] = (uint8_t)r;
    if (!NOST && P.stats) {
      sm.acc[ST_REASON0 + r] += 1;
      for (int k = 0; k < ST_REASON0; ++k) sm.acc[k] += sm.facc[k];
    }
  }
}

template <class G, class S>
__device__ __forceinline__ void flush_stats(const G& g, S& sm, unsigned long long* stats) {
  g.sync();
  if (stats)
    for (int k = g.rank(); k < ST_REASON0 + 8; k += G::N)
      if (sm.acc[k]) atomicAdd(stats + k, sm.acc[k]);
}

template <class G, class S>
__device__ __forceinline__ void clear_stats(const G& g, S& sm) {
  for (int k = g.rank(); k < ST_REASON0 + 8; k += G::N) sm.acc[k] = 0;
  g.sync();
}

// Launch, with pdl as a programmatic dependent of the kernel before it on the stream: the
// launch and the prologue overlap that kernel's end.
template <class... K, class... A>
cudaError_t launch_kernel(bool pdl, void (*k)(K...), int grid, int threads, size_t smem, cudaStream_t s, const A&... a) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, a...);
}

}  // namespace
}  // namespace m3e
