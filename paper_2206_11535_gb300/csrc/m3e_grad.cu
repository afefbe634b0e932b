// Gradient of the summed track chi2 of frozen candidates with respect to the
// rigid alignment of the four layers and the field scale (libm3e).
//
// A candidate is a quadruplet of hits (layers 0..3) whose track the selection
// found (Sec. "Track Reconstruction": two triplet fits and the global chi2 at the
// inverse-variance mean curvature).  The hit measured at nominal position x_nom
// on layer L sits at R(w_L) x_nom + d_L, R = Rz(wz) Ry(wy) Rx(wx); the field is
// scaled by params[24].  The selection of the quadruplet is discrete and stays
// fixed; chi2 is differentiable in the positions, so the gradient is exact for
// the frozen set.
//
// One thread per candidate: forward fit (the same fit_triplet as the selection,
// so that the chi2 equals the selection's at nominal alignment), then the
// reverse sweep by hand, recomputing each triplet's intermediate values instead
// of storing them, but for the arc angles and the small polar offset, which it takes
// from the forward fit (the only transcendental functions).  d chi2 / d(field scale) =
// 2 chi2 / scale exactly: the scale enters only through sigma_MS ~ 1/p and the two
// triplets' weights scale alike.
// Sums: per thread FP32 with its rounding errors kept beside it, per block FP64, then
// one block in a fixed order (deterministic for a given grid).
#include "m3e_device.cuh"

namespace m3e {
namespace {

constexpr int GT = 128;            // threads per block
constexpr int NS = 26;             // chi2, 24 alignment sums, chi2 of the finite gradients
constexpr int NG = NS + 1;         // and the number of valid candidates

// A running sum and the sum of its rounding errors (Knuth's two-sum), so that the sum of a
// thread's candidates is as good however many they are.  The gradient's 26 sums live in shared
// memory: 971,437 candidates take 82 us (81 with plain sums in registers), 88 with 3 blocks per
// SM instead of 4, 101 with both parts in registers.
__device__ __forceinline__ void add_to(float2& s, float v) {
  const float t = __fadd_rn(s.x, v), b = __fsub_rn(t, s.x);
  s.y = __fadd_rn(s.y, __fadd_rn(__fsub_rn(s.x, __fsub_rn(t, b)), __fsub_rn(v, b)));
  s.x = t;
}
// (a sum beyond FP32's range is infinite, as a plain one, and has no error)
__device__ __forceinline__ float error_of(const float2& s) { return isfinite(s.x) ? s.y : 0.f; }

struct AlignSm {
  float R[4][9];                   // rotation of each layer (row-major)
  float d[4][3];
  float scale;
};

__device__ void rotation(const float* w, float* R) {  // Rz(w[2]) Ry(w[1]) Rx(w[0])
  float sx, cx, sy, cy, sz, cz;
  sincosf(w[0], &sx, &cx);
  sincosf(w[1], &sy, &cy);
  sincosf(w[2], &sz, &cz);
  R[0] = cz * cy;
  R[1] = cz * sy * sx - sz * cx;
  R[2] = cz * sy * cx + sz * sx;
  R[3] = sz * cy;
  R[4] = sz * sy * sx + cz * cx;
  R[5] = sz * sy * cx - cz * sx;
  R[6] = -sy;
  R[7] = cy * sx;
  R[8] = cy * cx;
}

// ------------------------------------------------------------------ reverse sweep

// One segment of the circle solution (segment_core in the shared device code):
// adjoints of (R_C, theta_C, dPhi/dR, dtheta/dR) to adjoints of (d, z, R_t, Phi).
// The outputs are written as functions of d, z, R_t and the arc angle Phi, with
// sh = sin(Phi/2) and ch = cos(Phi/2) functions of Phi: the arc angle is a smooth
// function of the hits (twice the triangle's angle at the third hit), whereas its
// form 2 asin(d / 2 R_t) has an infinite slope at a half turn, where the branch
// switches.  Every quotient shares the reciprocals of Phi, sh, R_C and the two
// denominators, computed once with the forward values of the segment.
struct SegB {
  float d, z, sh, ch, ph;              // inputs
  float iph, ish, zp, RC, iRC, A2, iQ, g, gp, iDz, T, dphi, dth;
};

__device__ __forceinline__ SegB segment_values(float d, float z, float Rct, float sh, float ch, float ph) {
  SegB s;
  s.d = d;
  s.z = z;
  s.sh = sh;
  s.ch = ch;
  s.ph = ph;
  s.iph = 1.f / ph;
  s.ish = 1.f / sh;
  s.zp = z * s.iph;
  const float r2 = Rct * Rct + s.zp * s.zp;
  s.RC = sqrtf(r2);
  s.iRC = 1.f / s.RC;
  const float ish2 = s.ish * s.ish;
  s.A2 = 0.25f * d * ish2 * s.ish;
  s.iQ = 1.f / (0.5f * d * s.A2 * ch + s.zp * s.zp * s.iph);
  s.dphi = -s.RC * s.iQ;
  s.g = 0.5f * ph * s.ish;
  s.gp = 0.5f * sin_minus_xcos(0.5f * ph, sh, ch) * ish2;
  const float dg = d * s.g;
  s.iDz = 1.f / (z * z + dg * dg);
  s.T = z * d * s.gp * s.iDz;
  s.dth = s.T * s.dphi;
  return s;
}

__device__ __forceinline__ void segment_bwd(const SegB& s, float Rct, float RC_b, float th_b, float dphi_b, float dth_b,
                                            float& d_b, float& z_b, float& Rct_b, float& phi_b) {
  // dth = T dphi, T = z d gp / Dz, Dz = z^2 + (d g)^2, g = ph / (2 sh)
  const float T_b = dth_b * s.dphi;
  dphi_b += dth_b * s.T;
  const float tD = T_b * s.iDz;
  const float Dz_b = -tD * s.T;
  z_b = tD * s.d * s.gp + 2.f * s.z * Dz_b;
  d_b = tD * s.z * s.gp;
  const float gp_b = tD * s.z * s.d;
  const float dg_b = 2.f * s.d * s.g * Dz_b;
  d_b += dg_b * s.g;
  const float g_b = dg_b * s.d;
  float ph_b = 0.5f * g_b * s.ish;
  float sh_b = -s.ish * (g_b * s.g + 2.f * gp_b * s.gp);
  // gp = (sin x - x cos x) / (2 sh^2), x = ph / 2: d/dph (sin x - x cos x) = (ph / 4) sh
  ph_b += 0.125f * gp_b * s.ph * s.ish;
  // dphi = -RC / Q, Q = A ch + zp^2 / ph, A = d^2 / (8 sh^3)
  RC_b += dphi_b * s.dphi * s.iRC;
  const float Q_b = -dphi_b * s.dphi * s.iQ;
  const float QA = Q_b * s.A2, ch_b = 0.5f * s.d * QA;
  d_b += QA * s.ch;
  sh_b -= 3.f * ch_b * s.ch * s.ish;
  const float zi = s.zp * s.iph;
  float zp_b = 2.f * Q_b * zi;
  ph_b -= Q_b * zi * zi;
  // th = atan2(Rct, zp), RC = |(Rct, zp)|
  const float tr = th_b * s.iRC * s.iRC, cr = RC_b * s.iRC;
  Rct_b = tr * s.zp + cr * Rct;
  zp_b += cr * s.zp - tr * Rct;
  // zp = z / ph
  z_b += zp_b * s.iph;
  ph_b -= zp_b * zi;
  // sh = sin(ph / 2), ch = cos(ph / 2) on both branches (ch carries the sign)
  phi_b = ph_b + 0.5f * (sh_b * s.ch - ch_b * s.sh);
}

struct TripBar {                   // adjoints of a triplet fit's outputs
  float alpha, a0p, beta, b0p, s2, Rref, kappa, w;
};

// Reverse sweep of fit_triplet for hits a -> b -> c: adds the adjoints of the nine
// coordinates.  The two arc angles and the small offset b0p come from the forward
// fit (its only transcendental functions); everything else is recomputed from the
// coordinates.  w is the forward's weight 1 / sigma_kappa^2.
__device__ __forceinline__ void fit_triplet_bwd(const float* a, const float* b, const float* c, const TFitF& f, float w,
                                                const TripBar& o, float* ga, float* gb, float* gc) {
  const float ux = a[0] - b[0], uy = a[1] - b[1], vx = c[0] - b[0], vy = c[1] - b[1];
  const float wx = c[0] - a[0], wy = c[1] - a[1];
  const float cross = ux * vy - uy * vx, acr = fabsf(cross);
  const float d01 = sqrtf(ux * ux + uy * uy), d12 = sqrtf(vx * vx + vy * vy), d20 = sqrtf(wx * wx + wy * wy);
  const float id01 = 1.f / d01, id12 = 1.f / d12, id20 = 1.f / d20;
  const float i2c = 0.5f / cross;
  const float rtc = d01 * d12 * d20 * i2c;
  const float Rct = fabsf(rtc);
  const float dotc = wx * vx + wy * vy, dota = -(ux * wx + uy * wy);
  const float il0 = id20 * id12, il1 = id01 * id20;
  const SegB s0 = segment_values(d01, b[2] - a[2], Rct, acr * il0, dotc * il0, f.ph0);
  const SegB s1 = segment_values(d12, c[2] - b[2], Rct, acr * il1, dota * il1, f.ph1);
  const float dR = s0.RC - s1.RC;
  const float alpha = 0.5f * (s0.dphi + s1.dphi);
  const float a0p = 0.5f * s1.dphi * dR;
  const float beta = s1.dth - s0.dth;
  const float b0p = f.b0p;
  const float iRR = s0.iRC * s1.iRC;
  const float s2 = 0.5f * (1.f - (s0.zp * s1.zp - Rct * Rct) * iRR);
  const float sin2m = Rct * (s0.zp + s1.zp) * iRR;  // sin(theta0 + theta1) = d s2 / d m, m the mean angle
  const float den = alpha * alpha * s2 + beta * beta;
  const float iden = 1.f / den;
  const float u = -(alpha * a0p * s2 + beta * b0p) * iden;
  const float iRs = fabsf(f.kappa);
  // kappa = eps / Rs, w = kB^2 Rs^6 den / hl^2
  const float Rs_b = iRs * (6.f * o.w * w - o.kappa * f.kappa);
  const float Rref_b = o.Rref + Rs_b;  // Rs = R_C0 + u
  const float N_b = -Rs_b * iden;      // u = -N / den
  const float den_b = iden * (o.w * w - Rs_b * u);
  const float alpha_b = o.alpha + N_b * a0p * s2 + den_b * 2.f * alpha * s2;
  const float a0p_b = o.a0p + N_b * alpha * s2;
  const float s2_b = o.s2 + N_b * alpha * a0p + den_b * alpha * alpha;
  const float beta_b = o.beta + N_b * b0p + den_b * 2.f * beta;
  const float b0p_b = o.b0p + N_b * beta;
  const float m_b = s2_b * sin2m;
  const float dR_b = b0p_b * s1.dth + 0.5f * a0p_b * s1.dphi;
  float d01_b, z01_b, Rct0_b, d12_b, z12_b, Rct1_b, phi0_b, phi1_b;
  segment_bwd(s0, Rct, Rref_b + dR_b, 0.5f * m_b - b0p_b, 0.5f * alpha_b, -beta_b, d01_b, z01_b, Rct0_b, phi0_b);
  segment_bwd(s1, Rct, -dR_b, 0.5f * m_b + b0p_b, 0.5f * a0p_b * dR + 0.5f * alpha_b, b0p_b * dR + beta_b, d12_b, z12_b,
              Rct1_b, phi1_b);
  // R_t = |rtc|, rtc = d01 d12 d20 / (2 cross)
  const float rr = (Rct0_b + Rct1_b) * Rct;
  const float e01 = (d01_b + rr * id01) * id01, e12 = (d12_b + rr * id12) * id12, e20 = rr * id20 * id20;
  // arc angles (inscribed-angle theorem): Phi_01 = 2 atan2(|cross|, dotc) at c, Phi_12 =
  // 2 atan2(|cross|, dota) at a, where cross^2 + dot^2 is the squared product of the lengths
  const float q0 = 2.f * phi0_b * il0 * il0, q1 = 2.f * phi1_b * il1 * il1;
  const float acr_b = q0 * dotc + q1 * dota;
  const float cross_b = (cross > 0.f ? acr_b : -acr_b) - 2.f * rr * i2c;
  const float dotc_b = -q0 * acr, dota_b = -q1 * acr;
  // cross = u x v, dotc = w . v, dota = -u . w; u = a - b, v = c - b, w = c - a
  const float ux_b = e01 * ux + cross_b * vy - dota_b * wx, uy_b = e01 * uy - cross_b * vx - dota_b * wy;
  const float vx_b = e12 * vx - cross_b * uy + dotc_b * wx, vy_b = e12 * vy + cross_b * ux + dotc_b * wy;
  const float wx_b = e20 * wx + dotc_b * vx - dota_b * ux, wy_b = e20 * wy + dotc_b * vy - dota_b * uy;
  ga[0] += ux_b - wx_b;
  ga[1] += uy_b - wy_b;
  ga[2] -= z01_b;
  gb[0] -= ux_b + vx_b;
  gb[1] -= uy_b + vy_b;
  gb[2] += z01_b - z12_b;
  gc[0] += vx_b + wx_b;
  gc[1] += vy_b + wy_b;
  gc[2] += z12_b;
}

struct GradParams {
  const int32_t* hits;
  const int64_t* off;              // off[n_frames] = number of hits (bound of the indices)
  int64_t n_frames;
  const int4* cand;
  int64_t n_cand;
  const float* params;             // 25
  const float4* col_lut;
  const float* row_lut;
  double* partial;                 // [NG][gridDim.x]
  float* chi2_each;                // or nullptr
  float* kappa_each;               // or nullptr: the weighted mean curvature of each fit
};

template <bool GRAD>
__global__ void __launch_bounds__(GT, GRAD ? 4 : 8)
    k_fit_grad(const __grid_constant__ DevCfg C, const __grid_constant__ GradParams G) {
  __shared__ AlignSm A;
  __shared__ float2 sums[GRAD ? NS : 1][GT];  // the threads' running sums
  __shared__ double wsum[GT / 32];
  __shared__ unsigned wvalid[GT / 32];
  pdl_trigger();
  if (threadIdx.x < 4) {
    const int L = threadIdx.x;
    float w[3] = {G.params[6 * L + 3], G.params[6 * L + 4], G.params[6 * L + 5]};
    rotation(w, A.R[L]);
    for (int k = 0; k < 3; ++k) A.d[L][k] = G.params[6 * L + k];
  }
  if (threadIdx.x == 0) A.scale = G.params[24];
  __syncthreads();
  const int64_t n_hits = G.off[G.n_frames];
  const float kB = C.kB * A.scale;
  // chi2; per layer the gradient and its moment; chi2 of the candidates in the gradient
#pragma unroll
  for (int k = 0; k < (GRAD ? NS : 0); ++k) sums[k][threadIdx.x] = make_float2(0.f, 0.f);
  const auto add = [&](int k, float v) {
    float2 s = sums[k][threadIdx.x];
    add_to(s, v);
    sums[k][threadIdx.x] = s;
  };
  float2 csum = make_float2(0.f, 0.f);
  unsigned valid = 0;
  for (int64_t i = blockIdx.x * (int64_t)GT + threadIdx.x; i < G.n_cand; i += (int64_t)gridDim.x * GT) {
    const int4 q = __ldg(G.cand + i);
    const int qi[4] = {q.x, q.y, q.z, q.w};
    uint32_t ad[4];
    bool ok = true;
#pragma unroll
    for (int L = 0; L < 4; ++L) {
      const bool in = qi[L] >= 0 && qi[L] < n_hits;
      ok = ok && in;
      ad[L] = in ? (uint32_t)__ldg(G.hits + qi[L]) : 0u;
    }
    float P[4][3];                 // R X + d
#pragma unroll
    for (int L = 0; L < 4; ++L) {
      // the layer is known, so its constants are; an address of another layer is refused
      const int lad = (ad[L] >> 21) & 31, col = (ad[L] >> 13) & 255, row = ad[L] & 8191;
      const bool good = (ad[L] >> 26) == (uint32_t)L && lad < C.nlad[L] && col < C.ncol[L] && row < C.nrow[L];
      ok = ok && good;
      float X[3] = {0.f, 0.f, 0.f};
      if (good) {
        const float4 cl = __ldg(G.col_lut + C.col_off[L] + lad * C.ncol[L] + col);
        X[0] = cl.x;
        X[1] = cl.y;
        X[2] = __ldg(G.row_lut + C.row_off[L] + row);
      }
      const float* R = A.R[L];
#pragma unroll
      for (int r = 0; r < 3; ++r) P[L][r] = R[3 * r] * X[0] + R[3 * r + 1] * X[1] + R[3 * r + 2] * X[2] + A.d[L][r];
    }
    float chi2 = __int_as_float(0x7fc00000);  // NaN unless the fit succeeds
    float kb_out = __int_as_float(0x7fc00000);
    if (ok) {
      const TFitF f1 = fit_triplet(P[0][0], P[0][1], P[0][2], P[1][0], P[1][1], P[1][2], P[2][0], P[2][1], P[2][2],
                                   C.hl[1], kB);
      const TFitF f2 = fit_triplet(P[1][0], P[1][1], P[1][2], P[2][0], P[2][1], P[2][2], P[3][0], P[3][1], P[3][2],
                                   C.hl[2], kB);
      ok = f1.valid && f2.valid;
      float kb = 0.f, w1 = 0.f, w2 = 0.f;
      if (ok) {
        w1 = 1.f / (f1.skappa * f1.skappa);
        w2 = 1.f / (f2.skappa * f2.skappa);
        kb = (f1.kappa * w1 + f2.kappa * w2) / (w1 + w2);
        ok = kb != 0.f && isfinite(kb);
      }
      if (ok) {
        kb_out = kb;
        const float Rb = 1.f / fabsf(kb);
        const float pb = kB * Rb;
        chi2 = kink_chi2(f1, Rb, pb * C.ihl[1]) + kink_chi2(f2, Rb, pb * C.ihl[2]);
        ok = isfinite(chi2);
        if (GRAD && ok) {
          // chi2 = sum_t (A_t^2 s2_t + B_t^2) q_t, A = alpha u + a0p, B = beta u + b0p,
          // u = Rb - Rref, q = (kB Rb / hl)^2
          const TFitF* ft[2] = {&f1, &f2};
          TripBar tb[2];
          float Rb_b = 0.f;
          const float iRb = fabsf(kb);
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const TFitF& f = *ft[t];
            const float u = Rb - f.Rref;
            const float Aq = f.alpha * u + f.a0p, Bq = f.beta * u + f.b0p;
            const float kq = pb * (t == 0 ? C.ihl[1] : C.ihl[2]);
            const float qt = kq * kq;
            tb[t].a0p = 2.f * Aq * f.s2 * qt;
            tb[t].alpha = tb[t].a0p * u;
            tb[t].b0p = 2.f * Bq * qt;
            tb[t].beta = tb[t].b0p * u;
            tb[t].s2 = Aq * Aq * qt;
            const float lin = tb[t].a0p * f.alpha + tb[t].b0p * f.beta;
            tb[t].Rref = -lin;
            Rb_b += lin + (tb[t].s2 * f.s2 + Bq * Bq * qt) * 2.f * iRb;
          }
          // Rb = 1 / |kb|, kb = (k1 w1 + k2 w2) / (w1 + w2)
          const float kb_b = -Rb_b * Rb * Rb * (kb > 0.f ? 1.f : -1.f) / (w1 + w2);
          tb[0].kappa = kb_b * w1;
          tb[1].kappa = kb_b * w2;
          tb[0].w = kb_b * (f1.kappa - kb);
          tb[1].w = kb_b * (f2.kappa - kb);
          float g[4][3] = {};
          fit_triplet_bwd(P[0], P[1], P[2], f1, w1, tb[0], g[0], g[1], g[2]);
          fit_triplet_bwd(P[1], P[2], P[3], f2, w2, tb[1], g[1], g[2], g[3]);
          // validity and the chi2 sum are the forward's; a gradient that is not finite
          // (coincident hits) is left out of the gradient only
          bool fin = true;
#pragma unroll
          for (int L = 0; L < 4; ++L)
#pragma unroll
            for (int r = 0; r < 3; ++r) fin = fin && isfinite(g[L][r]);
          if (fin) {
            // P = R(w) X + d: dP/dd = I; dP/dw_k is the cross product of the rotation's axis
            // k with R X, so the moment (R X) x g is summed and projected on the three axes
            // once at the end
#pragma unroll
            for (int L = 0; L < 4; ++L) {
              const float qx = P[L][0] - A.d[L][0], qy = P[L][1] - A.d[L][1], qz = P[L][2] - A.d[L][2];
              add(1 + 6 * L, g[L][0]);
              add(2 + 6 * L, g[L][1]);
              add(3 + 6 * L, g[L][2]);
              add(4 + 6 * L, qy * g[L][2] - qz * g[L][1]);
              add(5 + 6 * L, qz * g[L][0] - qx * g[L][2]);
              add(6 + 6 * L, qx * g[L][1] - qy * g[L][0]);
            }
            add(25, chi2);
          }
        }
      }
    }
    if (ok) {
      add_to(csum, chi2);
      ++valid;
    }
    if (G.chi2_each) G.chi2_each[i] = ok ? chi2 : __int_as_float(0x7fc00000);
    if (G.kappa_each) G.kappa_each[i] = ok ? kb_out : __int_as_float(0x7fc00000);
  }
  // block sums in FP64, fixed order
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  double v = 0.0;
  if (GRAD) {
    sums[0][threadIdx.x] = csum;
    __syncthreads();
    // four threads per output, each adding 32 of the sums (8 times fewer FP64 additions, which
    // are slow here, than a shuffle tree per output), from its own lane on: no bank conflicts
    const int k = threadIdx.x >> 2, part = threadIdx.x & 3;
    float e = 0.f;
    if (k < NS) {
#pragma unroll 8
      for (int j = 0; j < 32; ++j) {
        const float2 q = sums[k][32 * part + ((j + lane) & 31)];
        v += (double)q.x;
        e += error_of(q);
      }
    }
    v += (double)e;
    v += __shfl_xor_sync(FULL, v, 1);
    v += __shfl_xor_sync(FULL, v, 2);
    if (k < NS && part == 0) G.partial[(int64_t)k * gridDim.x + blockIdx.x] = v;
  } else {
    v = (double)csum.x + (double)error_of(csum);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if (lane == 0) wsum[wp] = v;
  }
  valid = __reduce_add_sync(FULL, valid);
  if (lane == 0) wvalid[wp] = valid;
  __syncthreads();
  if (threadIdx.x == 32) {
    unsigned n = 0;
    for (int k = 0; k < GT / 32; ++k) n += wvalid[k];
    G.partial[(int64_t)NS * gridDim.x + blockIdx.x] = (double)n;
  }
  if (!GRAD && threadIdx.x == 0) {
    v = 0.0;
    for (int k = 0; k < GT / 32; ++k) v += wsum[k];
    G.partial[blockIdx.x] = v;
  }
}

// Sum of the block partials: a warp per output, its lanes over the blocks, in a fixed
// order; then the rotations' components from the moments.
__global__ void __launch_bounds__(32 * NG)
    k_fit_reduce(const double* partial, int nblocks, const float* __restrict__ params,
                 unsigned long long* n_valid, float* chi2_sum, float* grad) {
  __shared__ double sum[NG];
  // without the gradient two warps: the sum and the count
  const int k = grad ? threadIdx.x >> 5 : (threadIdx.x >> 5) * NS, lane = threadIdx.x & 31;
  pdl_wait();
  double v = 0.0;
#pragma unroll 16
  for (int b = lane; b < nblocks; b += 32) v += __ldcg(partial + (int64_t)k * nblocks + b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  if (lane == 0) sum[k] = v;
  __syncthreads();
  const int t = threadIdx.x;
  if (t == 31) *n_valid = (unsigned long long)sum[NS];
  if (t == 0 && chi2_sum) *chi2_sum = (float)sum[0];
  if (!grad) return;
  // (no candidate is valid at a scale of 0, and the gradient of the empty sum is 0)
  if (t == 32) grad[24] = sum[25] != 0.0 ? (float)(2.0 * sum[25] / (double)params[24]) : 0.f;
  if (t >= 64 && t < 76) {
    const int L = (t - 64) / 3, r = (t - 64) % 3;
    grad[6 * L + r] = (float)sum[1 + 6 * L + r];
  }
  if (t >= 96 && t < 108) {
    // R = Rz Ry Rx: the axes of d/dwx, d/dwy, d/dwz are Rz Ry ex, Rz ey and ez
    const int L = (t - 96) / 3, r = (t - 96) % 3;
    float sy, cy, sz, cz;
    sincosf(params[6 * L + 4], &sy, &cy);
    sincosf(params[6 * L + 5], &sz, &cz);
    const double mx = sum[4 + 6 * L], my = sum[5 + 6 * L], mz = sum[6 + 6 * L];
    const double v = r == 0 ? (double)(cz * cy) * mx + (double)(sz * cy) * my - (double)sy * mz
                   : r == 1 ? (double)cz * my - (double)sz * mx
                            : mz;
    grad[6 * L + 3 + r] = (float)v;
  }
}

}  // namespace

// Resident blocks per SM of the gradient kernel (grad) or of the forward-only one.
int fit_grad_blocks_per_sm(bool grad) {
  int n = 0;
  const cudaError_t e = grad ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_fit_grad<true>, GT, 0)
                             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_fit_grad<false>, GT, 0);
  return e == cudaSuccess && n > 0 ? n : 1;
}

// One wave of resident blocks at most: each block ends with FP64 sums.
int fit_grad_blocks(int resident, int64_t n_cand) {
  const int64_t nb = (n_cand + GT - 1) / GT;
  return nb < 1 ? 1 : (nb > resident ? resident : (int)nb);
}

int fit_grad_partial_size() { return NG; }

cudaError_t launch_fit_grad(const DevCfg& c, const int32_t* hits, const int64_t* off, int64_t n_frames,
                            const int32_t* cand, int64_t n_cand, const float* params, const float4* col_lut,
                            const float* row_lut, double* partial, int nblocks, unsigned long long* n_valid,
                            float* chi2_each, float* kappa_each, float* chi2_sum, float* grad, cudaStream_t s) {
  GradParams g{};
  g.hits = hits;
  g.off = off;
  g.n_frames = n_frames;
  g.cand = reinterpret_cast<const int4*>(cand);
  g.n_cand = n_cand;
  g.params = params;
  g.col_lut = col_lut;
  g.row_lut = row_lut;
  g.partial = partial;
  g.chi2_each = chi2_each;
  g.kappa_each = kappa_each;
  if (grad) k_fit_grad<true><<<nblocks, GT, 0, s>>>(c, g);
  else k_fit_grad<false><<<nblocks, GT, 0, s>>>(c, g);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_kernel(true, k_fit_reduce, 1, grad ? 32 * NG : 64, 0, s, (const double*)partial, nblocks, params, n_valid, chi2_sum, grad);
}

}  // namespace m3e
