// The convective term of Eq. convdg (Rusanov space-time DG, Sec. 2.5) for 1 <= p <= 4, in binary32-pair
// arithmetic (pair.cuh):
//   Ups^c_i = - int_{T_i x slab} grad(phi~_k) . v_c v + int_{dT_i x slab} phi~_k F^RS_c . n_i
//
// Two kernels.  k_conv_face, once per face: the traces of both tets, the Rusanov flux at the face's quadrature
// points and its moments with the P_p basis of the triangle.  k_conv_tet, once per tet: the volume term, and
// the four faces' moments taken to the tet's basis.  What the arithmetic is spent on, per tet at p = p_t = 4
// in thousands of pair multiply-adds (a kernel per tet that evaluates every trace and flux from both sides and
// tests 9 products against grad(phi) at the cubic rule's 343 points takes 1,030):
//  * the volume integrand is a polynomial (degree 3p - 1 in space, 3p_t in time), so the smallest Gauss rule
//    that is exact for it gives the same integral: 216 points instead of 343 (the face integrand is not
//    polynomial and keeps its rule);
//  * int F_cd d_d phi_k: d_e phi_k lies in P_{p-1}, so the 6 products v_c v_d (symmetric) are tested against
//    the 20 functions of P_{p-1} and the exact derivative matrices D_e[k][l] = int phi_l d_e phi_k and the
//    Jacobian are applied to the moments: 130 + 31 instead of 540;
//  * a trace lies in P_p of the triangle (15 functions): restricted there once, evaluated at the 49 points
//    with 15 terms instead of 35, once per face for both tets, and the flux tested against 15 functions.
// In sum 560.  Bound: issue and latency at 25 to 30 % occupancy (the sums of a point fill the registers).
// Measured, one kernel per tet -> these two: 13,182 tets, p = 3, p_t = 1, 4.19 -> 0.70 ms (faces 0.38, tets 0.33); 10,368
// tets, p = p_t = 4, 10.0 -> 3.7 ms (1.3 and 2.4).  The face kernel spent 70 % of the binary64 pipe on splitting the
// velocities and on the square roots (0.51 ms): both are done without it now (pair_split_int, pair_sqrt).  Threads
// own quadrature points for the evaluation (all columns of a point in registers, the basis table
// coalesced over the points), and outputs for the tests; all pair
// products run two at a time in packed binary32 operations.
#include <cmath>
#include <vector>

#include "pair.cuh"
#include "solver.h"

namespace stdg {
namespace {

// n sums of products of pairs, two at a time: s + c, with FINE s - c - d (pair_fma2)
template <int n, bool FINE = false>
struct ConvSum {
  static constexpr int H = (n + 1) / 2;
  float2 s[H], c[H], d[FINE ? H : 1];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int m = 0; m < H; ++m) s[m] = c[m] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int m = 0; m < (FINE ? H : 1); ++m) d[m] = make_float2(0.0f, 0.0f);
  }
  // += a x[m * stride]
  __device__ __forceinline__ void axpy(float2 a, const float2* x, int stride = 1) {
    const float2 ah2 = make_float2(a.x, a.x), nah2 = make_float2(-a.x, -a.x), al2 = make_float2(a.y, a.y);
#pragma unroll
    for (int m = 0; m < H; ++m) {
      const float2 x0 = x[2 * m * stride], x1 = 2 * m + 1 < n ? x[(2 * m + 1) * stride] : make_float2(0.0f, 0.0f);
      const float2 xh = make_float2(x0.x, x1.x), xl = make_float2(x0.y, x1.y);
      if constexpr (FINE) pair_fma2(ah2, nah2, al2, xh, xl, s[m], c[m], d[m]);
      else pair_fma2(ah2, nah2, al2, xh, xl, s[m], c[m]);
    }
  }
  // += the sums t
  __device__ __forceinline__ void add(const ConvSum& t) {
    static_assert(!FINE, "fine sums are added up term by term");
#pragma unroll
    for (int m = 0; m < H; ++m) {
      float2 s2, e;
      df_two_diff2(s[m], make_float2(-t.s[m].x, -t.s[m].y), s2, e);
      s[m] = s2;
      c[m] = __fadd2_rn(__fadd2_rn(c[m], t.c[m]), e);
    }
  }
  __device__ __forceinline__ float2 get(int m) const {
    const float sm = (m & 1) ? s[m >> 1].y : s[m >> 1].x, cm = (m & 1) ? c[m >> 1].y : c[m >> 1].x;
    float2 v = pair_norm(sm, FINE ? -cm : cm);
    if constexpr (FINE) v.y -= (m & 1) ? d[m >> 1].y : d[m >> 1].x;
    return v;
  }
  __device__ __forceinline__ double value(int m) const {
    const float2 v = get(m);
    return pair_value(v.x, v.y);
  }
};
// S[m] = Sum_k tab[k * stride] V[m * N + k] for the NA coefficient rows of V, as normalised pairs
template <int N, int NA, bool FINE = false>
__device__ __forceinline__ void conv_contract(const float2* __restrict__ tab, int stride, const float2* V,
                                              float2 (&S)[NA]) {
  ConvSum<NA, FINE> sum;
  sum.zero();
#pragma unroll 2
  for (int k = 0; k < N; ++k) sum.axpy(__ldg(tab + (size_t)k * stride), V + k, N);
#pragma unroll
  for (int m = 0; m < NA; ++m) S[m] = sum.get(m);
}

template <int P, int NG>
struct ConvDim {
  static constexpr int N = (P + 1) * (P + 2) * (P + 3) / 6, N1 = P * (P + 1) * (P + 2) / 6, M = (P + 1) * (P + 2) / 2;
  static constexpr int NV1 = (3 * P + 1) / 2, NV = NV1 * NV1 * NV1;    // volume rule: degree 3p - 1
  static constexpr int NF1 = (3 * P + 3) / 2, NF = NF1 * NF1;          // face rule: that of all non-polynomial data
  static constexpr int NTV = (3 * (NG - 1) + 2) / 2, NTF = (3 * (NG - 1) + 3) / 2;   // time rules
  static constexpr int NA = 3 * NG, Nst = N * NG;
  // Sums of few terms add more rounding than the shorter sums save: fine sums for the traces, moments and outputs at
  // p = 1 and for the moments at p = 2.  Relative rms error against binary64 at p_t = 0, a kernel per tet that sums
  // over the points -> plain sums here -> as built: p = 1 5.1e-15 -> 6.6e-15 -> 4.5e-15, p = 2 1.0e-14 -> 9.3e-15 ->
  // 7.6e-15, p = 3 2.0e-14 -> 1.5e-14 -> 1.4e-14, p = 4 2.4e-14 -> 2.1e-14 -> 2.0e-14; with random coefficients of
  // order 1, plain sums were also worse at p = 2 (8.0e-15 -> 8.2e-15 -> 6.5e-15).  Cost at p_t = 0: 82,944 tets,
  // p = 1, 206 -> 228 us; 34,992 tets, p = 2, 256 -> 275 us; at p = 3 and 4 below 1 %.
  static constexpr bool FINE = P == 1, FINE_M = P <= 2;
  // faces per CTA of 256 threads: all points of a face side by side
  static constexpr int kFT = 256, FB = kFT / NF;
  static constexpr int face_in = FB * 2 * NA * N, face_g = FB * NF * NA;
  static constexpr size_t face_smem = (size_t)((face_in > face_g ? face_in : face_g) + FB * 2 * NA * M) * sizeof(float2);
  // tets per CTA
  static constexpr int kTT = P == 4 ? 224 : P == 3 ? 128 : 256, TB = kTT / NV;
  static constexpr int QS = kTT / (TB * N1 * NG) < NV ? kTT / (TB * N1 * NG) : NV;   // shares of the points in the test
  static constexpr int tet_v = TB * NA * N, tet_g = TB * NV * 6 * NG, tet_h = QS * TB * 6 * NG * N1;
  static constexpr int tet_u = TB * 9 * NG * N1, tet_f = TB * 4 * NA * M;
  static constexpr size_t tet_smem = (size_t)(tet_v + tet_h + (tet_g > tet_u + tet_f ? tet_g : tet_u + tet_f)) * sizeof(float2);
  static_assert(TB * N1 * NG <= kTT, "one thread per tested function and time column");
};

// tables (all as pairs) in one array
struct ConvTab {
  const float2 *vphi, *vphi1, *vw, *vtg, *vtw;    // volume: [N][NV], [NV][N1], [NV], [NTV][NG], [NTV]
  const float2* D;                                // [3][N1][N]: int phi_l d_e phi_k
  const float2 *Rt, *Rk;                          // restriction to the triangle [64][N][M], and back [64][M][N]
  const float2 *chiT, *chi, *fw, *ftg, *ftw;      // triangle basis [M][NF], [NF][M]; [NF], [NTF][NG], [NTF]
};
struct ConvIn {
  int ne, nf;
  const int *left, *right, *code_l, *code_r, *t2f, *t2code, *bidx;
  const double *detJ, *Jinv, *normal, *area, *fvx, *tri_st, *ttau;
  FieldArg fld;
  double t0, dt;
  int nq, bnpt;                                   // callback data: (nq + NF) NTF points per boundary face, face points last
  const double* vbar;                             // [3][ne][Nst]
  float2* hf;                                     // [nf][3][NG][M]: moments of the flux along n_j
  double* ups;
};

template <int P, int NG>
__global__ void __launch_bounds__(256, 2) k_conv_face(const __grid_constant__ ConvIn a, const __grid_constant__ ConvTab t) {
  using C = ConvDim<P, NG>;
  constexpr int N = C::N, M = C::M, NA = C::NA, NF = C::NF, FB = C::FB, Nst = C::Nst;
  extern __shared__ __align__(16) float2 cvs[];
  float2* V = cvs;                                // [face][side][c][b][k]
  float2* G = cvs;                                // [face][point][c][a], once V is used up
  float2* T = cvs + (C::face_in > C::face_g ? C::face_in : C::face_g);   // [face][side][c][b][m]
  __shared__ float2 tg[C::NTF * NG], tw[C::NTF];
  const int th = threadIdx.x, j0 = blockIdx.x * FB;
  for (int o = th; o < C::NTF * NG; o += C::kFT) tg[o] = t.ftg[o];
  if (th < C::NTF) tw[th] = t.ftw[th];
  for (int o = th; o < FB * 2 * NA * N; o += C::kFT) {
    const int fs = o / (NA * N), rem = o - fs * NA * N, j = j0 + (fs >> 1), c = rem / Nst, r = rem - c * Nst;
    const int tet = j < a.nf ? ((fs & 1) ? a.right[j] : a.left[j]) : -1;
    V[o] = tet >= 0 ? pair_split_int(a.vbar[((size_t)c * a.ne + tet) * Nst + r]) : make_float2(0.0f, 0.0f);
  }
  __syncthreads();
  // traces in the triangle's basis: thread (face, side, m)
  for (int o = th; o < FB * 2 * M; o += C::kFT) {
    const int fs = o / M, m = o - fs * M, j = j0 + (fs >> 1);
    if (j >= a.nf) break;
    const int code = (fs & 1) ? a.code_r[j] : a.code_l[j];
    if (code < 0) continue;                       // no tet at this side of a boundary face
    float2 S[NA];
    conv_contract<N, NA, C::FINE>(t.Rt + (size_t)code * N * M + m, M, V + fs * NA * N, S);
#pragma unroll
    for (int q = 0; q < NA; ++q) T[(fs * NA + q) * M + m] = S[q];
  }
  __syncthreads();
  // flux: thread (face, point)
  const int f = th / NF, q = th - f * NF, j = j0 + f;
  if (f < FB && j < a.nf) {
    const bool bd = a.right[j] < 0;
    float2 Sm[NA], Sp[NA];
    conv_contract<M, NA>(t.chiT + q, NF, T + (2 * f) * NA * M, Sm);
    double x[3] = {0.0, 0.0, 0.0};
    if (!bd) {
      conv_contract<M, NA>(t.chiT + q, NF, T + (2 * f + 1) * NA * M, Sp);
    } else {
      const double* fv = a.fvx + 9 * (size_t)j;
      const double s0 = a.tri_st[2 * q], t0 = a.tri_st[2 * q + 1];
      for (int d = 0; d < 3; ++d) x[d] = fv[d] + s0 * (fv[3 + d] - fv[d]) + t0 * (fv[6 + d] - fv[d]);
    }
    ConvSum<NG> gs[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) gs[c].zero();
    const float2 wq = pair_mul(pair_split(a.dt * 2.0 * a.area[j]), t.fw[q]);
    const float2 nP[3] = {pair_split_int(a.normal[3 * (size_t)j]), pair_split_int(a.normal[3 * (size_t)j + 1]),
                          pair_split_int(a.normal[3 * (size_t)j + 2])};
#pragma unroll 1
    for (int ti = 0; ti < C::NTF; ++ti) {
      const float2* g = tg + ti * NG;
      float2 vm[3], vp[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float ss = 0.0f, cc = 0.0f;
#pragma unroll
        for (int b = 0; b < NG; ++b) pair_fma(g[b], Sm[c * NG + b], ss, cc);
        vm[c] = pair_norm(ss, cc);
      }
      if (!bd) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float ss = 0.0f, cc = 0.0f;
#pragma unroll
          for (int b = 0; b < NG; ++b) pair_fma(g[b], Sp[c * NG + b], ss, cc);
          vp[c] = pair_norm(ss, cc);
        }
      } else {
        double vb[3];
        eval_field(a.fld, x, a.t0 + a.ttau[ti] * a.dt,
                   (int64_t)a.bidx[j] * a.bnpt + (int64_t)a.nq * C::NTF + (int64_t)q * C::NTF + ti, a.ttau[ti], vb);
#pragma unroll
        for (int c = 0; c < 3; ++c) vp[c] = pair_split_int(vb[c]);
      }
      // Rusanov flux, s_max = 2 max(|v+|, |v-|) pointwise
      float s1 = 0.0f, c1 = 0.0f, s2 = 0.0f, c2 = 0.0f, s3 = 0.0f, c3 = 0.0f, s4 = 0.0f, c4 = 0.0f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        pair_fma(vm[c], nP[c], s1, c1);
        pair_fma(vp[c], nP[c], s2, c2);
        pair_fma(vm[c], vm[c], s3, c3);
        pair_fma(vp[c], vp[c], s4, c4);
      }
      const float2 unm = pair_norm(s1, c1), unp = pair_norm(s2, c2);
      // s_max / 2 is the root of the larger square
      const float2 q3 = pair_norm(s3, c3), q4 = pair_norm(s4, c4);
      const float2 W = pair_mul(wq, tw[ti]);
      const float2 hs = pair_mul(W, pair_sqrt(q3.x > q4.x || (q3.x == q4.x && q3.y > q4.y) ? q3 : q4));
      const float2 Wh = make_float2(0.5f * W.x, 0.5f * W.y);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        // h = W (0.5 (v+_c un+ + v-_c un-) - 0.5 s_max (v+_c - v-_c))
        const float2 cen = pair_mul(Wh, pair_add(pair_mul(vp[c], unp), pair_mul(vm[c], unm)));
        const float2 h = pair_add(cen, pair_neg(pair_mul(hs, pair_add(vp[c], pair_neg(vm[c])))));
        gs[c].axpy(h, g);
      }
    }
    float2* Gu = G + (f * NF + q) * NA;           // V is used up (every thread passed the barrier after T)
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int b = 0; b < NG; ++b) Gu[c * NG + b] = gs[c].get(b);
  }
  __syncthreads();
  // moments: thread (face, c, m)
  for (int o = th; o < FB * 3 * M; o += C::kFT) {
    const int ff = o / (3 * M), rem = o - ff * 3 * M, c = rem / M, m = rem - c * M;
    if (j0 + ff >= a.nf) break;
    ConvSum<NG, C::FINE_M> s;
    s.zero();
#pragma unroll 4
    for (int v = 0; v < NF; ++v) s.axpy(__ldg(t.chi + v * M + m), G + (ff * NF + v) * NA + c * NG);
    float2* out = a.hf + (((size_t)(j0 + ff) * 3 + c) * NG) * M + m;
#pragma unroll
    for (int b = 0; b < NG; ++b) out[b * M] = s.get(b);
  }
}

template <int P, int NG>
__global__ void __launch_bounds__(ConvDim<P, NG>::kTT, P == 3 ? 4 : 2) k_conv_tet(const __grid_constant__ ConvIn a,
                                                                                 const __grid_constant__ ConvTab t) {
  using C = ConvDim<P, NG>;
  constexpr int N = C::N, N1 = C::N1, M = C::M, NA = C::NA, NV = C::NV, TB = C::TB, Nst = C::Nst, NT = C::kTT, QS = C::QS;
  constexpr int R6 = 6 * NG, HL = R6 * N1;
  extern __shared__ __align__(16) float2 cvs[];
  float2* V = cvs;                                // [tet][c][b][k]
  float2* H = cvs + C::tet_v;                     // [share][tet][l][a][cd]: moments of v_c v_d
  float2* G = H + C::tet_h;                       // [tet][point][a][cd]
  float2* U = G;                                  // then [tet][c][e][l][a]: Sum_d Jinv[e][d] H_cd
  float2* F = G + C::tet_u;                       // and [tet][face][c][a][m]
  __shared__ float2 tg[C::NTV * NG], tw[C::NTV];
  const int th = threadIdx.x, i0 = blockIdx.x * TB;
  for (int o = th; o < C::NTV * NG; o += NT) tg[o] = t.vtg[o];
  if (th < C::NTV) tw[th] = t.vtw[th];
  for (int o = th; o < TB * NA * N; o += NT) {
    const int tl = o / (NA * N), rem = o - tl * NA * N, c = rem / Nst, r = rem - c * Nst, i = i0 + tl;
    V[o] = i < a.ne ? pair_split_int(a.vbar[((size_t)c * a.ne + i) * Nst + r]) : make_float2(0.0f, 0.0f);
  }
  __syncthreads();
  {                                               // v_c v_d at thread (tet, point), folded in time
    const int tl = th / NV, q = th - tl * NV, i = i0 + tl;
    if (tl < TB && i < a.ne) {
      float2 S[NA];
      conv_contract<N, NA>(t.vphi + q, NV, V + tl * NA * N, S);
      ConvSum<NG> gs[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) gs[r].zero();
      const float2 wq = pair_mul(pair_split(a.dt * a.detJ[i]), t.vw[q]);
#pragma unroll 1
      for (int ti = 0; ti < C::NTV; ++ti) {
        const float2* g = tg + ti * NG;
        const float2 W = pair_mul(wq, tw[ti]);
        float2 v[3], Wv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float ss = 0.0f, cc = 0.0f;
#pragma unroll
          for (int b = 0; b < NG; ++b) pair_fma(g[b], S[c * NG + b], ss, cc);
          v[c] = pair_norm(ss, cc);
          Wv[c] = pair_mul(W, v[c]);
        }
        // cd = 00, 01, 02, 11, 12, 22
#pragma unroll
        for (int r = 0; r < 6; ++r) {
          constexpr int rc[6] = {0, 0, 0, 1, 1, 2}, rd[6] = {0, 1, 2, 1, 2, 2};
          gs[r].axpy(pair_mul(Wv[rc[r]], v[rd[r]]), g);
        }
      }
      float2* Gu = G + (tl * NV + q) * R6;
#pragma unroll
      for (int b = 0; b < NG; ++b)
#pragma unroll
        for (int r = 0; r < 6; ++r) Gu[b * 6 + r] = gs[r].get(b);
    }
  }
  __syncthreads();
  {                                               // moments with P_{p-1}: thread (share of the points, tet, a, l)
    const int sh = th / (TB * N1 * NG), rem = th - sh * TB * N1 * NG, tl = rem / (N1 * NG), al = rem - tl * N1 * NG;
    const int b = al / N1, l = al - b * N1;
    if (sh < QS) {
      ConvSum<6> s;
      s.zero();
#pragma unroll 2
      for (int v = sh; v < NV; v += QS) s.axpy(__ldg(t.vphi1 + v * N1 + l), G + (tl * NV + v) * R6 + b * 6);
      float2* out = H + (sh * TB + tl) * HL + (l * NG + b) * 6;
#pragma unroll
      for (int r = 0; r < 6; ++r) out[r] = s.get(r);
    }
  }
  __syncthreads();                                // G is free
  for (int o = th; o < TB * HL && QS > 1; o += NT) {   // the shares' sums, in a fixed order
    float2 v = H[o];
#pragma unroll
    for (int sh = 1; sh < QS; ++sh) v = pair_add(v, H[sh * TB * HL + o]);
    H[o] = v;
  }
  for (int o = th; o < TB * 4 * NA * M; o += NT) {     // the faces' moments, along the outward normal
    const int tl = o / (4 * NA * M), rem = o - tl * 4 * NA * M, f = rem / (NA * M), i = i0 + tl;
    if (i >= a.ne) break;
    const int j = a.t2f[4 * i + f];
    const float2 v = a.hf[(size_t)j * NA * M + rem - f * NA * M];
    F[o] = a.left[j] == i ? v : pair_neg(v);
  }
  __syncthreads();
  for (int o = th; o < TB * 9 * NG * N1; o += NT) {
    const int tl = o / (9 * NG * N1), rem = o - tl * 9 * NG * N1, c = rem / (3 * NG * N1), e = rem / (NG * N1) % 3;
    const int la = rem % (NG * N1), i = i0 + tl;
    if (i >= a.ne) break;
    const float2* h = H + tl * HL + la * 6;
    float s = 0.0f, r = 0.0f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int lo = c < d ? c : d, up = c < d ? d : c;
      pair_fma(pair_split_int(a.Jinv[9 * (size_t)i + 3 * e + d]), h[lo == 0 ? up : lo + up + 1], s, r);
    }
    U[o] = pair_norm(s, r);
  }
  __syncthreads();
  // outputs: thread (tet, c, k), all time columns
  for (int o = th; o < TB * 3 * N; o += NT) {
    const int tl = o / (3 * N), rem = o - tl * 3 * N, c = rem / N, k = rem - c * N, i = i0 + tl;
    if (i >= a.ne) break;
    // plain sums: every derivative and face by itself first (the error part c of a sum grows with its length,
    // and with it the rounding of c)
    ConvSum<NG, C::FINE> s, part;
    auto& sum = C::FINE ? s : part;
    s.zero();
    const float2* u = U + (tl * 3 + c) * 3 * N1 * NG;
#pragma unroll 1
    for (int e = 0; e < 3; ++e) {
      if constexpr (!C::FINE) part.zero();
#pragma unroll 4
      for (int l = 0; l < N1; ++l) sum.axpy(pair_neg(__ldg(t.D + (e * N1 + l) * N + k)), u + (e * N1 + l) * NG);
      if constexpr (!C::FINE) s.add(part);
    }
#pragma unroll 1
    for (int f = 0; f < 4; ++f) {
      const float2* R = t.Rk + (size_t)a.t2code[4 * i + f] * M * N + k;
      const float2* h = F + ((tl * 4 + f) * 3 + c) * NG * M;
      if constexpr (!C::FINE) part.zero();
#pragma unroll 3
      for (int m = 0; m < M; ++m) sum.axpy(__ldg(R + m * N), h + m, M);
      if constexpr (!C::FINE) s.add(part);
    }
    double* out = a.ups + ((size_t)c * a.ne + i) * Nst + k;
#pragma unroll
    for (int b = 0; b < NG; ++b) out[b * N] = s.value(b);
  }
}

template <int P, int NG>
cudaError_t conv_launch(const ConvIn& a, const ConvTab& t, cudaStream_t st) {
  using C = ConvDim<P, NG>;
  cudaError_t e = cudaFuncSetAttribute(k_conv_face<P, NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::face_smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_conv_tet<P, NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::tet_smem);
  if (e != cudaSuccess) return e;
  if (a.nf > 0) k_conv_face<P, NG><<<(a.nf + C::FB - 1) / C::FB, C::kFT, C::face_smem, st>>>(a, t);
  if (a.ne > 0) k_conv_tet<P, NG><<<(a.ne + C::TB - 1) / C::TB, C::kTT, C::tet_smem, st>>>(a, t);
  return cudaGetLastError();
}

// orthonormal Dubiner basis of the reference triangle {s, t >= 0, s + t <= 1}, order "n = 0..p, i = 0..n, (i, n - i)"
void tri_basis(int p, double s, double t, double* out) {
  auto jac = [](int n, double al, double x) {     // P_n of the Jacobi weight (al, 0)
    double a = 1.0, b = 0.5 * ((al + 2.0) * x + al);
    if (n == 0) return a;
    for (int k = 2; k <= n; ++k) {
      const double q = 2.0 * k + al;
      const double c = ((q - 1) * (q * (q - 2) * x + al * al) * b - 2 * (k + al - 1) * (k - 1) * q * a) / (2 * k * (k + al) * (q - 2));
      a = b; b = c;
    }
    return b;
  };
  int m = 0;
  for (int n = 0; n <= p; ++n)
    for (int i = 0; i <= n; ++i) {
      const int jj = n - i;
      out[m++] = std::sqrt((2.0 * i + 1) * (2.0 * i + 2.0 * jj + 2)) * jac(i, 0.0, 2 * s / (1 - t) - 1) * std::pow(1 - t, i) *
                 jac(jj, 2.0 * i + 1, 2 * t - 1);
    }
}

const double kVert[4][3] = {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}};

}  // namespace

// The tables of (p, p_t) on the device, built at the first call.
static stdg_status conv_tables(stdg_solver* s, ConvTab* t) {
  const int p = s->p, pt = s->pt, N = s->N, Ng = s->Ng, N1 = p * (p + 1) * (p + 2) / 6, M = (p + 1) * (p + 2) / 2;
  // points of the rules: volume, face, and in time
  const int nv = (3 * p + 1) / 2, nf = (3 * p + 3) / 2, mv = (3 * pt + 2) / 2, mf = (3 * pt + 3) / 2;
  const size_t V = (size_t)nv * nv * nv, F = (size_t)nf * nf;
  const size_t len[13] = {N * V, V * N1, V, (size_t)mv * Ng, (size_t)mv, (size_t)3 * N1 * N, (size_t)64 * N * M,
                          (size_t)64 * M * N, M * F, F * M, F, (size_t)mf * Ng, (size_t)mf};
  size_t off[14] = {0};
  for (int k = 0; k < 13; ++k) off[k + 1] = off[k] + len[k];
  if (!s->conv_tab) {
    const Rule vr = tet_rule(nv), fr = tri_rule(nf), lr = tri_rule(p + 1), mr = tet_rule(p + 1);
    const Rule vt = line_rule(mv), ft = line_rule(mf);
    std::vector<double> h(off[13], 0.0), phi(N), dphi(3 * N), chi(M), g(Ng), dg(Ng);
    for (int q = 0; q < vr.n; ++q) {
      dubiner_eval(p, &vr.x[3 * q], phi.data(), dphi.data());
      for (int k = 0; k < N; ++k) h[off[0] + (size_t)k * vr.n + q] = phi[k];
      for (int l = 0; l < N1; ++l) h[off[1] + (size_t)q * N1 + l] = phi[l];   // the first N1 functions span P_{p-1}
      h[off[2] + q] = vr.w[q];
    }
    auto time_rule = [&](const Rule& r, size_t og, size_t ow) {
      for (int q = 0; q < r.n; ++q) {
        legendre01(pt, r.x[q], g.data(), dg.data());
        for (int b = 0; b < Ng; ++b) h[og + (size_t)q * Ng + b] = g[b];
        h[ow + q] = r.w[q];
      }
    };
    time_rule(vt, off[3], off[4]);
    time_rule(ft, off[11], off[12]);
    for (int q = 0; q < mr.n; ++q) {
      dubiner_eval(p, &mr.x[3 * q], phi.data(), dphi.data());
      for (int e = 0; e < 3; ++e)
        for (int l = 0; l < N1; ++l)
          for (int k = 0; k < N; ++k) h[off[5] + ((size_t)e * N1 + l) * N + k] += mr.w[q] * phi[l] * dphi[e * N + k];
    }
    for (int a = 0; a < 4; ++a)
      for (int b = 0; b < 4; ++b)
        for (int c = 0; c < 4; ++c) {
          if (a == b || b == c || a == c) continue;
          const size_t code = (size_t)tri_code(a, b, c);
          for (int q = 0; q < lr.n; ++q) {
            const double u = lr.x[2 * q], v = lr.x[2 * q + 1];
            double xi[3];
            for (int d = 0; d < 3; ++d) xi[d] = kVert[a][d] + u * (kVert[b][d] - kVert[a][d]) + v * (kVert[c][d] - kVert[a][d]);
            dubiner_eval(p, xi, phi.data(), dphi.data());
            tri_basis(p, u, v, chi.data());
            for (int k = 0; k < N; ++k)
              for (int m = 0; m < M; ++m) {
                h[off[6] + (code * N + k) * M + m] += lr.w[q] * chi[m] * phi[k];
                h[off[7] + (code * M + m) * N + k] += lr.w[q] * chi[m] * phi[k];
              }
          }
        }
    for (int q = 0; q < fr.n; ++q) {
      tri_basis(p, fr.x[2 * q], fr.x[2 * q + 1], chi.data());
      for (int m = 0; m < M; ++m) h[off[8] + (size_t)m * fr.n + q] = h[off[9] + (size_t)q * M + m] = chi[m];
      h[off[10] + q] = fr.w[q];
    }
    std::vector<float2> hp(off[13]);
    for (size_t k = 0; k < hp.size(); ++k) {
      const float hi = (float)h[k];
      hp[k] = make_float2(hi, (float)(h[k] - (double)hi));
    }
    float2* d = nullptr;
    const stdg_status e = dev_alloc(s, (void**)&d, hp.size() * sizeof(float2));
    if (e != STDG_OK) return e;
    if (cudaMemcpyAsync(d, hp.data(), hp.size() * sizeof(float2), cudaMemcpyHostToDevice, s->stream) != cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess) {
      set_error("convection tables: upload failed");
      return STDG_ECUDA;
    }
    s->conv_tab = d;
  }
  const float2* d = s->conv_tab;
  *t = ConvTab{d + off[0], d + off[1], d + off[2], d + off[3], d + off[4], d + off[5], d + off[6],
               d + off[7], d + off[8], d + off[9], d + off[10], d + off[11], d + off[12]};
  return STDG_OK;
}

// STDG_EUNSUPPORTED at p = 0, where the caller uses the general kernel.
stdg_status convection_modal(stdg_solver* s, const FieldArg& fld, const double* vbar, double* ups) {
  if (s->p < 1 || s->p > 4) return STDG_EUNSUPPORTED;
  ConvTab t{};
  const stdg_status e = conv_tables(s, &t);
  if (e != STDG_OK) return e;
  const int M = (s->p + 1) * (s->p + 2) / 2;
  // the faces' moments take the room of the products' input vectors (3 nf Nst words), free between products
  if ((int64_t)s->nf * 3 * s->Ng * M > s->fxws.nvec * (int64_t)s->Nst) { set_error("convection: workspace"); return STDG_EINVAL; }
  const ConvIn a{(int)s->ne, (int)s->nf, s->dm.left, s->dm.right, s->dm.code_l, s->dm.code_r, s->dm.t2f, s->dm.t2code, s->bidx,
                 s->dm.detJ, s->dm.Jinv, s->dm.normal, s->dm.area, s->dm.fvx, s->dr.tri_nl_st, s->d_ttau,
                 fld, s->t, s->dt, s->nq_nl, (s->nq_nl + s->nqf_nl) * s->nt_nl, vbar,
                 static_cast<float2*>(s->fxws.w), ups};
  cudaError_t ce = cudaErrorInvalidValue;
  switch (s->p) {
    case 1: STDG_NG_SWITCH(s->Ng, (ce = conv_launch<1, G>(a, t, s->stream))); break;
    case 2: STDG_NG_SWITCH(s->Ng, (ce = conv_launch<2, G>(a, t, s->stream))); break;
    case 3: STDG_NG_SWITCH(s->Ng, (ce = conv_launch<3, G>(a, t, s->stream))); break;
    default: STDG_NG_SWITCH(s->Ng, (ce = conv_launch<4, G>(a, t, s->stream))); break;
  }
  s->nlaunch += 1;                                 // two kernels, one counted by the caller
  if (ce != cudaSuccess) { set_error("convection launch failed: %s", cudaGetErrorString(ce)); return STDG_ECUDA; }
  return STDG_OK;
}

}  // namespace stdg
