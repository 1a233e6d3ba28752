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
// In sum 560.  Bound: issue and latency with 24 to 27 % of the warps (the sums of a point fill the registers).
// Measured, one kernel per tet -> these two: 13,182 tets, p = 3, p_t = 1, 4.19 -> 0.73 ms (faces 0.39, tets 0.34); 10,368
// tets, p = p_t = 4, 10.0 -> 3.6 ms (1.2 and 2.4).  The face kernel kept 70 % of the binary64 pipe busy with splitting
// the velocities and with the square roots (0.51 ms); without them (pair_split_int, pair_sqrt) 51 %: conversions.  Threads
// own quadrature points for the evaluation (all columns of a point in registers, the basis table
// coalesced over the points), and outputs for the tests; all pair
// products run two at a time in packed binary32 operations.
#include <algorithm>
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
  // 7.9e-15, p = 3 2.0e-14 -> 1.5e-14 -> 1.4e-14, p = 4 2.4e-14 -> 2.1e-14 -> 2.0e-14; with random coefficients of
  // order 1, plain sums were also worse at p = 2 (8.0e-15 -> 8.2e-15 -> 7.3e-15).  Cost at p_t = 0: 82,944 tets,
  // p = 1, 206 -> 218 us; 34,992 tets, p = 2, 256 -> 267 us; at p = 3 and 4 below 1 %.  (Fine sums that keep the
  // rounding of c's two parts apart: 4.0e-15 and 227 us at p = 1.)
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

// ---- the tables, in binary64 on the device from the nonlinear-degree tables of the solver and the nodes of the
// (smaller) volume rule: evaluated on the host and uploaded they were 2.4 ms of the first call at p = p_t = 4
constexpr int kVNodes = 6, kTNodes = 7;           // points of the volume and time rules, at most
struct ConvNodes {
  int nv, mv;                                     // nodes per direction, in time
  double x[3][kVNodes], w[3][kVNodes];            // Gauss-Jacobi (1 - x)^0, (1 - x)^1, (1 - x)^2
  double tg[kTNodes * kMaxNg], tw[kTNodes];       // time basis at the time nodes
  MultiIdx mi;
};
struct ConvSrc {                                  // [nq][N], [nq][3][N], [nq]; [64][nqf][N], [nqf][2], [nqf]; [nt][Ng], [nt]
  const double *tet_phi, *tet_dphi, *tet_w, *face_phi, *tri_st, *tri_w, *tg, *tw;
  int nq, nqf, nt;
};
struct ConvOff { int o[14]; };                    // where each table starts (ConvTab's order)

// P_n of the Jacobi weight (al, 0)
__device__ double conv_jacobi(int n, double al, double x) {
  double a = 1.0, b = 0.5 * ((al + 2.0) * x + al);
  if (n == 0) return a;
  for (int k = 2; k <= n; ++k) {
    const double q = 2.0 * k + al;
    const double c = ((q - 1) * (q * (q - 2) * x + al * al) * b - 2 * (k + al - 1) * (k - 1) * q * a) / (2 * k * (k + al) * (q - 2));
    a = b; b = c;
  }
  return b;
}
__device__ double conv_pow(double x, int n) {
  double v = 1.0;
  for (int k = 0; k < n; ++k) v *= x;
  return v;
}
// orthonormal Dubiner basis function k of the tetrahedron at the collapsed coordinates (u, v, w)
__device__ double conv_phi(const MultiIdx& mi, int k, double u, double v, double w) {
  const int i = mi.e[3 * k], j = mi.e[3 * k + 1], l = mi.e[3 * k + 2];
  return sqrt((2.0 * i + 1) * (2.0 * i + 2 * j + 2) * (2.0 * i + 2 * j + 2 * l + 3)) * conv_jacobi(i, 0, 2 * u - 1) *
         conv_pow(1 - v, i) * conv_jacobi(j, 2.0 * i + 1, 2 * v - 1) * conv_pow(1 - w, i + j) *
         conv_jacobi(l, 2.0 * i + 2 * j + 2, 2 * w - 1);
}
// orthonormal Dubiner basis of the reference triangle {s, t >= 0, s + t <= 1}, order "n = 0..p, i = 0..n, (i, n - i)"
__device__ double conv_chi(int m, double s, double t) {
  int n = 0;
  while ((n + 1) * (n + 2) / 2 <= m) ++n;
  const int i = m - n * (n + 1) / 2, j = n - i;
  return sqrt((2.0 * i + 1) * (2.0 * i + 2.0 * j + 2)) * conv_jacobi(i, 0, 2 * s / (1 - t) - 1) * conv_pow(1 - t, i) *
         conv_jacobi(j, 2.0 * i + 1, 2 * t - 1);
}

__global__ void __launch_bounds__(256) k_conv_tables(int N, int N1, int M, int Ng, const __grid_constant__ ConvNodes nd,
                                                     const ConvSrc a, const ConvOff off, float2* __restrict__ out) {
  __shared__ double chi[49 * 15];                 // at the face points
  const int F = a.nqf, nv = nd.nv, V = nv * nv * nv;
  for (int e = threadIdx.x; e < F * M; e += 256) chi[e] = conv_chi(e % M, a.tri_st[2 * (e / M)], a.tri_st[2 * (e / M) + 1]);
  __syncthreads();
  for (int g = blockIdx.x * 256 + threadIdx.x; g < off.o[13]; g += gridDim.x * 256) {
    int t = 0;
    while (g >= off.o[t + 1]) ++t;
    const int e = g - off.o[t];
    double v = 0.0;
    if (t <= 2) {                                 // at point q of the volume rule: phi_k, and the weight
      const int q = t == 0 ? e % V : t == 1 ? e / N1 : e, k = t == 0 ? e / V : e % N1;
      const int qa = q / (nv * nv), qb = q / nv % nv, qc = q % nv;
      v = t == 2 ? nd.w[0][qa] * nd.w[1][qb] * nd.w[2][qc] : conv_phi(nd.mi, k, nd.x[0][qa], nd.x[1][qb], nd.x[2][qc]);
    } else if (t == 3) {
      v = nd.tg[e];
    } else if (t == 4) {
      v = nd.tw[e];
    } else if (t == 5) {                          // int phi_l d_e phi_k
      const int d = e / (N1 * N), l = e / N % N1, k = e % N;
      for (int q = 0; q < a.nq; ++q) v = fma(a.tet_w[q] * a.tet_phi[(size_t)q * N + l], a.tet_dphi[((size_t)q * 3 + d) * N + k], v);
    } else if (t <= 7) {                          // int chi_m phi_k over the face with these vertices
      const int code = e / (N * M), r = e % (N * M), k = t == 6 ? r / M : r % N, m = t == 6 ? r % M : r / N;
      const int va = code >> 4, vb = code >> 2 & 3, vc = code & 3;
      if (va != vb && vb != vc && va != vc)
        for (int q = 0; q < F; ++q) v = fma(a.tri_w[q] * chi[q * M + m], a.face_phi[((size_t)code * F + q) * N + k], v);
    } else if (t <= 9) {
      v = t == 8 ? chi[e % F * M + e / F] : chi[e];
    } else {
      v = t == 10 ? a.tri_w[e] : t == 11 ? a.tg[e] : a.tw[e];
    }
    out[g] = pair_split(v);
  }
}

}  // namespace

// The tables of (p, p_t) on the device, built at the first call, in the solver's stream.
static stdg_status conv_tables(stdg_solver* s, ConvTab* t) {
  const int p = s->p, pt = s->pt, N = s->N, Ng = s->Ng, N1 = p * (p + 1) * (p + 2) / 6, M = (p + 1) * (p + 2) / 2;
  // points of the rules: volume, face, and in time
  const int nv = (3 * p + 1) / 2, nf = (3 * p + 3) / 2, mv = (3 * pt + 2) / 2, mf = (3 * pt + 3) / 2;
  const int V = nv * nv * nv, F = nf * nf;
  if (nv > kVNodes || mv > kTNodes || F != s->nqf_nl || mf != s->nt_nl || F * M > 49 * 15) {
    set_error("convection: unexpected quadrature rules");
    return STDG_EINVAL;
  }
  const int len[13] = {N * V, V * N1, V, mv * Ng, mv, 3 * N1 * N, 64 * N * M, 64 * M * N, M * F, F * M, F, mf * Ng, mf};
  ConvOff off{};
  for (int k = 0; k < 13; ++k) off.o[k + 1] = off.o[k] + len[k];
  if (!s->conv_tab) {
    ConvNodes nd{};
    nd.nv = nv; nd.mv = mv;
    std::vector<double> x, w, g(Ng), dg(Ng);
    for (int al = 0; al < 3; ++al) {
      gauss_jacobi01(nv, al, x, w);
      for (int q = 0; q < nv; ++q) { nd.x[al][q] = x[q]; nd.w[al][q] = w[q]; }
    }
    gauss_jacobi01(mv, 0, x, w);
    for (int q = 0; q < mv; ++q) {
      legendre01(pt, x[q], g.data(), dg.data());
      for (int b = 0; b < Ng; ++b) nd.tg[q * Ng + b] = g[b];
      nd.tw[q] = w[q];
    }
    const std::vector<int> ex = multi_indices(p);
    for (size_t k = 0; k < ex.size(); ++k) nd.mi.e[k] = (unsigned char)ex[k];
    const ConvSrc src{s->dr.tet_nl_phi, s->dr.tet_nl_dphi, s->dr.tet_nl_w, s->dr.face_nl_phi, s->dr.tri_nl_st, s->dr.tri_nl_w,
                      s->d_tg, s->d_tw, s->nq_nl, F, mf};
    float2* d = nullptr;
    const stdg_status e = dev_alloc(s, (void**)&d, (size_t)off.o[13] * sizeof(float2));
    if (e != STDG_OK) return e;
    ++s->nlaunch;
    k_conv_tables<<<std::min(304, (off.o[13] + 255) / 256), 256, 0, s->stream>>>(N, N1, M, Ng, nd, src, off, d);
    STDG_LAUNCH_CHECK();
    s->conv_tab = d;
  }
  const float2* d = s->conv_tab;
  *t = ConvTab{d + off.o[0], d + off.o[1], d + off.o[2], d + off.o[3], d + off.o[4], d + off.o[5], d + off.o[6],
               d + off.o[7], d + off.o[8], d + off.o[9], d + off.o[10], d + off.o[11], d + off.o[12]};
  return STDG_OK;
}

// STDG_EUNSUPPORTED at p = 0, where the caller uses the general kernel.
stdg_status convection_modal(stdg_solver* s, const FieldArg& fld, const double* vbar, double* ups) {
  if (s->p < 1 || s->p > 4) return STDG_EUNSUPPORTED;
  ConvTab t{};
  std::lock_guard<std::mutex> lock(*s->fxws.order);
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
