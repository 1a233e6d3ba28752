// The products of per-tet and per-face binary64 blocks with space-time vectors, in 64-bit fixed point
// (fixed.cuh): the five-point operator (Eq. CS_19 / A1_mod), the pressure right-hand side (Eq. A2_mod),
// the face gradient and velocity update (Eq. prevpress, A3_mod), averaging and the go back (Eq. average,
// goback).  All are one shape: a unit (tet or face) has SLOTS blocks of N x N; thread (unit, slot, row)
// multiplies its row of its block with the NCOL columns of the slot's vector, and the slots of an output
// group are added in 128-bit integers.
//
// What bounds them: the binary64 kernels they replace were bound by sm_103a's binary64 pipe (64 cycles
// per warp FMA, every block entry used for up to 15 columns).  Here an entry costs about 20 integer
// instructions to scale and split, once, and 3 IMAD.WIDE (2 cycles each) per column, so the integer
// pipe binds at many columns and the block traffic from HBM at one or two.  Layout: vectors as limbs in
// shared memory, [set][column][row], two rows per 16-byte broadcast load; blocks read by rows are staged
// through shared memory in rows of odd stride (64-bit accesses at odd strides hit every bank once)
// by 8-byte cp.async, blocks read by columns (the transposed products) come straight from global
// memory, coalesced over the threads of a slot.
#include <algorithm>
#include <cmath>

#include "fixed.cuh"
#include "lp_ptx.cuh"
#include "solver.h"

namespace stdg {
namespace {

// ---- the operations.  For unit u: mat() the block of a slot (nullptr: absent), its exponent and
// whether it is read by columns; vec() the column-0 pointer of a vector set and the distance between
// columns; store() one output.
struct FxSlot { const double* m; int e; bool col; };
struct FxVec { const double* p; int64_t stride_c, stride_q; };   // column (c, q) at p + c stride_c + q stride_q

// y_i = scale Sum over the diagonal and the four face blocks (T x)_nbr (+ mass term)
struct FxApply {
  static constexpr int SLOTS = 5, SETS = 5, GROUPS = 1, C = 1;
  static constexpr bool STAGED = true, MIX = true;
  int n;                                    // units
  const int4 *gface, *gnbr;
  const double *B, *A, *x, *detJ;
  const uint16_t *eB, *eA;
  double* y;
  double scale, mass_coef, pin_diag;
  int pinned;
  double K[kMaxNg * kMaxNg];
  __device__ int4 pick(const int4* t, int u) const { return t[u]; }
  __device__ static int at(const int4& v, int f) { return f == 0 ? v.x : f == 1 ? v.y : f == 2 ? v.z : v.w; }
  template <int N>
  __device__ FxSlot mat(int u, int sl) const {
    if (sl == 0) return {B + (size_t)u * N * N, eB[u], true};        // symmetric: its columns are its rows
    const int g = at(gface[u], sl - 1);
    if (g < 0) return {nullptr, 0, false};
    return {A + (size_t)(g >> 1) * N * N, eA[g >> 1], (g & 1) != 0};  // A_rl = A_lr^T
  }
  template <int N, int NG>
  __device__ FxVec vec(int u, int set) const {
    const int nb = set == 0 ? u : at(gnbr[u], set - 1);
    if (nb < 0) return {nullptr, 0, 0};
    return {x + (size_t)nb * N * NG, 0, N};
  }
  // pinned entries (constant mode of tet 0, every time column) read as 0
  __device__ bool zero(int u, int set, int k) const {
    return pinned && k == 0 && (set == 0 ? u : at(gnbr[u], set - 1)) == 0;
  }
  __device__ static int set_of(int sl) { return sl; }
  __device__ static int group_of(int) { return 0; }
  __device__ double unit_scale(int u) const { return mass_coef != 0.0 ? mass_coef * detJ[u] : 0.0; }
  template <int N, int NG>
  __device__ void store(int u, int, int, int q, int k, double v, double us) const {
    const double* xu = x + (size_t)u * N * NG + k;
    if (scale != 1.0) v *= scale;
    if (mass_coef != 0.0) {
      double m = 0.0;
      for (int b = 0; b < NG; ++b) m = fma(K[q * NG + b], xu[b * N], m);
      v = fma(us, m, v);
    }
    if (pinned && u == 0 && k == 0) v = pin_diag * xu[q * N];
    y[((size_t)u * NG + q) * N + k] = v;
  }
};

// b_i = coef Sum_f Sum_c Q^c_f(i)^T F_f^c
struct FxRhs {
  static constexpr int SLOTS = 12, SETS = 12, GROUPS = 1, C = 1;
  static constexpr bool STAGED = false, MIX = false;
  int n;
  const int *t2f, *left;
  const double *Q, *F;
  const uint16_t* eQ;
  double* b;
  double coef;
  int pinned;
  template <int N>
  __device__ FxSlot mat(int u, int sl) const {
    const int f = sl / 3, c = sl - 3 * f, j = t2f[4 * u + f], s = left[j] == u ? 0 : 1;
    return {Q + ((size_t)j * 6 + 3 * s + c) * N * N, eQ[2 * j + s], true};
  }
  template <int N, int NG>
  __device__ FxVec vec(int u, int set) const {
    const int f = set / 3, c = set - 3 * f;
    return {F + ((size_t)t2f[4 * u + f] * 3 + c) * N * NG, 0, N};
  }
  __device__ bool zero(int, int, int) const { return false; }
  __device__ static int set_of(int sl) { return sl; }
  __device__ static int group_of(int) { return 0; }
  __device__ double unit_scale(int) const { return 0.0; }
  template <int N, int NG>
  __device__ void store(int u, int, int, int q, int k, double v, double) const {
    b[((size_t)u * NG + q) * N + k] = pinned && u == 0 && k == 0 ? 0.0 : v * coef;
  }
};

// out_j^c = in_j^c - dt Sum_s Q^c_s (K^-1 p)_s  (velocity update: boundary faces copy `in`), or with
// grad the face gradient out_j^c = dt Sum_s Q^c_s (K^-1 p)_s (boundary faces: the volume block of slot 1
// with the left tet)
struct FxFace {
  static constexpr int SLOTS = 6, SETS = 2, GROUPS = 3, C = 1;
  static constexpr bool STAGED = true, MIX = true;
  int n;
  const int *left, *right;
  const double *Q, *p, *in;
  const uint16_t* eQ;
  double* out;
  double dt;
  int grad;
  template <int N>
  __device__ FxSlot mat(int u, int sl) const {
    const int s = sl / 3, c = sl - 3 * s;
    if (right[u] < 0 && !(grad && s == 1)) return {nullptr, 0, false};
    return {Q + ((size_t)u * 6 + 3 * s + c) * N * N, eQ[2 * u + s], false};
  }
  template <int N, int NG>
  __device__ FxVec vec(int u, int set) const {
    const int r = right[u];
    if (r < 0 && !(grad && set == 1)) return {nullptr, 0, 0};
    const int tet = set == 1 && r >= 0 ? r : left[u];
    return {p + (size_t)tet * N * NG, 0, N};
  }
  __device__ bool zero(int, int, int) const { return false; }
  __device__ static int set_of(int sl) { return sl / 3; }
  __device__ static int group_of(int sl) { return sl % 3; }
  __device__ double unit_scale(int) const { return 0.0; }
  template <int N, int NG>
  __device__ void store(int u, int g, int, int q, int k, double v, double) const {
    const size_t o = (((size_t)u * 3 + g) * NG + q) * N + k;
    out[o] = grad ? dt * v : right[u] < 0 ? in[o] : in[o] - dt * v;
  }
};

// out^c_i = 1/|J_i| Sum_f M_f(i) in_f^c
struct FxAverage {
  static constexpr int SLOTS = 4, SETS = 4, GROUPS = 1, C = 3;
  static constexpr bool STAGED = true, MIX = false;
  int n;
  const int *t2f, *left;
  const double *M, *in, *detJ;
  const uint16_t* eM;
  double* out;
  template <int N>
  __device__ FxSlot mat(int u, int f) const {
    const int j = t2f[4 * u + f], s = left[j] == u ? 0 : 1;
    return {M + ((size_t)j * 2 + s) * N * N, eM[2 * j + s], false};
  }
  template <int N, int NG>
  __device__ FxVec vec(int u, int f) const {
    return {in + (size_t)t2f[4 * u + f] * 3 * N * NG, N * NG, N};
  }
  __device__ bool zero(int, int, int) const { return false; }
  __device__ static int set_of(int sl) { return sl; }
  __device__ static int group_of(int) { return 0; }
  __device__ double unit_scale(int u) const { return 1.0 / detJ[u]; }
  template <int N, int NG>
  __device__ void store(int u, int, int c, int q, int k, double v, double us) const {
    out[(((size_t)c * n + u) * NG + q) * N + k] = v * us;
  }
};

// F_j^c = Sum_s M_s^T vbar_s^c, boundary faces the prescribed velocity
struct FxGoback {
  static constexpr int SLOTS = 2, SETS = 2, GROUPS = 1, C = 3;
  static constexpr bool STAGED = false, MIX = false;
  int n;
  int64_t ne;
  const int *left, *right;
  const double *M, *vbar, *Vbc;
  const uint16_t* eM;
  double* F;
  template <int N>
  __device__ FxSlot mat(int u, int s) const {
    if (right[u] < 0) return {nullptr, 0, false};
    return {M + ((size_t)u * 2 + s) * N * N, eM[2 * u + s], true};
  }
  template <int N, int NG>
  __device__ FxVec vec(int u, int s) const {
    const int r = right[u];
    if (r < 0) return {nullptr, 0, 0};
    return {vbar + (size_t)(s ? r : left[u]) * N * NG, ne * N * NG, N};
  }
  __device__ bool zero(int, int, int) const { return false; }
  __device__ static int set_of(int sl) { return sl; }
  __device__ static int group_of(int) { return 0; }
  __device__ double unit_scale(int) const { return 0.0; }
  template <int N, int NG>
  __device__ void store(int u, int, int c, int q, int k, double v, double) const {
    const size_t o = (((size_t)u * 3 + c) * NG + q) * N + k;
    F[o] = right[u] < 0 ? Vbc[o] : v;
  }
};

// units per CTA: about 200 to 320 threads, most lanes of the last warp used
template <class P, int N>
struct FxTile {
  static constexpr int per = P::SLOTS * N;
  static constexpr int TB = per >= 160 ? 1 : 256 / per;
  static constexpr int threads = (TB * per + 31) / 32 * 32;
};
template <class P, int N, int NG>
struct FxSmem {
  static constexpr int TB = FxTile<P, N>::TB, NC = P::C * NG, NS = N | 1, NX = (N + 1) & ~1;
  static constexpr size_t stage = P::STAGED ? (size_t)TB * P::SLOTS * N * NS * 8 : 0;
  static constexpr size_t red = (size_t)TB * P::SLOTS * NC * N * 16;
  static constexpr size_t xs = (size_t)TB * P::SETS * NC * NX * 8;
  // the partial sums take the place of the staged blocks and the vectors
  static constexpr size_t bytes = ((stage + xs > red ? stage + xs : red) + 15) / 16 * 16;
};

template <class P, int N, int NG>
__global__ void __launch_bounds__(FxTile<P, N>::threads) k_fx(P a, FxMat mix) {
  using T = FxTile<P, N>;
  using S = FxSmem<P, N, NG>;
  constexpr int TB = T::TB, NC = S::NC, NS = S::NS, NX = S::NX, NT = T::threads;
  extern __shared__ __align__(16) unsigned char fxs[];
  int2* xs = reinterpret_cast<int2*>(fxs);                        // [unit][set][column][NX]
  double* stage = reinterpret_cast<double*>(fxs + S::xs);         // [unit][slot][N][NS]
  longlong2* red = reinterpret_cast<longlong2*>(fxs);             // [unit][slot][column][N]
  __shared__ int ex[TB][P::SETS][NC];                             // exponents of the vector columns
  __shared__ int slow[TB];                                        // the unit takes the binary64 path
  __shared__ int es[TB][P::SLOTS];                                // exponents of the blocks (-1: absent)
  __shared__ double us[TB];
  const int t = threadIdx.x, u0 = blockIdx.x * TB;
  for (int o = t; o < TB * P::SETS * NC; o += NT) (&ex[0][0][0])[o] = 0;
  if (t < TB) slow[t] = 0;
  const int tl = t / T::per, sk = t - tl * T::per, sl = sk / N, k = sk - sl * N, u = u0 + tl;
  const bool act = tl < TB && u < a.n;
  FxSlot m{nullptr, 0, false};
  if (act) m = a.template mat<N>(u, sl);
  const bool have = m.m != nullptr;
  if constexpr (P::STAGED) {
    if (have) {
      double* st = stage + (size_t)(tl * P::SLOTS + sl) * N * NS + k;
#pragma unroll 5
      for (int j = 0; j < N; ++j) cp_async<8>(st + j * NS, m.m + j * N + k);
    }
  }
  __syncthreads();
  // vectors: thread (unit, set, row) loads its columns; their largest exponents (with mixing one per
  // set, as the columns are combined)
  constexpr int XP = P::SETS * N, XR = (TB * XP + NT - 1) / NT;
  double xv[XR][NC];
#pragma unroll
  for (int r = 0; r < XR; ++r) {
    const int o = t + r * NT, xl = o / XP, xr = o - xl * XP, set = xr / N, xk = xr - set * N;
#pragma unroll
    for (int c = 0; c < NC; ++c) xv[r][c] = 0.0;
    if (xl >= TB || u0 + xl >= a.n) continue;
    const FxVec v = a.template vec<N, NG>(u0 + xl, set);
    if (v.p && !a.zero(u0 + xl, set, xk)) {
#pragma unroll
      for (int c = 0; c < NC; ++c) xv[r][c] = v.p[(c / NG) * v.stride_c + (c % NG) * v.stride_q + xk];
    }
    if (P::MIX && mix.on) {
      int e = 0;
#pragma unroll
      for (int c = 0; c < NC; ++c) e = max(e, fx_exp(xv[r][c]));
      if (e) atomicMax(&ex[xl][set][0], e);
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int e = fx_exp(xv[r][c]);
        if (e) atomicMax(&ex[xl][set][c], e);
      }
    }
  }
  if (act && k == 0) {
    es[tl][sl] = have ? m.e : -1;
    if (have && !fx_ok(m.e)) slow[tl] = 1;
    if (sl == 0) us[tl] = a.unit_scale(u);
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < XR; ++r) {
    const int o = t + r * NT, xl = o / XP, xr = o - xl * XP, set = xr / N, xk = xr - set * N;
    if (xl >= TB) continue;
    int2* xd = xs + (size_t)(xl * P::SETS + set) * NC * NX + xk;
    if (P::MIX && mix.on) {
      const int e = ex[xl][set][0];
      if (!fx_ok(e) || !fx_ok(mix.e)) slow[xl] = 1;
      int h[NC], l[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) fx_limbs<kFxX>(xv[r][c], e, h[c], l[c]);
#pragma unroll 1
      for (int c = 0; c < NC; ++c) {          // (T x)_c: |S0| < 5 2^55, kept to 2^-56 of the full scale
        long long S0 = 0, S1 = 0;
#pragma unroll
        for (int b = 0; b < NC; ++b) fx_mad(mix.h[c * NC + b], mix.l[c * NC + b], h[b], l[b], S0, S1);
        const long long V = (S0 + ((S1 + (1 << 28)) >> kFxL) + 2) >> 2;
        xd[c * NX] = e ? fx_limbs_int(V) : make_int2(0, 0);
      }
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int e = ex[xl][set][c];
        if (!fx_ok(e)) slow[xl] = 1;
        int2 v = make_int2(0, 0);
        if (e) fx_limbs<kFxX>(xv[r][c], e, v.x, v.y);
        xd[c * NX] = v;
      }
    }
  }
  if constexpr (P::STAGED) cp_async_wait_all();
  __syncthreads();
  // products: row k of the slot's block with every column of the slot's vector
  const bool dbl = act && slow[tl] != 0;
  long long S0[NC], S1[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) S0[c] = S1[c] = 0;
  if (have && !dbl) {
    const int2* xr = xs + (size_t)(tl * P::SETS + P::set_of(sl)) * NC * NX;
    const double* mp = P::STAGED ? stage + (size_t)(tl * P::SLOTS + sl) * N * NS + (m.col ? k : k * NS) : m.m + k;
    const int step = P::STAGED ? (m.col ? NS : 1) : N;
    const int e = m.e ? m.e : kFxMinExp;
#pragma unroll (NC > 5 ? 2 : N <= 10 ? 5 : 4)
    for (int l = 0; l + 1 < N; l += 2) {
      int h0, l0, h1, l1;
      fx_limbs<kFxA>(mp[l * step], e, h0, l0);
      fx_limbs<kFxA>(mp[(l + 1) * step], e, h1, l1);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int4 v = *reinterpret_cast<const int4*>(xr + c * NX + l);
        fx_mad(h0, l0, v.x, v.y, S0[c], S1[c]);
        fx_mad(h1, l1, v.z, v.w, S0[c], S1[c]);
      }
    }
    if constexpr (N & 1) {
      int h0, l0;
      fx_limbs<kFxA>(mp[(N - 1) * step], e, h0, l0);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int2 v = xr[c * NX + N - 1];
        fx_mad(h0, l0, v.x, v.y, S0[c], S1[c]);
      }
    }
  }
  __syncthreads();                                     // the stage and the vectors are free
  if (have && dbl) {                                   // binary64 multiply-adds (non-finite or tiny operands)
    const FxVec v = a.template vec<N, NG>(u, P::set_of(sl));
#pragma unroll 1
    for (int c = 0; c < NC; ++c) {
      double s = 0.0;
#pragma unroll 1
      for (int l = 0; l < N; ++l) {
        const double* p = v.p + (c / NG) * v.stride_c + l;
        double xc = 0.0;
        if (!a.zero(u, P::set_of(sl), l)) {
          if (P::MIX && mix.on)
            for (int b = 0; b < NG; ++b) xc = fma(mix.v[(c % NG) * NG + b], p[b * v.stride_q], xc);
          else
            xc = p[(c % NG) * v.stride_q];
        }
        s = fma(m.m[m.col ? l * N + k : k * N + l], xc, s);
      }
      red[((size_t)(tl * P::SLOTS + sl) * NC + c) * N + k] = make_longlong2(__double_as_longlong(s), 0);
    }
  } else if (have) {
#pragma unroll
    for (int c = 0; c < NC; ++c) red[((size_t)(tl * P::SLOTS + sl) * NC + c) * N + k] = make_longlong2(S0[c], S1[c]);
  }
  __syncthreads();
  // outputs: the slots of each group added with aligned exponents
  constexpr int per_out = P::GROUPS * NC * N;
  for (int o = t; o < TB * per_out; o += NT) {
    const int ol = o / per_out, rem = o - ol * per_out, g = rem / (NC * N), c = rem / N % NC, ok = rem % N;
    const int ou = u0 + ol;
    if (ou >= a.n) continue;
    const longlong2* rp = red + ((size_t)ol * P::SLOTS * NC + c) * N + ok;
    double v;
    if (slow[ol]) {
      v = 0.0;
      for (int s = 0; s < P::SLOTS; ++s)
        if (P::group_of(s) == g && es[ol][s] >= 0) v += __longlong_as_double(rp[(size_t)s * NC * N].x);
    } else {
      int top = 0;
      for (int s = 0; s < P::SLOTS; ++s) {
        if (P::group_of(s) != g || es[ol][s] <= 0) continue;
        const int xe = ex[ol][P::set_of(s)][P::MIX && mix.on ? 0 : c];
        if (xe > 0) top = max(top, es[ol][s] + xe);
      }
      __int128 sum = 0;
      for (int s = 0; s < P::SLOTS; ++s) {
        if (P::group_of(s) != g || es[ol][s] <= 0) continue;
        const int xe = ex[ol][P::set_of(s)][P::MIX && mix.on ? 0 : c];
        if (xe <= 0) continue;
        const longlong2 r = rp[(size_t)s * NC * N];
        sum += (((__int128)r.x << kFxL) + r.y) >> min(top - es[ol][s] - xe, 127);
      }
      v = fx_value(sum, fx_unit(top, P::MIX && mix.on ? mix.e - 1019 : 0));
    }
    a.template store<N, NG>(ou, g, c / NG, c % NG, ok, v, us[ol]);
  }
}

template <class P, int N, int NG>
cudaError_t fx_launch_t(const P& a, const FxMat& mix, cudaStream_t st) {
  constexpr int smem = (int)FxSmem<P, N, NG>::bytes;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_fx<P, N, NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  constexpr int TB = FxTile<P, N>::TB;
  if (a.n > 0) k_fx<P, N, NG><<<(a.n + TB - 1) / TB, FxTile<P, N>::threads, smem, st>>>(a, mix);
  return cudaGetLastError();
}
template <class P, int N>
cudaError_t fx_launch_n(int Ng, const P& a, const FxMat& mix, cudaStream_t st) {
  switch (Ng) {
    case 1: return fx_launch_t<P, N, 1>(a, mix, st);
    case 2: return fx_launch_t<P, N, 2>(a, mix, st);
    case 3: return fx_launch_t<P, N, 3>(a, mix, st);
    case 4: return fx_launch_t<P, N, 4>(a, mix, st);
    case 5: return fx_launch_t<P, N, 5>(a, mix, st);
  }
  return cudaErrorInvalidValue;
}
template <class P>
cudaError_t fx_launch(int N, int Ng, const P& a, const FxMat& mix, cudaStream_t st) {
  switch (N) {
    case 1: return fx_launch_n<P, 1>(Ng, a, mix, st);
    case 4: return fx_launch_n<P, 4>(Ng, a, mix, st);
    case 10: return fx_launch_n<P, 10>(Ng, a, mix, st);
    case 20: return fx_launch_n<P, 20>(Ng, a, mix, st);
    case 35: return fx_launch_n<P, 35>(Ng, a, mix, st);
  }
  return cudaErrorInvalidValue;
}

// exponent of the largest entry of each block of `len` entries (fx_exp), one warp per block
__global__ void k_fx_exps(int64_t nblk, int len, const double* __restrict__ in, uint16_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  for (int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; b < nblk;
       b += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    int e = 0;
    for (int o = lane; o < len; o += 32) e = max(e, fx_exp(in[b * len + o]));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) out[b] = (uint16_t)e;
  }
}

// host: an n x n matrix in limbs
FxMat fx_mat(const double* v, int n) {
  FxMat m{};
  m.on = 1;
  double big = 0.0;
  for (int q = 0; q < n * n; ++q) {
    m.v[q] = v[q];
    big = std::isfinite(v[q]) ? std::fmax(big, std::fabs(v[q])) : INFINITY;
    if (!std::isfinite(big)) { m.e = 2047; return m; }
  }
  int E = 0;
  std::frexp(big, &E);
  m.e = big > 0.0 ? std::max(E + 1022, 1) : 0;
  if (m.e < kFxMinExp) return m;
  for (int q = 0; q < n * n; ++q) {
    const long long w = (long long)std::ldexp(v[q], kFxA - E);        // |w| < 2^kFxA
    const long long h = (w + (1 << (kFxL - 1))) >> kFxL;
    m.h[q] = (int)h;
    m.l[q] = (int)(w - h * (1LL << kFxL));
  }
  return m;
}

}  // namespace

cudaError_t launch_block_exps(int64_t nblk, int len, const double* blocks, uint16_t* exps, cudaStream_t st) {
  if (nblk > 0) k_fx_exps<<<1216, 256, 0, st>>>(nblk, len, blocks, exps);
  return cudaGetLastError();
}

cudaError_t launch_apply(const ApplyArgs& a, const double* x, double* y, cudaStream_t st) {
  FxApply p{};
  p.n = a.ne;
  p.gface = reinterpret_cast<const int4*>(a.gface); p.gnbr = reinterpret_cast<const int4*>(a.gnbr);
  p.B = a.B; p.A = a.Aoff; p.eB = a.eB; p.eA = a.eA; p.detJ = a.detJ;
  p.x = x; p.y = y;
  p.scale = a.scale; p.mass_coef = a.mass_coef; p.pin_diag = a.pin_diag; p.pinned = a.pinned;
  for (int q = 0; q < a.Ng * a.Ng; ++q) p.K[q] = a.Kmass[q];
  return fx_launch(a.N, a.Ng, p, a.tacc_identity ? FxMat{} : fx_mat(a.Tacc, a.Ng), st);
}

cudaError_t launch_rhs(const FaceOps& f, const double* F, double coef, int pinned, double* b, cudaStream_t st) {
  FxRhs p{};
  p.n = f.ne; p.t2f = f.t2f; p.left = f.left; p.Q = f.Q; p.eQ = f.eQ; p.F = F; p.b = b; p.coef = coef; p.pinned = pinned;
  return fx_launch(f.N, f.Ng, p, FxMat{}, st);
}

static FxFace fx_face(const FaceOps& f, const double* x, double dt) {
  FxFace p{};
  p.n = f.nf; p.left = f.left; p.right = f.right; p.Q = f.Q; p.eQ = f.eQ; p.p = x; p.dt = dt;
  return p;
}
cudaError_t launch_update(const FaceOps& f, const double* F, const double* dp, double dt, const double* Kinv, double* V,
                          cudaStream_t st) {
  FxFace p = fx_face(f, dp, dt);
  p.in = F; p.out = V;
  return fx_launch(f.N, f.Ng, p, fx_mat(Kinv, f.Ng), st);
}
cudaError_t launch_face_grad(const FaceOps& f, const double* P, double dt, const double* Kinv, double* G, cudaStream_t st) {
  FxFace p = fx_face(f, P, dt);
  p.grad = 1; p.out = G;
  return fx_launch(f.N, f.Ng, p, fx_mat(Kinv, f.Ng), st);
}

cudaError_t launch_average(const FaceOps& f, const double* detJ, const double* in, double* out, cudaStream_t st) {
  FxAverage p{};
  p.n = f.ne; p.t2f = f.t2f; p.left = f.left; p.M = f.Mij; p.eM = f.eM; p.in = in; p.detJ = detJ; p.out = out;
  return fx_launch(f.N, f.Ng, p, FxMat{}, st);
}
cudaError_t launch_goback(const FaceOps& f, const double* vbar, const double* Vbc, double* F, cudaStream_t st) {
  FxGoback p{};
  p.n = f.nf; p.ne = f.ne; p.left = f.left; p.right = f.right; p.M = f.Mij; p.eM = f.eM; p.vbar = vbar; p.Vbc = Vbc; p.F = F;
  return fx_launch(f.N, f.Ng, p, FxMat{}, st);
}

}  // namespace stdg
