// The products of per-tet and per-face binary64 blocks with space-time vectors, in 64-bit fixed point
// (fixed.cuh): the five-point operator (Eq. CS_19 / A1_mod), the pressure right-hand side (Eq. A2_mod),
// the face gradient and velocity update (Eq. prevpress, A3_mod), averaging and the go back (Eq. average,
// goback), the velocity moments (Eq. vis3).  All are one shape: a unit (tet or face) has SLOTS blocks of
// N x N; thread (unit, slot, row) multiplies its row of its block with the NCOL columns of the slot's vector,
// and the slots of an output group are added in 96-bit integers.
//
// What bounds them: binary64 kernels of this shape are bound by sm_103a's binary64 pipe (64 cycles per
// warp FMA, every block entry used for up to 15 columns).  Here a product costs 3 IMAD.WIDE (4 cycles
// each), with two of the integer ALU's additions per product, and the operands come through shared memory,
// which returns 128 bytes a cycle to an SM (8 cycles of each scheduler per 64-bit operand, also when all
// lanes read the same word).  Thread tiles of 2 or 3 rows save such reads and were slower: the
// blocks of a CTA fill the shared memory, so fewer threads per CTA are fewer warps per SM (N = 35, NG = 5
// at 24,576 tets: 1.4 times the time with two rows, 1.8 times with three).  Measured, start of a pass to its
// end, binary64 kernels before -> now: operator at 20,250 tets, p = 3, p_t = 0, 198 -> 80 us; at 24,576 tets,
// p = p_t = 4, 766 (binary32 pairs) -> 579 us; right-hand side at 7,986 tets, p = p_t = 4, 1,597 -> 442 us;
// velocity update at 20,250 tets, p = p_t = 2, 164 -> 107 us.
//
// Two launches: k_fx_vec scales the vector to limbs once, with one exponent per column of every tet (face,
// component), and applies the time matrix to it where the operation has one; k_fx starts at the same time
// (programmatic dependent launch) and first copies its blocks, which do not depend on the vector, into
// shared memory (8-byte cp.async; rows of odd stride, as 64-bit accesses at odd strides hit every bank
// once).  Blocks read by columns only (rhs, go back) come straight from global memory instead, coalesced
// over the threads of a slot.  Scaling the vectors inside k_fx instead, every one in all the units that
// use it, took as many instructions as the products (N = 35, NG = 5).
#include <algorithm>
#include <cmath>

#include "fixed.cuh"
#include "lp_ptx.cuh"
#include "solver.h"

namespace stdg {
namespace {

// ---- the operations.  For unit u: mat() the block of a slot (nullptr: absent), its exponent and
// whether it is read by columns; vec() the index of the vector (NG columns of N) of a set and component
// in the operation's input (-1: absent); store() one output.
struct FxSlot { const int2* m; int e; bool col; };

// y_i = scale Sum over the diagonal and the four face blocks (T x)_nbr (+ mass term)
struct FxApply {
  static constexpr int SLOTS = 5, SETS = 5, GROUPS = 1, C = 1;
  static constexpr bool STAGED = true;
  int n;                                    // units
  const int4 *gface, *gnbr;
  FxBlocks B, A;
  const double *x, *detJ;
  double* y;
  double scale, mass_coef, pin_diag;
  int unscaled, mass, pinned;               // scale is 1 (1) or -1 (-1), else 0; mass_coef is not 0 (comparing
                                            // them in the kernel would take the binary64 pipe)
  double K[kMaxNg * kMaxNg];
  __device__ int4 pick(const int4* t, int u) const { return t[u]; }
  __device__ static int at(const int4& v, int f) { return f == 0 ? v.x : f == 1 ? v.y : f == 2 ? v.z : v.w; }
  template <int N>
  __device__ FxSlot mat(int u, int sl) const {
    if (sl == 0) return {B.w + (size_t)u * N * N, B.e[u], true};        // symmetric: its columns are its rows
    const int g = at(gface[u], sl - 1);
    if (g < 0) return {nullptr, 0, false};
    return {A.w + (size_t)(g >> 1) * N * N, A.e[g >> 1], (g & 1) != 0};  // A_rl = A_lr^T
  }
  __device__ int vec(int u, int set, int) const { return set == 0 ? u : at(gnbr[u], set - 1); }
  template <int N>
  __device__ double entry(int u, int sl, int idx) const {
    return sl == 0 ? fx_entry(B, N * N, u, idx, N) : fx_entry(A, N * N, at(gface[u], sl - 1) >> 1, idx, N);
  }
  __device__ const FxScale& out_scale() const { return B.r; }
  __device__ static int set_of(int sl) { return sl; }
  __device__ static int group_of(int) { return 0; }
  __device__ static int slot_of(int, int j) { return j; }
  __device__ static bool copies(int) { return true; }
  __device__ double unit_scale(int u) const { return mass ? mass_coef * detJ[u] : 0.0; }
  template <int N, int NG>
  __device__ void store(int u, int, int, int q, int k, double v, double us) const {
    const double* xu = x + (size_t)u * N * NG + k;
    if (unscaled == 0) v *= scale;
    else if (unscaled < 0) v = -v;
    if (mass) {
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
  static constexpr bool STAGED = false;
  int n;
  const int4* tface;                        // per tet: its faces, (face << 1 | the tet is r)
  FxBlocks Q;
  double* b;
  double coef;
  int pinned;
  template <int N>
  __device__ FxSlot mat(int u, int sl) const {
    const int f = sl / 3, g = FxApply::at(tface[u], f);
    const size_t b = (size_t)g * 3 + sl - 3 * f;
    return {Q.w + b * N * N, Q.e[b], true};
  }
  __device__ int vec(int u, int set, int) const { return 3 * (FxApply::at(tface[u], set / 3) >> 1) + set % 3; }
  template <int N>
  __device__ double entry(int u, int sl, int idx) const {
    return fx_entry(Q, N * N, (size_t)FxApply::at(tface[u], sl / 3) * 3 + sl % 3, idx, N);
  }
  __device__ const FxScale& out_scale() const { return Q.c; }
  __device__ static int set_of(int sl) { return sl; }
  __device__ static int group_of(int) { return 0; }
  __device__ static int slot_of(int, int j) { return j; }
  __device__ static bool copies(int) { return true; }
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
  static constexpr bool STAGED = true;
  int n;
  const int *left, *right;
  FxBlocks Q;
  const double* in;
  double* out;
  double dt;
  int grad;
  template <int N>
  __device__ FxSlot mat(int u, int sl) const {
    const int s = sl / 3, c = sl - 3 * s;
    if (right[u] < 0 && !(grad && s == 1)) return {nullptr, 0, false};
    const size_t b = (size_t)u * 6 + 3 * s + c;
    return {Q.w + b * N * N, Q.e[b], false};
  }
  __device__ int vec(int u, int set, int) const {
    const int r = right[u];
    if (r < 0 && !(grad && set == 1)) return -1;
    return set == 1 && r >= 0 ? r : left[u];
  }
  template <int N>
  __device__ double entry(int u, int sl, int idx) const {
    return fx_entry(Q, N * N, 6 * (size_t)u + sl, idx, N);
  }
  __device__ const FxScale& out_scale() const { return Q.r; }
  __device__ static int set_of(int sl) { return sl / 3; }
  __device__ static int group_of(int sl) { return sl % 3; }
  __device__ static int slot_of(int g, int j) { return 3 * j + g; }
  __device__ static bool copies(int sl) { return sl % 3 == 0; }
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
  static constexpr bool STAGED = true;
  int n;
  const int4* tface;
  FxBlocks M;
  const double* detJ;
  double* out;
  template <int N>
  __device__ FxSlot mat(int u, int f) const {
    const int g = FxApply::at(tface[u], f);
    return {M.w + (size_t)g * N * N, M.e[g], false};
  }
  __device__ int vec(int u, int f, int c) const { return 3 * (FxApply::at(tface[u], f) >> 1) + c; }
  template <int N>
  __device__ double entry(int u, int f, int idx) const { return fx_entry(M, N * N, FxApply::at(tface[u], f), idx, N); }
  __device__ const FxScale& out_scale() const { return M.r; }
  __device__ static int set_of(int sl) { return sl; }
  __device__ static int group_of(int) { return 0; }
  __device__ static int slot_of(int, int j) { return j; }
  __device__ static bool copies(int) { return true; }
  __device__ double unit_scale(int u) const { return 1.0 / detJ[u]; }
  template <int N, int NG>
  __device__ void store(int u, int, int c, int q, int k, double v, double us) const {
    out[(((size_t)c * n + u) * NG + q) * N + k] = v * us;
  }
};

// F_j^c = Sum_s M_s^T vbar_s^c, boundary faces the prescribed velocity
struct FxGoback {
  static constexpr int SLOTS = 2, SETS = 2, GROUPS = 1, C = 3;
  static constexpr bool STAGED = false;
  int n, ne;
  const int *left, *right;
  FxBlocks M;
  const double* Vbc;
  double* F;
  template <int N>
  __device__ FxSlot mat(int u, int s) const {
    if (right[u] < 0) return {nullptr, 0, false};
    return {M.w + ((size_t)u * 2 + s) * N * N, M.e[2 * u + s], true};
  }
  __device__ int vec(int u, int s, int c) const {
    const int r = right[u];
    return r < 0 ? -1 : c * ne + (s ? r : left[u]);
  }
  template <int N>
  __device__ double entry(int u, int s, int idx) const { return fx_entry(M, N * N, 2 * (size_t)u + s, idx, N); }
  __device__ const FxScale& out_scale() const { return M.c; }
  __device__ static int set_of(int sl) { return sl; }
  __device__ static int group_of(int) { return 0; }
  __device__ static int slot_of(int, int j) { return j; }
  __device__ static bool copies(int) { return true; }
  __device__ double unit_scale(int) const { return 0.0; }
  template <int N, int NG>
  __device__ void store(int u, int, int c, int q, int k, double v, double) const {
    const size_t o = (((size_t)u * 3 + c) * NG + q) * N + k;
    F[o] = right[u] < 0 ? Vbc[o] : v;
  }
};

// U_j^(s)c = dt M_s V_j^c (boundary faces: 0 in the place of the absent side)
struct FxMoments {
  static constexpr int SLOTS = 2, SETS = 1, GROUPS = 2, C = 3;
  static constexpr bool STAGED = true;
  int n;
  const int* right;
  FxBlocks M;
  double* U;
  double dt;
  template <int N>
  __device__ FxSlot mat(int u, int s) const {
    if (s == 1 && right[u] < 0) return {nullptr, 0, false};
    return {M.w + ((size_t)u * 2 + s) * N * N, M.e[2 * u + s], false};
  }
  __device__ int vec(int u, int, int c) const { return 3 * u + c; }
  template <int N>
  __device__ double entry(int u, int s, int idx) const { return fx_entry(M, N * N, 2 * (size_t)u + s, idx, N); }
  __device__ const FxScale& out_scale() const { return M.r; }
  __device__ static int set_of(int) { return 0; }
  __device__ static int group_of(int sl) { return sl; }
  __device__ static int slot_of(int g, int) { return g; }
  __device__ static bool copies(int sl) { return sl == 0; }
  __device__ double unit_scale(int) const { return 0.0; }
  template <int N, int NG>
  __device__ void store(int u, int g, int c, int q, int k, double v, double) const {
    U[((((size_t)u * 2 + g) * 3 + c) * NG + q) * N + k] = dt * v;
  }
};

template <class P, int N, int NG>
struct FxTile {
  static constexpr int NC = P::C * NG, NS = N | 1, NX = (N + 1) & ~1;
  static constexpr int per = P::SLOTS * P::C * N;                // threads per unit
  // shared memory of TB units: the vectors and the staged blocks, whose place the partial sums take
  static constexpr size_t bytes(int TB) {
    const size_t in = (size_t)TB * (P::SETS * NC * NX * 8 + (P::STAGED ? P::SLOTS * N * NS * 8 : 0));
    const size_t red = (size_t)TB * P::SLOTS * NC * N * 12;
    return ((in > red ? in : red) + 15) / 16 * 16;
  }
  // units per CTA: the fewest idle lanes with at most 256 threads and 40 KB
  static constexpr int units() {
    int best = 1;
    for (int b = 2; b <= 32; ++b) {
      const int nt = (b * per + 31) / 32 * 32, ot = (best * per + 31) / 32 * 32;
      if (nt <= 256 && bytes(b) <= 40 * 1024 && b * per * ot > best * per * nt) best = b;
    }
    return best;
  }
  static constexpr int TB = units();
  static constexpr int threads = (TB * per + 31) / 32 * 32;
  // CTAs per SM to compile for: 6 NG accumulators and 28 more registers per thread where the blocks are read
  // straight from global memory (loads in flight come from many warps), 48 where they are staged, as
  // far as the shared memory goes
  static constexpr int regs = 6 * NG + (P::STAGED ? 48 : 28), fit = 65536 / (threads * regs);
  static constexpr int room = (int)(227 * 1024 / (bytes(TB) + 2048));
  static constexpr int blocks = fit < 1 ? 1 : fit < room ? fit : room;
  static constexpr size_t xs = (size_t)TB * P::SETS * NC * NX * 8, smem = bytes(TB);
};

// The input vector x as limbs: vector v (n of them, NG columns of N), column q, row k at w[(v NG + q) N + k],
// the (scaled) column's exponent in e[v NG + q]; with mix.on the columns of (mix x), all with the vector's one
// exponent.  pinned: row 0 of vector 0 reads as 0.
struct FxInput {
  FxScale sc;                                 // row k times 2^sc.s[k], the scaling of the blocks' columns
  const double* x;
  int2* w;
  uint16_t* e;
  int n, pinned;
};
__device__ __forceinline__ double fx_in(const FxInput& in, int v, size_t o, int k) {
  return in.pinned && v == 0 && k == 0 ? 0.0 : in.x[o];
}

template <int N>
struct FxLanes {                              // lanes per vector: a power of two that holds N rows, at most 32
  static constexpr int G = N <= 1 ? 1 : N <= 4 ? 4 : N <= 16 ? 16 : 32, K = (N + G - 1) / G;
};
template <int N, int NG>
__global__ void __launch_bounds__(256) k_fx_vec(const __grid_constant__ FxInput in, const __grid_constant__ FxMat mix) {
  constexpr int G = FxLanes<N>::G, K = FxLanes<N>::K;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int t = blockIdx.x * 256 + threadIdx.x, v = t / G, k0 = t % G;
  if ((t - (int)(threadIdx.x & 31)) / G >= in.n) return;      // whole warps past the end
  const bool have = v < in.n;
  double x[K][NG];
  int e[NG], sc[K];
#pragma unroll
  for (int q = 0; q < NG; ++q) e[q] = 0;
#pragma unroll
  for (int j = 0; j < K; ++j) sc[j] = k0 + j * G < N ? in.sc.s[k0 + j * G] : 0;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const int k = k0 + j * G;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      x[j][q] = have && k < N ? fx_in(in, v, ((size_t)v * NG + q) * N + k, k) : 0.0;
      const int ek = fx_exp(x[j][q]);
      e[q] = max(e[q], ek == 0 || ek == 2047 ? ek : min(max(ek + sc[j], 1), 2046));
    }
  }
  if (mix.on) {
#pragma unroll
    for (int q = 1; q < NG; ++q) e[0] = max(e[0], e[q]);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) e[0] = max(e[0], __shfl_xor_sync(0xffffffffu, e[0], o));
    if (!have) return;
    // exponents: of the columns before mixing where that takes the binary64 path (2047), else mixed
    const bool ok = fx_ok(e[0]) && fx_ok(mix.e);
#pragma unroll
    for (int q = 0; q < NG; ++q)
      if (k0 == q % G) in.e[v * NG + q] = (uint16_t)(e[0] == 0 ? 0 : ok ? e[0] : 2047);
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const int k = k0 + j * G;
      if (k >= N) continue;
      int2 w[NG];
#pragma unroll
      for (int q = 0; q < NG; ++q) w[q] = fx_limbs_x(x[j][q], (e[0] ? e[0] : kFxMinExp) - sc[j]);
#pragma unroll
      for (int q = 0; q < NG; ++q) {          // (T x)_q, below 5 2^122: its leading bits fit in 61
        FxAcc T{};
#pragma unroll
        for (int b = 0; b < NG; ++b) fx_mad1(make_int2(mix.h[q * NG + b], mix.l[q * NG + b]), w[b], T);
        const FxSum u = fx_sum(T, NG);        // 2^-37 of the sum of the products: 27 bits less are 2^-64
        in.w[((size_t)v * NG + q) * N + k] =
            fx_split((long long)((unsigned long long)__funnelshift_r(u.b, u.c, 27) << 32 | __funnelshift_r(u.a, u.b, 27)));
      }
    }
  } else {
#pragma unroll
    for (int q = 0; q < NG; ++q) {
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) e[q] = max(e[q], __shfl_xor_sync(0xffffffffu, e[q], o));
    }
    if (!have) return;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      if (k0 == q % G) in.e[v * NG + q] = (uint16_t)(fx_ok(e[q]) ? e[q] : 2047);
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const int k = k0 + j * G;
        if (k < N) in.w[((size_t)v * NG + q) * N + k] = fx_limbs_x(x[j][q], (e[q] ? e[q] : kFxMinExp) - sc[j]);
      }
    }
  }
}

template <class P, int N, int NG>
__global__ void __launch_bounds__(FxTile<P, N, NG>::threads, FxTile<P, N, NG>::blocks) k_fx(const __grid_constant__ P a,
                                                                                         const __grid_constant__ FxInput in,
                                                                                         const __grid_constant__ FxMat mix) {
  using T = FxTile<P, N, NG>;
  constexpr int TB = T::TB, NC = T::NC, NS = T::NS, NX = T::NX, NT = T::threads, C = P::C;
  extern __shared__ __align__(16) unsigned char fxs[];
  int2* xs = reinterpret_cast<int2*>(fxs);                        // [unit][set][column][NX]
  int2* stage = reinterpret_cast<int2*>(fxs + T::xs);             // [unit][slot][N][NS]
  constexpr int kRed = TB * P::SLOTS * NC * N;
  long long* redl = reinterpret_cast<long long*>(fxs);            // [unit][slot][column][N]: low 64 bits of the sums
  int* redh = reinterpret_cast<int*>(redl + kRed);                // and the high 32
  __shared__ int ex[TB][P::SETS][NC];                             // exponents of the vector columns
  __shared__ int slow[TB];                                        // the unit takes the binary64 path
  __shared__ int es[TB][P::SLOTS];                                // exponents of the blocks (0: absent or zero)
  __shared__ double us[TB];
  const int t = threadIdx.x, u0 = blockIdx.x * TB;
  if (t < TB) slow[t] = 0;
  const int tl = t / T::per, sk = t - tl * T::per, sl = sk / (C * N), ck = sk - sl * C * N, cg = ck / N, k0 = ck - cg * N;
  const int u = u0 + tl;
  const bool act = tl < TB && u < a.n;
  FxSlot m{nullptr, 0, false};
  if (act) m = a.template mat<N>(u, sl);
  const bool have = m.m != nullptr;
  if constexpr (P::STAGED) {
    // the threads of a slot copy its block: column k0, the rows dealt to the components
    if (have) {
      int2* st = stage + (size_t)(tl * P::SLOTS + sl) * N * NS + k0;
#pragma unroll 5
      for (int j = cg; j < N; j += C) cp_async<8>(st + j * NS, m.m + j * N + k0);
    }
  }
  if (act && ck == 0) {
    es[tl][sl] = have ? m.e : 0;
    if (sl == 0) us[tl] = a.unit_scale(u);
  }
  __syncthreads();                                     // slow is clear
  if (have && ck == 0 && !fx_ok(m.e)) slow[tl] = 1;
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the limbs are complete
  // the vectors: a thread copies its row of its component's NG columns (one slot of each set)
  if (act && P::copies(sl)) {
    const int set = P::set_of(sl), v = a.vec(u, set, cg);
    int2* xd = xs + ((size_t)(tl * P::SETS + set) * NC + cg * NG) * NX;
    if (v >= 0) {
      const int2* src = in.w + (size_t)v * NG * N;
#pragma unroll
      for (int q = 0; q < NG; ++q) cp_async<8>(xd + q * NX + k0, src + q * N + k0);
    }
    if (k0 == 0) {
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const int e = v >= 0 ? in.e[v * NG + q] : 0;
        ex[tl][set][cg * NG + q] = e;
        if (e == 2047) slow[tl] = 1;
      }
    }
  }
  cp_async_wait_all();
  __syncthreads();
  // products: row k of the slot's block with the NG columns of one component of the slot's vector
  const bool dbl = act && slow[tl] != 0;
  FxAcc acc[NG];
#pragma unroll
  for (int q = 0; q < NG; ++q) acc[q] = FxAcc{};
  if (have && !dbl) {
    const int2* xr = xs + ((size_t)(tl * P::SETS + P::set_of(sl)) * NC + cg * NG) * NX;
    const int2* mr = P::STAGED ? stage + (size_t)(tl * P::SLOTS + sl) * N * NS + k0 * (m.col ? 1 : NS) : m.m + k0;
    const int step = P::STAGED ? (m.col ? NS : 1) : N;           // along the sum
#pragma unroll (NG >= 4 ? 2 : 5)
    for (int l = 0; l + 1 < N; l += 2) {
      const int2 m0 = mr[l * step], m1 = mr[(l + 1) * step];
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const int4 v = *reinterpret_cast<const int4*>(xr + q * NX + l);
        fx_mad2(m0, make_int2(v.x, v.y), m1, make_int2(v.z, v.w), acc[q]);
      }
    }
    if constexpr (N & 1) {
      const int2 m0 = mr[(N - 1) * step];
#pragma unroll
      for (int q = 0; q < NG; ++q) fx_mad1(m0, xr[q * NX + N - 1], acc[q]);
    }
  }
  __syncthreads();                                     // the stage and the vectors are free
  const int rbase = ((tl * P::SLOTS + sl) * NC + cg * NG) * N;
  if (have && dbl) {                                   // binary64 multiply-adds (non-finite or tiny operands)
    const int v = a.vec(u, P::set_of(sl), cg);
#pragma unroll 1
    for (int q = 0; q < NG; ++q) {
      double s = 0.0;
#pragma unroll 1
      for (int l = 0; l < N; ++l) {
        double xc = 0.0;
        if (mix.on) {
          for (int b = 0; b < NG; ++b) xc = fma(mix.v[q * NG + b], fx_in(in, v, ((size_t)v * NG + b) * N + l, l), xc);
        } else {
          xc = fx_in(in, v, ((size_t)v * NG + q) * N + l, l);
        }
        s = fma(a.template entry<N>(u, sl, m.col ? l * N + k0 : k0 * N + l), xc, s);
      }
      redl[rbase + q * N + k0] = __double_as_longlong(s);
    }
  } else if (have) {
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const FxSum w = fx_sum(acc[q], (N + 1) / 2);
      redl[rbase + q * N + k0] = (long long)((unsigned long long)w.b << 32 | w.a);
      redh[rbase + q * N + k0] = (int)w.c;
    }
  }
  __syncthreads();
  // outputs: the slots of each group added with aligned exponents
  constexpr int per_out = P::GROUPS * NC * N;
  for (int o = t; o < TB * per_out; o += NT) {
    const int ol = o / per_out, rem = o - ol * per_out, g = rem / (NC * N), c = rem / N % NC, ok = rem % N;
    const int ou = u0 + ol;
    if (ou >= a.n) continue;
    const int rp = (ol * P::SLOTS * NC + c) * N + ok;
    double v;
    if (slow[ol]) {
      v = 0.0;
      for (int s = 0; s < P::SLOTS; ++s)
        if (P::group_of(s) == g && es[ol][s] > 0) v += __longlong_as_double(redl[rp + s * NC * N]);
    } else {
      // the exponent of each slot's sum, -1 where it is absent or zero
      constexpr int SG = P::SLOTS / P::GROUPS;
      int se[SG], top = 0;
#pragma unroll
      for (int j = 0; j < SG; ++j) {
        const int s = P::slot_of(g, j), be = es[ol][s], xe = ex[ol][P::set_of(s)][c];
        se[j] = be > 0 && xe > 0 ? be + xe : -1;
        top = max(top, se[j]);
      }
      FxSum sum{0, 0, 0};
#pragma unroll
      for (int j = 0; j < SG; ++j) {
        if (se[j] < 0) continue;
        const int p = rp + P::slot_of(g, j) * NC * N;
        const unsigned long long lo = (unsigned long long)redl[p];
        fx_add(sum, FxSum{(uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)redh[p]}, top - se[j]);
      }
      v = fx_value(sum, fx_unit(top, (mix.on ? mix.e - 1019 : 0) + a.out_scale().s[ok]));
    }
    a.template store<N, NG>(ou, g, c / NG, c % NG, ok, v, us[ol]);
  }
}

template <class P, int N, int NG>
cudaError_t fx_launch_t(const P& a, const FxInput& in, const FxMat& mix, cudaStream_t st) {
  using T = FxTile<P, N, NG>;
  if (a.n <= 0) return cudaSuccess;
  if (T::smem > 40 * 1024) {                  // with the static part above the 48 KB that need no opt-in
    const cudaError_t e = cudaFuncSetAttribute(k_fx<P, N, NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::smem);
    if (e != cudaSuccess) return e;
  }
  // (errors as the launches return them: asking for CUDA's last error between the two delayed the second by a
  // microsecond)
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(((int64_t)in.n * FxLanes<N>::G + 255) / 256));
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  const cudaError_t ev = cudaLaunchKernelEx(&cfg, k_fx_vec<N, NG>, in, mix);
  if (ev != cudaSuccess) return ev;
  cfg.gridDim = dim3((a.n + T::TB - 1) / T::TB);
  cfg.blockDim = dim3(T::threads);
  cfg.dynamicSmemBytes = T::smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_fx<P, N, NG>, a, in, mix);
}
template <class P, int N>
cudaError_t fx_launch_n(int Ng, const P& a, const FxInput& in, const FxMat& mix, cudaStream_t st) {
  switch (Ng) {
    case 1: return fx_launch_t<P, N, 1>(a, in, mix, st);
    case 2: return fx_launch_t<P, N, 2>(a, in, mix, st);
    case 3: return fx_launch_t<P, N, 3>(a, in, mix, st);
    case 4: return fx_launch_t<P, N, 4>(a, in, mix, st);
    case 5: return fx_launch_t<P, N, 5>(a, in, mix, st);
  }
  return cudaErrorInvalidValue;
}
// x: the input, nvec vectors, sc the scaling of its rows; ws: room for its limbs and exponents
template <class P>
cudaError_t fx_launch(int N, int Ng, const P& a, const double* x, int nvec, const FxScale& sc, const FxWork& ws, int pinned,
                      const FxMat& mix, cudaStream_t st) {
  const FxInput in{sc, x, static_cast<int2*>(ws.w), ws.e, nvec, pinned};
  if (!in.w || !in.e || (int64_t)nvec > ws.nvec) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lock(*ws.order);
  ++*ws.launches;
  switch (N) {
    case 1: return fx_launch_n<P, 1>(Ng, a, in, mix, st);
    case 4: return fx_launch_n<P, 4>(Ng, a, in, mix, st);
    case 10: return fx_launch_n<P, 10>(Ng, a, in, mix, st);
    case 20: return fx_launch_n<P, 20>(Ng, a, in, mix, st);
    case 35: return fx_launch_n<P, 35>(Ng, a, in, mix, st);
  }
  return cudaErrorInvalidValue;
}

// blocks of `len` binary64 entries to limbs in place, with their exponents; one warp per block
__global__ void __launch_bounds__(256) k_fx_encode(int64_t nblk, int len, int N, double* __restrict__ blocks,
                                                   uint16_t* __restrict__ exps, FxScale r, FxScale c) {
  const int lane = threadIdx.x & 31;
  for (int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; b < nblk;
       b += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    double* p = blocks + b * len;
    int e = 0;
    for (int o = lane; o < len; o += 32) {
      p[o] = scalbn(p[o], -(r.s[o / N % N] + c.s[o % N]));
      e = max(e, fx_exp(p[o]));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) exps[b] = (uint16_t)e;
    for (int o = lane; o < len; o += 32) reinterpret_cast<int2*>(p)[o] = fx_encode(p[o], e);
  }
}
__global__ void __launch_bounds__(256) k_fx_decode(int64_t first, int64_t n, int len, int N, const __grid_constant__ FxBlocks in,
                                                   double* __restrict__ out) {
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < n; o += (int64_t)gridDim.x * blockDim.x)
    out[o] = fx_entry(in, len, (first + o) / len, (int)((first + o) % len), N);
}
// top[l]: largest exponent of the diagonal entries (l, l) of the blocks B
__global__ void __launch_bounds__(256) k_fx_diag(int64_t ne, int N, const double* __restrict__ B, int* top) {
  __shared__ int m[kMaxN];
  if (threadIdx.x < kMaxN) m[threadIdx.x] = 0;
  __syncthreads();
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < ne * N; o += (int64_t)gridDim.x * blockDim.x) {
    const int l = (int)(o % N);
    atomicMax(&m[l], fx_exp(B[o / N * N * N + l * N + l]));
  }
  __syncthreads();
  if (threadIdx.x < N) atomicMax(&top[threadIdx.x], m[threadIdx.x]);
}
// top[m]: largest exponent in row m of the nq blocks Q with their columns scaled by c
__global__ void __launch_bounds__(256) k_fx_rows(int64_t nq, int N, const double* __restrict__ Q, FxScale c, int* top) {
  __shared__ int m[kMaxN];
  if (threadIdx.x < kMaxN) m[threadIdx.x] = 0;
  __syncthreads();
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < nq * N; o += (int64_t)gridDim.x * blockDim.x) {
    int e = 0;
    for (int l = 0; l < N; ++l) {
      const int el = fx_exp(Q[o * N + l]);
      if (el != 0 && el != 2047) e = max(e, el - c.s[l]);
    }
    atomicMax(&m[o % N], e);
  }
  __syncthreads();
  if (threadIdx.x < N) atomicMax(&top[threadIdx.x], m[threadIdx.x]);
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
    const long long w = std::llrint(std::ldexp(v[q], kFx - E));        // |w| <= 2^kFx
    const long long h = (w + (1LL << (kFxL - 1))) >> kFxL;
    m.h[q] = (int)h;
    m.l[q] = (int)(w - h * (1LL << kFxL));
  }
  return m;
}

}  // namespace

cudaError_t launch_fx_encode(int64_t nblk, int len, int N, double* blocks, uint16_t* exps, const FxScale& r,
                             const FxScale& c, cudaStream_t st) {
  if (nblk > 0) k_fx_encode<<<1216, 256, 0, st>>>(nblk, len, N, blocks, exps, r, c);
  return cudaGetLastError();
}
cudaError_t launch_fx_decode(int64_t first, int64_t n, int len, int N, const FxBlocks& in, double* out, cudaStream_t st) {
  if (n > 0) k_fx_decode<<<1216, 256, 0, st>>>(first, n, len, N, in, out);
  return cudaGetLastError();
}

cudaError_t fx_scales(int64_t ne, int64_t nq, int N, const double* B, const double* Q, int* top, FxScale* s, FxScale* t,
                      cudaStream_t st) {
  int h[kMaxN];
  // exponents relative to the largest, halved for the diagonal (a diagonal entry is a sum of squares)
  auto fetch = [&](const int* from, int div, FxScale* out) {
    cudaError_t e = cudaMemcpyAsync(h, from, N * sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    int big = 0;
    for (int l = 0; l < N; ++l)
      if (h[l] < 2047) big = std::max(big, h[l]);
    *out = FxScale{};
    for (int l = 0; l < N; ++l)
      if (h[l] > 0 && h[l] < 2047) out->s[l] = (signed char)std::max(-60, (h[l] - big) / div);
    return e;
  };
  cudaError_t e = cudaMemsetAsync(top, 0, 2 * N * sizeof(int), st);
  if (e != cudaSuccess) return e;
  k_fx_diag<<<304, 256, 0, st>>>(ne, N, B, top);
  if ((e = cudaGetLastError()) != cudaSuccess || (e = fetch(top, 2, s)) != cudaSuccess) return e;
  k_fx_rows<<<1216, 256, 0, st>>>(nq, N, Q, *s, top + N);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return fetch(top + N, 1, t);
}

cudaError_t launch_apply(const ApplyArgs& a, const double* x, double* y, cudaStream_t st) {
  FxApply p{};
  p.n = a.ne;
  p.gface = reinterpret_cast<const int4*>(a.gface); p.gnbr = reinterpret_cast<const int4*>(a.gnbr);
  p.B = a.B; p.A = a.A; p.detJ = a.detJ;
  p.x = x; p.y = y;
  p.scale = a.scale; p.mass_coef = a.mass_coef; p.pin_diag = a.pin_diag; p.pinned = a.pinned;
  p.unscaled = a.scale == 1.0 ? 1 : a.scale == -1.0 ? -1 : 0;
  p.mass = a.mass_coef != 0.0;
  for (int q = 0; q < a.Ng * a.Ng; ++q) p.K[q] = a.Kmass[q];
  return fx_launch(a.N, a.Ng, p, x, a.ne, a.B.c, a.ws, a.pinned, a.tacc_identity ? FxMat{} : fx_mat(a.Tacc, a.Ng), st);
}

cudaError_t launch_rhs(const FaceOps& f, const double* F, double coef, int pinned, double* b, cudaStream_t st) {
  FxRhs p{};
  p.n = f.ne; p.tface = reinterpret_cast<const int4*>(f.tface); p.Q = f.Q; p.b = b; p.coef = coef; p.pinned = pinned;
  return fx_launch(f.N, f.Ng, p, F, 3 * f.nf, f.Q.r, f.ws, 0, FxMat{}, st);
}

cudaError_t launch_update(const FaceOps& f, const double* F, const double* dp, double dt, const double* Kinv, double* V,
                          cudaStream_t st) {
  FxFace p{};
  p.n = f.nf; p.left = f.left; p.right = f.right; p.Q = f.Q; p.dt = dt; p.in = F; p.out = V;
  return fx_launch(f.N, f.Ng, p, dp, f.ne, f.Q.c, f.ws, 0, fx_mat(Kinv, f.Ng), st);
}
cudaError_t launch_face_grad(const FaceOps& f, const double* P, double dt, const double* Kinv, double* G, cudaStream_t st) {
  FxFace p{};
  p.n = f.nf; p.left = f.left; p.right = f.right; p.Q = f.Q; p.dt = dt; p.grad = 1; p.out = G;
  return fx_launch(f.N, f.Ng, p, P, f.ne, f.Q.c, f.ws, 0, fx_mat(Kinv, f.Ng), st);
}

cudaError_t launch_average(const FaceOps& f, const double* detJ, const double* in, double* out, cudaStream_t st) {
  FxAverage p{};
  p.n = f.ne; p.tface = reinterpret_cast<const int4*>(f.tface); p.M = f.Mij; p.detJ = detJ; p.out = out;
  return fx_launch(f.N, f.Ng, p, in, 3 * f.nf, f.Mij.c, f.ws, 0, FxMat{}, st);
}
cudaError_t launch_goback(const FaceOps& f, const double* vbar, const double* Vbc, double* F, cudaStream_t st) {
  FxGoback p{};
  p.n = f.nf; p.ne = f.ne; p.left = f.left; p.right = f.right; p.M = f.Mij; p.Vbc = Vbc; p.F = F;
  return fx_launch(f.N, f.Ng, p, vbar, 3 * f.ne, f.Mij.r, f.ws, 0, FxMat{}, st);
}

// One launch for the blocks of p <= 1, where two launches are what k_fx costs (750 tets, p = 1, p_t = 0: 18.0 ->
// 14.4 us); a block per face, binary64 multiply-adds, the face's blocks decoded to shared memory.
__global__ void __launch_bounds__(128) k_moments_small(int N, int Ng, const __grid_constant__ FxBlocks M,
                                                       const double* __restrict__ V, double dt, double* __restrict__ U) {
  __shared__ double Ms[2 * 16];
  const int j = blockIdx.x, Nst = N * Ng, NN = N * N;
  for (int e = threadIdx.x; e < 2 * NN; e += 128) Ms[e] = fx_entry(M, NN, 2 * (size_t)j + e / NN, e % NN, N);
  __syncthreads();
  for (int o = threadIdx.x; o < 6 * Nst; o += 128) {
    const int s = o / (3 * Nst), rem = o - s * 3 * Nst, k = rem % N;
    const double* v = V + (size_t)j * 3 * Nst + rem - k;
    double acc = 0.0;
    for (int l = 0; l < N; ++l) acc = fma(Ms[s * NN + k * N + l], v[l], acc);
    U[(size_t)j * 6 * Nst + o] = dt * acc;
  }
}
cudaError_t launch_moments(const FaceOps& f, const double* V, double dt, double* U, cudaStream_t st) {
  if (f.N <= 4) {
    if (f.nf > 0) k_moments_small<<<f.nf, 128, 0, st>>>(f.N, f.Ng, f.Mij, V, dt, U);
    return cudaGetLastError();
  }
  FxMoments p{};
  p.n = f.nf; p.right = f.right; p.M = f.Mij; p.U = U; p.dt = dt;
  return fx_launch(f.N, f.Ng, p, V, 3 * f.nf, f.Mij.c, f.ws, 0, FxMat{}, st);
}

}  // namespace stdg
