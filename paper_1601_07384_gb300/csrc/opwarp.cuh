// Warp-per-tet five-point operator kernel template (shared by the per-policy translation units).
#pragma once
#include <cuda_bf16.h>

#include <type_traits>

#include "lp_ptx.cuh"
#include "solver.h"

namespace stdg {

constexpr long kWarpSpin = 20000;   // x <= 1 ms suspend per try_wait

struct WF32 { using TB = float; using XIn = float; using YOut = float; using Real = float; static constexpr int kPlanes = 1; };
struct WBF16 { using TB = __nv_bfloat16; using XIn = float; using YOut = float; using Real = float; static constexpr int kPlanes = 1; };
struct WDF { using TB = float; using XIn = double; using YOut = double; using Real = double; static constexpr int kPlanes = 2; };

struct WarpArgs {
  int ne, N, NR, NP, Nst, S, pinned, kron;
  const int4* gface;            // per tet: (face << 1 | tet is r) or -1, 4 faces
  const int4* gnbr;             // per tet: neighbour tet or -1
  const void* Bd;               // diagonal blocks, padded layout
  const void* Ao;               // face blocks A_lr, padded layout
  uint32_t blk_bytes;           // one padded block (all planes)
  uint32_t plane_elems;         // NR * NP
  uint32_t xraw_off, stage_bytes, z_off, bar_off, warp_bytes;
  double scale, pin_diag;
  double Tacc[kMaxNg * kMaxNg];
  // viscous operator (Eq. A1_mod): + mass_coef |J_i| (K (x) I) x_i, exact in the input precision
  const double* detJ;
  double mass_coef;
  double Kmass[kMaxNg * kMaxNg];
  double* dotpart;              // optional: per block and column, Sum of x_i . y_i over its tets
  int* err;
};

// four consecutive entries of a row (element index idx, a multiple of 4)
__device__ __forceinline__ void load_row4(const float* B, int idx, float (&b)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(B + idx);
  b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
}
__device__ __forceinline__ void load_row4(const __nv_bfloat16* B, int idx, float (&b)[4]) {
  const uint2 v = *reinterpret_cast<const uint2*>(B + idx);
  b[0] = __uint_as_float(v.x << 16); b[1] = __uint_as_float(v.x & 0xFFFF0000u);
  b[2] = __uint_as_float(v.y << 16); b[3] = __uint_as_float(v.y & 0xFFFF0000u);
}
__device__ __forceinline__ float load_one(const float* B, int idx) { return B[idx]; }
__device__ __forceinline__ float load_one(const __nv_bfloat16* B, int idx) { return __bfloat162float(B[idx]); }

__host__ __device__ constexpr int warp_np_c(int N) { return N % 8 == 4 ? N : warp_np_c(N + 1); }
__host__ __device__ constexpr int warp_nr_c(int N) { return (N + 3) / 4 * 4; }

// Binary64-accurate multiply-add from binary32 pairs, (h, l) += (bh + bl)(zh + zl) with the bl zl
// term (relative size 2^-48) left out: the product bh zh split exactly by a fused multiply-add, its
// high part added to h by an error-free sum.  Two independent accumulators at once (the halves of
// the float2 values), in packed binary32 operations (f32x2, sm_100 and later).  nbh = -bh, formed
// once per chunk: pn = nbh zh is the rounded product negated exactly, so no negation per product.
__device__ __forceinline__ void df_fma2(float2& h, float2& l, float2 bh, float2 nbh, float2 bl, float2 zh, float2 zl) {
  const float2 pn = __fmul2_rn(nbh, zh);
  float2 e = __ffma2_rn(bh, zh, pn);              // bh zh - p, exact
  e = __ffma2_rn(bh, zl, e);
  e = __ffma2_rn(bl, zh, e);
  float2 s, t;
  df_two_diff2(h, pn, s, t);                      // h + p = h - pn, error-free
  h = s;
  l = __fadd2_rn(l, __fadd2_rn(t, e));
}

// pair policy: four entries of a block row (stride 1: vector loads of the hi and lo planes) or
// column (stride NP) times the matching z entries; entries (0, 1) and (2, 3) through the two halves
// of (h, l), one accumulator pair per time column
template <int NG, typename TB>
__device__ __forceinline__ void warp_chunk_df2(const TB* B, int stride, uint32_t plane, const float* z, int NR,
                                               int zplane, float2 (&h)[NG], float2 (&l)[NG]) {
  float bh[4], bl[4];
  if (stride == 1) {
    load_row4(B, 0, bh);
    load_row4(B + plane, 0, bl);
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      bh[u] = load_one(B, u * stride);
      bl[u] = load_one(B + plane, u * stride);
    }
  }
  const float2 bh01 = make_float2(bh[0], bh[1]), bh23 = make_float2(bh[2], bh[3]);
  const float2 nb01 = make_float2(-bh[0], -bh[1]), nb23 = make_float2(-bh[2], -bh[3]);
  const float2 bl01 = make_float2(bl[0], bl[1]), bl23 = make_float2(bl[2], bl[3]);
#pragma unroll
  for (int q = 0; q < NG; ++q) {
    const float4 zh = *reinterpret_cast<const float4*>(z + q * NR);
    const float4 zl = *reinterpret_cast<const float4*>(z + zplane + q * NR);
    df_fma2(h[q], l[q], bh01, nb01, bl01, make_float2(zh.x, zh.y), make_float2(zl.x, zl.y));
    df_fma2(h[q], l[q], bh23, nb23, bl23, make_float2(zh.z, zh.w), make_float2(zl.z, zl.w));
  }
}

// binary32 policies: the same four-entry chunk with packed multiply-adds, entries (0, 1) and (2, 3)
// in the two halves of one float2 accumulator per time column (fma.rn.f32x2: half the issue slots of
// four scalar multiply-adds, the same binary32 rounding)
template <int NG, typename TB>
__device__ __forceinline__ void warp_chunk2(const TB* B, int stride, const float* z, int NR, float2 (&acc)[NG]) {
  float b[4];
  if (stride == 1) {
    load_row4(B, 0, b);
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) b[u] = load_one(B, u * stride);
  }
  const float2 b01 = make_float2(b[0], b[1]), b23 = make_float2(b[2], b[3]);
#pragma unroll
  for (int q = 0; q < NG; ++q) {
    const float4 zv = *reinterpret_cast<const float4*>(z + q * NR);
    acc[q] = __ffma2_rn(b01, make_float2(zv.x, zv.y), acc[q]);
    acc[q] = __ffma2_rn(b23, make_float2(zv.z, zv.w), acc[q]);
  }
}

// One warp per tet, persistent over a strided stream of tets.  Lane 0 stages the tet's five blocks
// (its diagonal block and the face blocks of its interior faces) by 1-D TMA bulk copies; all lanes
// stage the x rows of the tet and its neighbours by cp.async.  binary32 x goes straight into rows of
// NR entries ([slot][time column][NR], the padding entries zeroed once and never written), the layout
// the products read; binary64 x (pair policy) is split into (hi, lo) planes of the same layout.
// Rows 0..31 of the output: lane k owns row k over all five blocks and all time columns.  Rows
// 32..N-1 (N = 35 at p = 4): one group of 8 lanes per row, each lane summing its share of the four-
// entry chunks, the group reduced by shuffles at the end.  No block-wide barrier anywhere.
template <typename W, int NG, int NC>
__global__ void __launch_bounds__(128, 1) k_apply_warp(WarpArgs a, const typename W::XIn* __restrict__ x,
                                                    typename W::YOut* __restrict__ y) {
  using TB = typename W::TB;
  using XIn = typename W::XIn;
  using Real = typename W::Real;
  constexpr bool kDF = W::kPlanes == 2;
  constexpr bool kRoll = kDF && (NC == 0 || NC > 20);   // large pair kernels: rolled loops
  constexpr bool kPrefetch = kRoll;                     // there: the blocks two tets ahead go to L2 (measured
                                                        // slower for the binary32 kernel)
  extern __shared__ __align__(128) unsigned char wsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpc = blockDim.x >> 5;
  unsigned char* base = wsm + (size_t)warp * a.warp_bytes;
  float* zs = reinterpret_cast<float*>(base + a.z_off);        // pair policy: (hi, lo) planes of z
  uint64_t* bar = reinterpret_cast<uint64_t*>(base + a.bar_off);
  // NC != 0: N known at compile time (row loops fully unrolled, shared-memory offsets immediate)
  const int N = NC ? NC : a.N, NR = NC ? warp_nr_c(NC) : a.NR, NP = NC ? warp_np_c(NC) : a.NP;
  const int Nst = NC ? NC * NG : a.Nst, S = a.S;
  // kernel parameters in the arithmetic type, converted once (a binary64 conversion or compare per
  // output row would go through the 1/64-rate binary64 pipe)
  const Real scale = (Real)a.scale;
  const bool has_mass = a.mass_coef != 0.0, kron = a.kron != 0, pinned = a.pinned != 0;
  Real tacc[NG * NG];
#pragma unroll
  for (int c = 0; c < NG * NG; ++c) tacc[c] = (Real)a.Tacc[c];
  const int zplane = 5 * NG * NR;
  if constexpr (kDF) {
    for (int e = lane; e < 2 * zplane; e += 32) zs[e] = 0.0f;            // padding entries stay 0
  } else {
    for (int st = 0; st < S; ++st) {
      float* xz = reinterpret_cast<float*>(base + (size_t)st * a.stage_bytes + a.xraw_off);
      for (int e = lane; e < zplane; e += 32) xz[e] = 0.0f;
    }
  }
  if (lane == 0) {
    for (int s = 0; s < S; ++s) mbar_init(&bar[s], 33);   // lane 0's expect_tx + 32 cp.async arrivals
    fence_async_smem();
  }
  __syncwarp();

  auto issue = [&](int i, int st, const int4& gf, const int4& gn) {
    unsigned char* sb = base + (size_t)st * a.stage_bytes;
    XIn* xr = reinterpret_cast<XIn*>(sb + a.xraw_off);
    const int fj[4] = {gf.x, gf.y, gf.z, gf.w};
    const int nn[4] = {gn.x, gn.y, gn.z, gn.w};
    if (lane == 0) {
      uint32_t bytes = a.blk_bytes;
#pragma unroll
      for (int f = 0; f < 4; ++f)
        if (fj[f] >= 0) bytes += a.blk_bytes;
      fence_async_smem();                         // earlier generic reads of this stage before the copies
      mbar_expect_tx(&bar[st], bytes);
      tma_load_1d(sb, static_cast<const unsigned char*>(a.Bd) + (size_t)i * a.blk_bytes, a.blk_bytes, &bar[st]);
#pragma unroll
      for (int f = 0; f < 4; ++f)
        if (fj[f] >= 0)
          tma_load_1d(sb + (size_t)(f + 1) * a.blk_bytes,
                      static_cast<const unsigned char*>(a.Ao) + (size_t)(fj[f] >> 1) * a.blk_bytes, a.blk_bytes,
                      &bar[st]);
    }
#pragma unroll
    for (int sl = 0; sl < 5; ++sl) {
      const int nb = sl == 0 ? i : (fj[sl - 1] >= 0 ? nn[sl - 1] : -1);
      if (nb < 0) continue;
      const XIn* src = x + (size_t)nb * Nst;
      if constexpr (kDF) {
        for (int o = lane; o < Nst; o += 32) cp_async<sizeof(XIn)>(xr + sl * Nst + o, src + o);
      } else {
#pragma unroll
        for (int q = 0; q < NG; ++q)
          for (int l = lane; l < N; l += 32) cp_async<sizeof(XIn)>(xr + (sl * NG + q) * NR + l, src + q * N + l);
      }
    }
    cp_async_mbar_arrive_noinc(&bar[st]);
  };

  const int nw = gridDim.x * wpc;
  float dacc[NG];                                 // x_i . y_i of this lane's rows (dotpart)
#pragma unroll
  for (int q = 0; q < NG; ++q) dacc[q] = 0.0f;
  int i = blockIdx.x * wpc + warp;
  const int4 none = make_int4(-1, -1, -1, -1);
  int4 gf_c = none, gn_c = none, gf_n = none, gn_n = none;
  // iteration it uses stage it % S in its use number it / S (mbarrier phase parity (it / S) & 1)
  bool abort = false, next_issued = false;
  int it = 0;
  if (i < a.ne) {
    gf_c = a.gface[i]; gn_c = a.gnbr[i];
    issue(i, 0, gf_c, gn_c);
    if (S == 2 && i + nw < a.ne) { gf_n = a.gface[i + nw]; gn_n = a.gnbr[i + nw]; }
  }
  for (; i < a.ne; i += nw, ++it) {
    const int st = S == 2 ? (it & 1) : 0;
    const int inx = i + nw;
    const int4 gf = gf_c, gn = gn_c;
    next_issued = false;
    if (S == 2 && inx < a.ne) {                   // next tet's copies run while this one computes
      issue(inx, st ^ 1, gf_n, gn_n);
      next_issued = true;
      gf_c = gf_n; gn_c = gn_n;
      if (inx + nw < a.ne) { gf_n = a.gface[inx + nw]; gn_n = a.gnbr[inx + nw]; }
    }
    {                                             // warp_wait_gave_up written out: as a call it takes 26 registers
      long spins = 0;                             // more at Ng = 5 (bfloat16, N = 20: 170 -> 196), and fewer warps fit
      const uint32_t par = (uint32_t)((it / S) & 1);
      while (!mbar_wait_hint(&bar[st], par))
        if (++spins > kWarpSpin) { abort = true; break; }
    }
    if (__any_sync(0xffffffffu, abort)) { abort = true; break; }
    __syncwarp();
    if (kPrefetch && lane == 0 && i + S * nw < a.ne) {   // the blocks after the next staged tet: towards L2
      const int ip = i + S * nw;
      const int4 gp = a.gface[ip];
      const int fp[4] = {gp.x, gp.y, gp.z, gp.w};
      bulk_prefetch_l2(static_cast<const unsigned char*>(a.Bd) + (size_t)ip * a.blk_bytes, a.blk_bytes);
#pragma unroll
      for (int f = 0; f < 4; ++f)
        if (fp[f] >= 0)
          bulk_prefetch_l2(static_cast<const unsigned char*>(a.Ao) + (size_t)(fp[f] >> 1) * a.blk_bytes, a.blk_bytes);
    }
    unsigned char* sb = base + (size_t)st * a.stage_bytes;
    XIn* xr = reinterpret_cast<XIn*>(sb + a.xraw_off);
    const int fj[4] = {gf.x, gf.y, gf.z, gf.w};
    const int nn[4] = {gn.x, gn.y, gn.z, gn.w};
    // pinned entries (constant mode of tet 0, every time column) read as 0
    if constexpr (kDF) {
#pragma unroll
      for (int sl = 0; sl < 5; ++sl) {
        const int nb = sl == 0 ? i : (fj[sl - 1] >= 0 ? nn[sl - 1] : -1);
        if (nb < 0) continue;
#pragma unroll
        for (int q = 0; q < NG; ++q)
          for (int l = lane; l < N; l += 32) {
            XIn v = xr[sl * Nst + q * N + l];
            if (pinned && nb == 0 && l == 0) v = (XIn)0;
            const float2 hl = df_split(v);
            float* zq = zs + (sl * NG + q) * NR + l;
            zq[0] = hl.x;
            zq[zplane] = hl.y;
          }
      }
    } else if (pinned) {
#pragma unroll
      for (int sl = 0; sl < 5; ++sl) {
        const int nb = sl == 0 ? i : (fj[sl - 1] >= 0 ? nn[sl - 1] : -1);
        if (nb == 0 && lane < NG) xr[(sl * NG + lane) * NR] = (XIn)0;
      }
    }
    __syncwarp();
    const float* zb = kDF ? zs : reinterpret_cast<const float*>(xr);   // z rows [slot][q][NR]
    const TB* blk = reinterpret_cast<const TB*>(sb);
    const int blk_elems = (int)(a.blk_bytes / sizeof(TB));
    int pres = 1, trm = 0;                        // per slot: block present / read transposed
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      pres |= (fj[f] >= 0 ? 1 : 0) << (f + 1);
      trm |= (fj[f] >= 0 && (fj[f] & 1) ? 1 : 0) << (f + 1);
    }
    // output row k of tet i from its sums v over the five blocks: time mixing, scale, mass term,
    // pin, store, x.y partials
    auto finish = [&](int k, const Real (&v)[NG]) {
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        Real o = v[q];
        if (!kron) {
          o = 0;
#pragma unroll
          for (int b = 0; b < NG; ++b) o += tacc[q * NG + b] * v[b];
        }
        o *= scale;
        if (has_mass) {                           // x_i as staged (binary64 for the pair policy)
          Real m = 0;
#pragma unroll
          for (int b = 0; b < NG; ++b)
            m += (Real)a.Kmass[q * NG + b] * (Real)(kDF ? xr[b * N + k] : xr[b * NR + k]);
          o += (Real)(a.mass_coef * a.detJ[i]) * m;
        }
        if (pinned && i == 0 && k == 0) o = (Real)a.pin_diag * (Real)x[q * N];
        y[(size_t)i * Nst + q * N + k] = (typename W::YOut)o;
        if (a.dotpart) dacc[q] += (float)((Real)x[(size_t)i * Nst + q * N + k] * o);
      }
    };
    const int nmain = N < 32 ? N : 32;
    if (lane < nmain) {
      const int k = lane;
      float2 dh[NG], dl[NG];                      // pair policy: packed (hi, lo) accumulators per column
      float2 c0[NG], c1[NG];                      // binary32 policies: two packed accumulators per column
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        dh[q] = dl[q] = make_float2(0.0f, 0.0f);
        c0[q] = c1[q] = make_float2(0.0f, 0.0f);
      }
      // pair policy at N > 20 (about 200 instructions per chunk): the block and chunk loops stay rolled,
      // as fully unrolled code outgrows the instruction cache
      auto block_main = [&](int sl) {
        if (!((pres >> sl) & 1)) return;
        const TB* B = blk + sl * blk_elems;
        const float* z = zb + sl * NG * NR;
        if (!((trm >> sl) & 1)) {                 // row k of the block, 4 entries per vector load
          const TB* Br = B + k * NP;
#pragma unroll (kRoll ? 1 : 8)
          for (int l = 0; l < NR; l += 8) {
            if constexpr (kDF) {
              warp_chunk_df2<NG>(Br + l, 1, a.plane_elems, z + l, NR, zplane, dh, dl);
              if (l + 4 < NR) warp_chunk_df2<NG>(Br + l + 4, 1, a.plane_elems, z + l + 4, NR, zplane, dh, dl);
            } else {
              warp_chunk2<NG>(Br + l, 1, z + l, NR, c0);
              if (l + 4 < NR) warp_chunk2<NG>(Br + l + 4, 1, z + l + 4, NR, c1);
            }
          }
        } else {                                  // column k: A_rl = A_lr^T, one word per lane
          const TB* Bc = B + k;
#pragma unroll (kRoll ? 1 : 8)
          for (int l = 0; l < NR; l += 8) {
            if constexpr (kDF) {
              warp_chunk_df2<NG>(Bc + l * NP, NP, a.plane_elems, z + l, NR, zplane, dh, dl);
              if (l + 4 < NR) warp_chunk_df2<NG>(Bc + (l + 4) * NP, NP, a.plane_elems, z + l + 4, NR, zplane, dh, dl);
            } else {
              warp_chunk2<NG>(Bc + l * NP, NP, z + l, NR, c0);
              if (l + 4 < NR) warp_chunk2<NG>(Bc + (l + 4) * NP, NP, z + l + 4, NR, c1);
            }
          }
        }
      };
      if constexpr (kRoll) {
#pragma unroll 1
        for (int sl = 0; sl < 5; ++sl) block_main(sl);
      } else {
        for (int sl = 0; sl < 5; ++sl) block_main(sl);
      }
      Real v[NG];
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        if constexpr (kDF) {
          float s, t;
          df_two_sum(dh[q].x, dh[q].y, s, t);
          v[q] = (double)s + (double)(t + (dl[q].x + dl[q].y));   // the error terms are ~2^-24 of s
        } else {
          v[q] = (c0[q].x + c0[q].y) + (c1[q].x + c1[q].y);
        }
      }
      finish(k, v);
    }
    if (N > 32) {                                 // rows 32 .. N-1: 8 lanes per row, chunks split
      const int g = lane >> 3, c = lane & 7, r = 32 + g;
      const int nch = NR / 4;
      float2 eh[NG], el[NG], ec[NG];
#pragma unroll
      for (int q = 0; q < NG; ++q) eh[q] = el[q] = ec[q] = make_float2(0.0f, 0.0f);
      if (r < N) {
#pragma unroll (kRoll ? 1 : 5)
        for (int sl = 0; sl < 5; ++sl) {
          if (!((pres >> sl) & 1)) continue;
          const TB* B = blk + sl * blk_elems;
          const float* z = zb + sl * NG * NR;
          const bool tr = (trm >> sl) & 1;
          for (int ch = c; ch < nch; ch += 8) {
            const int l = 4 * ch;
            if constexpr (kDF) {
              if (!tr) warp_chunk_df2<NG>(B + r * NP + l, 1, a.plane_elems, z + l, NR, zplane, eh, el);
              else warp_chunk_df2<NG>(B + l * NP + r, NP, a.plane_elems, z + l, NR, zplane, eh, el);
            } else {
              if (!tr) warp_chunk2<NG>(B + r * NP + l, 1, z + l, NR, ec);
              else warp_chunk2<NG>(B + l * NP + r, NP, z + l, NR, ec);
            }
          }
        }
      }
      Real v[NG];
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        float h, e;
        if constexpr (kDF) {
          df_two_sum(eh[q].x, eh[q].y, h, e);
          e += el[q].x + el[q].y;
        } else {
          h = ec[q].x + ec[q].y;
          e = 0.0f;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {         // within the 8-lane group
          const float oh = __shfl_xor_sync(0xffffffffu, h, o), oe = __shfl_xor_sync(0xffffffffu, e, o);
          if constexpr (kDF) {
            float s, t;
            df_two_sum(h, oh, s, t);
            h = s;
            e = e + oe + t;
          } else {
            h += oh;
          }
        }
        if constexpr (kDF) v[q] = (double)h + (double)e;
        else v[q] = h;
      }
      if (c == 0 && r < N) finish(r, v);
    }
    __syncwarp();
    if (S == 1 && inx < a.ne) {                   // one stage: the next tet's copies start now
      gf_c = a.gface[inx]; gn_c = a.gnbr[inx];
      issue(inx, 0, gf_c, gn_c);
    }
  }
  if (a.dotpart) {                                // fixed order: lanes by shuffle, warps by index
    __shared__ float wdot[4][kMaxNg];
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      float v = dacc[q];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) wdot[warp][q] = v;
    }
    __syncthreads();                              // every warp of the block reaches this point
    if (threadIdx.x < NG) {
      double t = 0.0;
      for (int w = 0; w < wpc; ++w) t += (double)wdot[w][threadIdx.x];
      a.dotpart[(size_t)blockIdx.x * NG + threadIdx.x] = t;
    }
  }
  if (abort) {
    if (lane == 0) atomicExch(a.err, 1);
    // bounded wait for this warp's copies in flight: the stage of iteration it and, when it was
    // issued, the stage of iteration it + 1
    const int st = S == 2 ? (it & 1) : 0;
    long spins = 0;
    while (!mbar_wait_hint(&bar[st], (uint32_t)((it / S) & 1)) && ++spins < kWarpSpin) {
    }
    if (next_issued) {
      spins = 0;
      while (!mbar_wait_hint(&bar[st ^ 1], (uint32_t)(((it + 1) / S) & 1)) && ++spins < kWarpSpin) {
      }
    }
  }
}

// Five warps per tet, one per block, for the blocks of p = 4 in binary32 or bfloat16: a CTA runs a
// strided stream of tets with two stages, warp w staging and multiplying block w (0: the diagonal one).  The
// kernel with a warp per tet needs a stage of all five blocks per warp: 7 warps per SM at p = 4, too few to
// cover their own shared-memory latency and loads; here 15 at p = 4 with the next tet's blocks always in flight,
// and a fifth of the work between two waits.  One barrier per tet: after it the stage is free and the five
// partial rows are complete (two buffers of these, so that the sums of one tet and the products of the next
// overlap).
template <typename W, int NG, int N>
struct CtaDim {
  static constexpr int NR = warp_nr_c(N), NP = warp_np_c(N), T = 160;
  static_assert(N > 32 && N <= 35, "rows: one per lane and the rest in groups of 8 lanes");
  static constexpr uint32_t blk = (uint32_t)(NR * NP * sizeof(typename W::TB));
  static constexpr uint32_t xrow = (uint32_t)(NG * NR * sizeof(float));             // one slot's x
  static constexpr uint32_t stage = 5 * blk + 5 * xrow, red = 5 * NG * NR * sizeof(float);
  static constexpr uint32_t smem = 2 * stage + 2 * red + 16;
  static_assert(blk % 16 == 0 && xrow % 16 == 0 && red % 16 == 0, "bulk copies and vector loads");
};
template <typename W, int NG, int N>
__global__ void __launch_bounds__(160, 3) k_apply_cta(const __grid_constant__ WarpArgs a,
                                                                   const float* __restrict__ x, float* __restrict__ y) {
  using TB = typename W::TB;
  using D = CtaDim<W, NG, N>;
  constexpr int NR = D::NR, NP = D::NP, Nst = N * NG;
  extern __shared__ __align__(128) unsigned char wsm[];
  const int lane = threadIdx.x & 31, slot = threadIdx.x >> 5, G = gridDim.x;
  float* red = reinterpret_cast<float*>(wsm + 2 * D::stage);                       // [2][slot][q][NR]
  uint64_t* bar = reinterpret_cast<uint64_t*>(wsm + 2 * D::stage + 2 * D::red);
  for (int st = 0; st < 2; ++st) {
    float* xz = reinterpret_cast<float*>(wsm + st * D::stage + 5 * D::blk);
    for (int e = threadIdx.x; e < 5 * NG * NR; e += D::T) xz[e] = 0.0f;             // padding entries stay 0
  }
  // parameters in binary32, converted once (every binary64 conversion or compare takes 64 cycles per warp)
  __shared__ float tacc[NG * NG], kmass[NG * NG];
  const float scale = (float)a.scale;
  const bool has_mass = a.mass_coef != 0.0;
  if (threadIdx.x < NG * NG) {
    tacc[threadIdx.x] = (float)a.Tacc[threadIdx.x];
    kmass[threadIdx.x] = (float)a.Kmass[threadIdx.x];
  }
  if (threadIdx.x == 0) {
    for (int st = 0; st < 2; ++st) mbar_init(&bar[st], 5 + D::T);                   // five expect_tx, all cp.async arrivals
    fence_async_smem();
  }
  __syncthreads();
  // this warp's block of tet i: f = index << 1 | transposed, or -1; nb the tet whose x it multiplies
  auto fetch = [&](int i, int& f, int& nb) {
    f = -1; nb = -1;
    if (i >= a.ne) return;
    if (slot == 0) { f = i << 1; nb = i; return; }
    f = reinterpret_cast<const int*>(a.gface)[4 * (size_t)i + slot - 1];
    nb = reinterpret_cast<const int*>(a.gnbr)[4 * (size_t)i + slot - 1];
  };
  auto issue = [&](int st, int f, int nb) {
    unsigned char* sb = wsm + st * D::stage;
    if (lane == 0) {
      fence_async_smem();                         // earlier generic reads of this stage before the copy
      mbar_expect_tx(&bar[st], f >= 0 ? D::blk : 0);
      if (f >= 0)
        tma_load_1d(sb + slot * D::blk, static_cast<const unsigned char*>(slot == 0 ? a.Bd : a.Ao) + (size_t)(f >> 1) * D::blk,
                    D::blk, &bar[st]);
    }
    if (f >= 0) {
      float* xr = reinterpret_cast<float*>(sb + 5 * D::blk + slot * D::xrow);
      const float* src = x + (size_t)nb * Nst;
#pragma unroll
      for (int q = 0; q < NG; ++q)
        for (int l = lane; l < N; l += 32) cp_async<4>(xr + q * NR + l, src + q * N + l);
    }
    cp_async_mbar_arrive_noinc(&bar[st]);
  };
  float dacc[NG];
#pragma unroll
  for (int q = 0; q < NG; ++q) dacc[q] = 0.0f;
  int i = blockIdx.x, it = 0, f0, n0, f1, n1, f2, n2;
  bool abort = false;
  fetch(i, f0, n0);
  fetch(i + G, f1, n1);
  fetch(i + 2 * G, f2, n2);
  if (i < a.ne) issue(0, f0, n0);
  if (i + G < a.ne) issue(1, f1, n1);
  for (; i < a.ne; i += G, ++it) {
    const int st = it & 1;
    abort = warp_wait_gave_up(&bar[st], (uint32_t)(it >> 1) & 1, kWarpSpin);   // one path for the whole warp
    __syncwarp();
    float* rd = red + (st * 5 + slot) * NG * NR;
    if (!abort) {
      const TB* B = reinterpret_cast<const TB*>(wsm + st * D::stage + slot * D::blk);
      float* z = reinterpret_cast<float*>(wsm + st * D::stage + 5 * D::blk + slot * D::xrow);
      if (a.pinned && n0 == 0) {                  // the constant mode of tet 0 reads as 0
        if (lane < NG) z[lane * NR] = 0.0f;
        __syncwarp();
      }
      float2 c0[NG], c1[NG];
#pragma unroll
      for (int q = 0; q < NG; ++q) c0[q] = c1[q] = make_float2(0.0f, 0.0f);
      if (f0 >= 0) {                              // row `lane`
        if (f0 & 1) {                             // column: A_rl = A_lr^T
#pragma unroll
          for (int l = 0; l < NR; l += 8) {
            warp_chunk2<NG>(B + l * NP + lane, NP, z + l, NR, c0);
            if (l + 4 < NR) warp_chunk2<NG>(B + (l + 4) * NP + lane, NP, z + l + 4, NR, c1);
          }
        } else {
#pragma unroll
          for (int l = 0; l < NR; l += 8) {
            warp_chunk2<NG>(B + lane * NP + l, 1, z + l, NR, c0);
            if (l + 4 < NR) warp_chunk2<NG>(B + lane * NP + l + 4, 1, z + l + 4, NR, c1);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < NG; ++q) rd[q * NR + lane] = (c0[q].x + c0[q].y) + (c1[q].x + c1[q].y);
      const int g = lane >> 3, c = lane & 7, r = 32 + g;   // rows 32 .. 34: 8 lanes per row, chunks split
      float2 ec[NG];
#pragma unroll
      for (int q = 0; q < NG; ++q) ec[q] = make_float2(0.0f, 0.0f);
      if (f0 >= 0 && r < N) {
        for (int l = 4 * c; l < NR; l += 32) {
          if (f0 & 1) warp_chunk2<NG>(B + l * NP + r, NP, z + l, NR, ec);
          else warp_chunk2<NG>(B + r * NP + l, 1, z + l, NR, ec);
        }
      }
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        float h = ec[q].x + ec[q].y;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
        if (c == 0 && r < N) rd[q * NR + r] = h;
      }
    }
    if (__syncthreads_or(abort)) { abort = true; break; }
    // the stage is free: the tet after the next one
    if (i + 2 * G < a.ne) issue(st, f2, n2);
    f0 = f1; n0 = n1; f1 = f2; n1 = n2;
    fetch(i + 3 * G, f2, n2);
    const int k = threadIdx.x;
    if (k < N) {                                  // row k: the five sums, time mixing, scale, mass term, pin
      const float* rk = red + st * 5 * NG * NR + k;
      float v[NG];
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        v[q] = 0.0f;
#pragma unroll
        for (int sl = 0; sl < 5; ++sl) v[q] += rk[(sl * NG + q) * NR];
      }
      const float* xi = x + (size_t)i * Nst + k;
      const float mj = has_mass ? (float)(a.mass_coef * a.detJ[i]) : 0.0f;
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        float o = v[q];
        if (!a.kron) {
          o = 0.0f;
#pragma unroll
          for (int b = 0; b < NG; ++b) o += tacc[q * NG + b] * v[b];
        }
        o *= scale;
        if (has_mass) {
          float m = 0.0f;
#pragma unroll
          for (int b = 0; b < NG; ++b) m += kmass[q * NG + b] * xi[b * N];
          o += mj * m;
        }
        if (a.pinned && i == 0 && k == 0) o = (float)a.pin_diag * x[q * N];
        y[(size_t)i * Nst + q * N + k] = o;
        if (a.dotpart) dacc[q] += xi[q * N] * o;
      }
    }
  }
  if (a.dotpart) {                                // fixed order: lanes by shuffle, warps by index
    __shared__ float wdot[5][NG];
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      float v = dacc[q];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) wdot[slot][q] = v;
    }
    __syncthreads();
    if (threadIdx.x < NG) {
      double t = 0.0;
      for (int w = 0; w < 5; ++w) t += (double)wdot[w][threadIdx.x];
      a.dotpart[(size_t)blockIdx.x * NG + threadIdx.x] = t;
    }
  }
  if (abort) {
    if (threadIdx.x == 0) atomicExch(a.err, 1);
    // bounded wait for the copies in flight: those of tets it and, where there is one, it + 1
    for (int j = it; j < it + 2; ++j) {
      if (i + (j - it) * G >= a.ne) break;
      long spins = 0;
      while (!mbar_wait_hint(&bar[j & 1], (uint32_t)(j >> 1) & 1) && ++spins < kWarpSpin) {
      }
    }
  }
}

// padded block copies: dst block b = planes x NR x NP, zero outside N x N.  A CTA takes whole blocks, about 4,096
// entries at a time, indices by divisions with constants and the scaling from shared memory (a constant-bank read
// with an index per thread is repeated for each value); one plane is rounded to binary32 without the binary64
// pipe.  Bound by memory: 82,944 tets, p = 3, 8 bytes read and 4 written per entry, both copies.
template <typename TB, int PLANES, int N>
__global__ void __launch_bounds__(256) k_to_padded(int64_t nblk, const __grid_constant__ FxBlocks src, TB* __restrict__ dst) {
  constexpr int NR = warp_nr_c(N), NP = warp_np_c(N), pl = NR * NP, per = PLANES * pl, cta = per < 4096 ? 4096 / per : 1;
  __shared__ signed char rs[NR], cs[NP];
  if (threadIdx.x < NR) rs[threadIdx.x] = threadIdx.x < N ? src.r.s[threadIdx.x] : 0;
  if (threadIdx.x < NP) cs[threadIdx.x] = threadIdx.x < N ? src.c.s[threadIdx.x] : 0;
  __syncthreads();
  for (int64_t b0 = (int64_t)blockIdx.x * cta; b0 < nblk; b0 += (int64_t)gridDim.x * cta) {
    const int cnt = (nblk - b0 < cta ? (int)(nblk - b0) : cta) * per;
#pragma unroll 4
    for (int e = threadIdx.x; e < cnt; e += 256) {
      const int b = e / per, rem = e - b * per, plane = rem / pl, rc = rem - plane * pl, r = rc / NP, c = rc - r * NP;
      const bool in = r < N && c < N;
      TB* out = dst + b0 * per + e;
      if constexpr (PLANES == 2) {
        const double v = in ? fx_entry(src, (size_t)N * N, b0 + b, r * N + c, N) : 0.0;
        const float hi = (float)v;
        *out = plane == 0 ? hi : (float)(v - (double)hi);
      } else {
        *out = (TB)(in ? fx_entry_f32(src, (size_t)N * N, b0 + b, r * N + c, rs[r] + cs[c]) : 0.0f);
      }
    }
  }
}
template <typename TB, int PLANES>
static cudaError_t to_padded(stdg_solver* s, int64_t nblk, const FxBlocks& src, void* dst) {
  TB* d = static_cast<TB*>(dst);
  switch (s->N) {
    case 1: k_to_padded<TB, PLANES, 1><<<1216, 256, 0, s->stream>>>(nblk, src, d); break;
    case 4: k_to_padded<TB, PLANES, 4><<<1216, 256, 0, s->stream>>>(nblk, src, d); break;
    case 10: k_to_padded<TB, PLANES, 10><<<1216, 256, 0, s->stream>>>(nblk, src, d); break;
    case 20: k_to_padded<TB, PLANES, 20><<<1216, 256, 0, s->stream>>>(nblk, src, d); break;
    case 35: k_to_padded<TB, PLANES, 35><<<1216, 256, 0, s->stream>>>(nblk, src, d); break;
    default: return cudaErrorInvalidValue;
  }
  ++s->nlaunch;
  return cudaGetLastError();
}

static uint32_t a16(size_t b) { return (uint32_t)((b + 15) & ~(size_t)15); }

template <typename W>
static cudaError_t ensure_warp_blocks(stdg_solver* s, void** Bd, void** Ao) {
  if (*Bd) return cudaSuccess;
  using TB = typename W::TB;
  const int N = s->N, NR = warp_nr_c(N), NP = warp_np_c(N);
  const size_t per = (size_t)W::kPlanes * NR * NP;
  cudaError_t e = dev_alloc_cuda(s, Bd, (size_t)s->ne * per * sizeof(TB));
  if (e != cudaSuccess) return e;
  e = dev_alloc_cuda(s, Ao, (size_t)s->nf * per * sizeof(TB));
  if (e != cudaSuccess) return e;
  e = to_padded<TB, W::kPlanes>(s, s->ne, blocks_B(s), *Bd);
  return e != cudaSuccess ? e : to_padded<TB, W::kPlanes>(s, s->nf, blocks_A(s), *Ao);
}

// padded copy of the viscous diagonal blocks (Eq. A1_mod, with the face blocks A_lr)
template <typename W>
static cudaError_t ensure_warp_visc_diag(stdg_solver* s, void** Bv) {
  if (*Bv) return cudaSuccess;
  using TB = typename W::TB;
  const int N = s->N, NR = warp_nr_c(N), NP = warp_np_c(N);
  cudaError_t e = dev_alloc_cuda(s, Bv, (size_t)s->ne * W::kPlanes * NR * NP * sizeof(TB));
  if (e != cudaSuccess) return e;
  return to_padded<TB, W::kPlanes>(s, s->ne, blocks_Bv(s), *Bv);
}

// Per warp: S stages of [5 blocks | x], then (pair policy only) the (hi, lo) z planes, then the S
// mbarriers.  binary32 x is staged in rows of NR entries per time column, binary64 x as it is.
static WarpArgs warp_layout(const stdg_solver* s, size_t tb, int planes, size_t xin, int S) {
  WarpArgs a{};
  a.ne = (int)s->ne; a.N = s->N; a.NR = warp_nr_c(s->N); a.NP = warp_np_c(s->N); a.Nst = s->Nst; a.S = S;
  a.plane_elems = (uint32_t)(a.NR * a.NP);
  a.blk_bytes = (uint32_t)(planes * a.plane_elems * tb);
  a.xraw_off = 5 * a.blk_bytes;
  const bool df = planes == 2;
  a.stage_bytes = a.xraw_off + (df ? a16((size_t)5 * s->Nst * xin) : a16((size_t)5 * s->Ng * a.NR * xin));
  a.z_off = S * a.stage_bytes;
  a.bar_off = a.z_off + (df ? a16((size_t)planes * 5 * s->Ng * a.NR * sizeof(float)) : 0);
  a.warp_bytes = a16(a.bar_off + 2 * sizeof(uint64_t));
  return a;
}

template <typename W>
static WarpArgs warp_args(const stdg_solver* s) {
  // two stages when ten warps fit on an SM with them, else one (more warps hide the latency)
  WarpArgs a = warp_layout(s, sizeof(typename W::TB), W::kPlanes, sizeof(typename W::XIn), 2);
  if ((size_t)a.warp_bytes * 10 > 228 * 1024) a = warp_layout(s, sizeof(typename W::TB), W::kPlanes, sizeof(typename W::XIn), 1);
  return a;
}

template <typename W>
static constexpr int warp_kind() { return W::kPlanes == 2 ? 2 : (sizeof(typename W::TB) == 4 ? 1 : 0); }

template <typename W>
using WarpKernel = void (*)(WarpArgs, const typename W::XIn*, typename W::YOut*);

// p = 4: k_apply_cta with binary32 blocks at every size (us per application, the warp-per-tet kernel -> this one, L2
// flushed; p_t = 0: 750 tets 10.9 -> 10.9, 2,058 17.1 -> 15.0, 10,368 47.8 -> 45.7; p_t = 2: 13.0 -> 11.9, 21.2 -> 17.0,
// 64.2 -> 51.9; p_t = 4: 13.0 -> 12.9, 21.2 -> 21.1, 66.2 -> 66.2), with bfloat16 blocks, of which twice as many warps
// fit, only where few tets leave those without work (p_t = 2: 2,058 tets 21.2 -> 15.0, 4,374 29.3 -> 25.2; but p_t = 0:
// 4,374 19.1 -> 19.1, 10,368 31.4 -> 33.4).  p = 3 keeps the warp per tet: 82,944 tets, p_t = 1, 99 us against 127.
template <typename W>
static bool cta_serves(const stdg_solver* s) {
  return W::kPlanes == 1 && s->N == 35 && (sizeof(typename W::TB) == 4 || s->ne <= 32 * 152);
}

// the instantiation for this N: compile-time N for p = 2, 3, 4, runtime N otherwise
template <typename W, int NG>
static WarpKernel<W> warp_kernel(const stdg_solver* s) {
  if constexpr (W::kPlanes == 1) {
    if (cta_serves<W>(s)) return k_apply_cta<W, NG, 35>;
  }
  switch (s->N) {
    case 10: return k_apply_warp<W, NG, 10>;
    case 20: return k_apply_warp<W, NG, 20>;
    case 35:
      if constexpr (W::kPlanes == 2 || sizeof(typename W::TB) == 2) return k_apply_warp<W, NG, 35>;
      else break;                                 // cta_serves at every size
    default: return k_apply_warp<W, NG, 0>;
  }
  return nullptr;
}

// Launch shape (warps per CTA, persistent grid) from the occupancy of this layout; sets the
// kernel's dynamic shared-memory limit.  Host-side setup: must not run during stream capture.
template <typename W, int NG>
static cudaError_t warp_configure(stdg_solver* s) {
  const WarpArgs a = warp_args<W>(s);
  const WarpKernel<W> kern = warp_kernel<W, NG>(s);
  int& grid = s->warp_grid[warp_kind<W>() * 8 + NG];
  int& wpc = s->warp_wpc[warp_kind<W>() * 8 + NG];
  if (grid != 0) return cudaSuccess;
  int nsm = 152;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, s->device);
  if (cta_serves<W>(s)) {
    const int smem = (int)CtaDim<W, NG, 35>::smem;
    int per = 0;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, 160, smem);
    if (e != cudaSuccess || per == 0) return e != cudaSuccess ? e : cudaErrorInvalidConfiguration;
    wpc = 5;
    grid = nsm * (per < 8 ? per : 8);             // at most 1,216 rows of x . y partials
    return cudaSuccess;
  }
  int best = 0, bw = 1;
  for (int c : {4, 2, 1}) {
    const size_t smem = (size_t)c * a.warp_bytes;
    if (smem > 227 * 1024) continue;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) continue;
    int per = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, 32 * c, smem);
    if (per * c > best) { best = per * c; bw = c; }
  }
  cudaGetLastError();
  if (best == 0) return cudaErrorInvalidConfiguration;      // the blocks of one tet do not fit on an SM
  wpc = bw;
  grid = nsm * (best / bw);
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)((size_t)wpc * a.warp_bytes));
}

template <typename W>
static cudaError_t warp_prepare_t(stdg_solver* s, void** Bd, void** Ao) {
  cudaError_t e = ensure_warp_blocks<W>(s, Bd, Ao);
  if (e != cudaSuccess) return e;
  switch (s->Ng) {
    case 1: return warp_configure<W, 1>(s);
    case 2: return warp_configure<W, 2>(s);
    case 3: return warp_configure<W, 3>(s);
    case 4: return warp_configure<W, 4>(s);
    default: return warp_configure<W, 5>(s);
  }
}

template <typename W, int NG>
static cudaError_t launch_warp_ng(stdg_solver* s, const WarpArgs& a, const typename W::XIn* x, typename W::YOut* y) {
  const int grid = s->warp_grid[warp_kind<W>() * 8 + NG], wpc = s->warp_wpc[warp_kind<W>() * 8 + NG];
  if (grid == 0) return cudaErrorNotReady;                  // warp_prepare has not run
  const size_t smem = cta_serves<W>(s) ? CtaDim<W, NG, 35>::smem : (size_t)wpc * a.warp_bytes;
  warp_kernel<W, NG>(s)<<<grid, 32 * wpc, smem, s->stream>>>(a, x, y);
  return cudaGetLastError();
}

template <typename W>
static cudaError_t launch_warp(stdg_solver* s, const void* Bd, const void* Ao, const typename W::XIn* x,
                               typename W::YOut* y, int pinned, int kron, double scale, double pin_diag,
                               double mass_coef = 0.0, const double* Kmass = nullptr, double* dotpart = nullptr) {
  if (!Bd) return cudaErrorNotReady;
  WarpArgs a = warp_args<W>(s);
  a.gface = reinterpret_cast<const int4*>(s->gface);
  a.gnbr = reinterpret_cast<const int4*>(s->gnbr);
  a.Bd = Bd; a.Ao = Ao;
  a.pinned = pinned; a.kron = kron; a.scale = scale; a.pin_diag = pin_diag;
  for (int q = 0; q < s->Ng * s->Ng; ++q) a.Tacc[q] = s->tm.Tp[q];
  a.detJ = s->dm.detJ;
  a.mass_coef = Kmass ? mass_coef : 0.0;
  a.dotpart = dotpart;
  for (int q = 0; Kmass && q < s->Ng * s->Ng; ++q) a.Kmass[q] = Kmass[q];
  a.err = s->derr;
  switch (s->Ng) {
    case 1: return launch_warp_ng<W, 1>(s, a, x, y);
    case 2: return launch_warp_ng<W, 2>(s, a, x, y);
    case 3: return launch_warp_ng<W, 3>(s, a, x, y);
    case 4: return launch_warp_ng<W, 4>(s, a, x, y);
    default: return launch_warp_ng<W, 5>(s, a, x, y);
  }
}

}  // namespace stdg
