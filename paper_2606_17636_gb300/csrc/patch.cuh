// A level of the fused FP32 V-cycle whose error stays in registers: thread
// (k, pr) of 512 holds the patch of PR rows x 4 columns at row PR pr, column
// 4 k (nr = 16 .. 128, 4096 or 8192 cells).  Included by k_vsmem.cu.
//
// A radial line is then nr / 4 neighbouring lanes of one warp, so its sweeps
// pass one value per row and half-sweep through shuffles; a polar line runs
// through nt / PR threads in different warps, whose half-sweeps pass the
// patches' first and last rows through shared memory (one block barrier per
// half-sweep).  The right-hand side and the inverse diagonal lie in shared
// memory where only their own thread reads them, as whole 16-byte words.
// Bound by the instruction issue and shared-memory traffic of one SM, and by
// the chain of half-sweeps.  With the error in shared memory a pass moved 40
// bytes per cell of it and formed the diagonal anew; here 16 to 24.  A radial
// pass of 128 x 64 cells takes 3 100 cycles and a polar one 3 800 (4 700 on
// average before; the multiply-adds alone are 1 300), restriction 2 300
// (5 000), prolongation 2 500 (5 600); a V-cycle with two cycles each way
// 24.4 us with up to 152 planes (41.1), 48.4 with 257 (80.6); 64 x 128:
// 26.5 (44.8); patches of two rows, 128 x 32: 16.3 (30.9), 64 x 64: 16.4
// (26.0), 32 x 128: 17.3 (34.5).
// Every relaxation receives the operands and operations of relax_r / relax_t,
// and the transfers those of s_restrict_f32 / s_prolong_f32, so the results are
// bitwise those of the line-by-line schedule.
#pragma once
#include "lines.cuh"

namespace ps {

constexpr int kPatchThreads = 512;

// 32 bytes of one row (32-byte aligned): a whole sector per lane.
__device__ __forceinline__ void ld_run(float2 (&d)[4], const float2* p) {
  asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(d[0].x), "=f"(d[0].y), "=f"(d[1].x), "=f"(d[1].y), "=f"(d[2].x), "=f"(d[2].y), "=f"(d[3].x), "=f"(d[3].y)
               : "l"(p));
}
__device__ __forceinline__ void st_run(float2* p, const float2 (&d)[4]) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(d[0].x), "f"(d[0].y), "f"(d[1].x),
               "f"(d[1].y), "f"(d[2].x), "f"(d[2].y), "f"(d[3].x), "f"(d[3].y)
               : "memory");
}

template <int PR>
struct Patch {
  float2 E[PR][4];
  float nE[4], nW[4], nP[4], nw[4];    // the columns' couplings and polar omega, negated
  const float *rt, *tt, *omr;          // the level's tables and row omegas (shared memory)
  int nr, nt, k, pr, lpr;
  bool first, last, low, high;         // patch at the first / last column or row of the plane
  float s2;
  float4* f;                           // right-hand side, [2 row + colour][thread]: columns colour and colour + 2
  float4 *top, *bot;                   // first and last rows of the patches, [colour][thread]
  float2* dia;                         // negated inverse diagonal, [2 row + colour][thread]

  // tab: the level's packed tables; space: of its error array (8 bytes per
  // cell), the exchanged rows, then the diagonal (PR = 2: in its own space)
  __device__ __forceinline__ Patch(const LevelDev& L, float s2_, const float* tab, float2* f_, float2* space, float2* dia_) {
    nr = L.nr; nt = L.nt; lpr = nr >> 2; s2 = s2_;
    rt = tab;
    tt = rt + RT_N * (nr + 2);
    omr = tt + TT_N * (nt + 2);
    k = threadIdx.x & (lpr - 1);
    pr = threadIdx.x / lpr;
    first = k == 0; last = k == lpr - 1;
    low = pr == 0; high = (pr + 1) * PR == nt;
    f = reinterpret_cast<float4*>(f_) + threadIdx.x;
    top = reinterpret_cast<float4*>(space) + threadIdx.x;
    bot = top + 2 * kPatchThreads;
    dia = dia_ + threadIdx.x;
  }
  __device__ __forceinline__ void r4(float (&d)[4], int id_) const {   // radial table entries of the columns
    const float2* p = reinterpret_cast<const float2*>(rt + id_ * (nr + 2) + 4 * k + 1);
    const float2 a = p[0], b = p[1];
    d[0] = a.x; d[1] = a.y; d[2] = b.x; d[3] = b.y;
  }
  __device__ __forceinline__ void tR(float (&d)[PR], int id_) const {   // polar table entries of the rows
    const float2* p = reinterpret_cast<const float2*>(tt + id_ * (nt + 2) + PR * pr + 1);
#pragma unroll
    for (int q = 0; q < PR / 2; ++q) {
      const float2 a = p[q];
      d[2 * q] = a.x;
      d[2 * q + 1] = a.y;
    }
  }
  // once the tables are there
  __device__ __forceinline__ void coefficients() {
    r4(nE, RT_AE); r4(nW, RT_AW); r4(nP, RT_P);
    const float* o = omr + nt + 4 * k;
#pragma unroll
    for (int c = 0; c < 4; ++c) { nE[c] = -nE[c]; nW[c] = -nW[c]; nP[c] = -nP[c]; nw[c] = -o[c]; }
  }
  __device__ __forceinline__ static void join(float2 (&d)[4], float4 a, float4 b) {   // colours 0 and 1 -> columns
    d[0] = make_float2(a.x, a.y); d[1] = make_float2(b.x, b.y);
    d[2] = make_float2(a.z, a.w); d[3] = make_float2(b.z, b.w);
  }
  __device__ __forceinline__ static float4 half(const float2 (&d)[4], int c) {
    return make_float4(d[c].x, d[c].y, d[c + 2].x, d[c + 2].y);
  }
  __device__ __forceinline__ void ld_f(float2 (&g)[4], int r) const { join(g, f[2 * r * kPatchThreads], f[(2 * r + 1) * kPatchThreads]); }
  __device__ __forceinline__ void st_f(const float2 (&g)[4], int r) const {
    f[2 * r * kPatchThreads] = half(g, 0);
    f[(2 * r + 1) * kPatchThreads] = half(g, 1);
  }
  // rows of the patches below (their last) and above (their first); zero beyond the plane
  __device__ __forceinline__ float4 below(int c) const {
    return low ? make_float4(0.f, 0.f, 0.f, 0.f) : bot[c * kPatchThreads - lpr];
  }
  __device__ __forceinline__ float4 above(int c) const {
    return high ? make_float4(0.f, 0.f, 0.f, 0.f) : top[c * kPatchThreads + lpr];
  }
  __device__ __forceinline__ void put(float4* to, int c, int r) const { to[c * kPatchThreads] = half(E[r], c); }
  __device__ __forceinline__ float2 left(float2 v) const {    // the left neighbour's value
    float2 l;
    l.x = __shfl_up_sync(0xffffffffu, v.x, 1);
    l.y = __shfl_up_sync(0xffffffffu, v.y, 1);
    return first ? make_float2(0.f, 0.f) : l;
  }
  __device__ __forceinline__ float2 right(float2 v) const {
    float2 l;
    l.x = __shfl_down_sync(0xffffffffu, v.x, 1);
    l.y = __shfl_down_sync(0xffffffffu, v.y, 1);
    return last ? make_float2(0.f, 0.f) : l;
  }
  // the diagonal's negated inverse, for its own thread
  __device__ __forceinline__ void set_dia() {
    float Q[4], D[4], T[PR], dt[PR];
    r4(Q, RT_Q); r4(D, RT_DR);
    tR(T, TT_T); tR(dt, TT_DT);
#pragma unroll
    for (int r = 0; r < PR; ++r) {
      float d[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) d[c] = -rcp_diag(fmac(-(s2 * Q[c]), T[r], fmac(-nP[c], dt[r], D[c])));
      dia[2 * r * kPatchThreads] = make_float2(d[0], d[2]);
      dia[(2 * r + 1) * kPatchThreads] = make_float2(d[1], d[3]);
    }
  }

  // Radial lines of rows C, C + 2, ..
  template <int C>
  __device__ __forceinline__ void radial_rows(int n_sor) {
    constexpr int H = PR / 2;
    float aN[PR], aS[PR], w[H], nid[H][4];
    float2 g[H][4];
    tR(aN, TT_AN);
    tR(aS, TT_AS);
    auto source = [&](int h, const float2 (&x)[4]) {   // x: the row of the neighbouring patch
      const int r = 2 * h + C;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float2 un = r + 1 < PR ? E[r + 1 < PR ? r + 1 : 0][c] : x[c];
        const float2 us = r > 0 ? E[r > 0 ? r - 1 : 0][c] : x[c];
        g[h][c] = fma2(nP[c], fma2(aS[r], us, mul2(aN[r], un)), g[h][c]);
      }
    };
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const int r = 2 * h + C;
      ld_f(g[h], r);
      const float2 a = dia[2 * r * kPatchThreads], b = dia[(2 * r + 1) * kPatchThreads];
      nid[h][0] = a.x; nid[h][1] = b.x; nid[h][2] = a.y; nid[h][3] = b.y;
      w[h] = -omr[PR * pr + r];
      if (h != (C ? H - 1 : 0)) source(h, g[h]);   // a row inside the patch: x is not read
    }
    __syncthreads();   // the neighbouring patches' rows are there
    {
      float2 x[4];
      if constexpr (C == 0) join(x, below(0), below(1));
      else join(x, above(0), above(1));
      source(C ? H - 1 : 0, x);
    }
#pragma unroll 1
    for (int it = 0; it < n_sor; ++it) {
#pragma unroll
      for (int par = 0; par < 2; ++par) {
        float2 y[H];
#pragma unroll
        for (int h = 0; h < H; ++h) y[h] = par ? right(E[2 * h + C][0]) : left(E[2 * h + C][3]);
#pragma unroll
        for (int q = 0; q < 2; ++q)   // the cells inside the patch first
#pragma unroll
          for (int h = 0; h < H; ++h) {
            const int c = par ? 1 + 2 * q : 2 - 2 * q;
            float2(&e)[4] = E[2 * h + C];
            const float2 em = c > 0 ? e[c > 0 ? c - 1 : 0] : y[h], ep = c < 3 ? e[c < 3 ? c + 1 : 0] : y[h];
            const float2 r = fma2(nW[c], em, fma2(nE[c], ep, g[h][c]));
            e[c] = fma2(w[h], fma2(nid[h][c], r, e[c]), e[c]);
          }
      }
    }
  }
  // Both colours; needs the patches' last rows in bot, leaves first and last
  // rows in top and bot (the next reader takes the barrier).
  __device__ __forceinline__ void radial(int n_sor) {
    radial_rows<0>(n_sor);
    put(top, 0, 0);
    put(top, 1, 0);
    radial_rows<1>(n_sor);
    put(bot, 0, PR - 1);
    put(bot, 1, PR - 1);
  }

  // Polar lines of columns C, C + 2.
  template <int C>
  __device__ __forceinline__ void polar_cols(int n_sor) {
    float up[PR][2], dn[PR][2];
    float2 g[PR][2], nid[PR];
    {
      float aN[PR], aS[PR];
      tR(aN, TT_AN);
      tR(aS, TT_AS);
#pragma unroll
      for (int r = 0; r < PR; ++r) {
        const float2 x = C ? right(E[r][0]) : left(E[r][3]);
        const float4 fr = f[(2 * r + C) * kPatchThreads];
        nid[r] = dia[(2 * r + C) * kPatchThreads];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int c = C + 2 * q;
          const float2 ue = c < 3 ? E[r][c < 3 ? c + 1 : 0] : x, uw = c > 0 ? E[r][c > 0 ? c - 1 : 0] : x;
          g[r][q] = fma2(nW[c], uw, fma2(nE[c], ue, q ? make_float2(fr.z, fr.w) : make_float2(fr.x, fr.y)));
          up[r][q] = nP[c] * aN[r];
          dn[r][q] = nP[c] * aS[r];
        }
      }
    }
    auto relax = [&](int r, const float2 (&y)[2]) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int c = C + 2 * q;
        const float2 em = r > 0 ? E[r > 0 ? r - 1 : 0][c] : y[q], ep = r + 1 < PR ? E[r + 1 < PR ? r + 1 : 0][c] : y[q];
        const float2 s = fma2(dn[r][q], em, fma2(up[r][q], ep, g[r][q]));
        E[r][c] = fma2(nw[c], fma2(q ? nid[r].y : nid[r].x, s, E[r][c]), E[r][c]);
      }
    };
    float2 y[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 1
    for (int it = 0; it < n_sor; ++it) {
      // even rows, then odd rows; the ones inside the patch before the barrier
#pragma unroll
      for (int r = 2; r < PR; r += 2) relax(r, y);
      if (C == 0 || it > 0) __syncthreads();
      {
        const float4 v = below(C);
        y[0] = make_float2(v.x, v.y);
        y[1] = make_float2(v.z, v.w);
      }
      relax(0, y);
      put(top, C, 0);
#pragma unroll
      for (int r = 1; r < PR - 1; r += 2) relax(r, y);
      __syncthreads();
      {
        const float4 v = above(C);
        y[0] = make_float2(v.x, v.y);
        y[1] = make_float2(v.z, v.w);
      }
      relax(PR - 1, y);
      put(bot, C, PR - 1);
    }
  }
  __device__ __forceinline__ void polar(int n_sor) {
    polar_cols<0>(n_sor);
    polar_cols<1>(n_sor);
  }

  // Area-weighted restriction of the defect (values in the layout of vslot);
  // needs current rows in top and bot.  PR / 2 x 2 coarse cells per thread.
  // The signs sit in the coefficients: f + (-L e), rounded like f - L e.
  template <typename Slot>
  __device__ __forceinline__ void restrict_to(float2* fc, Slot slot) {
    float DR[4], Q[4], RW[4], AN[PR], AS[PR], DT[PR], T[PR], TW[PR];
    r4(DR, RT_DR); r4(Q, RT_Q); r4(RW, RT_RW);
    tR(AN, TT_AN); tR(AS, TT_AS); tR(DT, TT_DT); tR(T, TT_T); tR(TW, TT_RW);
    float2 S[4], N[4];
    join(S, below(0), below(1));
    join(N, above(0), above(1));
#pragma unroll
    for (int h = 0; h < PR / 2; ++h) {
      float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int r = 2 * h + b;
        const float2 W = left(E[r][3]), X = right(E[r][0]);
        float2 fr[4];
        ld_f(fr, r);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float2 n = r + 1 < PR ? E[r + 1 < PR ? r + 1 : 0][c] : N[c], s = r > 0 ? E[r > 0 ? r - 1 : 0][c] : S[c];
          const float2 w = c > 0 ? E[r][c > 0 ? c - 1 : 0] : W, x = c < 3 ? E[r][c < 3 ? c + 1 : 0] : X;
          const float aN = nP[c] * AN[r], aS = nP[c] * AS[r];
          const float d = -fmac(-(s2 * Q[c]), T[r], fmac(-nP[c], DT[r], DR[c]));
          const float2 t = fma2(d, E[r][c], fma2(aS, s, fma2(aN, n, fma2(nW[c], w, mul2(nE[c], x)))));
          acc[c >> 1] = fma2(RW[c] * TW[r], make_float2(fr[c].x + t.x, fr[c].y + t.y), acc[c >> 1]);
        }
      }
      st_pair(fc + slot((PR / 2) * pr + h, 2 * k), acc[0], acc[1]);
    }
  }

  // Bilinear correction from the coarse level C: this patch's coarse columns
  // 2 k, 2 k + 1 as pairs, the ones beside them from the neighbouring lanes.
  template <typename Slot>
  __device__ __forceinline__ void prolong_from(const LevelDev& C, const float2* ec, bool odd, Slot slot) {
    constexpr int R = PR / 2 + 2;   // coarse rows of the neighbourhood
    float P1[4], P2[4], Q1[PR], Q2[PR];
    r4(P1, RT_P1); r4(P2, RT_P2);
    tR(Q1, TT_P1); tR(Q2, TT_P2);
    const int rl = first ? C.gL : -1, rr_ = last ? C.gR : -1;   // ghost rules of the columns outside
    const bool zl = rl == GH_ZERO, zr = rr_ == GH_ZERO, nl = rl == GH_PARITY && odd, nrt = rr_ == GH_PARITY && odd;
    auto flip = [](float2 v, bool zero, bool neg) {
      return zero ? make_float2(0.f, 0.f) : (neg ? make_float2(-v.x, -v.y) : v);
    };
    auto row = [&](float2 (&d)[4], int v) {   // 1-based coarse row (PR / 2) pr + v
      const int y = (PR / 2) * pr + v, rule = y == 0 ? C.gB : (y == C.nt + 1 ? C.gT : -1);
      const int jc = min(max(y, 1), C.nt) - 1;
      const bool zy = rule == GH_ZERO, ny = rule == GH_PARITY && odd;
      float2 a, b, l, r;
      ld_pair(a, b, ec + slot(jc, 2 * k));
      l.x = __shfl_up_sync(0xffffffffu, b.x, 1);
      l.y = __shfl_up_sync(0xffffffffu, b.y, 1);
      r.x = __shfl_down_sync(0xffffffffu, a.x, 1);
      r.y = __shfl_down_sync(0xffffffffu, a.y, 1);
      if (first) l = a;   // a ghost mirrors its neighbour inside
      if (last) r = b;
      d[0] = flip(l, zl || zy, nl != ny);
      d[1] = flip(a, zy, ny);
      d[2] = flip(b, zy, ny);
      d[3] = flip(r, zr || zy, nrt != ny);
    };
    float2 a[4], b[4];
    row(a, 0);
#pragma unroll
    for (int v = 0; v + 1 < R; ++v) {   // coarse rows v (a) and v + 1 (b) correct fine rows 2 v - 1 and 2 v
      row(b, v + 1);
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const int r = 2 * v - 1 + o;
        if (r >= 0 && r < PR) {
          const int q = r >= 0 && r < PR ? r : 0;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int u = (c + 1) >> 1;   // columns (u, u + 1) of the neighbourhood
            const float w11 = P1[c] * Q1[q], w21 = P2[c] * Q1[q], w12 = P1[c] * Q2[q], w22 = P2[c] * Q2[q];
            const float2 t = fma2(w22, b[u + 1], fma2(w12, b[u], fma2(w21, a[u + 1], mul2(w11, a[u]))));
            E[q][c].x += t.x;
            E[q][c].y += t.y;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = b[u];
    }
  }
};

}  // namespace ps
