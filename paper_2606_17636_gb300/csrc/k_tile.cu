// Several smoothing passes of a level in one launch (Sec. 3.2), FP32.
//
// A block holds a window of WX x WY cells of one plane (error, right-hand side
// and inverse diagonal) in shared memory and runs `npass` consecutive passes
// on it, radial and polar lines in turn, both zebra colours each.  A line's
// n_sor even-odd SOR sweeps reach at most 2 n_sor cells along it, and the
// second colour also sees the first colour's result, so a pass reaches
// 4 n_sor - 1 cells along its lines and 2 lines across: after a whole cycle
// only cells within 4 n_sor + 1 of an inner window edge differ from the
// passes over the whole plane.  The windows overlap by that halo and each
// block stores the cells it owns, which are bitwise those of the passes over
// the whole plane.  Before the passes a launch may add the prolongated coarse
// correction; after them it may restrict the defect or add the result to the
// FP64 solution.
//
// For the last planes of a solve: a level-wide pass costs 4 us of latency with
// one plane active whatever it computes.  With one plane of 256 x 128 cells two
// cycles and the restriction take 11 us in one launch (four passes and a
// restriction: 19 us and four launches' gaps more), the prolongation, a cycle
// and the update 13 us.  The halos cost 4.5 times the work (two cycles on 64 x 64
// windows), so many planes keep the level-wide passes: 129 planes take 150 us
// here against 107.
//
// Inner loop: a thread holds 8 consecutive cells of two neighbouring lines
// (one of each colour), so a half-sweep needs one shuffle per 4 cells, and
// the two components of a cell move through packed FP32 multiply-adds.
// Shared-memory layout: cell (j, i) in 16-byte chunk (i >> 1), the chunk index
// XORed so that both the radial accesses (8 lanes, 4 chunks apart, one row)
// and the polar ones (chunks of neighbouring columns in rows 8 apart) of a
// quarter-warp fall on 8 different bank groups.
#include "lines.cuh"

namespace ps {

namespace {


template <int WX>
__device__ __forceinline__ int chunk_at(int j, int q) {   // 16-byte chunk index of columns 2q, 2q + 1 of row j
  constexpr int M = WX / 2;
  int s = q ^ ((j >> 1) & 4);
  if constexpr (WX >= 64) s ^= (q >> 3) & 3;
  else s ^= ((q >> 3) & 1) ^ (j & 2);
  return j * M + s;
}
template <int WX>
__device__ __forceinline__ int pair_at(int j, int q) {    // 8-byte pair index of the inverse diagonal's columns 2q, 2q + 1
  int s = q ^ (((j >> 3) & 3) << 2);
  if constexpr (WX >= 64) s ^= ((q >> 4) & 1) << 1;
  else s ^= j & 2;
  return j * (WX / 2) + s;
}

// Window tables in shared memory (floats): radial entries of WX columns,
// polar entries of WY rows; the couplings and the diagonal's polar part
// negated (see sor_run).
template <int WX, int WY>
struct Tab {
  enum { nAE = 0, nAW = WX, nP = 2 * WX, Q = 3 * WX, DR = 4 * WX, RW = 5 * WX, P1 = 6 * WX, P2 = 7 * WX,
         OMT = 8 * WX, AN = 9 * WX, AS = AN + WY, T = AN + 2 * WY, nDT = AN + 3 * WY, TRW = AN + 4 * WY,
         TP1 = AN + 5 * WY, TP2 = AN + 6 * WY, OMR = AN + 7 * WY, N = AN + 8 * WY };
};

__device__ __forceinline__ void ld8(float (&d)[8], const float* p) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  d[0] = a.x; d[1] = a.y; d[2] = a.z; d[3] = a.w;
  d[4] = b.x; d[5] = b.y; d[6] = b.z; d[7] = b.w;
}
template <int WX>
__device__ __forceinline__ void ld_row8(float2 (&d)[8], const float4* s, int j, int k) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float4 v = s[chunk_at<WX>(j, 4 * k + q)];
    d[2 * q] = make_float2(v.x, v.y);
    d[2 * q + 1] = make_float2(v.z, v.w);
  }
}
template <int WX>
__device__ __forceinline__ void st_row8(float4* s, int j, int k, const float2 (&d)[8]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    s[chunk_at<WX>(j, 4 * k + q)] = make_float4(d[2 * q].x, d[2 * q].y, d[2 * q + 1].x, d[2 * q + 1].y);
}
template <int WX>
__device__ __forceinline__ void ld_id_row(float (&d)[8], const float2* id, int j, int k) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float4 v = *reinterpret_cast<const float4*>(id + pair_at<WX>(j, 4 * k + 2 * q));
    d[4 * q] = v.x; d[4 * q + 1] = v.y; d[4 * q + 2] = v.z; d[4 * q + 3] = v.w;
  }
}
__device__ __forceinline__ void zero8(float2 (&d)[8]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) d[c] = make_float2(0.f, 0.f);
}

// Radial lines, both colours: thread (row pair, k) holds columns 8k .. 8k + 7
// of rows 2 rp (colour 0) and 2 rp + 1 (colour 1).
template <int WX, int WY>
__device__ __forceinline__ void pass_r(float4* se, const float4* sf, const float2* sid, const float* tb, int n_sor) {
  typedef Tab<WX, WY> TB;
  constexpr int LPL = WX / 8;
  const int k = threadIdx.x % LPL, j0 = 2 * (threadIdx.x / LPL), j1 = j0 + 1;
  const bool first = k == 0, last = k == LPL - 1;
  float nup[8], ndn[8], np[8], nid[8];
  float2 e0[8], e1[8], g[8], nb[8];
  ld_row8<WX>(e0, se, j0, k);
  ld_row8<WX>(e1, se, j1, k);
  ld_row8<WX>(g, sf, j0, k);
  if (j0 > 0) ld_row8<WX>(nb, se, j0 - 1, k);
  else zero8(nb);
  ld8(np, tb + TB::nP + 8 * k);
  {
    const float aN = tb[TB::AN + j0], aS = tb[TB::AS + j0];
#pragma unroll
    for (int c = 0; c < 8; ++c) g[c] = fma2(np[c], fma2(aS, nb[c], mul2(aN, e1[c])), g[c]);
  }
  ld8(nup, tb + TB::nAE + 8 * k);
  ld8(ndn, tb + TB::nAW + 8 * k);
  ld_id_row<WX>(nid, sid, j0, k);
  sor_run<8>(e0, g, nup, ndn, nid, -tb[TB::OMR + j0], first, last, n_sor);
  st_row8<WX>(se, j0, k, e0);
  ld_row8<WX>(g, sf, j1, k);
  ld_id_row<WX>(nid, sid, j1, k);
  __syncthreads();
  if (j1 + 1 < WY) ld_row8<WX>(nb, se, j1 + 1, k);
  else zero8(nb);
  {
    const float aN = tb[TB::AN + j1], aS = tb[TB::AS + j1];
#pragma unroll
    for (int c = 0; c < 8; ++c) g[c] = fma2(np[c], fma2(aS, e0[c], mul2(aN, nb[c])), g[c]);
  }
  sor_run<8>(e1, g, nup, ndn, nid, -tb[TB::OMR + j1], first, last, n_sor);
  st_row8<WX>(se, j1, k, e1);
  __syncthreads();
}

// Polar / vertical lines, both colours: thread (column pair, b) holds rows
// 8b .. 8b + 7 of columns 2 cp (colour 0) and 2 cp + 1 (colour 1); the lanes of
// a column lie 32 / (WY / 8) apart.
template <int WX, int WY>
__device__ __forceinline__ void pass_t(float4* se, const float4* sf, const float2* sid, const float* tb, int n_sor) {
  typedef Tab<WX, WY> TB;
  constexpr int LPC = WY / 8, CPW = 32 / LPC;
  const int lane = threadIdx.x & 31, b = lane / CPW, cp = (threadIdx.x >> 5) * CPW + lane % CPW;
  const int i0 = 2 * cp, i1 = i0 + 1, jb = 8 * b;
  const bool first = b == 0, last = b == LPC - 1;
  float2* s2 = reinterpret_cast<float2*>(se);
  float2 e0[8], e1[8], g[8], nb[8];
  float an[8], as[8], nid0[8], nid1[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float4 v = se[chunk_at<WX>(jb + c, cp)];
    e0[c] = make_float2(v.x, v.y);
    e1[c] = make_float2(v.z, v.w);
    g[c] = *reinterpret_cast<const float2*>(sf + chunk_at<WX>(jb + c, cp));
    nb[c] = cp > 0 ? s2[2 * chunk_at<WX>(jb + c, cp - 1) + 1] : make_float2(0.f, 0.f);
    const float2 d = sid[pair_at<WX>(jb + c, cp)];
    nid0[c] = d.x;
    nid1[c] = d.y;
  }
  ld8(an, tb + TB::AN + jb);
  ld8(as, tb + TB::AS + jb);
  {
    const float naE = tb[TB::nAE + i0], naW = tb[TB::nAW + i0], np = tb[TB::nP + i0];
    float nup[8], ndn[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      g[c] = fma2(naW, nb[c], fma2(naE, e1[c], g[c]));
      nup[c] = np * an[c];
      ndn[c] = np * as[c];
    }
    sor_run<8, CPW>(e0, g, nup, ndn, nid0, -tb[TB::OMT + i0], first, last, n_sor);
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    s2[2 * chunk_at<WX>(jb + c, cp)] = e0[c];
    g[c] = *(reinterpret_cast<const float2*>(sf + chunk_at<WX>(jb + c, cp)) + 1);
  }
  __syncthreads();
  {
    const float naE = tb[TB::nAE + i1], naW = tb[TB::nAW + i1], np = tb[TB::nP + i1];
    float nup[8], ndn[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      nb[c] = cp + 1 < WX / 2 ? s2[2 * chunk_at<WX>(jb + c, cp + 1)] : make_float2(0.f, 0.f);
      g[c] = fma2(naW, e0[c], fma2(naE, nb[c], g[c]));
      nup[c] = np * an[c];
      ndn[c] = np * as[c];
    }
    sor_run<8, CPW>(e1, g, nup, ndn, nid1, -tb[TB::OMT + i1], first, last, n_sor);
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) s2[2 * chunk_at<WX>(jb + c, cp) + 1] = e1[c];
  __syncthreads();
}

// e += P ec on the window whose first cell is (y0, x0): thread (coarse column,
// strip of four coarse rows); the formulas, ghost rules and order of
// operations of k_prolong.
template <int WX, int WY>
__device__ __forceinline__ void add_coarse(float4* se, const float* tb, const LevelDev& C,
                                           const float2* __restrict__ ec, int x0, int y0, bool odd) {
  typedef Tab<WX, WY> TB;
  const int Il = threadIdx.x % (WX / 2), Jl = 4 * (threadIdx.x / (WX / 2));
  const int I = x0 / 2 + Il, J0 = y0 / 2 + Jl;
  int ic[3];
  bool zc[3], nc[3];
#pragma unroll
  for (int u = 0; u < 3; ++u) {   // 1-based coarse column I + u
    const int x = I + u, rule = x == 0 ? C.gL : (x == C.nr + 1 ? C.gR : -1);
    ic[u] = min(max(x, 1), C.nr) - 1;
    zc[u] = rule == GH_ZERO;
    nc[u] = rule == GH_PARITY && odd;
  }
  float2 r[6][3];   // 1-based coarse rows J0 .. J0 + 5
#pragma unroll
  for (int v = 0; v < 6; ++v) {
    const int y = J0 + v, rule = y == 0 ? C.gB : (y == C.nt + 1 ? C.gT : -1);
    const int jc = min(max(y, 1), C.nt) - 1;
    const bool zr = rule == GH_ZERO, nrw = rule == GH_PARITY && odd;
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const float2 x = ec[size_t(jc) * C.nr + ic[u]];
      r[v][u] = (zc[u] || zr) ? make_float2(0.f, 0.f) : ((nc[u] != nrw) ? make_float2(-x.x, -x.y) : x);
    }
  }
  const float2 p1v = *reinterpret_cast<const float2*>(tb + TB::P1 + 2 * Il);
  const float2 p2v = *reinterpret_cast<const float2*>(tb + TB::P2 + 2 * Il);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int j = 2 * (Jl + q) + b;
      const float q1 = tb[TB::TP1 + j], q2 = tb[TB::TP2 + j];
      float4* cell = se + chunk_at<WX>(j, Il);
      const float4 v = *cell;
      float2 uu[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const float p1 = a ? p1v.y : p1v.x, p2 = a ? p2v.y : p2v.x;
        const float2 A = r[q + b][a], Bv = r[q + b][a + 1], Cv = r[q + b + 1][a], D = r[q + b + 1][a + 1];
        const float w11 = p1 * q1, w21 = p2 * q1, w12 = p1 * q2, w22 = p2 * q2;
        uu[a].x += fmac(w22, D.x, fmac(w12, Cv.x, fmac(w21, Bv.x, w11 * A.x)));
        uu[a].y += fmac(w22, D.y, fmac(w12, Cv.y, fmac(w21, Bv.y, w11 * A.y)));
      }
      *cell = make_float4(uu[0].x, uu[0].y, uu[1].x, uu[1].y);
    }
  }
}

// Defect restriction of the owned coarse cells: the operations of k_restrict.
template <int WX, int WY>
__device__ __forceinline__ void restrict_own(const float4* se, const float4* sf, const float* tb,
                                             const LevelDev& C, float2* __restrict__ fc, float s2v, int x0,
                                             int y0, int xa, int xb, int ya, int yb) {
  typedef Tab<WX, WY> TB;
  const float2* e2 = reinterpret_cast<const float2*>(se);
  const int nx = (xb - xa) / 2, ny = (yb - ya) / 2;
  const float2 z = make_float2(0.f, 0.f);
  auto two = [](const float* p) { return *reinterpret_cast<const float2*>(p); };
  for (RowWalk w(threadIdx.x, blockDim.x, nx); w.j < ny; w.next()) {
    const int i0 = xa - x0 + 2 * w.c, j0 = ya - y0 + 2 * w.j, cq = i0 / 2;   // window coordinates
    float4 r[4], fv[2];
    float2 W[2], E[2];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = j0 - 1 + q;
      r[q] = j >= 0 && j < WY ? se[chunk_at<WX>(j, cq)] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      W[b] = i0 > 0 ? e2[2 * chunk_at<WX>(j0 + b, cq - 1) + 1] : z;
      E[b] = i0 + 2 < WX ? e2[2 * chunk_at<WX>(j0 + b, cq + 1)] : z;
      fv[b] = sf[chunk_at<WX>(j0 + b, cq)];
    }
    const float2 nAE = two(tb + TB::nAE + i0), nAW = two(tb + TB::nAW + i0), nP = two(tb + TB::nP + i0);
    const float2 DR = two(tb + TB::DR + i0), QQ = two(tb + TB::Q + i0), RW = two(tb + TB::RW + i0);
    const float2 AN = two(tb + TB::AN + j0), AS = two(tb + TB::AS + j0), nDT = two(tb + TB::nDT + j0);
    const float2 TT = two(tb + TB::T + j0), TW = two(tb + TB::TRW + j0);
    float ax = 0.f, ay = 0.f;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        auto cell = [&](int q) { return a ? make_float2(r[q].z, r[q].w) : make_float2(r[q].x, r[q].y); };
        const float2 c = cell(b + 1), N = cell(b + 2), S = cell(b);
        const float2 Ev = a ? E[b] : make_float2(r[b + 1].z, r[b + 1].w);
        const float2 Wv = a ? make_float2(r[b + 1].x, r[b + 1].y) : W[b];
        const float2 fc2 = a ? make_float2(fv[b].z, fv[b].w) : make_float2(fv[b].x, fv[b].y);
        const float aE = -(a ? nAE.y : nAE.x), aW = -(a ? nAW.y : nAW.x), P = -(a ? nP.y : nP.x);
        const float aN = P * (b ? AN.y : AN.x), aS = P * (b ? AS.y : AS.x);
        const float d = fmac(-(s2v * (a ? QQ.y : QQ.x)), b ? TT.y : TT.x, fmac(P, -(b ? nDT.y : nDT.x), a ? DR.y : DR.x));
        const float rx = fc2.x - fmac(d, c.x, fmac(aS, S.x, fmac(aN, N.x, fmac(aW, Wv.x, aE * Ev.x))));
        const float ry = fc2.y - fmac(d, c.y, fmac(aS, S.y, fmac(aN, N.y, fmac(aW, Wv.y, aE * Ev.y))));
        const float wgt = (a ? RW.y : RW.x) * (b ? TW.y : TW.x);
        ax = fmac(wgt, rx, ax);
        ay = fmac(wgt, ry, ay);
      }
    fc[size_t(ya / 2 + w.j) * C.nr + xa / 2 + w.c] = make_float2(ax, ay);
  }
}

template <int WX, int WY>
constexpr size_t tile_smem() {
  return size_t(WX) * WY * 20 + size_t(Tab<WX, WY>::N) * 4;
}

// First cell of window t along a dimension of n cells, and the cells it owns.
__device__ __forceinline__ void window(int t, int nt, int n, int W, int H, int& x0, int& xa, int& xb) {
  const int s = W - 2 * H;
  x0 = nt == 1 ? 0 : min(t * s, n - W);
  xa = t == 0 ? 0 : t * s + H;
  xb = t == nt - 1 ? n : t * s + W - H;
}

template <int WX, int WY>
__global__ void __launch_bounds__(WX * WY / 16, 8192 / (WX * WY)) k_tile(LevelDev L, LevelDev C, Batch B, TileStep a) {
  typedef Tab<WX, WY> TB;
  constexpr int NTH = WX * WY / 16;
  extern __shared__ __align__(16) unsigned char traw[];
  float4* se = reinterpret_cast<float4*>(traw);
  float4* sf = se + WX * WY / 2;
  float2* sid = reinterpret_cast<float2*>(sf + WX * WY / 2);
  float* tb = reinterpret_cast<float*>(sid + WX * WY / 2);
  const int nact = *B.nact, per = a.ntx * a.nty;
  // the first item's plane, fetched beside the count
  const int pf = B.act[min(int(blockIdx.x) / per, B.max_planes - 1)];
  const int nr = L.nr, nt = L.nt, tid = threadIdx.x;
  for (int w = blockIdx.x; w < nact * per; w += gridDim.x) {
    const int k = w / per, t = w - k * per, ty = t / a.ntx, tx = t - ty * a.ntx;
    const int p = w == int(blockIdx.x) ? pf : B.act[k];
    const int slot = B.slot ? B.slot[p] : p;
    int x0, xa, xb, y0, ya, yb;
    window(tx, a.ntx, nr, WX, a.halo, x0, xa, xb);
    window(ty, a.nty, nt, WY, a.halo, y0, ya, yb);
    const size_t base = size_t(p) * nr * nt, org = base + size_t(y0) * nr + x0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int idx = tid + q * NTH, j = idx / (WX / 2), c = idx % (WX / 2);
      const size_t g = org + size_t(j) * nr + 2 * c;
      cp_async_v(sf + chunk_at<WX>(j, c), reinterpret_cast<const float4*>(a.f + g), true);
      if (a.src) cp_async_v(se + chunk_at<WX>(j, c), reinterpret_cast<const float4*>(a.src + g), true);
      else se[chunk_at<WX>(j, c)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    {
      // the window's table rows, all loads in flight before the first store:
      // radial AE, AW, P, Q, D_r, weights, then omega of the polar lines;
      // polar aN, aS, T, D_theta, weights, then omega of the radial lines
      const float* rt = L.rf + 1 + x0;
      const float* tt = L.tf + 1 + y0;
      constexpr int NX = 9 * WX, NE = (TB::N + NTH - 1) / NTH;
      float x[NE];
#pragma unroll
      for (int q = 0; q < NE; ++q) {
        const int e = tid + q * NTH;
        if (e < NX) {
          const int row = e / WX, i = e % WX;
          x[q] = row == 8 ? L.omt_f[size_t(slot) * nr + x0 + i] : rt[(row < 5 ? row : row + 1) * (nr + 2) + i];
          if (row < 3) x[q] = -x[q];
        } else if (e < TB::N) {
          const int row = (e - NX) / WY, j = (e - NX) % WY;
          x[q] = row == 7 ? L.omr_f[size_t(slot) * nt + y0 + j] : tt[(row < 4 ? row : row + 1) * (nt + 2) + j];
          if (row == 3) x[q] = -x[q];
        }
      }
#pragma unroll
      for (int q = 0; q < NE; ++q)
        if (tid + q * NTH < TB::N) tb[tid + q * NTH] = x[q];
    }
    const float s2v = B.s2f[slot];
    cp_async_wait_all();
    __syncthreads();
    {   // inverse diagonal of the window, negated: 8 columns of a row pair per thread
      constexpr int LPL = WX / 8;
      const int kk = tid % LPL, j0 = 2 * (tid / LPL);
      float np[8], q[8], dr[8];
      ld8(np, tb + TB::nP + 8 * kk);
      ld8(q, tb + TB::Q + 8 * kk);
      ld8(dr, tb + TB::DR + 8 * kk);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const float Tj = tb[TB::T + j0 + b], ndt = tb[TB::nDT + j0 + b];
        float d[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) d[c] = -rcp_diag(fmac(-(s2v * q[c]), Tj, fmac(np[c], ndt, dr[c])));
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<float4*>(sid + pair_at<WX>(j0 + b, 4 * kk + 2 * h)) =
              make_float4(d[4 * h], d[4 * h + 1], d[4 * h + 2], d[4 * h + 3]);
      }
    }
    if (a.op & TILE_PROLONG)
      add_coarse<WX, WY>(se, tb, C, a.ec + size_t(p) * C.nr * C.nt, x0, y0, (B.mode[slot] & 1) != 0);
    __syncthreads();
    for (int q = 0; q < a.npass; ++q) {
      if (q & 1) pass_t<WX, WY>(se, sf, sid, tb, a.n_sor);
      else pass_r<WX, WY>(se, sf, sid, tb, a.n_sor);
    }
    const int nx2 = (xb - xa) / 2, ny = yb - ya;
    if (a.op & TILE_UPDATE) {
      for (RowWalk wk(tid, NTH, nx2); wk.j < ny; wk.next()) {
        const float4 x = se[chunk_at<WX>(ya - y0 + wk.j, (xa - x0) / 2 + wk.c)];
        double2* o = a.u + base + size_t(ya + wk.j) * nr + xa + 2 * wk.c;
        double2 s = o[0], r = o[1];
        s.x += widen(x.x);
        s.y += widen(x.y);
        r.x += widen(x.z);
        r.y += widen(x.w);
        o[0] = s;
        o[1] = r;
      }
    } else {
      for (RowWalk wk(tid, NTH, nx2); wk.j < ny; wk.next())
        *reinterpret_cast<float4*>(a.dst + base + size_t(ya + wk.j) * nr + xa + 2 * wk.c) =
            se[chunk_at<WX>(ya - y0 + wk.j, (xa - x0) / 2 + wk.c)];
    }
    if (a.op & TILE_RESTRICT)
      restrict_own<WX, WY>(se, sf, tb, C, a.fc + size_t(p) * C.nr * C.nt, s2v, x0, y0, xa, xb, ya, yb);
    __syncthreads();
  }
}

int tile_count(int n, int W, int H) { return n <= W ? 1 : (n - 2 * H + (W - 2 * H) - 1) / (W - 2 * H); }

int win(int n) { return n >= 64 ? 64 : 32; }

template <int WX, int WY>
void launch_wxy(const LevelDev& L, const LevelDev& C, const Batch& B, const TileStep& a, cudaStream_t st) {
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_tile<WX, WY>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(tile_smem<WX, WY>()));
    attr = true;
  }
  const long occ = 8192 / (WX * WY);
  const long items = long(a.ntx) * a.nty * B.max_planes;
  const long cap = long(sm_count()) * occ;
  k_tile<WX, WY><<<unsigned(items < cap ? items : cap), WX * WY / 16, tile_smem<WX, WY>(), st>>>(L, C, B, a);
}

}  // namespace

// A cycle reaches 4 n_sor + 1 cells in both directions, the defect of a
// restriction one more; even window origins keep the zebra and SOR colours.
bool tile_step(int nr, int nt, int n_sor, int cycles, bool restricts, TileStep& t) {
  if (nr < 32 || nt < 32 || n_sor < 1) return false;
  t.n_sor = n_sor;
  t.npass = 2 * cycles;
  t.halo = (cycles * (4 * n_sor + 1) + (restricts ? 1 : 0) + 1) / 2 * 2;
  const int wx = win(nr), wy = win(nt);
  if ((nr > wx && wx - 2 * t.halo < 16) || (nt > wy && wy - 2 * t.halo < 16)) return false;
  t.ntx = tile_count(nr, wx, t.halo);
  t.nty = tile_count(nt, wy, t.halo);
  return true;
}

int tile_slots(int nr, int nt) { return sm_count() * (8192 / (win(nr) * win(nt))); }

void launch_tile(const LevelDev& L, const LevelDev& C, const Batch& B, const TileStep& a, cudaStream_t st) {
  if (L.nr >= 64) {
    if (L.nt >= 64) launch_wxy<64, 64>(L, C, B, a, st);
    else launch_wxy<64, 32>(L, C, B, a, st);
  } else {
    if (L.nt >= 64) launch_wxy<32, 64>(L, C, B, a, st);
    else launch_wxy<32, 32>(L, C, B, a, st);
  }
}

}  // namespace ps
