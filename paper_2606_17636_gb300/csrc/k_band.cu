// Fused-colour line smoothing of FP32 levels in global memory, in bands held in
// registers (Sec. 3.2; the passes of k_smooth.cu for lines of 32 to 512 cells).
//
// Radial: a group of n / CPL lanes (n the line's cells; CPL = 8, or 16 for 512)
// walks a band of W pairs of neighbouring lines, an even and an odd one: it
// relaxes the next pair's even line, then the odd line between it and the last
// even one, stores the finished pair and moves on.  Each line is read once into
// a ring in shared memory that only its group uses, and nothing is shared
// between groups, so there is no block barrier and no halo copy: the even line
// behind the band's last odd line belongs to the next band and is relaxed twice
// (17/16 of the work at W = 8).  With few planes W falls to 1, so that the
// groups spread over the SMs.  A band's result does not depend on W: every
// relaxation receives the operands of the line-by-line schedule.
// Polar: see k_march below.
//
// Bound by instructions (about 20 a cell and sweep with packed FP32 pairs)
// rather than by bytes.  With 129 planes of 256 x 128 cells a radial pass takes
// 21 us and a polar one 22 (staged passes of k_smooth.cu: 34 and 37; the bytes
// take 15); with 257 planes of 512 x 256, 280 and 143 us (334 and 848; 121).
#include "lines.cuh"

namespace ps {

namespace {

constexpr int kBandThreads = 128;

template <int CPL>
__device__ __forceinline__ void zero_run(float2 (&d)[CPL]) {
#pragma unroll
  for (int c = 0; c < CPL; ++c) d[c] = make_float2(0.f, 0.f);
}
// Entries of cells CPL k .. of a table row (entry of cell i at i + 1).
template <int CPL>
__device__ __forceinline__ void tab_run(float (&d)[CPL], const float* __restrict__ tab, int k) {
#pragma unroll
  for (int q = 0; q < CPL / 2; ++q) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(tab + CPL * k + 2 * q + 1));
    d[2 * q] = v.x;
    d[2 * q + 1] = v.y;
  }
}

// Radial pass.  The lines of the next pairs travel by asynchronous copies into a
// ring of kStages pairs per group (error and right-hand side of both lines), so
// that a pair's latency is hidden behind the relaxations of the one before.
// A line's 16-byte chunk q lies at q ^ ((q >> 3) & 3): the lanes of a
// quarter-warp, CPL / 2 chunks apart, read 8 different bank groups.
constexpr int kStages = 3;
template <int CPL>
__global__ void __launch_bounds__(kBandThreads, CPL == 8 ? 2 : 1)
    k_band(LevelDev L, Batch B, const float2* __restrict__ ein, float2* __restrict__ eout, const float2* __restrict__ f,
           int zero_init, int n_sor, int target) {
  extern __shared__ float4 ring[];
  const int nr = L.nr, nt = L.nt, NR = nr + 2, NT = nt + 2;
  const int pairs = nt / 2, lpl = nr / CPL, gpw = 32 / lpl, hn = nr / 2;
  const int lane = threadIdx.x & 31, k = lane & (lpl - 1), sub = lane / lpl;
  const bool first = k == 0, last = k == lpl - 1;
  const int nact = *B.nact;
  // pairs per band: as many as leave `target` groups
  int W = 1;
  while (W < 8 && 2 * W <= pairs && nact * pairs >= 2 * W * target) W *= 2;
  const int bands = pairs / W, total = nact * bands;
  const int warp = (blockIdx.x * kBandThreads + threadIdx.x) >> 5, warps = gridDim.x * (kBandThreads / 32);
  float4* mine = ring + size_t((threadIdx.x >> 5) * gpw + sub) * kStages * 4 * hn;   // [stage][e0 e1 f0 f1][hn]
  const float* rt = L.rf;
  const float* tt = L.tf;
  float ca[CPL], cb[CPL], cc[CPL], cd[CPL], ce[CPL];   // coefficients that all lines share
  tab_run<CPL>(ca, rt + RT_AE * NR, k);
  tab_run<CPL>(cb, rt + RT_AW * NR, k);
  tab_run<CPL>(cc, rt + RT_P * NR, k);
  tab_run<CPL>(cd, rt + RT_DR * NR, k);
  tab_run<CPL>(ce, rt + RT_Q * NR, k);
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    ca[c] = -ca[c];
    cb[c] = -cb[c];
  }
  auto chunk = [](int q) { return q ^ ((q >> 3) & 3); };
  auto take = [&](float2 (&d)[CPL], const float4* a) {
#pragma unroll
    for (int c = 0; c < CPL / 2; ++c) {
      const float4 v = a[chunk(CPL / 2 * k + c)];
      d[2 * c] = make_float2(v.x, v.y);
      d[2 * c + 1] = make_float2(v.z, v.w);
    }
  };
  for (int w0 = warp * gpw; w0 < total; w0 += warps * gpw) {
    const int item = w0 + sub;
    const bool live = item < total;
    const int kp = live ? item / bands : 0, p0 = live ? (item - kp * bands) * W : 0;
    const int p = B.act[kp];
    const int slot = B.slot ? B.slot[p] : p;
    const float s2 = B.s2f[slot];
    const float* om = L.omr_f + size_t(slot) * nt;
    const size_t base = size_t(p) * nr * nt;
    const float4* ep = reinterpret_cast<const float4*>(ein + base);
    const float4* fp = reinterpret_cast<const float4*>(f + base);
    // pair q of the band into stage (q - p0) % kStages (past the plane: nothing)
    auto fetch = [&](int q) {
      if (q <= p0 + W && q < pairs) {
        float4* d = mine + ((q - p0) % kStages) * 4 * hn;
#pragma unroll
        for (int m = 0; m < CPL / 2; ++m) {
          const int c = k + lpl * m, o = chunk(c);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const size_t g = size_t(2 * q + h) * hn + c;
            if (!zero_init) cp_async_v(d + h * hn + o, ep + g, true);
            cp_async_v(d + (2 + h) * hn + o, fp + g, true);
          }
        }
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    // relax line x (e) with its right-hand side at g0 from the lines after (un) and before (us)
    auto relax = [&](int x, const float4* g0, float2 (&e)[CPL], const float2 (&un)[CPL], const float2 (&us)[CPL]) {
      float2 g[CPL];
      float nid[CPL];
      const float nw = -__ldg(om + x);
      const float aN = __ldg(tt + TT_AN * NT + x + 1), aS = __ldg(tt + TT_AS * NT + x + 1);
      const float Tj = __ldg(tt + TT_T * NT + x + 1), dtj = __ldg(tt + TT_DT * NT + x + 1);
      take(g, g0);
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        g[c] = fma2(-cc[c], fma2(aS, us[c], mul2(aN, un[c])), g[c]);
        nid[c] = -rcp_diag(fmac(-(s2 * ce[c]), Tj, fmac(cc[c], dtj, cd[c])));
      }
      sor_run<CPL>(e, g, ca, cb, nid, nw, first, last, n_sor);
    };
    __syncwarp();   // the last band's reads of the ring are done
    float2 E[CPL], O[CPL], R[CPL], S[CPL];   // the current pair (E relaxed), the next pair
    zero_run<CPL>(S);
    if (p0 > 0 && !zero_init) {   // the line before the band
      const float4* a = ep + size_t(2 * p0 - 1) * hn + CPL / 2 * k;
#pragma unroll
      for (int c = 0; c < CPL / 2; ++c) {
        const float4 v = a[c];
        S[2 * c] = make_float2(v.x, v.y);
        S[2 * c + 1] = make_float2(v.z, v.w);
      }
    }
    fetch(p0);
    fetch(p0 + 1);
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncwarp();
    if (zero_init) {
      zero_run<CPL>(E);
      zero_run<CPL>(O);
    } else {
      take(E, mine);
      take(O, mine + hn);
    }
    relax(2 * p0, mine + 2 * hn, E, O, S);
#pragma unroll 1
    for (int q = p0; q < p0 + W; ++q) {
      const float4* cur = mine + ((q - p0) % kStages) * 4 * hn;
      const float4* nxt = mine + ((q + 1 - p0) % kStages) * 4 * hn;
      fetch(q + 2);   // over the pair before this one, whose reads are done (__syncwarp below)
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      __syncwarp();
      if (zero_init || q + 1 >= pairs) {
        zero_run<CPL>(R);
        zero_run<CPL>(S);
      } else {
        take(R, nxt);
        take(S, nxt + hn);
      }
      // past the plane: a line of zeros whose relaxation is dropped
      relax(min(2 * q + 2, nt - 2), q + 1 < pairs ? nxt + 2 * hn : cur + 2 * hn, R, S, O);
      if (q + 1 == pairs) zero_run<CPL>(R);
      relax(2 * q + 1, cur + 3 * hn, O, R, E);
      __syncwarp();
      if (live) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float4* o = reinterpret_cast<float4*>(eout + base + size_t(2 * q + h) * nr + CPL * k);
#pragma unroll
          for (int c = 0; c < CPL / 2; ++c)
            o[c] = h ? make_float4(O[2 * c].x, O[2 * c].y, O[2 * c + 1].x, O[2 * c + 1].y)
                     : make_float4(E[2 * c].x, E[2 * c].y, E[2 * c + 1].x, E[2 * c + 1].y);
        }
      }
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        E[c] = R[c];
        O[c] = S[c];
      }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  }
}

// Polar / vertical pass as a march (both colours, NS sweeps): a warp takes up to
// 30 pairs of neighbouring columns, one pair per lane, and walks down the rows
// two at a time, so every access is a run of 16 bytes per lane along r and
// nothing is shared but by shuffles.  The even-odd sweeps of a column become a
// pipeline along it: with rows up to r (odd) in, sweep stage s = 1 .. 2 NS updates
// row r - s; the even columns are final 2 NS rows behind, the odd ones, whose
// source needs the final even columns on both sides (own lane and the next),
// 4 NS rows behind.  A lane on either side holds the neighbouring pair (the right
// one relaxes its even column again).  Rows are cut into segments of H when few
// planes are active; a segment starts 4 NS rows early and ends 4 NS rows late,
// the reach of the sweeps, so its rows are bitwise those of the whole columns.
// Rows arrive by asynchronous copies, kAhead pairs ahead, each lane's own.
//
// The staged column tiles of k_smooth.cu take 37 us with 129 planes of 256 x 128
// cells and 848 us with 257 planes of 512 x 256 (one 151 KB block an SM); the
// march 22 and 143 (the bytes take 15 and 121).  A step is bound by its chain of
// dependent multiply-adds with 8 to 12 warps an SM.
constexpr int kAhead = 4;   // row pairs in flight
template <int NS>
__global__ void __launch_bounds__(kBandThreads, 3)
    k_march(LevelDev L, Batch B, const float2* __restrict__ ein, float2* __restrict__ eout, const float2* __restrict__ f,
            int tiles, int width, int target) {
  constexpr int W = 4 * NS + 2, D = 2 * NS, kPad = 2 * D;
  constexpr int kRow = 4;    // float4 per lane and row pair: e, f of both rows
  // per row aN, aS, T, -D_theta, zero beyond the plane (a zero row stays zero
  // through its relaxation); then every warp's ring
  extern __shared__ float4 rowtab[];
  const int nr = L.nr, nt = L.nt, NR = nr + 2, NT = nt + 2, pairs = nr / 2;
  const int lane = threadIdx.x & 31;
  const int nact = *B.nact;
  for (int t = threadIdx.x; t < nt + 2 * kPad; t += kBandThreads) {
    const int j = t - kPad;
    const float* tt = L.tf + j + 1;
    rowtab[t] = j >= 0 && j < nt ? make_float4(tt[TT_AN * NT], tt[TT_AS * NT], tt[TT_T * NT], -tt[TT_DT * NT])
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  int segs = 1;   // segments per column: as many as fill the chip, at least 8 rows each
  while (nt / (2 * segs) >= 8 && nact * tiles * segs * 2 <= target) segs *= 2;
  const int H = nt / segs, per = tiles * segs, total = nact * per;
  const int warp = (blockIdx.x * kBandThreads + threadIdx.x) >> 5, warps = gridDim.x * (kBandThreads / 32);
  const float2 z = make_float2(0.f, 0.f);
  float4* mine = rowtab + nt + 2 * kPad + size_t(threadIdx.x >> 5) * kAhead * kRow * 32 + lane;   // [pair % kAhead][value][lane]
  for (int item = warp; item < total; item += warps) {
    const int kp = item / per, rest = item - kp * per, seg = rest / tiles, tile = rest - seg * tiles;
    const int p = B.act[kp];
    const int slot = B.slot ? B.slot[p] : p;
    const float s2 = B.s2f[slot];
    const int q = tile * width + lane - 1;                         // this lane's pair
    const bool in = q >= 0 && q < pairs, own = in && lane >= 1 && lane <= width;
    const size_t base = size_t(p) * nr * nt + 2 * size_t(in ? q : 0);
    const int hr = nr / 2;                                          // row stride in float4
    // a lane beyond the plane holds zeros: no couplings, any diagonal
    float naE[2], naW[2], nP[2], dr[2], nsQ[2], nw[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = in ? 2 * q + c : 0;
      const float* rt = L.rf + i + 1;
      naE[c] = in ? -rt[RT_AE * NR] : 0.f;
      naW[c] = in ? -rt[RT_AW * NR] : 0.f;
      nP[c] = in ? -rt[RT_P * NR] : 0.f;
      dr[c] = in ? rt[RT_DR * NR] : 1.f;
      nsQ[c] = in ? -(s2 * rt[RT_Q * NR]) : 0.f;
      nw[c] = -L.omt_f[size_t(slot) * nr + i];
    }
    const int r0 = seg * H, r1 = r0 + H;
    // windows by distance from the newest row: errors of both columns, the odd
    // column's right-hand side, sources and coefficients of the rows in flight
    float2 E[W], O[W], F1[D + 2], G0[D + 1], G1[D + 1];
    float id0[D + 1], up0[D + 1], dn0[D + 1], id1[D + 1], up1[D + 1], dn1[D + 1];
#pragma unroll
    for (int d = 0; d < W; ++d) E[d] = O[d] = z;
#pragma unroll
    for (int d = 0; d < D + 2; ++d) F1[d] = z;
#pragma unroll
    for (int d = 0; d <= D; ++d) {
      G0[d] = G1[d] = z;
      id0[d] = up0[d] = dn0[d] = id1[d] = up1[d] = dn1[d] = 0.f;
    }
    const int x0 = max(r0 - 2 * D, 0), x1 = r1 + 2 * D;   // rows x, x + 1 enter, x - 2 D and the next leave
    // rows x, x + 1 of e and f (zeros beyond the plane); every lane reads only its own copies
    const float4* ge = reinterpret_cast<const float4*>(ein + base) + size_t(x0) * hr;
    const float4* gf = reinterpret_cast<const float4*>(f + base) + size_t(x0) * hr;
    int fx = x0;
    auto fetch = [&]() {
      float4* d = mine + ((fx >> 1) % kAhead) * kRow * 32;
      const bool ok = in && fx < nt;
      const size_t o = ok ? hr : 0;
      cp_async_v(d, ok ? ge : reinterpret_cast<const float4*>(ein), ok);
      cp_async_v(d + 32, (ok ? ge : reinterpret_cast<const float4*>(ein)) + o, ok);
      cp_async_v(d + 64, ok ? gf : reinterpret_cast<const float4*>(f), ok);
      cp_async_v(d + 96, (ok ? gf : reinterpret_cast<const float4*>(f)) + o, ok);
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      ge += 2 * hr;
      gf += 2 * hr;
      fx += 2;
    };
    auto coeff = [&](const float4& t, int c, float& id, float& up, float& dn) {
      id = -rcp_diag(fmac(nsQ[c], t.z, fmac(nP[c], t.w, dr[c])));
      up = nP[c] * t.x;
      dn = nP[c] * t.y;
    };
#pragma unroll
    for (int a = 0; a < kAhead - 1; ++a) fetch();
    float4* out = reinterpret_cast<float4*>(eout + base) + size_t(x0) * hr - size_t(2 * D) * hr;
    constexpr int kSteps = 4;   // unrolled: the windows move by renaming
#pragma unroll kSteps
    for (int x = x0; x < x1; x += 2) {
      const int s0 = x - 2 * D;
      fetch();   // over the pair that left the last step
      asm volatile("cp.async.wait_group %0;\n" ::"n"(kAhead - 1) : "memory");
      const float4* row = mine + ((x >> 1) % kAhead) * kRow * 32;
#pragma unroll
      for (int d = W - 1; d >= 2; --d) {
        E[d] = E[d - 2];
        O[d] = O[d - 2];
      }
#pragma unroll
      for (int d = D + 1; d >= 2; --d) F1[d] = F1[d - 2];
#pragma unroll
      for (int d = D; d >= 2; --d) {
        G0[d] = G0[d - 2]; id0[d] = id0[d - 2]; up0[d] = up0[d - 2]; dn0[d] = dn0[d - 2];
        G1[d] = G1[d - 2]; id1[d] = id1[d - 2]; up1[d] = up1[d - 2]; dn1[d] = dn1[d - 2];
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // h = 0: row x (distance 1), h = 1: row x + 1 (distance 0)
        const int d = 1 - h;
        const float4 ne = row[h * 32], nf = row[(2 + h) * 32];
        E[d] = make_float2(ne.x, ne.y);
        O[d] = make_float2(ne.z, ne.w);
        F1[d] = make_float2(nf.z, nf.w);
        float2 w;
        w.x = __shfl_up_sync(0xffffffffu, O[d].x, 1);
        w.y = __shfl_up_sync(0xffffffffu, O[d].y, 1);
        G0[d] = fma2(naW[0], w, fma2(naE[0], O[d], make_float2(nf.x, nf.y)));
        coeff(rowtab[x + h + kPad], 0, id0[d], up0[d], dn0[d]);
      }
#pragma unroll
      for (int s = 1; s <= D; ++s) {
        const float2 r = fma2(dn0[s], E[s + 1], fma2(up0[s], E[s - 1], G0[s]));
        E[s] = fma2(nw[0], fma2(id0[s], r, E[s]), E[s]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // the odd column's next rows: their even neighbours are final
        const int d = 1 - h;
        float2 e;
        e.x = __shfl_down_sync(0xffffffffu, E[D + d].x, 1);
        e.y = __shfl_down_sync(0xffffffffu, E[D + d].y, 1);
        G1[d] = fma2(naW[1], E[D + d], fma2(naE[1], e, F1[D + d]));
        coeff(rowtab[x + h - D + kPad], 1, id1[d], up1[d], dn1[d]);
      }
#pragma unroll
      for (int s = 1; s <= D; ++s) {
        const float2 r = fma2(dn1[s], O[D + s + 1], fma2(up1[s], O[D + s - 1], G1[s]));
        O[D + s] = fma2(nw[1], fma2(id1[s], r, O[D + s]), O[D + s]);
      }
      if (own && s0 >= r0 && s0 < r1) {
        out[0] = make_float4(E[W - 1].x, E[W - 1].y, O[W - 1].x, O[W - 1].y);
        out[hr] = make_float4(E[W - 2].x, E[W - 2].y, O[W - 2].x, O[W - 2].y);
      }
      out += 2 * hr;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  }
}

bool run_length(int n) { return n >= 32 && n <= 512; }

template <int CPL>
void radial(const LevelDev& L, const Batch& B, const float2* ein, float2* eout, const float2* f, bool zi, int n_sor,
            cudaStream_t st) {
  const int pairs = L.nt / 2, gpw = 32 / (L.nr / CPL);
  constexpr int kBlocks = CPL == 8 ? 2 : 1;
  const size_t sm = size_t(kBandThreads / 32) * gpw * kStages * 4 * (L.nr / 2) * sizeof(float4);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_band<CPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * kStages * 32 * CPL * 32);
    attr = true;
  }
  const int resident = sm_count() * kBlocks * (kBandThreads / 32) * gpw;   // groups at once
  const long most = long(B.max_planes) * pairs;                            // bands of one pair
  const long warps = ((most < resident ? most : resident) + gpw - 1) / gpw;
  k_band<CPL><<<unsigned((warps + kBandThreads / 32 - 1) / (kBandThreads / 32)), kBandThreads, sm, st>>>(
      L, B, ein, eout, f, zi ? 1 : 0, n_sor, resident);
}

template <int NS>
void march(const LevelDev& L, const Batch& B, const float2* ein, float2* eout, const float2* f, cudaStream_t st) {
  const int pairs = L.nr / 2, tiles = (pairs + 29) / 30, width = (pairs + tiles - 1) / tiles;
  const int resident = sm_count() * 3 * (kBandThreads / 32);
  const long most = long(B.max_planes) * tiles * (L.nt / 8);
  const long warps = most < resident ? most : resident;
  const size_t sm = (size_t(L.nt) + 8 * NS + (kBandThreads / 32) * kAhead * 4 * 32) * sizeof(float4);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_march<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024);
    attr = true;
  }
  k_march<NS><<<unsigned((warps + kBandThreads / 32 - 1) / (kBandThreads / 32)), kBandThreads, sm, st>>>(L, B, ein, eout, f, tiles, width, resident);
}

}  // namespace

// The lines held in registers, and enough of them to fill the chip: below about
// 1.5 M cells over all planes the staged passes' shorter way through a launch
// wins by 1 to 2 us a pass (64 x 64 x 33 planes, two cycles: 43 us against 44;
// 128 x 64 x 129: 62 against 67; above, 256 x 64 x 129: 88 against 79,
// 256 x 128 x 129: 168 against 116, 512 x 256 x 33: 206 against 150).  planes
// counts the batch, not the active ones: above the line the register passes also
// win with few planes active (an iteration's smoothing and update, staged against
// here: 17 of 129 planes of 256 x 128 92 and 65 us, 6 of 65 of 512 x 256 200 and
// 145, 33 of 257 of 256 x 64 84 and 64).
bool band_pays(int nr, int nt, int n_sor, int planes) {
  return run_length(nr) && run_length(nt) && n_sor >= 1 && n_sor <= 3 && long(planes) * nr * nt >= 1500000l;
}

void launch_band_radial(const LevelDev& L, const Batch& B, const float2* ein, float2* eout, const float2* f, bool zero_init,
                        int n_sor, cudaStream_t st) {
  if (L.nr > 256) radial<16>(L, B, ein, eout, f, zero_init, n_sor, st);
  else radial<8>(L, B, ein, eout, f, zero_init, n_sor, st);
}

void launch_march(const LevelDev& L, const Batch& B, const float2* ein, float2* eout, const float2* f, int n_sor,
                  cudaStream_t st) {
  if (n_sor == 1) march<1>(L, B, ein, eout, f, st);
  else if (n_sor == 2) march<2>(L, B, ein, eout, f, st);
  else march<3>(L, B, ein, eout, f, st);
}

}  // namespace ps
