// Azimuthal transforms (Sec. 2.2): real rows of n_phi values along phi, two
// rows packed as one complex sequence, split into the two half spectra
// (m = 0..N/2) and written transposed to the mode-major plane layout
// [m][j][i].  The inverse rebuilds the full Hermitian spectrum of two rows,
// transforms, and writes the real and imaginary outputs as the two rows.
//
// Arithmetic: block fixed point in 64-bit integers.  GB300 does two FP64
// operations a clock and SM, against 64 or more integer ones, and an FP64
// radix-2 transform kept that pipe 83 % busy: 282 us forward and 273 us inverse
// for 256 x 128 rows of 256 values (152 us of pipe time at best for
// 5 N log2 N operations), where the bytes take 20 us.  In fixed point an
// addition is two integer instructions and a twiddle product twelve 32-bit
// multiplies; the same transforms take 61 and 79 us, bound by the issue of 41 and
// 54 million warp instructions (integer ALU pipe 56 % busy, 16 warps an SM at 128
// registers).  Zero times a twiddle is zero, so that modes which cancel exactly,
// those of rows constant or periodic along phi, come out as zeros and retire at
// their first residual.
//
// Scaling: a row's values are aligned to its largest exponent (a power of two
// each, so scaling a row scales its spectrum exactly).  Every partial sum of a
// transform is bounded by the sum of the magnitudes that enter it, so a row is
// scaled to bring that sum (formed in FP32, rounded up) just below 2^61: no
// step can overflow, and a row with one dominant value keeps all its 53 bits with
// room below.  A flat row of N values would keep 61 - log2 N; from 128 values on
// the first pass is scaled by the smaller bound radix x maximum instead and the
// twiddle products shift the rest out, so that flat rows keep all 53 too.  What
// error remains is that of the twiddle products and the final rounding to FP64.
// Relative to a row's 2-norm, against extended precision, here and in FP64 radix 2
// (rms over 400 rows of 256 values, in 1e-17): white noise 5.3 and 34, a bump 5.3
// and 33, 1 + 1 % noise 4.5 and 14, 1 + 0.01 cos 1.6 and 2.8, constant rows 5.0
// and 4.9 (the final rounding alone); the inverse 4.1 to 5.5 and 4.1 to 48.
// A row pair with an infinity or NaN gives NaN, as FP64 arithmetic does.
//
// Work split: N / 16 threads per row pair, 16 values in a thread's registers;
// passes of radix 16, 8 or 4 with one exchange through shared memory between
// them.  A block takes several pairs, so that its transposed accesses cover
// whole sectors (16 rows: 256 contiguous bytes per mode).
#include <climits>
#include <cmath>
#include <cstdio>
#include <vector>

#include "kernels.h"

namespace ps {

namespace {

typedef long long i64;
typedef unsigned long long u64;

struct Z {
  i64 x, y;
};
__device__ __forceinline__ Z operator+(Z a, Z b) { return Z{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Z operator-(Z a, Z b) { return Z{a.x - b.x, a.y - b.y}; }

// Constants w = (h 2^32 + l) 2^-62, |w| <= 1, -2^31 <= l < 2^31.
constexpr int kR_h = 759250125, kR_l = -25716447;   // sqrt(1/2)
constexpr int kC_h = 992008094, kC_l = 1696238673;   // cos(pi / 8)
constexpr int kS_h = 410903207, kS_l = -1364630830;   // sin(pi / 8)

// x = h 2^32 + l with the same range of l: one instruction, l being the low word as
// it stands (with l unsigned, the product left out below had a mean to add: nonzero
// for x = 0, and 66 and 84 us against 59 and 78 for the transforms above).
__device__ __forceinline__ int hi32(i64 x) { return int(x >> 32) + int(unsigned(x) >> 31); }
__device__ __forceinline__ int lo32(i64 x) { return int(unsigned(x)); }
__device__ __forceinline__ i64 mulw(int a, int b) { return i64(a) * i64(b); }

// x w for |x| < 2^62.5, rounded but for the product of the low halves, which is
// left out: at most one unit, of either sign alike, and zero where x has no low
// half, so that zero times w is zero.
__device__ __forceinline__ i64 mulq(i64 x, int h, int l) {
  const int xh = hi32(x), xl = lo32(x);
  return (mulw(xh, h) << 2) + ((mulw(xh, l) + mulw(xl, h) + (1 << 29)) >> 30);
}
// z (wr + i wi) for |z| <= 2^62 and |w| <= 1: the sums of the mixed products stay
// below 2^62 + 2^61.5 (high half of z times low half of w, and the other way round).
__device__ __forceinline__ Z mulz(Z z, int rh, int rl, int ih, int il) {
  const int xh = hi32(z.x), xl = lo32(z.x), yh = hi32(z.y), yl = lo32(z.y);
  const i64 a = mulw(xh, rh) - mulw(yh, ih), b = mulw(xh, ih) + mulw(yh, rh);
  const i64 c = mulw(xh, rl) + mulw(xl, rh) - mulw(yh, il) - mulw(yl, ih);
  const i64 d = mulw(xh, il) + mulw(xl, ih) + mulw(yh, rl) + mulw(yl, rh);
  return Z{(a << 2) + ((c + (1 << 29)) >> 30), (b << 2) + ((d + (1 << 29)) >> 30)};
}

// SIGN < 0: e^{-2 pi i}, SIGN > 0: e^{+2 pi i}.
template <int SIGN>
__device__ __forceinline__ Z rot90(Z z) {   // z times e^{SIGN i pi / 2}
  return SIGN < 0 ? Z{z.y, -z.x} : Z{-z.y, z.x};
}
template <int SIGN>
__device__ __forceinline__ void fft4(Z& a, Z& b, Z& c, Z& d) {
  const Z s = a + c, t = a - c, u = b + d, v = rot90<SIGN>(b - d);
  a = s + u;
  b = t + v;
  c = s - u;
  d = t - v;
}
template <int SIGN>
__device__ __forceinline__ Z rot45(Z z) {   // z times e^{SIGN i pi / 4}
  const i64 s = mulq(z.x + z.y, kR_h, kR_l), d = mulq(z.y - z.x, kR_h, kR_l);
  return SIGN < 0 ? Z{s, d} : Z{-d, s};
}
template <int SIGN>
__device__ __forceinline__ Z rot225(Z z, bool swap) {   // z times e^{SIGN i pi / 8}, or of 3 pi / 8 with swap
  const int ch = swap ? kS_h : kC_h, cl = swap ? kS_l : kC_l, sh = swap ? kC_h : kS_h, sl = swap ? kC_l : kS_l;
  return SIGN < 0 ? mulz(z, ch, cl, -sh, -sl) : mulz(z, ch, cl, sh, sl);
}

// Radix-R butterflies on R registers, outputs in natural order.
template <int R, int SIGN>
__device__ __forceinline__ void butterfly(Z* v) {
  if constexpr (R == 4) {
    fft4<SIGN>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    Z e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    fft4<SIGN>(e[0], e[1], e[2], e[3]);
    fft4<SIGN>(o[0], o[1], o[2], o[3]);
    o[1] = rot45<SIGN>(o[1]);
    o[2] = rot90<SIGN>(o[2]);
    o[3] = rot45<SIGN>(rot90<SIGN>(o[3]));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = e[k] + o[k];
      v[k + 4] = e[k] - o[k];
    }
  } else {
    static_assert(R == 16, "radix");
#pragma unroll
    for (int i = 0; i < 4; ++i) fft4<SIGN>(v[i], v[i + 4], v[i + 8], v[i + 12]);   // v[i + 4 k]
    v[5] = rot225<SIGN>(v[5], false);                  // W^1
    v[9] = rot45<SIGN>(v[9]);                          // W^2
    v[13] = rot225<SIGN>(v[13], true);                 // W^3
    v[6] = rot45<SIGN>(v[6]);                          // W^2
    v[10] = rot90<SIGN>(v[10]);                        // W^4
    v[14] = rot45<SIGN>(rot90<SIGN>(v[14]));           // W^6
    v[7] = rot225<SIGN>(v[7], true);                   // W^3
    v[11] = rot45<SIGN>(rot90<SIGN>(v[11]));           // W^6
    {
      const Z w = rot225<SIGN>(v[15], false);          // W^9 = -W^1
      v[15] = Z{-w.x, -w.y};
    }
    Z o[16];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      fft4<SIGN>(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
#pragma unroll
      for (int l = 0; l < 4; ++l) o[k + 4 * l] = v[4 * k + l];
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = o[k];
  }
}

// Passes of a transform of N values: radix of pass p (1: no such pass).
__host__ __device__ constexpr int radix(int N, int p) {
  return N <= 16 ? (p == 0 ? N : 1)
       : N == 32 ? (p == 0 ? 8 : p == 1 ? 4 : 1)
       : N == 64 ? (p < 2 ? 8 : 1)
       : N == 128 ? (p == 0 ? 16 : p == 1 ? 8 : 1)
       : N == 256 ? (p < 2 ? 16 : 1)
       : N == 512 ? (p < 3 ? 8 : 1)
                  : (p == 0 ? 16 : p < 3 ? 8 : 1);
}
__host__ __device__ constexpr int length(int N, int p) { return p == 0 ? N : length(N, p - 1) / radix(N, p - 1); }
__host__ __device__ constexpr int ilog(int n) { return n <= 1 ? 0 : 1 + ilog(n / 2); }
__host__ __device__ constexpr int values(int N) { return N < 16 ? N : 16; }
// Offset of pass p's twiddles in the table: [r][t], r < radix, t < length / radix.
__host__ __device__ constexpr int table_at(int N, int p) { return p == 0 ? 0 : table_at(N, p - 1) + length(N, p - 1); }

// Position of element `pos` of a sequence in shared memory (16-byte units):
// padded so that the strided accesses of the passes and of the output fall on
// different bank groups.
template <int N>
__host__ __device__ constexpr int padded(int pos) {
  return N >= 512 ? pos + (pos >> 3) + (pos >> 6) : N == 256 ? pos + (pos >> 4) : N >= 64 ? pos + (pos >> 3) : pos + (pos >> 2);
}
template <int N>
__host__ __device__ constexpr int region() {   // per row pair; odd, at least the two raw half spectra
  return (padded<N>(N - 1) + 1 > N + 2 ? padded<N>(N - 1) + 1 : N + 2) | 1;
}
// Where output m lies after the passes (digit-reversed).
template <int N>
__device__ __forceinline__ int place(int m) {
  constexpr int R0 = radix(N, 0), R1 = radix(N, 1), M1 = N / R0, M2 = M1 / R1;
  const int r0 = m % R0, r1 = (m / R0) % R1, r2 = m / (R0 * R1);
  return padded<N>(r0 * M1 + r1 * M2 + r2);
}

__device__ __forceinline__ i64 shr_round(i64 v, int s) { return (v + ((1ll << s) >> 1)) >> s; }

// The passes from P on; the first takes its input in v (element q of
// butterfly g at g + (N / R) q), the others from shared memory S.  D: the bits
// that the twiddle products shift out over all passes.
template <int N, int SIGN, int P>
__device__ __forceinline__ void passes(Z (&v)[values(N)], longlong2* S, const int4* __restrict__ tw, int t, int D) {
  constexpr int V = values(N), T = N / V, R = radix(N, P), M = length(N, P), L = M / R, NB = V / R;
  constexpr bool last = radix(N, P + 1) == 1;
  if constexpr (P > 0) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int g = t + T * b, at = (g / L) * M + g % L;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const longlong2 s = S[padded<N>(at + L * q)];
        v[b * R + q] = Z{s.x, s.y};
      }
    }
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) butterfly<R, SIGN>(v + b * R);
  if constexpr (!last) {
    // two passes: all of D here; three: what the second pass does not need
    const int first = radix(N, 2) == 1 ? D : min(D, ilog(radix(N, 1)));
    const int s = P == 0 ? first : D - first;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int g = t + T * b;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int4 w = __ldg(tw + table_at(N, P) + r * L + g % L);
        Z z = mulz(v[b * R + r], w.x, w.y, w.z, w.w);
        if constexpr (N >= 128) z = Z{shr_round(z.x, s), shr_round(z.y, s)};
        v[b * R + r] = z;
      }
    }
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int g = t + T * b, at = (g / L) * M + g % L;
#pragma unroll
    for (int r = 0; r < R; ++r) S[padded<N>(at + L * r)] = make_longlong2(v[b * R + r].x, v[b * R + r].y);
  }
  __syncthreads();
  if constexpr (!last) passes<N, SIGN, P + 1>(v, S, tw, t, D);
}

// ---- binary64 <-> fixed point ---------------------------------------------------
__device__ __forceinline__ int exponent(u64 b) { return int((b >> 52) & 0x7ff); }
__device__ __forceinline__ u64 significand(u64 b) {
  const u64 f = b & 0xfffffffffffffull;
  return exponent(b) ? f | (1ull << 52) : f;
}
// The magnitude in units of 2^(em - 1023) as FP32, within 2^-23 below it (a
// subnormal value counts as the smallest normal one with its fraction).
__device__ __forceinline__ float magnitude(u64 b, int em) {
  const int d = em - max(exponent(b), 1);
  return d > 126 ? 0.f : __uint_as_float((unsigned(127 - d) << 23) | (unsigned(b >> 29) & 0x7fffffu));
}
// The value in units of 2^(em - 1075 - sh), rounded; sh <= 7.
__device__ __forceinline__ i64 to_fixed(u64 b, int em, int sh) {
  const int r = em - max(exponent(b), 1) + 7 - sh;
  const u64 m = r > 61 ? 0ull : (((significand(b) << 8) >> r) + 1ull) >> 1;
  return i64(b) < 0 ? -i64(m) : i64(m);
}
// v 2^e with |v| < 2^63, rounded to nearest even: in integer
// arithmetic where the value has more than 32 bits and e (safe: |e| < 900)
// keeps the result normal, else through the FP64 pipe.
__device__ __forceinline__ bool safe_exponent(int e) { return e > -900 && e < 900; }
__device__ __forceinline__ double to_double(i64 v, int e, bool safe) {
  const unsigned s = unsigned(v >> 63), hi0 = unsigned(v >> 32) ^ s, lo0 = unsigned(v) ^ s;
  const u64 u = ((u64(hi0) << 32) | lo0) + (s & 1u);   // |v|
  const unsigned hi = unsigned(u >> 32);
  if (hi == 0u || !safe) return v == 0 ? 0.0 : scalbn(__ll2double_rn(v), e);
  const int lz = __clz(int(hi)) - 1;                    // leading bit to position 62
  const u64 n = u << lz;
  const u64 m = (n + (0x1ffu + ((unsigned(n) >> 10) & 1u))) >> 10;   // 53 bits (2^53 when the rounding carries)
  const unsigned top = unsigned(e + 1023 + 61 - lz) << 20;   // biased exponent less one: the leading bit adds it
  return __hiloint2double(int((unsigned(m >> 32) + top) | (s << 31)), int(unsigned(m)));
}

// Largest exponent and sum of magnitudes over a row pair's T threads.
template <int T>
__device__ __forceinline__ int row_max(int x, int* red) {
  constexpr int W = T < 32 ? T : 32;
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
  if constexpr (T > 32) {   // two warps per row pair
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) red[w] = x;
    __syncthreads();
    x = max(red[w & ~1], red[w | 1]);
    __syncthreads();
  }
  return x;
}
template <int T>
__device__ __forceinline__ float row_sum(float x, int* red) {
  constexpr int W = T < 32 ? T : 32;
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if constexpr (T > 32) {
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) red[w] = __float_as_int(x);
    __syncthreads();
    x = __int_as_float(red[w & ~1]) + __int_as_float(red[w | 1]);
    __syncthreads();
  }
  return x;
}

// Left shift of a row's values from units of 2^(em - 1075), given the sum of
// their magnitudes in units of 2^(em - 1023), and the bits by which the whole
// sum then exceeds 2^61 (from 128 values on: the first pass only meets radix
// values below 2^(em - 1022) of each row, in the inverse transform with a factor
// sqrt(2) for their two parts, 2^61.5 in all; else 0).
struct RowScale {
  int sh, drop;
};
template <int N>
__device__ __forceinline__ RowScale row_scale(float sum) {
  // at most 1e-4 too small, whatever rounding down the magnitudes met
  const int top = int(__float_as_uint(fmaxf(sum, 1.f) * 1.0001f) >> 23) - 127;   // sum < 2^(top + 1)
  RowScale s;
  s.sh = min(8 - top, 7);
  s.drop = 0;
  if constexpr (N >= 128) {
    constexpr int cap = ilog(radix(N, 0)) + 1;
    if (top > cap) {
      s.sh = 8 - cap;
      s.drop = top - cap;
    }
  }
  return s;
}

// Marks in place of a row's exponent: a pair with an infinity or NaN, and a row
// of zeros (whose transform is exactly zero beside another row's rounding errors).
constexpr int kBadRow = INT_MAX, kZeroRow = INT_MIN;
__device__ __forceinline__ double from_row(i64 v, int e) {
  if (e == kBadRow) return __longlong_as_double(0x7ff8000000000000ll);
  if (e == kZeroRow) return 0.0;
  return to_double(v, e, safe_exponent(e));
}

template <int N>
struct Split {
  static constexpr int V = values(N), T = N / V;
  static constexpr int kPairs = T >= 64 ? 4 : (128 / T > 8 ? (128 / T > 64 ? 64 : 128 / T) : 8);   // row pairs per block
};

template <int N>
__global__ void __launch_bounds__(256, 2) k_fft_fwd(const double* __restrict__ rho, double2* __restrict__ out, int nr,
                                                    int nt, FftTables tab, int pairs) {
  constexpr int V = values(N), T = N / V, R = radix(N, 0), L = N / R, NB = V / R, M = N / 2 + 1;
  extern __shared__ __align__(16) unsigned char fraw[];
  longlong2* S = reinterpret_cast<longlong2*>(fraw);
  __shared__ int eo[128];
  __shared__ int redi[8];
  const int pair = threadIdx.x / T, t = threadIdx.x % T, j = blockIdx.y;
  const int i0 = blockIdx.x * 2 * pairs, ia = i0 + 2 * pair;
  const double* ra = rho + (size_t(min(ia, nr - 1)) * nt + j) * N;
  const double* rb = rho + (size_t(min(ia + 1, nr - 1)) * nt + j) * N;
  const bool oka = ia < nr, okb = ia + 1 < nr;
  u64 a[V], b[V];
  int ea = 0, eb = 0;
#pragma unroll
  for (int g = 0; g < NB; ++g)
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int n = t + T * g + L * q;
      a[g * R + q] = oka ? u64(__double_as_longlong(ra[n])) : 0ull;
      b[g * R + q] = okb ? u64(__double_as_longlong(rb[n])) : 0ull;
    }
#pragma unroll
  for (int q = 0; q < V; ++q) {
    ea = max(ea, exponent(a[q]));
    eb = max(eb, exponent(b[q]));
  }
  ea = max(row_max<T>(ea, redi), 1);
  eb = max(row_max<T>(eb, redi), 1);
  const bool bad = ea == 0x7ff || eb == 0x7ff || tab.bad;
  float sa = 0.f, sb = 0.f;
  u64 na = 0ull, nb = 0ull;   // nonzero values met
#pragma unroll
  for (int q = 0; q < V; ++q) {
    sa += magnitude(a[q], ea);
    sb += magnitude(b[q], eb);
    na |= a[q] << 1;
    nb |= b[q] << 1;
  }
  const int any_a = row_max<T>(na ? 1 : 0, redi), any_b = row_max<T>(nb ? 1 : 0, redi);
  const RowScale A = row_scale<N>(row_sum<T>(sa, redi)), B = row_scale<N>(row_sum<T>(sb, redi));
  const int D = max(A.drop, B.drop);
  Z v[V];
#pragma unroll
  for (int q = 0; q < V; ++q) v[q] = Z{to_fixed(a[q], ea, A.sh), to_fixed(b[q], eb, B.sh)};
  if (t == 0) {   // exponents of the spectra, the split's halving and the scale's power of two included
    eo[2 * pair] = bad ? kBadRow : any_a ? ea - 1075 - A.sh + D + tab.es - 1 : kZeroRow;
    eo[2 * pair + 1] = bad ? kBadRow : any_b ? eb - 1075 - B.sh + D + tab.es - 1 : kZeroRow;
  }
  passes<N, -1, 0>(v, S + size_t(pair) * region<N>(), tab.fwd, t, D);
  // X_a = (Z[m] + conj Z[N-m]) / 2,  X_b = (Z[m] - conj Z[N-m]) / (2i); a
  // pair's two rows are 32 contiguous bytes, the block's pairs lie side by side
  const int lg = 31 - __clz(pairs);
  for (int idx = threadIdx.x; idx < M * pairs; idx += blockDim.x) {
    const int m = idx >> lg, p = idx & (pairs - 1), i = i0 + 2 * p;
    if (i >= nr) continue;
    const longlong2* Sp = S + size_t(p) * region<N>();
    const longlong2 z = Sp[place<N>(m)], c = Sp[place<N>((N - m) & (N - 1))];
    const int xa = eo[2 * p], xb = eo[2 * p + 1];
    double2 ua = make_double2(from_row(z.x + c.x, xa), from_row(z.y - c.y, xa));
    double2 ub = make_double2(from_row(z.y + c.y, xb), from_row(c.x - z.x, xb));
    if constexpr (N <= 16) {   // no twiddles: the scale is still to come
      ua = make_double2(ua.x * tab.post, ua.y * tab.post);
      ub = make_double2(ub.x * tab.post, ub.y * tab.post);
    }
    double2* o = out + (size_t(m) * nt + j) * nr + i;
    o[0] = ua;
    if (i + 1 < nr) o[1] = ub;
  }
}

template <int N>
__global__ void __launch_bounds__(256, 2) k_fft_inv(const double2* __restrict__ fh, double* __restrict__ phi, int nr,
                                                    int nt, FftTables tab, int pairs) {
  constexpr int V = values(N), T = N / V, R = radix(N, 0), L = N / R, M = N / 2 + 1;
  extern __shared__ __align__(16) unsigned char fraw[];
  longlong2* S = reinterpret_cast<longlong2*>(fraw);
  __shared__ int eo[128], em[128];   // exponents of the outputs; of the inputs
  __shared__ float sum[128];
  __shared__ int some[128];   // a nonzero value met
  const int pair = threadIdx.x / T, t = threadIdx.x % T, j = blockIdx.y;
  const int i0 = blockIdx.x * 2 * pairs, lg = 32 - __clz(pairs), rows = 2 * pairs;
  for (int r = threadIdx.x; r < rows; r += blockDim.x) {
    em[r] = 1;
    sum[r] = 0.f;
    some[r] = 0;
  }
  __syncthreads();
  // the raw half spectra of the block's rows: row r of pair p at p region +
  // (r & 1) M + m; a thread meets rows r0, r0 + step, ... (one or two)
  constexpr int B8 = 8;   // loads in flight per thread
  for (int idx = threadIdx.x; idx < M * rows; idx += B8 * blockDim.x) {
    longlong2 v[B8];
#pragma unroll
    for (int q = 0; q < B8; ++q) {
      const int at = idx + q * blockDim.x, m = at >> lg, r = at & (rows - 1);
      v[q] = make_longlong2(0, 0);
      if (at < M * rows && i0 + r < nr) {
        const double2 x = fh[(size_t(m) * nt + j) * nr + i0 + r];
        v[q].x = __double_as_longlong(x.x);
        if (m != 0 && m != N / 2) v[q].y = __double_as_longlong(x.y);   // only real parts of m = 0, N/2
      }
    }
#pragma unroll
    for (int q = 0; q < B8; ++q) {
      const int at = idx + q * blockDim.x, m = at >> lg, r = at & (rows - 1);
      if (at >= M * rows) break;
      S[size_t(r >> 1) * region<N>() + (r & 1) * M + m] = v[q];
      const int e = max(exponent(u64(v[q].x)), exponent(u64(v[q].y)));
      if (e > em[r]) atomicMax(&em[r], e);
      if ((u64(v[q].x | v[q].y) << 1) && !some[r]) some[r] = 1;
    }
  }
  __syncthreads();
  {   // sums of magnitudes (both halves of the spectrum: twice the stored one's), in a fixed order
    constexpr int W = T < 32 ? T : 32;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 2 * pair + h, e = em[r];
      const longlong2* X = S + size_t(pair) * region<N>() + h * M;
      float s = 0.f;
      for (int m = t; m < M; m += T) s += magnitude(u64(X[m].x), e) + magnitude(u64(X[m].y), e);
#pragma unroll
      for (int o = W / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (t % W == 0) atomicAdd(&sum[r], s);   // at most two terms: any order gives the same sum
    }
  }
  __syncthreads();
  const bool bad = em[2 * pair] == 0x7ff || em[2 * pair + 1] == 0x7ff;
  const RowScale A = row_scale<N>(2.f * sum[2 * pair]), B = row_scale<N>(2.f * sum[2 * pair + 1]);
  const int D = max(A.drop, B.drop), ea = em[2 * pair], eb = em[2 * pair + 1];
  longlong2* Sp = S + size_t(pair) * region<N>();
  for (int m = t; m < M; m += T) {   // to fixed point, in place
    const longlong2 a = Sp[m], b = Sp[M + m];
    Sp[m] = make_longlong2(to_fixed(u64(a.x), ea, A.sh), to_fixed(u64(a.y), ea, A.sh));
    Sp[M + m] = make_longlong2(to_fixed(u64(b.x), eb, B.sh), to_fixed(u64(b.y), eb, B.sh));
  }
  if (t == 0) {
    eo[2 * pair] = bad ? kBadRow : some[2 * pair] ? ea - 1075 - A.sh + D : kZeroRow;
    eo[2 * pair + 1] = bad ? kBadRow : some[2 * pair + 1] ? eb - 1075 - B.sh + D : kZeroRow;
  }
  __syncthreads();
  Z v[V];
#pragma unroll
  for (int k = 0; k < V; ++k) {   // Z = X_a + i X_b, the upper half by conjugation
    const int n = t + T * (k / R) + L * (k % R), m = n < M ? n : N - n;
    const longlong2 a = Sp[m], b = Sp[M + m];
    v[k] = n < M ? Z{a.x - b.y, a.y + b.x} : Z{a.x + b.y, b.x - a.y};
  }
  __syncthreads();   // the spectra are read
  passes<N, +1, 0>(v, Sp, tab.inv, t, D);
  for (int idx = threadIdx.x; idx < N * pairs; idx += blockDim.x) {
    const int p = idx / N, n = idx % N, i = i0 + 2 * p;
    if (i >= nr) continue;
    const longlong2 z = S[size_t(p) * region<N>() + place<N>(n)];
    phi[(size_t(i) * nt + j) * N + n] = from_row(z.x, eo[2 * p]);
    if (i + 1 < nr) phi[(size_t(i + 1) * nt + j) * N + n] = from_row(z.y, eo[2 * p + 1]);
  }
}

// Row pairs per block for nr rows: the split's, fewer when the rows are fewer.
template <int N>
int pairs_for(int nr) {
  int p = Split<N>::kPairs;
  while (p > 1 && Split<N>::T * p > 32 && p >= nr) p /= 2;   // at least a warp, half of the pairs used
  return p;
}

template <int N>
void forward(const double* rho, double2* f, int nr, int nt, const FftTables& tab, cudaStream_t st) {
  const int pairs = pairs_for<N>(nr);
  const size_t sm = size_t(pairs) * region<N>() * sizeof(longlong2);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_fft_fwd<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
    attr = true;
  }
  k_fft_fwd<N><<<dim3((nr + 2 * pairs - 1) / (2 * pairs), nt), Split<N>::T * pairs, sm, st>>>(rho, f, nr, nt, tab, pairs);
}
template <int N>
void inverse(const double2* fh, double* phi, int nr, int nt, const FftTables& tab, cudaStream_t st) {
  const int pairs = pairs_for<N>(nr);
  const size_t sm = size_t(pairs) * region<N>() * sizeof(longlong2);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_fft_inv<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
    attr = true;
  }
  k_fft_inv<N><<<dim3((nr + 2 * pairs - 1) / (2 * pairs), nt), Split<N>::T * pairs, sm, st>>>(fh, phi, nr, nt, tab, pairs);
}

}  // namespace

// Twiddles of both transforms of length N as (h, l) pairs of cos and sin in
// units of 2^-62; the forward's first pass carries the scale's mantissa.
// Lengths of one pass have no twiddles: the output takes the scale.  A scale
// that is not finite gives NaN.
std::vector<int4> fft_tables(int N, double scale, FftTables* t, size_t* inv_at) {
  int e = 0;
  double ms = std::frexp(scale, &e);
  t->bad = std::isfinite(scale) ? 0 : 1;
  const bool fold = N > 16 && !t->bad;
  t->es = fold ? e : 0;
  t->post = scale;
  if (!fold) ms = 1.0;
  std::vector<int4> out;
  const long double pi = 3.14159265358979323846264338327950288L, unit = 4611686018427387904.0L;   // 2^62
  auto part = [&](long double x, int& h, int& l) {
    const i64 q = i64(std::floor(x * unit + 0.5L));
    l = int(static_cast<unsigned>(q));   // the low half with its sign
    h = int((q - l) / 4294967296ll);
  };
  for (int dir = 0; dir < 2; ++dir) {
    if (dir == 1) *inv_at = out.size();
    for (int p = 0; radix(N, p + 1) > 1; ++p) {
      const int M = length(N, p), R = radix(N, p), L = M / R;
      for (int r = 0; r < R; ++r)
        for (int x = 0; x < L; ++x) {
          // cos and sin of 2 pi k / M from the first octant
          const int k = (r * x) % M, oct = k * 8 / M;
          auto cs = [&](int kk, bool sine) {   // 0 <= kk <= M / 4
            const bool flip = 8 * kk > M;
            const long double a = 2.0L * pi * (flip ? M - 4 * kk : 4 * kk) / (4.0L * M);
            return (sine != flip) ? std::sin(a) : std::cos(a);
          };
          const int quad = oct / 2, kq = k - quad * M / 4;
          const long double c0 = cs(kq, false), s0 = cs(kq, true);
          const long double c = quad == 0 ? c0 : quad == 1 ? -s0 : quad == 2 ? -c0 : s0;
          const long double s = quad == 0 ? s0 : quad == 1 ? c0 : quad == 2 ? -s0 : -c0;
          const long double f = (dir == 0 && p == 0) ? static_cast<long double>(ms) : 1.0L;
          int4 w;
          part(c * f, w.x, w.y);
          part((dir == 0 ? -s : s) * f, w.z, w.w);
          out.push_back(w);
        }
    }
  }
  if (out.empty()) out.push_back(make_int4(0, 0, 0, 0));
  return out;
}

#define FFT_SIZES(F, ...)                                   \
  switch (N) {                                              \
    case 4: F<4>(__VA_ARGS__); break;                       \
    case 8: F<8>(__VA_ARGS__); break;                       \
    case 16: F<16>(__VA_ARGS__); break;                     \
    case 32: F<32>(__VA_ARGS__); break;                     \
    case 64: F<64>(__VA_ARGS__); break;                     \
    case 128: F<128>(__VA_ARGS__); break;                   \
    case 256: F<256>(__VA_ARGS__); break;                   \
    case 512: F<512>(__VA_ARGS__); break;                   \
    case 1024: F<1024>(__VA_ARGS__); break;                 \
    default: std::fprintf(stderr, "psolve: n_phi %d unsupported\n", N); \
  }

void launch_fft_forward(const double* rho, double2* f, int nr, int nt, int N, const FftTables& tab, cudaStream_t st) {
  FFT_SIZES(forward, rho, f, nr, nt, tab, st)
}

void launch_fft_inverse(const double2* fh, double* phi, int nr, int nt, int N, const FftTables& tab, cudaStream_t st) {
  FFT_SIZES(inverse, fh, phi, nr, nt, tab, st)
}

}  // namespace ps
