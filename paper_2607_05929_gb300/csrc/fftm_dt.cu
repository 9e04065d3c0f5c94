// Axis passes of the 3D discrete transforms (Sec. 2.7.2: a 3D DT is three 1D
// DTs, x then y then z; the inverse runs z, y, x).
//
// One CTA transforms a tile of 2 W real pencils of one component along one axis (one 128-byte
// line of consecutive x for the y and z axes, as many consecutive rows for the x axis), two
// real pencils (a, b) to a complex one z = a + i b:
//
//   global --pre--> buffer --stage--> buffer ... --out--> global
//
// The FFTs are Stockham stages of radix up to 16 held in registers, between two buffers in
// shared memory (natural order throughout, no permutation and no staging of the reals); on y and
// z a thread keeps one pencil pair and reads and writes global memory itself, 128 bytes a row.
//
// The complex FFT lengths of the Table 1 transforms of n voxels:
//   DFT      n: spectra of a and b split from Z_k and conj Z_(n-k), halfcomplex order
//   DCT-III, DST-III and their inverses (DCT-II, DST-II): n (Makhoul 1980: the real transform of a
//            reordered sequence with one twiddle per element; DST-III = (-1)^k DCT-III of the
//            reversed input)
//   DCT-I    its odd bins are a DCT-III of n / 2 on f_j - f_(n-j), its even bins a DCT-I of n / 2
//            on f_j + f_(n-j); split twice (n / 2 + n / 4), the rest as the even extension of a
//            DCT-I of n / 4: 5 n / 4 in all, where the even extension of the whole is 2 n
//   DST-I    likewise, sums and differences exchanged: DST-III of n / 2, of n / 4, odd extension
// (n / 2 + n if only one factor 2 divides n, 2 n if none does or n < 8).  The splits cost one
// addition per element and level.  FP64 data: the FP64 pipe bounds the pass, and half of the FFT's
// work goes (128^3: x 415 -> 225 us, y 385 -> 220, fused z 821 -> 436).  FP32 data: instruction
// issue and latency bound it, and the passes through shared memory and their barriers go (256^3: x
// 319 -> 230 us, y 352 -> 193, fused z 627 -> 221; the copy rate would allow 60).
//
// The fused z pass multiplies the z spectrum by the Green factor (Eqs.
// NSGO1_*, NSGO2_*) and runs the inverse z transform without leaving the SM.
#include "fftm_internal.cuh"

namespace fftm {

template <typename T>
using v2 = typename V2<T>::t;

template <typename T>
__device__ __forceinline__ v2<T> mk(T x, T y) {
  v2<T> r;
  r.x = x;
  r.y = y;
  return r;
}
__device__ __forceinline__ float2 ldg2(const float2* p) { return __ldg(p); }
__device__ __forceinline__ double2 ldg2(const double2* p) { return __ldg(p); }
template <typename T>
__device__ __forceinline__ v2<T> cadd(v2<T> a, v2<T> b) { return mk<T>(a.x + b.x, a.y + b.y); }
template <typename T>
__device__ __forceinline__ v2<T> csub(v2<T> a, v2<T> b) { return mk<T>(a.x - b.x, a.y - b.y); }
template <typename T>
__device__ __forceinline__ v2<T> cmul(v2<T> a, v2<T> b) {
  return mk<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename T>
__device__ __forceinline__ v2<T> mul_mi(v2<T> a) { return mk<T>(a.y, -a.x); }  // a * (-i)

// R-point forward DFTs (kernel exp(-2 pi i rt / R)) in registers.
template <typename T>
__device__ __forceinline__ void dft2(v2<T>* x) {
  v2<T> a = x[0], b = x[1];
  x[0] = cadd<T>(a, b);
  x[1] = csub<T>(a, b);
}
template <typename T>
__device__ __forceinline__ void dft4(v2<T>& x0, v2<T>& x1, v2<T>& x2, v2<T>& x3) {
  v2<T> t0 = cadd<T>(x0, x2), t1 = csub<T>(x0, x2);
  v2<T> t2 = cadd<T>(x1, x3), t3 = mul_mi<T>(csub<T>(x1, x3));
  x0 = cadd<T>(t0, t2);
  x2 = csub<T>(t0, t2);
  x1 = cadd<T>(t1, t3);
  x3 = csub<T>(t1, t3);
}
template <typename T>
__device__ __forceinline__ void dft3(v2<T>* x) {
  const T h = T(0.86602540378443864676);  // sqrt(3)/2
  v2<T> t1 = cadd<T>(x[1], x[2]), t2 = csub<T>(x[1], x[2]);
  v2<T> m = mk<T>(x[0].x - T(0.5) * t1.x, x[0].y - T(0.5) * t1.y);
  v2<T> s = mk<T>(h * t2.y, -h * t2.x);  // -i sqrt(3)/2 (x1 - x2)
  x[0] = cadd<T>(x[0], t1);
  x[1] = cadd<T>(m, s);
  x[2] = csub<T>(m, s);
}
template <typename T>
__device__ __forceinline__ void dft8(v2<T>* x) {
  const T c = T(0.70710678118654752440);  // sqrt(1/2)
  v2<T> e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
  v2<T> o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
  dft4<T>(e0, e1, e2, e3);
  dft4<T>(o0, o1, o2, o3);
  o1 = mk<T>(c * (o1.x + o1.y), c * (o1.y - o1.x));   // * e^{-i pi/4}
  o2 = mul_mi<T>(o2);                                 // * e^{-i pi/2}
  o3 = mk<T>(c * (o3.y - o3.x), -c * (o3.x + o3.y));  // * e^{-3 i pi/4}
  x[0] = cadd<T>(e0, o0);
  x[4] = csub<T>(e0, o0);
  x[1] = cadd<T>(e1, o1);
  x[5] = csub<T>(e1, o1);
  x[2] = cadd<T>(e2, o2);
  x[6] = csub<T>(e2, o2);
  x[3] = cadd<T>(e3, o3);
  x[7] = csub<T>(e3, o3);
}

// Larger DFTs from the small ones: 6 and 12 by the prime-factor map (no twiddles), 9 and 16 as
// 3 x 3 and 4 x 4.
template <typename T>
__device__ __forceinline__ void dft6(v2<T>* x) {  // input 3 a + 2 b, output 3 c + 4 d (mod 6)
  v2<T> u[3] = {x[0], x[2], x[4]}, v[3] = {x[3], x[5], x[1]};
  dft3<T>(u);
  dft3<T>(v);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    x[(4 * d) % 6] = cadd<T>(u[d], v[d]);
    x[(4 * d + 3) % 6] = csub<T>(u[d], v[d]);
  }
}
template <typename T>
__device__ __forceinline__ void dft12(v2<T>* x) {  // input 4 a + 3 b, output 4 d + 9 c (mod 12)
  v2<T> y[4][3];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
#pragma unroll
    for (int a = 0; a < 3; ++a) y[b][a] = x[(4 * a + 3 * b) % 12];
    dft3<T>(y[b]);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    dft4<T>(y[0][d], y[1][d], y[2][d], y[3][d]);
#pragma unroll
    for (int c = 0; c < 4; ++c) x[(4 * d + 9 * c) % 12] = y[c][d];
  }
}
template <typename T>
__device__ __forceinline__ void dft9(v2<T>* x) {
  // exp(-2 pi i k / 9), k = 1, 2, 4
  const v2<T> w1 = mk<T>(T(0.76604444311897803520), T(-0.64278760968653932632));
  const v2<T> w2 = mk<T>(T(0.17364817766693034885), T(-0.98480775301220805937));
  const v2<T> w4 = mk<T>(T(-0.93969262078590838405), T(-0.34202014332566873304));
  v2<T> y[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
#pragma unroll
    for (int a = 0; a < 3; ++a) y[b][a] = x[3 * a + b];
    dft3<T>(y[b]);
  }
  y[1][1] = cmul<T>(y[1][1], w1);
  y[1][2] = cmul<T>(y[1][2], w2);
  y[2][1] = cmul<T>(y[2][1], w2);
  y[2][2] = cmul<T>(y[2][2], w4);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    v2<T> t[3] = {y[0][k], y[1][k], y[2][k]};
    dft3<T>(t);
    x[k] = t[0];
    x[k + 3] = t[1];
    x[k + 6] = t[2];
  }
}
// a (c + cl + i s) for a constant whose real part is held in two parts: cos(pi / 8) lies half a unit
// from its FP32 value, on the same side in every product, so that two radix-16 stages shrink a spectrum
// by 2.7e-8 (stages of 8, 8 and 4: 2.1e-8) and an FP32 DFT of 256 points came out 1 % further from the
// exact sums than with those; with the low part 1.3e-8, and 4 % nearer (256 x 16 x 2 points, five kinds
// on the first axis: 1.17e-7 to 1.26e-7 against 1.22e-7 to 1.34e-7; 256^3 Green update 1122 -> 1128 us).
// FP64: cl adds nothing.
template <typename T>
__device__ __forceinline__ v2<T> cmul_hl(v2<T> a, T c, T cl, T s) {
  if constexpr (sizeof(T) == 8) return cmul<T>(a, mk<T>(c, s));
  else return mk<T>(fma(a.x, c, fma(-a.y, s, a.x * cl)), fma(a.y, c, fma(a.x, s, a.y * cl)));
}
template <typename T>
__device__ __forceinline__ void dft16(v2<T>* x) {
  constexpr double cd = 0.92387953251128675613;  // cos, sin of pi / 8
  const T c = T(cd), s = T(0.38268343236508977173), cl = T(cd - (double)T(cd));
  const T h = T(0.70710678118654752440);
  v2<T> y[4][4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
#pragma unroll
    for (int a = 0; a < 4; ++a) y[b][a] = x[4 * a + b];
    dft4<T>(y[b][0], y[b][1], y[b][2], y[b][3]);
  }
  y[1][1] = cmul_hl<T>(y[1][1], c, cl, -s);
  y[1][2] = mk<T>(h * (y[1][2].x + y[1][2].y), h * (y[1][2].y - y[1][2].x));
  y[1][3] = mul_mi<T>(cmul_hl<T>(y[1][3], c, cl, s));  // s - i c = -i (c + i s)
  y[2][1] = mk<T>(h * (y[2][1].x + y[2][1].y), h * (y[2][1].y - y[2][1].x));
  y[2][2] = mul_mi<T>(y[2][2]);
  y[2][3] = mk<T>(h * (y[2][3].y - y[2][3].x), -h * (y[2][3].x + y[2][3].y));
  y[3][1] = mul_mi<T>(cmul_hl<T>(y[3][1], c, cl, s));
  y[3][2] = mk<T>(h * (y[3][2].y - y[3][2].x), -h * (y[3][2].x + y[3][2].y));
  y[3][3] = cmul_hl<T>(y[3][3], -c, -cl, s);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    dft4<T>(y[0][k], y[1][k], y[2][k], y[3][k]);
#pragma unroll
    for (int m = 0; m < 4; ++m) x[k + 4 * m] = y[m][k];
  }
}
template <typename T, int R>
__device__ __forceinline__ void dft(v2<T>* x) {
  if (R == 2) dft2<T>(x);
  else if (R == 3) dft3<T>(x);
  else if (R == 4) dft4<T>(x[0], x[1], x[2], x[3]);
  else if (R == 6) dft6<T>(x);
  else if (R == 8) dft8<T>(x);
  else if (R == 9) dft9<T>(x);
  else if (R == 12) dft12<T>(x);
  else dft16<T>(x);
}

// Tile geometry: W complex pencils (2 W real ones, 128 bytes of T) per CTA.  Buffer element
// (row m, pencil pc) sits at m SP + pc: on y and z a warp walks the pencils (contiguous), on x it
// also walks the rows, and the pad keeps both free of bank conflicts.
template <typename T, int AXIS>
struct Tile {
  static constexpr int W = 64 / sizeof(T);
  static constexpr int SP = AXIS == 0 ? W + 1 : W;
};

// One butterfly of a Stockham stage: inputs b + r N / R, outputs at (b / Lp) Lp R + b % Lp + r Lp.
template <typename T, int R, int SP>
__device__ __forceinline__ void butterfly(const v2<T>* src, v2<T>* dst, const SegPlan& sg, int s, int b,
                                          const v2<T>* __restrict__ tw) {
  const int nb = sg.nb[s], Lp = sg.lp[s];
  v2<T> x[R];
#pragma unroll
  for (int r = 0; r < R; ++r) x[r] = src[(b + r * nb) * SP];
  int base = b * R;
  if (Lp > 1) {
    // b / Lp as a multiply-high: exact for b < 2^16 and 2 <= Lp <= 2^13 with
    // magic = ceil(2^32 / Lp) (the rounding excess b (magic Lp - 2^32) / 2^32 < 2^-16
    // stays below 1 / Lp)
    const int g = (int)__umulhi((unsigned)b, sg.magic[s]), k = b - g * Lp;
    base = g * Lp * R + k;
    const int t = k * sg.tstep[s];
#pragma unroll
    for (int r = 1; r < R; ++r) x[r] = cmul<T>(x[r], ldg2(tw + r * t));
  }
  dft<T, R>(x);
#pragma unroll
  for (int r = 0; r < R; ++r) dst[(base + r * Lp) * SP] = x[r];
}

// Butterfly f of a stage, counted over the segments one after the other (a warp mostly works on
// one of them).  src, dst: the buffers at the thread's pencil.
template <typename T, int SP>
__device__ __forceinline__ void stage_item(const v2<T>* src, v2<T>* dst, const AxisPlan<T>& pl, int s, int f) {
  int g = 0, b = f;
  if (pl.nseg > 1 && b >= pl.seg[0].nb[s]) {
    b -= pl.seg[0].nb[s];
    g = 1;
    if (pl.nseg > 2 && b >= pl.seg[1].nb[s]) {
      b -= pl.seg[1].nb[s];
      g = 2;
    }
  }
  const SegPlan& sg = pl.seg[g];
  src += sg.off * SP;
  dst += sg.off * SP;
  switch (sg.rad[s]) {
    case 2: butterfly<T, 2, SP>(src, dst, sg, s, b, pl.tw); break;
    case 3: butterfly<T, 3, SP>(src, dst, sg, s, b, pl.tw); break;
    case 4: butterfly<T, 4, SP>(src, dst, sg, s, b, pl.tw); break;
    case 6: butterfly<T, 6, SP>(src, dst, sg, s, b, pl.tw); break;
    case 8: butterfly<T, 8, SP>(src, dst, sg, s, b, pl.tw); break;
    case 9: butterfly<T, 9, SP>(src, dst, sg, s, b, pl.tw); break;
    case 12: butterfly<T, 12, SP>(src, dst, sg, s, b, pl.tw); break;
    default: butterfly<T, 16, SP>(src, dst, sg, s, b, pl.tw); break;
  }
}

template <typename T>
__device__ __forceinline__ int stage_items(const AxisPlan<T>& pl, int s) {
  int n = pl.seg[0].nb[s];
  if (pl.nseg > 1) n += pl.seg[1].nb[s];
  if (pl.nseg > 2) n += pl.seg[2].nb[s];
  return n;
}

// Output m of a DCT-III of length N in Makhoul's order, from an inverse FFT evaluated as
// swap(FFT(swap)); a DST-III changes the sign of the odd ones.
template <typename T, int SP>
__device__ __forceinline__ v2<T> out_c3(const v2<T>* z, int m, int N, bool dst) {
  const bool odd = m & 1;
  const v2<T> v = z[(odd ? N - 1 - (m >> 1) : m >> 1) * SP];
  const T sg = (dst && odd) ? T(-1) : T(1);
  return mk<T>(sg * v.y, sg * v.x);
}

// Row `row` of a transform whose outputs are FFT outputs one by one (all but those of post_item);
// z: the buffer at the thread's pencil, natural order in every segment.  Selects instead of
// branches: where lanes walk the rows, neighbours lie in different segments.
template <typename T, int SP>
__device__ __forceinline__ v2<T> out_row(const AxisPlan<T>& pl, const v2<T>* z, int row) {
  if (pl.kind == K_DFT) {  // inverse
    const v2<T> v = z[row * SP];
    return mk<T>(v.x, -v.y);
  }
  const bool dst = pl.kind == K_DST1 || pl.kind == K_DST3;
  if (pl.kind == K_DCT3 || pl.kind == K_DST3) return out_c3<T, SP>(z, row, pl.n, dst);
  const int k = row + (dst ? 1 : 0), lev = pl.lev;
  const bool s0 = lev >= 1 && (k & 1), s1 = lev >= 2 && (k & 3) == 2, c3 = s0 || s1;
  const int m = s0 ? k >> 1 : k >> 2;
  const bool odd = m & 1;
  const int N = s0 ? pl.seg[0].N : pl.seg[1].N, i3 = (s0 ? 0 : pl.seg[1].off) + (odd ? N - 1 - (m >> 1) : m >> 1);
  const int ie = pl.seg[lev].off + (k >> lev);
  const v2<T> v = z[(c3 ? i3 : ie) * SP];
  const bool swap = c3 || dst;
  const T sx = (dst && (c3 ? odd : true)) ? T(-1) : T(1), sy = (dst && c3 && odd) ? T(-1) : T(1);
  return mk<T>(sx * (swap ? v.y : v.x), sy * (swap ? v.x : v.y));
}

// The same, every row: items i0, i0 + istep, ... of each segment in turn (a row that looks its
// segment up costs three times the instructions).
template <typename T, int SP, typename Put>
__device__ __forceinline__ void out_rows(const AxisPlan<T>& pl, const v2<T>* z, int i0, int istep, Put&& put) {
  if (pl.kind == K_DFT) {
    for (int i = i0; i < pl.n; i += istep) {
      const v2<T> v = z[i * SP];
      put(i, mk<T>(v.x, -v.y));
    }
    return;
  }
  const bool type1 = pl.kind == K_DCT1 || pl.kind == K_DST1, dst = pl.kind == K_DST1 || pl.kind == K_DST3;
  const int nc3 = type1 ? pl.lev : 1, first = (type1 && dst) ? 1 : 0;
  for (int g = 0; g < nc3; ++g) {
    const int N = pl.seg[g].N, step = type1 ? 2 << g : 1, r0 = type1 ? (1 << g) - first : 0;
    const v2<T>* zs = z + pl.seg[g].off * SP;
    for (int m = i0; m < N; m += istep) put(r0 + step * m, out_c3<T, SP>(zs, m, N, dst));
  }
  if (type1) {
    const int N = pl.seg[pl.lev].N / 2;  // the extension's bins 0 .. N, those of the DST inside
    const v2<T>* zs = z + pl.seg[pl.lev].off * SP;
    for (int m = i0 + first; m <= N - first; m += istep) {
      const v2<T> v = zs[m * SP];
      put((m << pl.lev) - first, dst ? mk<T>(-v.y, v.x) : v);
    }
  }
}

// The pre-processing: rows of the transform's range (ld(row) = the pencil pair's values) to the
// FFT inputs (st(index, value)), in this many items.
template <typename T>
__device__ __forceinline__ int pre_items(const AxisPlan<T>& pl, bool inverse) {
  switch (pl.kind) {
    case K_DFT: return inverse ? pl.n / 2 + 1 : pl.n;
    case K_DCT1:
    case K_DST1: return pl.lev == 0 ? pl.n + 1 : pl.n / (2 << pl.lev) + 1;
    default: return inverse ? pl.n : pl.n / 2 + 1;
  }
}

// DCT-III inputs k and N - k of a segment from the sequence values zk, zn (exchanged for a DST-III,
// whose sequence is reversed): w_k (z_k - i z_(N-k)), w_k = exp(i pi k / 2N), stored with real and
// imaginary part swapped.
template <typename T, typename St>
__device__ __forceinline__ void pre_c3(bool dst, v2<T> v0, v2<T> v1, int k, int N, int wstep,
                                       const v2<T>* __restrict__ qw, int off, St&& st) {
  const v2<T> zk = dst ? v1 : v0, zn = dst ? v0 : v1;
  {
    const v2<T> w = ldg2(qw + k * wstep);
    const v2<T> d = k == 0 ? zk : mk<T>(zk.x + zn.y, zk.y - zn.x);
    const v2<T> h = cmul<T>(d, w);
    st(off + k, mk<T>(h.y, h.x));
  }
  if (k > 0 && 2 * k != N) {
    const v2<T> w = ldg2(qw + (N - k) * wstep);
    const v2<T> h = cmul<T>(mk<T>(zn.x + zk.y, zn.y - zk.x), w);
    st(off + N - k, mk<T>(h.y, h.x));
  }
}

// DCT-I or DST-I of n voxels, split LEV times: item j holds every element that the folds of j
// meet, 2^(LEV+1) of them.
template <typename T, int LEV, typename Ld, typename St>
__device__ __forceinline__ void pre_type1(const AxisPlan<T>& pl, int j, Ld&& ld, St&& st) {
  const int n = pl.n;
  const bool dst = pl.kind == K_DST1;
  const int first = dst ? 1 : 0;
  auto f = [&](int pos) -> v2<T> {  // node position 0 .. n (zero at both ends for the DST)
    return (!dst || (pos > 0 && pos < n)) ? ld(pos - first) : mk<T>(T(0), T(0));
  };
  // fold of a pair: the part that the odd bins take (difference for the DCT, sum for the DST) and
  // the part that goes on
  const T sg = dst ? T(1) : T(-1);
  auto odd = [&](v2<T> a, v2<T> b) { return mk<T>(a.x + sg * b.x, a.y + sg * b.y); };
  auto even = [&](v2<T> a, v2<T> b) { return mk<T>(a.x - sg * b.x, a.y - sg * b.y); };
  const int off = pl.seg[LEV].off, N2 = pl.seg[LEV].N;  // the extension, of length 2 (n >> LEV)
  auto ext = [&](v2<T> v, int k) {
    st(off + k, v);
    if (k > 0 && 2 * k != N2) st(off + N2 - k, mk<T>(-sg * v.x, -sg * v.y));
  };
  if (LEV == 0) {
    ext(f(j), j);
  } else if (LEV == 1) {
    const int h = n / 2;  // elements j, h - j and their mirrors
    const v2<T> a0 = f(j), a7 = f(n - j), a3 = f(h - j), a4 = f(h + j);
    pre_c3<T>(dst, odd(a0, a7), odd(a3, a4), j, h, 2, pl.qw, 0, st);
    ext(even(a0, a7), j);
    if (2 * j != h) ext(even(a3, a4), h - j);
  } else {
    const int h = n / 2, g = n / 4;
    const v2<T> a0 = f(j), a7 = f(n - j), a1 = f(g - j), a6 = f(n - g + j);
    const v2<T> a2 = f(g + j), a5 = f(n - g - j), a3 = f(h - j), a4 = f(h + j);
    pre_c3<T>(dst, odd(a0, a7), odd(a3, a4), j, h, 2, pl.qw, 0, st);
    if (2 * j != g) pre_c3<T>(dst, odd(a1, a6), odd(a2, a5), g - j, h, 2, pl.qw, 0, st);  // j = 0: k = h / 2
    const v2<T> e0 = even(a0, a7), e3 = even(a3, a4), e1 = even(a1, a6), e2 = even(a2, a5);
    pre_c3<T>(dst, odd(e0, e3), odd(e1, e2), j, g, 4, pl.qw, pl.seg[1].off, st);
    ext(even(e0, e3), j);
    if (2 * j != g) ext(even(e1, e2), g - j);
  }
}

template <typename T, typename Ld, typename St>
__device__ __forceinline__ void pre_item(const AxisPlan<T>& pl, bool inverse, int i, Ld&& ld, St&& st) {
  const int n = pl.n;
  if (pl.kind == K_DFT) {
    const v2<T> c = ld(i);
    if (!inverse) {
      st(i, c);
    } else if (i == 0 || 2 * i == n) {  // halfcomplex rows of a and b -> conj(A + i B) at i and n - i
      st(i, mk<T>(c.x, -c.y));
    } else {
      const v2<T> d = ld(n - i);
      st(i, mk<T>(c.x - d.y, -(d.x + c.y)));
      st(n - i, mk<T>(c.x + d.y, d.x - c.y));
    }
  } else if (pl.kind == K_DCT1 || pl.kind == K_DST1) {
    if (pl.lev == 2) pre_type1<T, 2>(pl, i, ld, st);
    else if (pl.lev == 1) pre_type1<T, 1>(pl, i, ld, st);
    else pre_type1<T, 0>(pl, i, ld, st);
  } else {
    const bool dst = pl.kind == K_DST3;
    if (!inverse) {  // sequence value k of the DCT: row k; node k of the DST: row k - 1
      const v2<T> v0 = (dst && i == 0) ? mk<T>(T(0), T(0)) : ld(dst ? i - 1 : i);
      const v2<T> v1 = (dst || i > 0) ? ld(dst ? n - 1 - i : n - i) : v0;
      pre_c3<T>(dst, v0, v1, i, n, 1, pl.qw, 0, st);
    } else {  // DCT-II in Makhoul's order; DST-II: of (-1)^m x_m
      v2<T> v = ld(i);
      if (dst && (i & 1)) v = mk<T>(-v.x, -v.y);
      st((i & 1) ? n - 1 - (i >> 1) : i >> 1, v);
    }
  }
}

// DFT forward, DCT-II and DST-II: an item of the pre-processing loads one row (the loads are issued
// PRE_BATCH items at a time, since one load per trip leaves a pass waiting for memory), and the outputs
// pair the FFT bins k and n - k: items 0 .. n / 2 of post_item, each the rows r0 and r1 (r1 < 0: only
// the first).
__device__ __forceinline__ bool rows_in_pairs_out(int kind, bool inverse) {
  return kind == K_DFT ? !inverse : (inverse && (kind == K_DCT3 || kind == K_DST3));
}
constexpr int PRE_BATCH = 8;

template <typename T, int SP>
__device__ __forceinline__ void post_item(const AxisPlan<T>& pl, const v2<T>* z, int k, int* r0, v2<T>* o0, int* r1,
                                          v2<T>* o1) {
  const int n = pl.n, c = k == 0 ? 0 : n - k;
  const v2<T> Zk = z[k * SP], Zc = z[c * SP];
  const T sx = Zk.x + Zc.x, dx = Zk.x - Zc.x, sy = Zk.y + Zc.y, dy = Zk.y - Zc.y;
  if (pl.kind == K_DFT) {
    *r0 = k;
    *r1 = (k > 0 && k != c) ? c : -1;
    *o0 = mk<T>(T(0.5) * sx, T(0.5) * sy);
    *o1 = mk<T>(T(0.5) * dy, T(-0.5) * dx);
  } else {
    const v2<T> w = ldg2(pl.qw + k);
    const bool dst = pl.kind == K_DST3;  // DST-II: item k belongs to node n - k, row n - 1 - k
    *r0 = dst ? n - 1 - k : k;
    *r1 = (k > 0 && k != c) ? (dst ? k - 1 : c) : -1;
    *o0 = mk<T>(sx * w.x + dy * w.y, sy * w.x - dx * w.y);
    *o1 = mk<T>(sx * w.y - dy * w.x, sy * w.y + dx * w.x);
  }
}

// The Green factor of one z line: with (kx, ky) fixed the B0 / 2 mu0 denominator is
// alpha cos^2 + beta sin^2 of the z frequency, each coefficient a sum of products that are exactly
// zero where a factor is, so a null denominator stays an exact zero.
template <typename T>
struct GreenLine {
  T alpha, beta;
  __device__ __forceinline__ T at(T s, T c, T g) const {
    const T den = alpha * c + beta * s;
    return den > T(0) ? g / den : T(0);
  }
};
template <typename T>
__device__ __forceinline__ GreenLine<T> green_line(const PassParams<T>& P, int q, int kx, int ky) {
  GreenLine<T> G;
  G.alpha = G.beta = T(0);
  if (kx < 0 || kx >= P.fL[q][0]) return G;
  const T sx = P.S2[q][0][kx], cx = P.C2[q][0][kx], sy = P.S2[q][1][ky], cy = P.C2[q][1][ky];
  const T t = P.tetra ? T(1) : T(0);
  const T c0 = P.hf[0] * sx * cy, s0 = t * P.hf[0] * cx * sy;
  const T c1 = P.hf[1] * cx * sy, s1 = t * P.hf[1] * sx * cy;
  const T c2 = t * P.hf[2] * sx * sy, s2 = P.hf[2] * cx * cy;
  G.alpha = P.two_mu0 * (c0 + c1 + c2) + P.lam0 * (q == 0 ? c0 : (q == 1 ? c1 : c2));
  G.beta = P.two_mu0 * (s0 + s1 + s2) + P.lam0 * (q == 0 ? s0 : (q == 1 ? s1 : s2));
  return G;
}

// Threads per CTA at most.  FP32 type-I passes along x and y have two CTAs an SM at 256 voxels
// (82 KB of buffers): 512 threads each (x 263 -> 230 us, y 208 -> 193); the fused z pass has three
// (z 238 us with 512, 221 with 256).
template <typename T, int FUSED>
constexpr int pass_threads() { return sizeof(T) == 4 && !FUSED ? 512 : 256; }
template <typename T, int FUSED>
constexpr int pass_ctas() { return sizeof(T) == 8 ? 1 : (FUSED ? 3 : 2); }

// The flat index over (pencil, item) of an x tile, items fastest, one division per thread.
struct RowItems {
  int items, p, i, dp, di;
  __device__ __forceinline__ explicit RowItems(int n) : items(n) {
    p = (int)threadIdx.x / n;
    i = (int)threadIdx.x - p * n;
    dp = (int)blockDim.x / n;
    di = (int)blockDim.x - dp * n;
  }
  __device__ __forceinline__ void next() {
    p += dp;
    i += di;
    if (i >= items) {
      i -= items;
      ++p;
    }
  }
};

template <typename T, int AXIS, int FUSED>
__global__ void __launch_bounds__(pass_threads<T, FUSED>(), pass_ctas<T, FUSED>())
    k_pass(const __grid_constant__ PassParams<T> P, int buf_rows) {
  if (P.stop && *P.stop) return;
  constexpr int W = Tile<T, AXIS>::W, SP = Tile<T, AXIS>::SP, WSH = W == 16 ? 4 : 3;
  const int q = blockIdx.y;
  const AxisPlan<T>& pl = P.plan[q];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  v2<T>* const buf0 = reinterpret_cast<v2<T>*>(smem_raw);
  const int buf_step = buf_rows * SP;
  auto buf = [&](int i) { return buf0 + i * buf_step; };  // the two buffers
  const int pc = threadIdx.x & (W - 1);  // this thread's pencil pair (fixed: W divides the block)
  const int i0 = threadIdx.x >> WSH, istep = blockDim.x >> WSH;

  const int N1 = P.N[0], N2 = P.N[1], N3 = P.N[2];
  const long long sy = P.stride[1], sz = P.stride[2];
  const T* in = P.in[q];  // may be out itself: a CTA reads its pencils before it writes them
  T* out = P.out[q];
  const int L = pl.L, lo = pl.lo;

  // ---- tile geometry ----
  const char* ip = nullptr;       // y, z: this thread's pair at row 0, and the byte stride of a row
  char* op = nullptr;
  int es = 0;
  bool va = false, vb = false;    // its two pencils exist and lie in the component's range
  int x0 = 0, yfix = 0;
  long long* rowoff = reinterpret_cast<long long*>(buf0 + 2 * buf_step);  // x: the tile's rows
  int* rowok = reinterpret_cast<int*>(rowoff + 2 * W);
  if (AXIS == 0) {
    if (threadIdx.x < 2 * W) {
      const int r = blockIdx.x * 2 * W + threadIdx.x;
      // rows past the last one read it again; they and the dismissed rows are not stored
      const int rc = min(r, N2 * N3 - 1), z = rc / N2, y = rc - z * N2;
      rowoff[threadIdx.x] = (long long)y * sy + (long long)z * sz + lo;
      rowok[threadIdx.x] = r < N2 * N3 && y >= P.flo[q][1] && y < P.flo[q][1] + P.fL[q][1] && z >= P.flo[q][2] &&
                           z < P.flo[q][2] + P.fL[q][2];
    }
    __syncthreads();
  } else {
    const int ntx = (N1 + 2 * W - 1) / (2 * W);
    const int other = blockIdx.x / ntx;
    x0 = (blockIdx.x - other * ntx) * 2 * W;
    const int x = x0 + 2 * pc;
    va = x >= P.flo[q][0] && x < P.flo[q][0] + P.fL[q][0];
    vb = x + 1 >= P.flo[q][0] && x + 1 < P.flo[q][0] + P.fL[q][0];
    const long long st = AXIS == 1 ? sy : sz, base = x + (long long)other * (AXIS == 1 ? sz : sy) + lo * st;
    yfix = other;
    es = (int)(st * (long long)sizeof(T));
    ip = reinterpret_cast<const char*>(in + base);
    op = reinterpret_cast<char*>(out + base);
    // Dismissed positions hold zeros and stay zero: a pencil of zeros packed with another one would
    // come out as that one's rounding, which no Green factor scales down afterwards.
    const int ko = other - P.flo[q][AXIS == 1 ? 2 : 1];
    if (ko < 0 || ko >= P.fL[q][AXIS == 1 ? 2 : 1]) return;
  }

  // ---- pre-processing: global -> buffer 0 ----
  const bool inv_first = (P.inverse != 0) && !FUSED;
  const v2<T> zero = mk<T>(T(0), T(0));
  {
    const int items = pre_items(pl, inv_first);
    if (AXIS == 0) {
      RowItems f(items);
      if (rows_in_pairs_out(pl.kind, inv_first)) {
        while (f.p < W) {
          v2<T> v[PRE_BATCH];
          int fp[PRE_BATCH], fi[PRE_BATCH];
#pragma unroll
          for (int k = 0; k < PRE_BATCH; ++k, f.next()) {
            fp[k] = f.p;
            fi[k] = f.i;
            if (f.p < W) v[k] = mk<T>(in[rowoff[2 * f.p] + f.i], in[rowoff[2 * f.p + 1] + f.i]);
          }
#pragma unroll
          for (int k = 0; k < PRE_BATCH; ++k) {
            auto st = [&](int m, const v2<T>& x) { buf0[m * SP + fp[k]] = x; };
            if (fp[k] < W) pre_item<T>(pl, inv_first, fi[k], [&](int) { return v[k]; }, st);
          }
        }
      } else {
        for (; f.p < W; f.next()) {
          const T* a = in + rowoff[2 * f.p];
          const T* b = in + rowoff[2 * f.p + 1];
          v2<T>* d = buf0 + f.p;
          pre_item<T>(pl, inv_first, f.i, [&](int row) { return mk<T>(a[row], b[row]); },
                      [&](int m, const v2<T>& v) { d[m * SP] = v; });
        }
      }
    } else {
      auto ld = [&](int row) {
        const char* a = ip + (long long)row * es;
        v2<T> v = zero;
        if (va && vb) v = *reinterpret_cast<const v2<T>*>(a);
        else if (va) v.x = *reinterpret_cast<const T*>(a);
        else if (vb) v.y = reinterpret_cast<const T*>(a)[1];
        return v;
      };
      auto st = [&](int m, const v2<T>& v) { buf0[m * SP + pc] = v; };
      if (rows_in_pairs_out(pl.kind, inv_first)) {
        for (int i = i0; i < items; i += PRE_BATCH * istep) {
          v2<T> v[PRE_BATCH];
#pragma unroll
          for (int k = 0; k < PRE_BATCH; ++k)
            if (i + k * istep < items) v[k] = ld(i + k * istep);
#pragma unroll
          for (int k = 0; k < PRE_BATCH; ++k)
            if (i + k * istep < items) pre_item<T>(pl, inv_first, i + k * istep, [&](int) { return v[k]; }, st);
        }
      } else {
        for (int i = i0; i < items; i += istep) pre_item<T>(pl, inv_first, i, ld, st);
      }
    }
  }
  __syncthreads();

  int cur = 0;  // the buffer that the next step reads
  bool inverse = inv_first;
#pragma unroll 1
  for (int half = 0; half < (FUSED ? 2 : 1); ++half) {
#pragma unroll 1
    for (int s = 0; s < pl.nst; ++s) {
      const int items = stage_items(pl, s);
      for (int f = i0; f < items; f += istep) stage_item<T, SP>(buf(cur) + pc, buf(cur ^ 1) + pc, pl, s, f);
      cur ^= 1;
      __syncthreads();
    }
    if (FUSED && half == 0) {
      // ---- forward spectrum times the Green factor -> inverse FFT inputs, in the other buffer ----
      const v2<T>* src = buf(cur) + pc;
      v2<T>* dst = buf(cur ^ 1) + pc;
      const int ky = yfix - P.flo[q][1], kx = x0 + 2 * pc - P.flo[q][0];
      const GreenLine<T> Ga = green_line<T>(P, q, kx, ky), Gb = green_line<T>(P, q, kx + 1, ky);
      const T gs = -P.gscale[q];
      const T* __restrict__ S2 = P.S2[q][2];
      const T* __restrict__ C2 = P.C2[q][2];
      if (pl.kind == K_DFT) {  // Z_k = A + i B, Z_(n-k) = conj A + i conj B: scale A and B, conjugate
        const int n = pl.n;
        for (int k = i0; k <= n / 2; k += istep) {
          const int c = k == 0 ? 0 : n - k;
          const v2<T> Zk = src[k * SP], Zc = src[c * SP];
          const T sn = __ldg(S2 + k), cs = __ldg(C2 + k);
          const T ga = T(0.5) * Ga.at(sn, cs, gs), gb = T(0.5) * Gb.at(sn, cs, gs);
          const T ax = ga * (Zk.x + Zc.x), ay = ga * (Zk.y - Zc.y);
          const T bx = gb * (Zk.y + Zc.y), by = gb * (Zc.x - Zk.x);
          dst[k * SP] = mk<T>(ax - by, -(ay + bx));
          if (k != c) dst[c * SP] = mk<T>(ax + by, ay - bx);
        }
      } else {
        auto ld = [&](int row) {
          const v2<T> v = out_row<T, SP>(pl, src, row);
          const T sn = __ldg(S2 + row), cs = __ldg(C2 + row);
          return mk<T>(v.x * Ga.at(sn, cs, gs), v.y * Gb.at(sn, cs, gs));
        };
        auto st = [&](int m, const v2<T>& v) { dst[m * SP] = v; };
        const int items = pre_items(pl, true);
        for (int i = i0; i < items; i += istep) pre_item<T>(pl, true, i, ld, st);
      }
      cur ^= 1;
      inverse = true;
      __syncthreads();
    }
  }

  // ---- results -> global ----
  const T sc = P.scale[q];
  const bool paired = rows_in_pairs_out(pl.kind, inverse);
  const int items = paired ? pl.n / 2 + 1 : L;
  if (AXIS != 0) {
    const v2<T>* z = buf(cur) + pc;
    auto put = [&](int row, const v2<T>& v) {
      char* o = op + (long long)row * es;
      if (va && vb) *reinterpret_cast<v2<T>*>(o) = mk<T>(sc * v.x, sc * v.y);
      else if (va) *reinterpret_cast<T*>(o) = sc * v.x;
      else if (vb) reinterpret_cast<T*>(o)[1] = sc * v.y;
    };
    if (!paired) {
      out_rows<T, SP>(pl, z, i0, istep, put);
    } else {
      for (int i = i0; i < items; i += istep) {
        int r0, r1;
        v2<T> o0, o1;
        post_item<T, SP>(pl, z, i, &r0, &o0, &r1, &o1);
        put(r0, o0);
        if (r1 >= 0) put(r1, o1);
      }
    }
    return;
  }
  // x: lanes walk the rows' elements; accumulated onto the base field where there is one
  const T* __restrict__ bh = P.base[q];
  const T* __restrict__ bl = P.base_lo[q];
  T* __restrict__ ol = P.out_lo[q];
  for (RowItems f(items); f.p < W; f.next()) {
    const v2<T>* z = buf(cur) + f.p;
    const long long off[2] = {rowoff[2 * f.p], rowoff[2 * f.p + 1]};
    const bool ok[2] = {rowok[2 * f.p] != 0, rowok[2 * f.p + 1] != 0};
    int r[2] = {f.i, -1};
    v2<T> o[2];
    if (paired) post_item<T, SP>(pl, z, f.i, &r[0], &o[0], &r[1], &o[1]);
    else o[0] = out_row<T, SP>(pl, z, f.i);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (r[e] < 0) continue;
      const T val[2] = {sc * o[e].x, sc * o[e].y};
      const long long at[2] = {off[0] + r[e], off[1] + r[e]};
      if (bh == nullptr) {
        if (ok[0]) out[at[0]] = val[0];
        if (ok[1]) out[at[1]] = val[1];
        continue;
      }
      T b0[2], b1[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        b0[c] = bh[at[c]];
        b1[c] = ol ? bl[at[c]] : T(0);
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (!ok[c]) continue;
        if (ol == nullptr) {
          out[at[c]] = b0[c] + val[c];
        } else {
          // (hi, lo) = (bh, bl) + v: error-free sum of the high parts (TwoSum), low parts
          // gathered, then renormalised so that |lo| stays below half an ulp of hi
          const T s1 = b0[c] + val[c];
          const T bb = s1 - b0[c];
          const T er = (b0[c] - (s1 - bb)) + (val[c] - bb);
          const T t = b1[c] + er;
          const T h = s1 + t;
          out[at[c]] = h;
          ol[at[c]] = t - (h - s1);
        }
      }
    }
  }
}

// Shared memory of a pass: two buffers of the longest segment sum of the three components, and on
// x the offsets of the tile's rows.
template <typename T, int AXIS, int FUSED>
static cudaError_t launch_one(const PassParams<T>& P, cudaStream_t s) {
  constexpr int W = Tile<T, AXIS>::W, SP = Tile<T, AXIS>::SP;
  int rows = 0, items = 0;
  for (int q = 0; q < 3; ++q) {
    rows = rows > P.plan[q].total ? rows : P.plan[q].total;
    for (int t = 0; t < P.plan[q].nst; ++t) {
      int m = 0;  // butterflies of the stage
      for (int g = 0; g < P.plan[q].nseg; ++g) m += P.plan[q].seg[g].nb[t];
      items = items > m ? items : m;
    }
  }
  const size_t smem = (size_t)2 * rows * SP * sizeof(v2<T>) + (AXIS == 0 ? 2 * W * (sizeof(long long) + sizeof(int)) : 0);
  if (smem > (size_t)kMaxDynSmem) return cudaErrorInvalidValue;
  // a thread per butterfly of the widest stage, at least 64 (short axes: more CTAs per SM instead)
  constexpr int most = pass_threads<T, FUSED>();
  int threads = (items * W + 31) / 32 * 32;
  threads = threads < 64 ? 64 : (threads > most ? most : threads);
  auto kern = k_pass<T, AXIS, FUSED>;
  // the same opt-in limit for every problem: the attribute is per function, so a
  // per-problem value could be lowered by another thread between its set and our launch
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
  if (e != cudaSuccess) return e;
  dim3 grid;
  if (AXIS == 0) grid.x = (unsigned)((P.N[1] * P.N[2] + 2 * W - 1) / (2 * W));
  else grid.x = (unsigned)(((P.N[0] + 2 * W - 1) / (2 * W)) * (AXIS == 1 ? P.N[2] : P.N[1]));
  grid.y = 3;
  kern<<<grid, threads, smem, s>>>(P, rows);
  return cudaGetLastError();
}

// The longest transforms taken: 512 voxels on a non-periodic axis, 768 on a periodic one (the
// problem's descriptor admits more; there a pass returns cudaErrorInvalidValue).
constexpr int MAX_PASS_BOUNDED = 512, MAX_PASS_PERIODIC = 768;

template <typename T>
cudaError_t launch_pass(const PassParams<T>& P, cudaStream_t s) {
  for (int q = 0; q < 3; ++q)
    if (P.plan[q].n > (P.plan[q].kind == K_DFT ? MAX_PASS_PERIODIC : MAX_PASS_BOUNDED)) return cudaErrorInvalidValue;
  if (P.fused) {
    if (P.axis != 2) return cudaErrorInvalidValue;
    return launch_one<T, 2, 1>(P, s);
  }
  if (P.axis == 0) return launch_one<T, 0, 0>(P, s);
  if (P.axis == 1) return launch_one<T, 1, 0>(P, s);
  return launch_one<T, 2, 0>(P, s);
}

template cudaError_t launch_pass<float>(const PassParams<float>&, cudaStream_t);
template cudaError_t launch_pass<double>(const PassParams<double>&, cudaStream_t);

// ---- standalone Green factor on a spectral field ----
template <typename T>
__global__ void k_green(GreenParams<T> P) {
  const int q = blockIdx.y;
  const long long total = (long long)P.N[0] * P.N[1] * P.N[2];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % P.N[0]);
    const long long r = i / P.N[0];
    const int y = (int)(r % P.N[1]);
    const int z = (int)(r / P.N[1]);
    const int kx = x - P.flo[q][0], ky = y - P.flo[q][1], kz = z - P.flo[q][2];
    const long long off = x + y * P.sy + z * P.sz;
    if (kx < 0 || ky < 0 || kz < 0 || kx >= P.fL[q][0] || ky >= P.fL[q][1] || kz >= P.fL[q][2]) {
      P.f[q][off] = T(0);
      continue;
    }
    const T sx = P.S2[q][0][kx], cx = P.C2[q][0][kx];
    const T sy = P.S2[q][1][ky], cy = P.C2[q][1][ky];
    const T sz = P.S2[q][2][kz], cz = P.C2[q][2][kz];
    T a0 = P.hf[0] * sx * cy * cz, a1 = P.hf[1] * cx * sy * cz, a2 = P.hf[2] * cx * cy * sz;
    if (P.tetra) {
      a0 += P.hf[0] * cx * sy * sz;
      a1 += P.hf[1] * sx * cy * sz;
      a2 += P.hf[2] * sx * sy * cz;
    }
    const T aq = (q == 0) ? a0 : ((q == 1) ? a1 : a2);
    const T den = P.two_mu0 * (a0 + a1 + a2) + P.lam0 * aq;
    P.f[q][off] *= (den > T(0) ? -P.gscale[q] / den : T(0));
  }
}

template <typename T>
cudaError_t launch_green(const GreenParams<T>& P, cudaStream_t s) {
  dim3 grid(1216, 3);
  k_green<T><<<grid, 256, 0, s>>>(P);
  return cudaGetLastError();
}
template cudaError_t launch_green<float>(const GreenParams<float>&, cudaStream_t);
template cudaError_t launch_green<double>(const GreenParams<double>&, cudaStream_t);

}  // namespace fftm
