// 64-bit fixed-point transforms for the FP64 sine-transform P_eps^{-1} (Sec. 4,
// eqs. ytild, blockdiaginv, zcompt).
//
// Why fixed point.  GB300 issues 2 FP64 operations per clock per SM.  Its
// integer units issue 53 64-bit additions and 49 32 x 32 -> 64-bit
// multiply-adds per clock per SM (measured), so an exact 64-bit integer
// addition costs 1/30 of an FP64 addition and a 64-bit product by a constant
// (three 32-bit products) about 1/9 of an FP64 product.  The transforms are
// bounded linear maps of one line at a time, so a common exponent per line
// pair is enough: the values are 62-bit integers, where FP64 carries 53 bits of
// each.  Measured for P_eps^{-1} against extended precision (2-norm, 63 cases: 1D to
// 3D, N = 64 to 1024, eps = 1e-3 to 1, a = 1e-5 to 1; flat, alternating and smooth
// data): from 0.01 to 1.2 times the error of the floating-point passes, below it
// in most cases.
//
// Representation.  A line pair (two real lines a, b packed as a + i b) holds
// 64-bit integers v with one exponent F: the value is v 2^F.
// Every stage keeps |v| < 2^62.  F comes from the data: with M the largest
// |component| and L the sum that bounds every partial result of a line's
// transform, the first radix-R pass can grow values to min(R C M, L), which
// fixes F; what the later passes can still grow (at most L) is taken off by
// the twiddle factors, which come from a table scaled by 2^-s with s chosen
// per line pair.  Lines that are far from flat (a single spike) so lose no
// bits to headroom they do not need.  Non-finite inputs set the exponent to
// kFxNan, which every pass hands on and the last one turns into NaN.
//
// The transforms are written as phases between block barriers, each a plain
// function of (thread, shared memory, registers), so that they also compile
// for the host.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

namespace bec {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

#define BEC_FX __host__ __device__ __forceinline__

struct cx {
  i64 x, y;
};

// a 64-bit constant w split as h 2^32 + l with l signed
struct alignas(8) W64 {
  int h, l;
};
struct alignas(16) CW64 {        // cosine and sine
  W64 c, d;
};

constexpr int kFxNan = 1 << 28;  // line exponent of lines with non-finite values
constexpr i64 kHalf = 0x80000000LL;

BEC_FX constexpr W64 split64(i64 w) { return W64{(int)((w + kHalf) >> 32), (int)w}; }

BEC_FX i64 madw(int a, int b, i64 c) { return (i64)a * b + c; }
BEC_FX int lo_w(i64 x) { return (int)x; }
// x = hi_r 2^32 + (signed low word)
BEC_FX int hi_r(i64 x) { return (int)(x >> 32) + (int)((unsigned)x >> 31); }

// round(x w / 2^64), |x| < 2^62, error below 1: the low x low product
// (|.| <= 2^-2 after the division) is left out
BEC_FX i64 mul64(i64 x, W64 w, i64 init = kHalf) {
  const int xh = hi_r(x), xl = (int)x;
  i64 m = madw(xh, w.l, init);
  m = madw(xl, w.h, m);
  return madw(xh, w.h, (i64)(int)(m >> 32));
}

// x c + y d and y c - x d, divided by 2^64 (rounded): the product of x + i y
// and c - i d.  The 64-bit sum of the four cross products stays below 2^63 for
// |x + i y| < 2^62 and |c + i d| <= 0.9 2^63.
BEC_FX cx cmul_conj(cx v, CW64 w, i64 ix = kHalf, i64 iy = kHalf) {
  const int xh = hi_r(v.x), xl = (int)v.x, yh = hi_r(v.y), yl = (int)v.y;
  const int nh = -w.d.h, nl = -w.d.l;
  i64 m = madw(xh, w.c.l, ix);
  m = madw(xl, w.c.h, m);
  m = madw(yh, w.d.l, m);
  m = madw(yl, w.d.h, m);
  i64 n = madw(yh, w.c.l, iy);
  n = madw(yl, w.c.h, n);
  n = madw(xh, nl, n);
  n = madw(xl, nh, n);
  cx r;
  r.x = madw(yh, w.d.h, madw(xh, w.c.h, (i64)(int)(m >> 32)));
  r.y = madw(xh, nh, madw(yh, w.c.h, (i64)(int)(n >> 32)));
  return r;
}
// SIGN -1: v (c - i d); +1: v (c + i d), over 2^64
template <int SIGN>
BEC_FX cx cmul_w(cx v, CW64 w, i64 ix, i64 iy) {
  if constexpr (SIGN > 0) {
    w.d.h = -w.d.h;              // no word of a table entry is -2^31
    w.d.l = -w.d.l;
  }
  return cmul_conj(v, w, ix, iy);
}

BEC_FX cx add(cx a, cx b) { return {a.x + b.x, a.y + b.y}; }
BEC_FX cx sub(cx a, cx b) { return {a.x - b.x, a.y - b.y}; }
// SIGN i a
template <int SIGN>
BEC_FX cx rot(cx a) { return SIGN < 0 ? cx{a.y, -a.x} : cx{-a.y, a.x}; }

// constants below 1/2 in magnitude, times 2^64
constexpr i64 kH1 = -5402926248376769404LL;   // sqrt(1/2) - 1
constexpr i64 kC1 = -1404174782535421627LL;   // cos(pi/8) - 1
constexpr i64 kS1 = 7059263338087549767LL;    // sin(pi/8)

// u sqrt(1/2)
BEC_FX i64 mul_h(i64 u) { return u + mul64(u, split64(kH1)); }
// (c + SIGN i s) v with c = cos(pi/8), s = sin(pi/8)
template <int SIGN>
BEC_FX cx rot8(cx v) {
  constexpr W64 c1 = split64(kC1), s1 = split64(SIGN < 0 ? kS1 : -kS1);
  const int xh = hi_r(v.x), xl = (int)v.x, yh = hi_r(v.y), yl = (int)v.y;
  i64 m = madw(xh, c1.l, kHalf);
  m = madw(xl, c1.h, m);
  m = madw(yh, s1.l, m);
  m = madw(yl, s1.h, m);
  i64 n = madw(yh, c1.l, kHalf);
  n = madw(yl, c1.h, n);
  n = madw(xh, -s1.l, n);
  n = madw(xl, -s1.h, n);
  cx r;
  r.x = v.x + madw(yh, s1.h, madw(xh, c1.h, (i64)(int)(m >> 32)));
  r.y = v.y + madw(xh, -s1.h, madw(yh, c1.h, (i64)(int)(n >> 32)));
  return r;
}

// In-register DFTs with kernel e^{SIGN 2 pi i r k / R}, natural order.
template <int SIGN>
BEC_FX void dft4(cx& a0, cx& a1, cx& a2, cx& a3) {
  const cx s = add(a0, a2), d = sub(a0, a2), t = add(a1, a3), w = rot<SIGN>(sub(a1, a3));
  a0 = add(s, t);
  a2 = sub(s, t);
  a1 = add(d, w);
  a3 = sub(d, w);
}

template <int R, int SIGN>
BEC_FX void dft(cx (&v)[R]) {
  if constexpr (R == 2) {
    const cx a = v[0], b = v[1];
    v[0] = add(a, b);
    v[1] = sub(a, b);
  } else if constexpr (R == 4) {
    dft4<SIGN>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    // X_k = E_k + w^k O_k, X_{k+4} = E_k - w^k O_k, w = e^{SIGN 2 pi i / 8}
    cx e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft4<SIGN>(e[0], e[1], e[2], e[3]);
    dft4<SIGN>(o[0], o[1], o[2], o[3]);
    const cx s1 = add(o[1], rot<SIGN>(o[1])), s3 = sub(rot<SIGN>(o[3]), o[3]);
    o[1] = {mul_h(s1.x), mul_h(s1.y)};
    o[2] = rot<SIGN>(o[2]);
    o[3] = {mul_h(s3.x), mul_h(s3.y)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = add(e[k], o[k]);
      v[k + 4] = sub(e[k], o[k]);
    }
  } else {
    static_assert(R == 16, "radix 2, 4, 8 or 16");
    // 4 x 4: DFTs over a + 4 b (b = 0..3) for each a, twiddles w16^{a kb},
    // DFTs over a; output kb + 4 ka
#pragma unroll
    for (int a = 0; a < 4; ++a) dft4<SIGN>(v[a], v[a + 4], v[a + 8], v[a + 12]);
    // v[a + 4 kb]; w16^m with m = a kb
    auto h45 = [](cx z) {                       // (1 + SIGN i) z / sqrt 2
      const cx u = add(z, rot<SIGN>(z));
      return cx{mul_h(u.x), mul_h(u.y)};
    };
    v[1 + 4] = rot8<SIGN>(v[1 + 4]);                              // m = 1
    v[1 + 8] = h45(v[1 + 8]);                                     // m = 2
    v[1 + 12] = rot<SIGN>(rot8<-SIGN>(v[1 + 12]));                // m = 3 = 4 - 1
    v[2 + 4] = h45(v[2 + 4]);                                     // m = 2
    v[2 + 8] = rot<SIGN>(v[2 + 8]);                               // m = 4
    v[2 + 12] = rot<SIGN>(h45(v[2 + 12]));                        // m = 6
    v[3 + 4] = rot<SIGN>(rot8<-SIGN>(v[3 + 4]));                  // m = 3
    v[3 + 8] = rot<SIGN>(h45(v[3 + 8]));                          // m = 6
    const cx z9 = rot8<SIGN>(v[3 + 12]);                          // m = 9 = 8 + 1
    v[3 + 12] = {-z9.x, -z9.y};
    cx o[16];
#pragma unroll
    for (int kb = 0; kb < 4; ++kb) {
      dft4<SIGN>(v[4 * kb], v[4 * kb + 1], v[4 * kb + 2], v[4 * kb + 3]);
#pragma unroll
      for (int ka = 0; ka < 4; ++ka) o[kb + 4 * ka] = v[4 * kb + ka];
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = o[k];
  }
}

// ------------------------------------------------------------ line layout
// A line of n = 2^LOGN complex values is transformed by TPL threads, EPT
// values each, in up to three radix passes (radices 2^radix_log).
constexpr int npass(int logn) { return logn <= 4 ? 1 : logn <= 8 ? 2 : 3; }
constexpr int radix_log(int logn, int p) {
  return logn == 3 ? 3
       : logn == 4 ? 4
       : logn == 5 ? (p == 0 ? 3 : 2)
       : logn == 6 ? 3
       : logn == 7 ? (p == 0 ? 4 : 3)
       : logn == 8 ? 4
       : logn == 9 ? 3
                   : (p == 0 ? 4 : 3);
}
// log2 of the product of the radices before pass p
constexpr int before_log(int logn, int p) {
  int s = 0;
  for (int i = 0; i < p; ++i) s += radix_log(logn, i);
  return s;
}

template <int LOGN>
struct Line {
  static constexpr int n = 1 << LOGN;
  static constexpr int EPT = n < 16 ? n : 16;
  static constexpr int TPL = n / EPT;
  static constexpr int NP = npass(LOGN);
  // complex slots from one line to the next: odd, so that the same element of
  // consecutive lines falls on different banks
  static constexpr int STRIDE = (n + n / 16 + 1) | 1;
};

// Slot of element i of a line: one pad slot every 16.  The indices of a pass
// are bit permutations of (thread, butterfly, element), so the slot of
// a | b with disjoint bits is slot(a) + slot(b): a thread computes the slot of
// its first element, the others are compile-time offsets from it.
BEC_FX constexpr int slot(int i) { return i + (i >> 4); }

// Butterfly b of pass P reads and writes (in place) elements base + step i.
template <int LOGN, int P>
BEC_FX void bfly_index(int b, int& base, int& step) {
  constexpr int lr = radix_log(LOGN, P), before = before_log(LOGN, P);
  constexpr int lm = LOGN - before - lr;          // log2 of the sub-length after the pass
  const int blk = b >> lm, i1 = b & ((1 << lm) - 1);
  base = (blk << (lm + lr)) + i1;
  step = 1 << lm;
}

// Natural output index of output l of butterfly b of the last pass: base + l step.
template <int LOGN>
BEC_FX void out_index(int b, int& base, int& step) {
  constexpr int NP = npass(LOGN);
  if constexpr (NP == 1) {
    base = 0;
    step = 1;
  } else if constexpr (NP == 2) {
    base = b;
    step = 1 << radix_log(LOGN, 0);
  } else {
    constexpr int r1 = radix_log(LOGN, 0), r2 = radix_log(LOGN, 1);
    base = (b >> r2) + ((b & ((1 << r2) - 1)) << r1);
    step = 1 << (r1 + r2);
  }
}

// Twiddle tables: for the pass P before the last, [s][l][i1] with the factors
// w^{i1 l 2^before} (w = e^{2 pi i / n}) times 2^(64 - s), s = 2 .. kFxShifts
// + 1: n >> before entries a scale, adjacent threads at adjacent i1.
constexpr int kFxShifts = 6;
constexpr int tw_count(int logn) {
  return npass(logn) < 2 ? 1
         : kFxShifts * ((1 << logn) + (npass(logn) > 2 ? 1 << (logn - before_log(logn, 1)) : 0));
}
// first entry of pass p's table
constexpr int tw_first(int logn, int p) { return p == 0 ? 0 : kFxShifts << logn; }

// The DFTs and twiddles of pass P on the thread's values: butterfly u of
// thread t is b = t + TPL u, its element i at v[u R + i]; s: the pass's shift;
// dx, dy: whether the real and the imaginary parts that are only shifted, and
// with TIES the products (many are by powers of two), round ties down (0 or 1).
// Ties that all go one way leave a mean, 1/8 of a unit an element at s = 2; lines
// that a later transform adds up take turns, so that these means cancel.
template <int LOGN, int P, int SIGN, bool TIES = false>
BEC_FX void pass_compute(cx (&v)[Line<LOGN>::EPT], const CW64* __restrict__ tw, int t, int s,
                         int dx = 0, int dy = 0) {
  using G = Line<LOGN>;
  constexpr int lr = radix_log(LOGN, P), R = 1 << lr, NB = G::EPT / R;
  constexpr int before = before_log(LOGN, P), lm = LOGN - before - lr;
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    cx w[R];
#pragma unroll
    for (int i = 0; i < R; ++i) w[i] = v[u * R + i];
    dft<R, SIGN>(w);
    if constexpr (P + 1 < G::NP) {
      const int i1 = (t + G::TPL * u) & ((1 << lm) - 1);
      const CW64* tp = tw + tw_first(LOGN, P) + ((s - 2) << (LOGN - before)) + i1;
      const i64 rnd = 1LL << (s - 1);
      w[0] = {(w[0].x + (rnd - dx)) >> s, (w[0].y + (rnd - dy)) >> s};
#pragma unroll
      for (int l = 1; l < R; ++l) w[l] = cmul_w<SIGN>(w[l], tp[l << lm], TIES ? kHalf - dx : kHalf, TIES ? kHalf - dy : kHalf);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) v[u * R + i] = w[i];
  }
}
// `swap`: real and imaginary parts change places (an inverse transform is the
// forward one between two such exchanges)
template <int LOGN, int P>
BEC_FX void pass_read(cx (&v)[Line<LOGN>::EPT], const cx* line, int t) {
  using G = Line<LOGN>;
  constexpr int R = 1 << radix_log(LOGN, P), NB = G::EPT / R;
  int b0, step;
  bfly_index<LOGN, P>(t, b0, step);
  const cx* p = line + slot(b0);
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    int bu, st;
    bfly_index<LOGN, P>(G::TPL * u, bu, st);
#pragma unroll
    for (int i = 0; i < R; ++i) v[u * R + i] = p[slot(bu + i * st)];
  }
}
template <int LOGN, int P>
BEC_FX void pass_write(const cx (&v)[Line<LOGN>::EPT], cx* line, int t) {
  using G = Line<LOGN>;
  constexpr int R = 1 << radix_log(LOGN, P), NB = G::EPT / R;
  int b0, step;
  bfly_index<LOGN, P>(t, b0, step);
  cx* p = line + slot(b0);
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    int bu, st;
    bfly_index<LOGN, P>(G::TPL * u, bu, st);
#pragma unroll
    for (int i = 0; i < R; ++i) p[slot(bu + i * st)] = v[u * R + i];
  }
}
template <int LOGN>
BEC_FX void write_natural(const cx (&v)[Line<LOGN>::EPT], cx* line, int t) {
  using G = Line<LOGN>;
  constexpr int R = 1 << radix_log(LOGN, G::NP - 1), NB = G::EPT / R;
  int b0, step;
  out_index<LOGN>(t, b0, step);
  cx* p = line + slot(b0);
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    int bu, st;
    out_index<LOGN>(G::TPL * u, bu, st);
#pragma unroll
    for (int i = 0; i < R; ++i) p[slot(bu + i * st)] = v[u * R + i];
  }
}

// ------------------------------------------------------------ line scale
BEC_FX float bits_f(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  std::memcpy(&f, &u, 4);
  return f;
#endif
}
BEC_FX unsigned f_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  unsigned u;
  std::memcpy(&u, &f, 4);
  return u;
#endif
}
// 2^e for e < 128, at least 2^-126
BEC_FX float exp2_f(int e) { return bits_f((unsigned)(e < -126 ? 1 : e + 127) << 23); }
BEC_FX int ilog2f(float f) { return (int)(f_bits(f) >> 23) - 127; }                       // f > 0

// v >> 32 >> d as a float's magnitude, in units 2^(32 + the reference exponent)
BEC_FX float mag(i64 v, int d = 0) {
#ifdef __CUDA_ARCH__
  int r;
  asm("shr.s32 %0, %1, %2;" : "=r"(r) : "r"((int)(v >> 32)), "r"(d));
  return fabsf((float)r);
#else
  return fabsf((float)((int)(v >> 32) >> (d > 31 ? 31 : d)));
#endif
}

// What the threads of a line pair know of its values: m the largest
// |component|, l the sum that bounds every partial result.
struct alignas(8) Stat {
  float m, l;
};
// The join over a line's threads, in two phases.  Lanes across lines (tid = t
// LPB + L): the 32 / LPB threads a line has in a warp join by shuffles, the
// warps through shared memory.  Lanes along a line (ROWS, tid = L TPL + t):
// shuffles alone, and for TPL = 64 the two warps through shared memory.
template <int LPB, int TPL, bool ROWS>
struct LineJoin {
  static constexpr int THREADS = LPB * TPL;
  static constexpr unsigned MASK = THREADS >= 32 ? 0xffffffffu : (1u << (THREADS & 31)) - 1u;
  static constexpr bool LOCAL = ROWS && TPL <= 32;            // no barrier between put and get
  static constexpr int LO = ROWS ? 1 : LPB;                   // lane distances of a line's threads
  static constexpr int HI = ROWS ? (TPL < 32 ? TPL : 32) : (THREADS < 32 ? THREADS : 32);
  static constexpr int CNT = ROWS ? (TPL > 32 ? TPL / 32 : 1) : (THREADS < 32 ? 1 : THREADS / 32);

  static BEC_FX void put(Stat* st, Stat& s, int tid, int L) {
#ifdef __CUDA_ARCH__
#pragma unroll
    for (int o = LO; o < HI; o <<= 1) {
      s.m = fmaxf(s.m, __shfl_xor_sync(MASK, s.m, o));
      s.l += __shfl_xor_sync(MASK, s.l, o);
    }
    if constexpr (!LOCAL) {
      if (ROWS ? (tid & 31) == 0 : (tid & 31) < LPB)
        st[ROWS ? tid >> 5 : (tid >> 5) * LPB + L] = s;
    }
#else
    st[tid] = s;
#endif
  }
  static BEC_FX Stat get(const Stat* st, Stat s, int tid, int L) {
#ifdef __CUDA_ARCH__
    if constexpr (LOCAL) return s;
    const Stat* p = ROWS ? st + (tid >> 5) / CNT * CNT : st + L;
    s = p[0];
#pragma unroll
    for (int w = 1; w < CNT; ++w) {
      const Stat q = p[ROWS ? w : w * LPB];
      s = {fmaxf(s.m, q.m), s.l + q.l};
    }
#else
    s = {0.f, 0.f};
    for (int t = 0; t < TPL; ++t) {
      const Stat q = st[ROWS ? L * TPL + t : t * LPB + L];
      s = {fmaxf(s.m, q.m), s.l + q.l};
    }
#endif
    return s;
  }
};
// the largest of the block's integers, likewise
template <int THREADS>
BEC_FX void max_put(int* mx, int tid, int v) {
#ifdef __CUDA_ARCH__
  const int m = __reduce_max_sync(THREADS >= 32 ? 0xffffffffu : (1u << (THREADS & 31)) - 1u, v);
  if ((tid & 31) == 0) mx[tid >> 5] = m;
#else
  mx[tid] = v;
#endif
}
template <int THREADS>
BEC_FX int max_get(const int* mx) {
#ifdef __CUDA_ARCH__
  constexpr int cnt = THREADS < 32 ? 1 : THREADS / 32;
#else
  constexpr int cnt = THREADS;
#endif
  int m = mx[0];
#pragma unroll
  for (int w = 1; w < cnt; ++w) m = m > mx[w] ? m : mx[w];
  return m;
}
// whether the condition holds on all lanes (on the host: for the thread)
template <int THREADS>
BEC_FX bool all_warp(bool c) {
#ifdef __CUDA_ARCH__
  return __all_sync(THREADS >= 32 ? 0xffffffffu : (1u << (THREADS & 31)) - 1u, c);
#else
  return c;
#endif
}
// running sums of more than 16 threads join in groups of kGroup
constexpr int kGroup = 8;

// The exponent F of a line pair and the shifts of its twiddle passes.
struct Scale {
  int F, s2, s3;
};
// grow: first-pass growth of one component (R C); bound: the sum no partial
// result exceeds, both in units 2^(32 + e) and at least 1.
template <int LOGN>
BEC_FX Scale line_scale(int e, float grow, float bound) {
  constexpr int NP = Line<LOGN>::NP;
  const float b = (NP == 1 || bound < grow) ? bound : grow;
  const int el = ilog2f(bound), eb = ilog2f(b);
  Scale r;
  r.F = e + eb - 29;                            // b 2^(32+e-F) < 2^62
  const int s = el - eb;                        // growth left to the later passes
  r.s2 = r.s3 = 0;
  if constexpr (NP == 2) {
    r.s2 = s < 2 ? 2 : s;
  } else if constexpr (NP == 3) {
    constexpr int r2 = radix_log(LOGN, 1);
    r.s2 = s < 2 ? 2 : s > r2 ? r2 : s;
    r.s3 = s - r.s2 < 2 ? 2 : s - r.s2;
  }
  return r;
}

// v 2^-r (rounded down) for r >= 0, 64-bit shifts that give 0 or -1 from 63 on
BEC_FX i64 shr(i64 v, int r) {
#ifdef __CUDA_ARCH__
  i64 d;
  asm("shr.s64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(r));
  return d;
#else
  return v >> (r > 63 ? 63 : r);
#endif
}
// v 2^r, 0 from r = 64 on
BEC_FX i64 shl(i64 v, int r) {
#ifdef __CUDA_ARCH__
  i64 d;
  asm("shl.b64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(r));
  return d;
#else
  return r > 63 ? 0 : (i64)((u64)v << r);
#endif
}
// v 2^-r for either sign of r
BEC_FX i64 shift(i64 v, int r) {
  const int l = r < 0 ? -r : 0, k = r < 0 ? 0 : r;
  return shr(shl(v, l), k);
}
// the same rounded to nearest, |v| < 2^62 (0 from r = 63 on)
BEC_FX i64 shr_rn(i64 v, int r) {
  const int k = r < 63 ? r : 63;
  return shr(v + (i64)((u64)shl(1, k) >> 1), k);
}
BEC_FX i64 shift_rn(i64 v, int r) {
  const int l = r < 0 ? -r : 0, k = r < 0 ? 0 : r;
  return shr_rn(shl(v, l), k);
}
BEC_FX u64 shr_u(u64 v, int r) {
#ifdef __CUDA_ARCH__
  u64 d;
  asm("shr.u64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(r));
  return d;
#else
  return r > 63 ? 0 : v >> r;
#endif
}

// ------------------------------------------------------------ conversions
BEC_FX u64 d_bits(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 u;
  std::memcpy(&u, &x, 8);
  return u;
#endif
}
BEC_FX double bits_d(u64 u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((i64)u);
#else
  double d;
  std::memcpy(&d, &u, 8);
  return d;
#endif
}
// high word of |x|; for finite x the exponent field is its top 11 bits
BEC_FX int d_habs(u64 b) { return (int)(b >> 32) & 0x7FFFFFFF; }
// x 2^-F as an integer (truncated towards zero); |x 2^-F| < 2^62.  Zero and
// subnormal numbers are read as if normal: below 2^-1022, they vanish for
// F >= kFxMin.
constexpr int kFxMin = -1010;
BEC_FX i64 d_to_fx(u64 b, int F) {
  const unsigned hi = (unsigned)(b >> 32);
  const int e = (int)(hi >> 20) & 0x7FF;
  const u64 m = ((u64)((hi & 0xFFFFFu) | 0x100000u) << 32) | (unsigned)b;
  const i64 a = (i64)shr_u(m << 10, F + 1085 - e);     // (m << 10) 2^(e - 1085) = |x|
  const i64 s = (i64)((int)hi >> 31);
  return (a ^ s) - s;
}
// the same for any F: zeros and subnormal numbers as they are
BEC_FX i64 d_to_fx_sub(u64 b, int F) {
  const int e = (int)(b >> 52) & 0x7FF;
  const u64 m = (b & 0xFFFFFFFFFFFFFULL) | (e != 0 ? 1ULL << 52 : 0);
  const i64 a = (i64)shr_u(m << 10, F + 1085 - (e != 0 ? e : 1));
  const i64 s = (i64)b >> 63;
  return (a ^ s) - s;
}
// v 2^F rounded to nearest (ties away from zero).  fx_round takes |v| >= 2^32 with
// a normal result (fx_normal(F)); fx_to_d sends the rest to fx_to_d_slow, which
// rounds to 53 bits the same way first.
BEC_FX bool fx_normal(int F) { return F > -1030 && F < 950; }
BEC_FX double fx_round(u64 a, i64 s, int F) {         // (s ? -a : a) 2^F, s 0 or -1
#ifdef __CUDA_ARCH__
  const int lz = __clz((int)(a >> 32));
#else
  const int lz = __builtin_clz((unsigned)(a >> 32));
#endif
  const u64 nrm = a << lz;
  // the 53-bit significand brings the exponent's last unit with it
  const u64 r = ((u64)(unsigned)(F + 1085 - lz) << 52) + (nrm >> 11) + ((nrm >> 10) & 1);
  return bits_d(r | ((u64)s & 0x8000000000000000ULL));
}
static __host__ __device__ __noinline__ double fx_to_d_slow(i64 v, int F) {
  const i64 s = v >> 63;
  const u64 a = (u64)((v ^ s) - s);
  return v == 0 ? 0.0 : ldexp(a >> 32 ? fx_round(a, s, 0) : (double)v, F);
}
BEC_FX double fx_to_d(i64 v, int F) {
  const i64 s = (i64)((int)(v >> 32) >> 31);
  const u64 a = (u64)((v ^ s) - s);
  if ((unsigned)(a >> 32) == 0) return fx_to_d_slow(v, F);
  return fx_round(a, s, F);
}

}  // namespace fx
}  // namespace bec
