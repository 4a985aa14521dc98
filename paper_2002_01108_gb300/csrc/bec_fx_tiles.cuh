// The passes of the fixed-point sine-transform P_eps^{-1} (bec_fx.cuh) as
// tiles: each tile is the work of one block, written as phases that a block
// barrier separates.  A phase sees the thread's index, the block's shared
// memory and the thread's registers (Reg), so that a host program can run the
// phases of a block thread by thread.
//
// Exponents between the passes.  A tile is 2 LPB adjacent columns (or modes)
// of one row of the slice, the same columns in every pass (xg, of XG a row),
// or 2 LPB rows in the x-DST; its lines have their own scales, but it writes
// all results with one exponent, the largest of its lines'.  The
// next pass, whose lines cross those tiles, copies the exponents of its lines'
// elements to shared memory, takes its statistics in the unit 2^ref of the
// largest one, from the high words shifted right by ref - exponent, and then
// shifts each element from its own exponent to the tile's scale.
#pragma once

#include "bec_fx.cuh"

namespace bec {
namespace fx {

enum DstKind {
  kRowsFwd = 0,     // x-DST of FP64 rows
  kColsY = 1,       // forward y-DST, after the x-DST
  kColsZ = 2,       // z-DST, forward or back, after the y-DST
  kColsYBack = 3,   // y-DST after the time pass
  kRowsBack = 4     // x-DST to FP64 rows
};

struct DstArgs {
  const void* in;
  void* out;
  int m, dim, kind, xg;                             // xg: tiles a row
  long long J, rows;                                // points a slice; rows in all
  const int* ein;
  const int* xadd;                                  // after the time pass: exponent a time step
  int* eout;                                        // one a tile
  const W64* sinw;                                  // 2 sin(j pi / n) - 1, j < n/2, times 2^63
  const CW64* tw;                                   // tw_count(logn) entries
};

// DST-I of line pairs: 4 S_k = 4 sum_j x_j sin(pi j k / n), the method of
// warp_dst_pair (bec_fft.cuh) on integers.  With w_j = 2 sin(j pi / n) - 1 the
// pre-pass is y_j = 2 (x_j + h), y_{n-j} = 2 (x_{n-j} + h), h = w_j (x_j +
// x_{n-j}) / 2: one product for two values and no 2 sin > 1 to represent; the
// factor 2 is the difference between the exponents of x (F - 1) and y (F).
// ROWS: lines run along x (rows 2 L, 2 L + 1 of the tile, lanes along the
// line); else down the columns L and LPB + L of the tile (lanes across).
template <int LOGN, int LPB, bool ROWS, bool IN_D, bool OUT_D>
struct DstTile {
  using G = Line<LOGN>;
  static constexpr int n = G::n, TPL = G::TPL, EPT = G::EPT, H = EPT / 2, W = 2 * LPB;
  static_assert(H == 8, "lines of at least 16");
  static constexpr int THREADS = LPB * TPL;
  static constexpr bool GROUPS = TPL > 16, kInD = IN_D;
  static constexpr int XG = n / W > 0 ? n / W : 1;  // tiles a row
  static constexpr int NE = ROWS ? W * XG : n;      // exponents of a tile's elements
  static constexpr size_t kBuf = (size_t)LPB * G::STRIDE * sizeof(cx);
  static constexpr size_t kTot = (size_t)THREADS * sizeof(cx);
  static constexpr size_t kStat = (size_t)THREADS * sizeof(Stat);
  static constexpr size_t kMax = (size_t)THREADS * sizeof(int);
  static constexpr size_t kFl = LPB * sizeof(int);
  static constexpr size_t kGt = GROUPS ? (size_t)LPB * (TPL / kGroup) * sizeof(cx) : 0;
  static constexpr size_t SMEM = kBuf + kTot + kStat + kMax + kGt + kFl + (IN_D ? 0 : NE * sizeof(int));
  using Join = LineJoin<LPB, TPL, ROWS>;
  static constexpr int RS = n + n / 16;             // real slots of a line (row pass output)

  struct Ctx {
    cx* line;
    cx *tot, *gt;
    Stat* st;
    int *mx, *fl, *se;                              // se[j - 1] (ROWS: se[row XG + (j - 1) / W])
    int L, t, tid;
    bool va, vb;
    long long la, lb;                               // offsets of x_1 of the two lines
    long long es;                                   // elements from x_j to x_{j+1}
    int ref, add, f;                                // f: exponent of the line's outputs
    int dx, dy;                                     // pass_compute; ROWS: constants
    Stat s;
    Scale sc;
  };
  struct Reg {
    i64 a[H], a2[H], b[H], b2[H];                   // x_p, x_{n-p} of both lines
    cx v[EPT];
  };

  static BEC_FX void init(Ctx& c, const DstArgs& g, unsigned char* smem, int tid, long long blk) {
    c.tid = tid;
    c.L = ROWS ? tid / TPL : tid % LPB;
    c.t = ROWS ? tid % TPL : tid / LPB;
    c.line = reinterpret_cast<cx*>(smem) + c.L * G::STRIDE;
    c.tot = reinterpret_cast<cx*>(smem + kBuf);
    c.st = reinterpret_cast<Stat*>(smem + kBuf + kTot);
    c.mx = reinterpret_cast<int*>(smem + kBuf + kTot + kStat);
    c.gt = reinterpret_cast<cx*>(smem + kBuf + kTot + kStat + kMax);
    c.fl = reinterpret_cast<int*>(smem + kBuf + kTot + kStat + kMax + kGt);
    c.se = c.fl + LPB;
    c.add = 0;
    const long long m = g.m;
    int e = -kFxNan;
    if constexpr (ROWS) {
      const long long r0 = blk * W, ra = r0 + 2 * c.L;
      c.va = ra < g.rows;
      c.vb = ra + 1 < g.rows;
      c.la = ra * m;
      c.lb = c.la + m;
      c.es = 1;
      c.dx = 0;                                     // rows in turn (m is odd: a row's steps too)
      c.dy = 1;
      if constexpr (!IN_D) {
        for (int k = tid; k < NE; k += THREADS) {
          const long long r = r0 + k / XG;
          int x = -kFxNan;
          if (r < g.rows) {
            const long long base = g.dim == 1 ? 0 : g.dim == 2 ? r / m : r / (m * m) * m + r % m;
            x = g.ein[base * XG + k % XG];
          }
          c.se[k] = x;
          e = e > x ? e : x;
        }
      }
    } else {
      const long long u = blk / XG;                 // 2D: time step; 3D: (step, z), z-DST (step, y)
      const int xg = (int)(blk - u * XG), ca = xg * W + c.L, cb = ca + LPB;
      c.va = ca < m;
      c.vb = cb < m;
      const bool z = g.kind == kColsZ;
      c.la = (z ? u / m * g.J + u % m * m : u * m * m) + ca;
      c.lb = c.la + LPB;
      c.es = z ? m * m : m;
      c.dx = c.dy = (int)((z || g.dim == 3 ? u / m : u) & 1);   // time steps in turn
      if (g.kind == kColsYBack) c.add = g.xadd[g.dim == 2 ? u : u / m];
      for (int k = tid; k < n - 1; k += THREADS) {
        const int x = g.kind == kColsY ? g.ein[(u * m + k) / W]
                      : g.kind == kColsZ ? g.ein[(u / m * m + k) * XG + xg]
                                         : g.ein[((g.dim == 2 ? 0 : u % m * m) + k) * XG + xg];
        c.se[k] = x;
        e = e > x ? e : x;
      }
    }
    if constexpr (!IN_D) max_put<THREADS>(c.mx, tid, e);
  }

  // loads the pairs (p, n - p), p = t + TPL u (p = 0 stands for the middle
  // element, alone); of FP64 values the largest high word is published
  static BEC_FX void load(Ctx& c, Reg& r, const DstArgs& g) {
    const i64* in = static_cast<const i64*>(g.in);   // FP64 bit patterns or integers
    // x_p from the front, x_{n-p} from the back of the line
    const int p0 = c.t == 0 ? n / 2 : c.t, q0 = c.t == 0 ? n / 2 : n - c.t;
    const i64 *fa = in + c.la + (c.t - 1) * c.es, *ba = in + c.la + (n - 1 - c.t) * c.es;
    const i64 *fb = fa + (c.lb - c.la), *bb = ba + (c.lb - c.la);
    const long long step = TPL * c.es;
#pragma unroll
    for (int u = 0; u < H; ++u) r.a[u] = r.a2[u] = r.b[u] = r.b2[u] = 0;
    if (c.va) {
      r.a[0] = fa[(p0 - c.t) * c.es];
      r.a2[0] = ba[(q0 - n + c.t) * c.es];
#pragma unroll
      for (int u = 1; u < H; ++u) {
        r.a[u] = fa[u * step];
        r.a2[u] = ba[-u * step];
      }
    }
    if (c.vb) {
      r.b[0] = fb[(p0 - c.t) * c.es];
      r.b2[0] = bb[(q0 - n + c.t) * c.es];
#pragma unroll
      for (int u = 1; u < H; ++u) {
        r.b[u] = fb[u * step];
        r.b2[u] = bb[-u * step];
      }
    }
    if constexpr (IN_D) {
      int m = 0;
#pragma unroll
      for (int u = 0; u < H; ++u) {
        const int x = d_habs((u64)r.a[u]), x2 = d_habs((u64)r.a2[u]);
        const int y = d_habs((u64)r.b[u]), y2 = d_habs((u64)r.b2[u]);
        const int xm = x > x2 ? x : x2, ym = y > y2 ? y : y2, w = xm > ym ? xm : ym;
        m = m > w ? m : w;
      }
      line_max_put(c, m);
    }
  }
  // largest high word of the line (FP64 input), in two phases like LineJoin
  static BEC_FX void line_max_put(Ctx& c, int v) {
#ifdef __CUDA_ARCH__
#pragma unroll
    for (int o = Join::LO; o < Join::HI; o <<= 1) {
      const int w = __shfl_xor_sync(Join::MASK, v, o);
      v = v > w ? v : w;
    }
    if (Join::LOCAL) c.ref = v;
    else if ((c.tid & 31) == 0) c.mx[c.tid >> 5] = v;
#else
    c.mx[c.tid] = v;
#endif
  }
  static BEC_FX int line_max_get(const Ctx& c) {
#ifdef __CUDA_ARCH__
    if (Join::LOCAL) return c.ref;
    const int* p = c.mx + (c.tid >> 5) / Join::CNT * Join::CNT;
    int m = p[0];
    for (int w = 1; w < Join::CNT; ++w) m = m > p[w] ? m : p[w];
#else
    int m = 0;
    for (int i = 0; i < TPL; ++i) m = m > c.mx[c.L * TPL + i] ? m : c.mx[c.L * TPL + i];
#endif
    return m;
  }
  // exponents of the pair u's elements in lines a and b
  struct Ex {
    int x, x2, y, y2;
  };
  static BEC_FX Ex exps(const Ctx& c, int u) {
    const int p = c.t + TPL * u, j = u == 0 && c.t == 0 ? n / 2 : p, j2 = u == 0 && c.t == 0 ? n / 2 : n - p;
    if constexpr (ROWS) {
      const int *ea = c.se + 2 * c.L * XG, *eb = ea + XG;
      const int k = (j - 1) / W, k2 = (j2 - 1) / W;
      return {ea[k], ea[k2], eb[k], eb[k2]};
    } else {
      const int x = c.se[j - 1], x2 = c.se[j2 - 1];
      return {x, x2, x, x2};
    }
  }

  // the block's unit (integers) or the line's (FP64 values, made integers on the
  // scale their largest one asks for), and the statistics
  static BEC_FX void measure(Ctx& c, Reg& r) {
    float m = 0.f, l = 0.f;
    if constexpr (IN_D) {
      const int em = line_max_get(c) >> 20;
      // |x| < 2^(em - 1022); the first pass's growth R1 5.66 |x|, on y's scale F
      // = ref + 1, stays below 2^62
      constexpr int lg = radix_log(LOGN, 0) + 3;    // R1 5.66 < 2^lg
      c.ref = em - 1022 + lg - 62 - 1;
      if (c.ref >= kFxMin) {
#pragma unroll
        for (int u = 0; u < H; ++u) {
          r.a[u] = d_to_fx((u64)r.a[u], c.ref);
          r.a2[u] = d_to_fx((u64)r.a2[u], c.ref);
          r.b[u] = d_to_fx((u64)r.b[u], c.ref);
          r.b2[u] = d_to_fx((u64)r.b2[u], c.ref);
        }
      } else {                                      // zeros, or next to the subnormal numbers
#pragma unroll
        for (int u = 0; u < H; ++u) {
          r.a[u] = d_to_fx_sub((u64)r.a[u], c.ref);
          r.a2[u] = d_to_fx_sub((u64)r.a2[u], c.ref);
          r.b[u] = d_to_fx_sub((u64)r.b[u], c.ref);
          r.b2[u] = d_to_fx_sub((u64)r.b2[u], c.ref);
        }
      }
#pragma unroll
      for (int u = 0; u < H; ++u) l += mag(r.a[u]) + mag(r.a2[u]) + mag(r.b[u]) + mag(r.b2[u]);
      if (em == 0x7FF) c.ref = kFxNan;
    } else {
      const int mx = max_get<THREADS>(c.mx);
      c.ref = mx;
#pragma unroll
      for (int u = 0; u < H; ++u) {
        const Ex e = exps(c, u);
        const float x = mag(r.a[u], mx - e.x), x2 = mag(r.a2[u], mx - e.x2);
        const float y = mag(r.b[u], mx - e.y), y2 = mag(r.b2[u], mx - e.y2);
        m = fmaxf(m, fmaxf(fmaxf(x, x2), fmaxf(y, y2)));
        l += (x + x2) + (y + y2);
      }
    }
    c.s = {m, l};
    Join::put(c.st, c.s, c.tid, c.L);
  }

  // the line's scale, the values on it, the pre-pass
  static BEC_FX void prepass(Ctx& c, Reg& r, const DstArgs& g) {
    const Stat s = Join::get(c.st, c.s, c.tid, c.L);
    constexpr float R1 = (float)(1 << radix_log(LOGN, 0));
    // |y_j| <= 4 max|x| a line, 5.66 max|x| for a + i b; sum |y_j| <= 4 sum |x_j|.
    // The statistics come from high words (one unit of slack each), the sum from
    // float additions.  With 4 (sum |a| + sum |b|) < 2^62 the sums C + C' of the
    // last step stay below 2^63.
    const float bound = 4.004f * (s.l + (float)(2 * n));
    if constexpr (IN_D) {
      // F = ref + 1 (a growth of less than 2^31 high words of 2^ref) unless the
      // line is sparse
      c.sc = line_scale<LOGN>(c.ref, 1073741824.f, bound);
    } else {
      c.sc = line_scale<LOGN>(c.ref, R1 * 5.66f * (s.m + 1.f), bound);
    }
    const int fi = c.sc.F - 1, k = fi - c.ref;      // right shift from the unit ref
    c.f = (c.ref > kFxNan / 2 ? kFxNan : c.sc.F + c.sc.s2 + c.sc.s3) + c.add;
    if (c.t == 0) c.fl[c.L] = c.f;
    if constexpr (IN_D) {
#pragma unroll
      for (int u = 0; u < H; ++u)
        if (k < 0)
          pair(c, g, u, r.a[u] << -k, r.a2[u] << -k, r.b[u] << -k, r.b2[u] << -k, 0);
        else
          pair(c, g, u, r.a[u], r.a2[u], r.b[u], r.b2[u], 0);
    } else {
      // integers are shifted rounding down by k (and more), which takes (1 - 2^-k) / 2
      // of a unit from x_j and x_{n-j} in the mean and 1 + w_j times that from y_j: h
      // gets it back.  A mean left in y would meet in the lowest modes, which the time
      // pass amplifies.
      if (all_warp<THREADS>(k >= 0)) {              // right shifts only
#pragma unroll
        for (int u = 0; u < H; ++u) {
          const Ex e = exps(c, u);
          pair(c, g, u, shr(r.a[u], fi - e.x), shr(r.a2[u], fi - e.x2), shr(r.b[u], fi - e.y),
               shr(r.b2[u], fi - e.y2), k > 0 ? k : 0);
        }
      } else {
#pragma unroll
        for (int u = 0; u < H; ++u) {
          const Ex e = exps(c, u);
          pair(c, g, u, shift(r.a[u], fi - e.x), shift(r.a2[u], fi - e.x2), shift(r.b[u], fi - e.y),
               shift(r.b2[u], fi - e.y2), k > 0 ? k : 0);
        }
      }
    }
  }
  // y_p and y_{n-p}, p = t + TPL u, to shared memory
  static BEC_FX void pair(const Ctx& c, const DstArgs& g, int u, i64 a, i64 a2, i64 b, i64 b2, int k) {
    const W64 w = g.sinw[c.t + TPL * u];
    const unsigned back = 0x80000000u + (unsigned)w.h;    // (1 + w) / 2
    const i64 init = kHalf + (i64)(back - (back >> (k < 31 ? k : 31)));
    const i64 sa = a + a2, sb = b + b2;
    const i64 ha = mul64(sa, w, init), hb = mul64(sb, w, init);   // s w / 2
    if (u == 0) {                                   // p = 0: y_{n/2} = 4 x_{n/2}, y_0 = 0
      const bool mid = c.t == 0;
      c.line[slot(mid ? n / 2 : c.t)] = cx{mid ? sa : a + ha, mid ? sb : b + hb};
      c.line[slot(mid ? 0 : n - c.t)] = cx{mid ? 0 : a2 + ha, mid ? 0 : b2 + hb};
    } else {
      c.line[slot(c.t) + slot(TPL * u)] = cx{a + ha, b + hb};
      c.line[slot(n - c.t - TPL * u)] = cx{a2 + ha, b2 + hb};
    }
  }

  // pass P of the FFT: read, transform; all but the last write in place
  template <int P>
  static BEC_FX void pass(Ctx& c, Reg& r, const DstArgs& g) {
    pass_read<LOGN, P>(r.v, c.line, c.t);
    pass_compute<LOGN, P, -1, ROWS>(r.v, g.tw, c.t, P == 0 ? c.sc.s2 : c.sc.s3, c.dx, c.dy);
    if constexpr (P + 1 < G::NP) pass_write<LOGN, P>(r.v, c.line, c.t);
  }
  static BEC_FX void natural(Ctx& c, Reg& r) { write_natural<LOGN>(r.v, c.line, c.t); }

  // the chunk k = H t .. H t + H - 1 < n/2: even outputs (v[2 i + 1]) and the
  // running sums of the odd ones (v[2 i])
  static BEC_FX void chunk(Ctx& c, Reg& r) {
    const cx* fp = c.line + slot(H * c.t);
    const cx* bp = c.line + slot(n - H - H * c.t);
    cx run{0, 0};
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const cx C = fp[slot(i)];
      cx rv = C, ev{0, 0};
      if (i > 0 || c.t > 0) {
        const cx Cn = i > 0 ? bp[slot(H - i)] : c.line[slot(n - H * c.t)];
        rv = add(C, Cn);
        ev = cx{Cn.y - C.y, C.x - Cn.x};
      }
      run = add(run, rv);
      r.v[2 * i] = run;
      r.v[2 * i + 1] = ev;
    }
    c.tot[c.t * LPB + c.L] = run;
  }
  // group sums of the chunk totals (TPL > 16 only)
  static BEC_FX void chunk_group(Ctx& c) {
    if (c.t >= TPL / kGroup) return;
    cx s = c.tot[c.t * kGroup * LPB + c.L];
    for (int i = 1; i < kGroup; ++i) s = add(s, c.tot[(c.t * kGroup + i) * LPB + c.L]);
    c.gt[c.t * LPB + c.L] = s;
  }
  // outputs: 4 S_{2k+1} at index 2k, 4 S_{2k} at 2k - 1 (index 0: x_1)
  static BEC_FX void store(Ctx& c, Reg& r, const DstArgs& g) {
    cx off{0, 0};
    if constexpr (GROUPS) {
      for (int k = 0; k < c.t / kGroup; ++k) off = add(off, c.gt[k * LPB + c.L]);
      for (int t = c.t / kGroup * kGroup; t < c.t; ++t) off = add(off, c.tot[t * LPB + c.L]);
    } else {
      for (int t = 0; t < c.t; ++t) off = add(off, c.tot[t * LPB + c.L]);
    }
    // the tile's exponent is the largest of its lines'
    int fm = c.fl[0];
#pragma unroll
    for (int i = 1; i < LPB; ++i) fm = fm > c.fl[i] ? fm : c.fl[i];
    const int d = fm - c.f;
    c.f = fm;
    const i64 half = d > 0 ? 1LL << ((d > 62 ? 62 : d) - 1) : 0;
    const cx rnd = d > 0 ? cx{half - c.dx, half - c.dy} : cx{0, 0};
    off = add(off, rnd);
    auto dn = [d](i64 v) { return shr(v, d); };
    if constexpr (ROWS) {
      // line a, then line b, a pad slot every 16
      i64* ob = reinterpret_cast<i64*>(c.line) + (2 * H + 1) * c.t;
#pragma unroll
      for (int i = 0; i < H; ++i) {
        const cx od = add(r.v[2 * i], off), ev = add(r.v[2 * i + 1], rnd);
        ob[2 * i] = dn(od.x);
        ob[RS + 2 * i] = dn(od.y);
        if (i > 0) {
          ob[2 * i - 1] = dn(ev.x);
          ob[RS + 2 * i - 1] = dn(ev.y);
        } else if (c.t > 0) {
          ob[-2] = dn(ev.x);
          ob[RS - 2] = dn(ev.y);
        }
      }
    } else {
      i64 *oa = static_cast<i64*>(g.out) + c.la + 2 * H * c.t * c.es, *ob = oa + LPB;
      if (c.va) {
#pragma unroll
        for (int i = 0; i < H; ++i) {
          oa[2 * i * c.es] = dn(r.v[2 * i].x + off.x);
          if (i > 0 || c.t > 0) oa[(2 * i - 1) * c.es] = dn(r.v[2 * i + 1].x + rnd.x);
        }
      }
      if (c.vb) {
#pragma unroll
        for (int i = 0; i < H; ++i) {
          ob[2 * i * c.es] = dn(r.v[2 * i].y + off.y);
          if (i > 0 || c.t > 0) ob[(2 * i - 1) * c.es] = dn(r.v[2 * i + 1].y + rnd.y);
        }
      }
    }
  }
  static BEC_FX void store_exp(const Ctx& c, const DstArgs& g, long long blk) {
    if (!OUT_D && c.tid == 0) g.eout[blk] = c.f;
  }
  // row pass: the rows of the tile to global memory, in order
  static BEC_FX void store_rows(Ctx& c, const DstArgs& g, unsigned char* smem, long long blk) {
    const i64* buf = reinterpret_cast<const i64*>(smem);
    // a thread keeps its places j (mod THREADS) in the rows it visits
    constexpr int PER = THREADS >= n ? 1 : n / THREADS;   // places of a thread in a row
    constexpr int RPI = THREADS >= n ? THREADS / n : 1;   // rows visited at once
    const int j0 = c.tid & (n - 1), row0 = THREADS >= n ? c.tid >> LOGN : 0;
#pragma unroll 4
    for (int row = row0; row < W; row += RPI) {
      const long long R = blk * W + row;
      if (R >= g.rows) break;
      const i64* src = buf + (row >> 1) * (2 * G::STRIDE) + (row & 1) * RS;
      const int f = OUT_D ? c.f + (g.dim == 1 ? g.xadd[R] : 0) : 0;
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int j = j0 + q * THREADS;
        if (j < g.m) {
          const i64 v = src[j + (j >> 4)];
          if constexpr (OUT_D) {
            static_cast<double*>(g.out)[R * g.m + j] =
                fx_normal(f) ? fx_to_d(v, f)
                             : f > kFxNan / 2 ? bits_d(0x7FF8000000000000ULL) : fx_to_d_slow(v, f);
          } else {
            static_cast<i64*>(g.out)[R * g.m + j] = v;
          }
        }
      }
    }
  }
};

// ---------------------------------------------------------------- time pass
struct TimeArgs {
  i64* data;                   // [N][J]
  long long J;
  int m, dim;                  // modes a row; rows: 1 (1D), m, m^2
  const int* ein;              // exponents of the input tiles
  int* eout;                   // [row][xg] exponents of the outputs, less the step's xadd[j]
  int* xadd;                   // [N], written here
  const W64* esm;              // eps^{j/N} = esm 2^-63 2^ese
  const int* ese;
  const double* eis;           // eps^{-j/N}
  const double* scale_dev;     // null: 1
  const CW64* q;               // [N/2+1][J]: scale conj(d) / |d|^2, times 2^(63 - qe)
  const int* qe;               // [tile][N/2+1]
  const CW64* tw;
};

// d = w 2^-63 2^x with |w| < 2^63 - 2^31 (two words); non-finite: x = kFxNan
BEC_FX W64 mant_of(double d, int& x) {
  const u64 b = d_bits(d);
  const int ef = (int)(b >> 52) & 0x7FF;
  if (ef == 0x7FF) {
    x = kFxNan;
    return W64{0, 0};
  }
  const u64 m = (b & 0xFFFFFFFFFFFFFULL) | (ef != 0 ? 1ULL << 52 : 0);
  x = (ef < 1 ? 1 : ef) - 1022;
  i64 w = (i64)(m << 10);
  if (w > 0x7FFFFFFF00000000LL) {                   // next to 1: half of it
    w >>= 1;
    ++x;
  }
  return split64((i64)b < 0 ? -w : w);
}

// Modes x0 + L (real part) and x0 + LPB + L (imaginary part) of a row are a
// line; lanes run across lines.  Scale by eps^{j/N} (Step 1), FFT, divide by
// lambda'_k mu^M + tau mu^K (Step 2), inverse FFT, unscale (Step 3).  The
// inverse transform is the forward one with real and imaginary parts
// exchanged before and after, so both run the same instructions.
template <int LOGN, int LPB>
struct TimeTile {
  using G = Line<LOGN>;
  static constexpr int N = G::n, TPL = G::TPL, EPT = G::EPT, H = EPT / 2, W = 2 * LPB;
  static constexpr int THREADS = LPB * TPL;
  static constexpr size_t kBuf = (size_t)LPB * G::STRIDE * sizeof(cx);
  static constexpr size_t kStat = (size_t)THREADS * sizeof(Stat);
  static constexpr size_t kMax = (size_t)THREADS * sizeof(int);
  static constexpr size_t SMEM = kBuf + kStat + kMax + (size_t)N * (sizeof(W64) + sizeof(int)) +
                                 (LPB + N / 2 + 1) * sizeof(int);
  using Join = LineJoin<LPB, TPL, false>;
  static constexpr int R1 = 1 << radix_log(LOGN, 0);
  static constexpr int RL = 1 << radix_log(LOGN, G::NP - 1);

  struct Ctx {
    cx* line;
    Stat* st;
    int *mx, *fl, *se;                              // se[j]: exponent of time step j's values
    W64* eim;                                       // eps^{-j/N} scale, as mantissas
    int* qx;                                        // qe[k] - qe[0]; null: no factors
    int L, t, tid;
    bool va, vb;
    long long qa, qb, tile;
    int ref, f;                                     // f: exponent of the values in registers
    Scale sc;
    Stat s;
  };
  struct Reg {
    cx v[EPT];
  };

  // the thread's place in the block's lines; returns the tile's index in its row
  static BEC_FX int place(Ctx& c, int m, unsigned char* smem, int tid, long long blk) {
    c.tid = tid;
    c.L = tid % LPB;
    c.t = tid / LPB;
    c.tile = blk;
    c.line = reinterpret_cast<cx*>(smem) + c.L * G::STRIDE;
    c.st = reinterpret_cast<Stat*>(smem + kBuf);
    c.mx = reinterpret_cast<int*>(smem + kBuf + kStat);
    c.eim = reinterpret_cast<W64*>(smem + kBuf + kStat + kMax);
    c.se = reinterpret_cast<int*>(c.eim + N);
    c.fl = c.se + N;
    c.qx = nullptr;
    const int XG = (m + W) / W;                     // m + 1 = a power of two >= W, or 1
    const long long row = blk / XG;
    const int xg = (int)(blk - row * XG), x0 = xg * W + c.L;
    c.qa = row * m + x0;
    c.qb = c.qa + LPB;
    c.va = x0 < m;
    c.vb = x0 + LPB < m;
    return xg;
  }
  static BEC_FX void init(Ctx& c, const TimeArgs& g, unsigned char* smem, int tid, long long blk) {
    const int XG = (g.m + W) / W, xg = place(c, g.m, smem, tid, blk);
    const long long row = blk / XG;
    const double s = g.scale_dev ? g.scale_dev[0] : 1.0;
    const long long eb = g.dim == 3 ? (row % g.m) * XG + xg : xg;
    const long long es = g.dim == 3 ? (long long)g.m * XG : XG;
    int e = -kFxNan;
    for (int j = tid; j < N; j += THREADS) {
      int x;
      c.eim[j] = mant_of(g.eis[j] * s, x);
      if (blk == 0) g.xadd[j] = x;
      x = (g.dim == 1 ? g.ein[j / W] : g.ein[eb + j * es]) + g.ese[j];
      c.se[j] = x;
      e = e > x ? e : x;
    }
    max_put<THREADS>(c.mx, tid, e);
  }

  // the exponents of the factors; after load(), whose loads are then on their way
  static BEC_FX void factors(Ctx& c, const TimeArgs& g) {
    c.qx = c.fl + LPB;
    const int* qe = g.qe + c.tile * (N / 2 + 1);
    for (int k = c.tid; k < N / 2 + 1; k += THREADS) c.qx[k] = qe[k] - qe[0];
  }
  template <typename Args>
  static BEC_FX void load(Ctx& c, Reg& r, const Args& g) {
    int b0, step;
    bfly_index<LOGN, 0>(c.t, b0, step);
    const i64 *pa = g.data + b0 * g.J + c.qa, *pb = pa + LPB;
#pragma unroll
    for (int i = 0; i < EPT; ++i) r.v[i] = cx{0, 0};
    if (c.va) {
#pragma unroll
      for (int i = 0; i < EPT; ++i) {
        int bu, st;
        bfly_index<LOGN, 0>(TPL * (i / R1), bu, st);
        r.v[i].x = pa[(bu + (i % R1) * st) * g.J];
      }
    }
    if (c.vb) {
#pragma unroll
      for (int i = 0; i < EPT; ++i) {
        int bu, st;
        bfly_index<LOGN, 0>(TPL * (i / R1), bu, st);
        r.v[i].y = pb[(bu + (i % R1) * st) * g.J];
      }
    }
  }
  // the block's unit and statistics, as in DstTile
  static BEC_FX void measure(Ctx& c, Reg& r) {
    c.ref = max_get<THREADS>(c.mx);
    int b0, step;
    bfly_index<LOGN, 0>(c.t, b0, step);
    float m = 0.f, la = 0.f, lb = 0.f;
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      int bu, st;
      bfly_index<LOGN, 0>(TPL * (i / R1), bu, st);
      const int d = c.ref - c.se[b0 + bu + (i % R1) * st];
      const float x = mag(r.v[i].x, d), y = mag(r.v[i].y, d);
      m = fmaxf(m, fmaxf(x, y));
      la += x;
      lb += y;
    }
    // one sum that bounds both lines' (max over a and b of each thread's part)
    c.s = {m, fmaxf(la, lb)};
    Join::put(c.st, c.s, c.tid, c.L);
  }

  // the line's scale and D_eps (Step 1)
  static BEC_FX void first(Ctx& c, Reg& r, const TimeArgs& g) {
    const Stat s = Join::get(c.st, c.s, c.tid, c.L);
    // the separated spectra (times 2) are bounded by 2 sum |a| and 2 sum |b|
    c.sc = line_scale<LOGN>(c.ref, (float)R1 * 1.4143f * (s.m + 1.f), 2.f * (s.l + (float)N));
    const int fi = c.sc.F - 1;                      // eps^{j/N} times 2^63: half
    const int k = fi - c.ref;
    // shifts round to nearest: a mean left here is frequency 0's, whose factor is
    // the largest
    int b0, step;
    bfly_index<LOGN, 0>(c.t, b0, step);
    const W64* wp = g.esm + b0;
    const int* ep = c.se + b0;
    if (all_warp<THREADS>(k >= 0)) {                // right shifts only
#pragma unroll
      for (int i = 0; i < EPT; ++i) {
        int bu, st;
        bfly_index<LOGN, 0>(TPL * (i / R1), bu, st);
        const int j = bu + (i % R1) * st, d = fi - ep[j];
        const W64 w = wp[j];
        r.v[i] = cx{mul64(shr_rn(r.v[i].x, d), w), mul64(shr_rn(r.v[i].y, d), w)};
      }
    } else {
#pragma unroll
      for (int i = 0; i < EPT; ++i) {
        int bu, st;
        bfly_index<LOGN, 0>(TPL * (i / R1), bu, st);
        const int j = bu + (i % R1) * st, d = fi - ep[j];
        const W64 w = wp[j];
        r.v[i] = cx{mul64(shift_rn(r.v[i].x, d), w), mul64(shift_rn(r.v[i].y, d), w)};
      }
    }
    c.f = (c.ref > kFxNan / 2 ? kFxNan : c.sc.F) + c.sc.s2 + c.sc.s3;
  }
  static BEC_FX void read0(Ctx& c, Reg& r) { pass_read<LOGN, 0>(r.v, c.line, c.t); }
  template <typename Args>
  static BEC_FX void pass0(Ctx& c, Reg& r, const Args& g) {
    pass_compute<LOGN, 0, -1>(r.v, g.tw, c.t, c.sc.s2);
    if constexpr (G::NP > 1) pass_write<LOGN, 0>(r.v, c.line, c.t);
  }
  template <int P, typename Args>
  static BEC_FX void pass(Ctx& c, Reg& r, const Args& g) {
    pass_read<LOGN, P>(r.v, c.line, c.t);
    pass_compute<LOGN, P, -1>(r.v, g.tw, c.t, c.sc.s3);
    if constexpr (P + 1 < G::NP) pass_write<LOGN, P>(r.v, c.line, c.t);
  }
  static BEC_FX void natural(Ctx& c, Reg& r) { write_natural<LOGN>(r.v, c.line, c.t); }

  // the packed results at k and N - k from the spectrum there
  static BEC_FX void divide(cx C, cx Cn, CW64 qa, CW64 qb, cx& nc, cx& nn) {
    const cx A1{C.x + Cn.x, C.y - Cn.y}, A2{C.y + Cn.y, Cn.x - C.x};
    const cx B1 = cmul_conj(A1, qa), B2 = cmul_conj(A2, qb);
    nc = cx{B1.x - B2.y, B1.y + B2.x};
    nn = cx{B1.x + B2.y, B2.x - B1.y};
  }
  // Step 2 on the pairs (k, N - k), k = t + TPL u; thread 0's k = 0 stands
  // for the two self-paired frequencies 0 and N/2 (real, B_k = A_k q_k)
  static BEC_FX void solve(Ctx& c, Reg& r, const TimeArgs& g) {
    // lines past the end read mode J - 1's factors (their values are zeros)
    const CW64 *qa = g.q + (c.va ? c.qa : g.J - 1) + c.t * g.J,
               *qb = g.q + (c.vb ? c.qb : g.J - 1) + c.t * g.J;
    const cx* fp = c.line + slot(c.t);
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const cx C = fp[slot(TPL * u)];
      const cx Cn = c.line[slot(u == 0 && c.t == 0 ? 0 : N - c.t - TPL * u)];
      divide(C, Cn, qa[TPL * u * g.J], qb[TPL * u * g.J], r.v[2 * u], r.v[2 * u + 1]);
    }
    if (c.t == 0) {
      const cx C = c.line[slot(N / 2)];
      cx nc;
      divide(C, C, qa[N / 2 * g.J], qb[N / 2 * g.J], nc, r.v[1]);
    }
    // the products at k count in the unit 2^qe[k], the statistics in 2^qe[0]
    float m = 0.f, l = 0.f;
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const float w = exp2_f(c.qx[c.t + TPL * u]);
      const float w1 = u == 0 && c.t == 0 ? exp2_f(c.qx[N / 2]) : w;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float x = mag(r.v[2 * u + i].x), y = mag(r.v[2 * u + i].y);
        // one unit of slack each
        m = fmaxf(m, (fmaxf(x, y) + 1.f) * (i == 0 ? w : w1));
        l += (x + y + 2.f) * (i == 0 ? w : w1);
      }
    }
    c.s = {m, l};
    Join::put(c.st, c.s, c.tid, c.L);
  }
  // the solution spectrum on the inverse transform's scale, parts exchanged
  static BEC_FX void rescale(Ctx& c, Reg& r) {
    const Stat s = Join::get(c.st, c.s, c.tid, c.L);
    const Scale k = line_scale<LOGN>(0, (float)R1 * 1.4143f * s.m, s.l);
    c.sc = k;
    c.f += 1 + k.F + k.s2 + k.s3;                   // 1: q halves
    if (c.t == 0) c.fl[c.L] = c.f;
    cx* fp = c.line + slot(c.t);
#pragma unroll
    for (int u = 0; u < H; ++u) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const bool mid = i == 1 && u == 0 && c.t == 0;
        const int d = c.qx ? k.F - c.qx[mid ? N / 2 : c.t + TPL * u] : k.F;
        const cx v = r.v[2 * u + i], w{shift_rn(v.y, d), shift_rn(v.x, d)};
        if (i == 0) fp[slot(TPL * u)] = w;
        else c.line[slot(mid ? N / 2 : N - c.t - TPL * u)] = w;
      }
    }
  }
  // D_eps^{-1} (Step 3): the last pass's outputs are in registers, output i of
  // butterfly u is time step base + i step
  static BEC_FX void store(Ctx& c, Reg& r, const TimeArgs& g) {
    int b0, step;
    out_index<LOGN>(c.t, b0, step);
    i64 *pa = g.data + b0 * g.J + c.qa, *pb = pa + LPB;
    const W64* ep = c.eim + b0;
    // on the tile's exponent, the largest of its lines'
    int fm = c.fl[0];
#pragma unroll
    for (int i = 1; i < LPB; ++i) fm = fm > c.fl[i] ? fm : c.fl[i];
    const int d = fm - c.f;
    const i64 rnd = d > 0 ? 1LL << ((d > 62 ? 62 : d) - 1) : 0;
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      int bu, st;
      out_index<LOGN>(TPL * (i / RL), bu, st);
      const int j = bu + (i % RL) * st;
      const W64 w = ep[j];                          // half
      if (c.va) pa[j * g.J] = mul64(shr(r.v[i].y + rnd, d), w);
      if (c.vb) pb[j * g.J] = mul64(shr(r.v[i].x + rnd, d), w);
    }
    if (c.tid == 0) g.eout[c.tile] = fm + 1 + g.qe[c.tile * (N / 2 + 1)];
  }
};

// ------------------------------------------- time transforms of the multigrid route
struct SpecArgs {
  i64* data;                   // [N][J] FP64 bit patterns
  double2* spec;               // [N/2+1][J] half spectrum
  long long J;
  int m;
  const double* w;             // eps^{j/N}, inverse: eps^{-j/N}
  double scale;
  const double* scale_dev;     // null: 1
  const CW64* tw;
};

// The time pass cut open (FP64 in and out): Step 1 to the half spectrum, and
// Step 3 from one.  A line's unit comes from its largest value alone, so lines
// of different size in a tile do not lose bits to each other.
template <int LOGN, int LPB>
struct SpecTile : TimeTile<LOGN, LPB> {
  using B = TimeTile<LOGN, LPB>;
  using typename B::Ctx;
  using typename B::Reg;
  using G = Line<LOGN>;
  using Join = LineJoin<LPB, G::TPL, false>;
  static constexpr int N = G::n, TPL = G::TPL, EPT = G::EPT, H = EPT / 2, THREADS = B::THREADS;
  static constexpr int R1 = B::R1, RL = B::RL;

  static BEC_FX double to_d(i64 v, int f) {
    return fx_normal(f) ? fx_to_d(v, f) : f > kFxNan / 2 ? bits_d(0x7FF8000000000000ULL) : fx_to_d_slow(v, f);
  }
  static BEC_FX void init(Ctx& c, const SpecArgs& g, unsigned char* smem, int tid, long long blk) {
    B::place(c, g.m, smem, tid, blk);
    const double s = g.scale_dev ? g.scale * g.scale_dev[0] : g.scale;
    int e = -kFxNan;
    for (int j = tid; j < N; j += THREADS) {
      int x;
      c.eim[j] = mant_of(g.w[j] * s, x);
      c.se[j] = x;
      e = e > x ? e : x;
    }
    max_put<THREADS>(c.mx, tid, e);
  }
  // the largest exponent field of the line, in two phases; the lines' shared
  // memory is free until the first pass
  static BEC_FX Stat* scratch(const Ctx& c) { return reinterpret_cast<Stat*>(c.line - c.L * G::STRIDE); }
  static BEC_FX void max_in(Ctx& c, const Reg& r) {
    int h = 0;
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      const int x = d_habs((u64)r.v[i].x), y = d_habs((u64)r.v[i].y), w = x > y ? x : y;
      h = h > w ? h : w;
    }
    c.s = {(float)(h >> 20), 0.f};
    Join::put(scratch(c), c.s, c.tid, c.L);
  }
  // the line's values as integers below 2^bits; returns their exponent
  static BEC_FX int to_fixed(Ctx& c, Reg& r, int bits) {
    const int em = (int)Join::get(scratch(c), c.s, c.tid, c.L).m;
    const int f = em - 1022 - bits;
    if (f >= kFxMin) {
#pragma unroll
      for (int i = 0; i < EPT; ++i) r.v[i] = cx{d_to_fx((u64)r.v[i].x, f), d_to_fx((u64)r.v[i].y, f)};
    } else {
#pragma unroll
      for (int i = 0; i < EPT; ++i) r.v[i] = cx{d_to_fx_sub((u64)r.v[i].x, f), d_to_fx_sub((u64)r.v[i].y, f)};
    }
    c.f = em == 0x7FF ? kFxNan : 0;
    return f;
  }

  // forward: values, then the statistics as in TimeTile::measure
  static BEC_FX void measure(Ctx& c, Reg& r) {
    c.ref = to_fixed(c, r, 62);
    const int e = max_get<THREADS>(c.mx);
    int b0, step;
    bfly_index<LOGN, 0>(c.t, b0, step);
    float m = 0.f, la = 0.f, lb = 0.f;
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      int bu, st;
      bfly_index<LOGN, 0>(TPL * (i / R1), bu, st);
      const int d = e - c.se[b0 + bu + (i % R1) * st];
      const float x = mag(r.v[i].x, d), y = mag(r.v[i].y, d);
      m = fmaxf(m, fmaxf(x, y));
      la += x;
      lb += y;
    }
    c.s = {m, fmaxf(la, lb)};
    Join::put(c.st, c.s, c.tid, c.L);
  }
  static BEC_FX void first(Ctx& c, Reg& r) {
    const Stat s = Join::get(c.st, c.s, c.tid, c.L);
    const int e = max_get<THREADS>(c.mx);
    c.sc = line_scale<LOGN>(c.ref + e, (float)R1 * 1.4143f * (s.m + 1.f), 2.f * (s.l + (float)N));
    const int fi = c.sc.F - 1;                      // w times 2^63: half
    int b0, step;
    bfly_index<LOGN, 0>(c.t, b0, step);
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      int bu, st;
      bfly_index<LOGN, 0>(TPL * (i / R1), bu, st);
      const int j = b0 + bu + (i % R1) * st, d = fi - c.ref - c.se[j];
      r.v[i] = cx{mul64(shift_rn(r.v[i].x, d), c.eim[j]), mul64(shift_rn(r.v[i].y, d), c.eim[j])};
    }
    if (e > kFxNan / 2) c.f = kFxNan;
    c.f += (c.f == kFxNan ? 0 : c.sc.F) + c.sc.s2 + c.sc.s3;
  }
  // the two lines' spectra at k, separated
  static BEC_FX void put(const Ctx& c, const SpecArgs& g, int k, cx C, cx Cn) {
    const int f = c.f - 1;
    double2* p = g.spec + k * g.J;
    if (c.va) p[c.qa] = make_double2(to_d(C.x + Cn.x, f), to_d(C.y - Cn.y, f));
    if (c.vb) p[c.qb] = make_double2(to_d(C.y + Cn.y, f), to_d(Cn.x - C.x, f));
  }
  static BEC_FX void store(Ctx& c, const SpecArgs& g) {
    const cx* fp = c.line + slot(c.t);
#pragma unroll
    for (int u = 0; u < H; ++u)
      put(c, g, c.t + TPL * u, fp[slot(TPL * u)], c.line[slot(u == 0 && c.t == 0 ? 0 : N - c.t - TPL * u)]);
    if (c.t == 0) put(c, g, N / 2, c.line[slot(N / 2)], c.line[slot(N / 2)]);
  }

  // inverse: v[2 u], v[2 u + 1] = the two lines' values at k = t + TPL u; of the
  // real frequencies 0 and N/2 the real parts, side by side
  static BEC_FX void load_spec(Ctx& c, Reg& r, const SpecArgs& g) {
    const i64 *pa = reinterpret_cast<const i64*>(g.spec + c.t * g.J + c.qa), *pb = pa + 2 * LPB;
#pragma unroll
    for (int i = 0; i < EPT; ++i) r.v[i] = cx{0, 0};
    if (c.va) {
#pragma unroll
      for (int u = 0; u < H; ++u) r.v[2 * u] = cx{pa[2 * TPL * u * g.J], pa[2 * TPL * u * g.J + 1]};
      if (c.t == 0) r.v[0].y = pa[N * g.J];
    }
    if (c.vb) {
#pragma unroll
      for (int u = 0; u < H; ++u) r.v[2 * u + 1] = cx{pb[2 * TPL * u * g.J], pb[2 * TPL * u * g.J + 1]};
      if (c.t == 0) r.v[1].y = pb[N * g.J];
    }
  }
  // A + i B at k and conj(A) + i conj(B) at N - k, and what rescale() wants
  static BEC_FX void measure_spec(Ctx& c, Reg& r) {
    const int f = to_fixed(c, r, 61);
    c.f += c.f == kFxNan ? 0 : f - 1;               // rescale() counts a factor 2
    float m = 0.f, l = 0.f;
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const cx A = r.v[2 * u], Bv = r.v[2 * u + 1];
      const bool real = u == 0 && c.t == 0;
      r.v[2 * u] = real ? cx{A.x, Bv.x} : cx{A.x - Bv.y, A.y + Bv.x};
      r.v[2 * u + 1] = real ? cx{A.y, Bv.y} : cx{A.x + Bv.y, Bv.x - A.y};
    }
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      const float x = mag(r.v[i].x), y = mag(r.v[i].y);
      m = fmaxf(m, fmaxf(x, y) + 1.f);              // one unit of slack each
      l += x + y + 2.f;
    }
    c.s = {m, l};
    Join::put(c.st, c.s, c.tid, c.L);
  }
  static BEC_FX void store_time(Ctx& c, Reg& r, const SpecArgs& g) {
    int b0, step;
    out_index<LOGN>(c.t, b0, step);
    double *pa = reinterpret_cast<double*>(g.data) + b0 * g.J + c.qa, *pb = pa + LPB;
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      int bu, st;
      out_index<LOGN>(TPL * (i / RL), bu, st);
      const int j = bu + (i % RL) * st, f = c.f + 1 + c.se[b0 + j];
      const W64 w = c.eim[b0 + j];                  // half
      if (c.va) pa[j * g.J] = to_d(mul64(r.v[i].y, w), f);
      if (c.vb) pb[j * g.J] = to_d(mul64(r.v[i].x, w), f);
    }
  }
};

}  // namespace fx
}  // namespace bec
