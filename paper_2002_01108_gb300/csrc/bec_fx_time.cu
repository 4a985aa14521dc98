// Time pass of the fixed-point P_eps^{-1} (bec_fx_tiles.cuh), its tables, and
// the choice of the fixed-point route.
//
// The division by lambda'_k + tau mu is a product by a table of reciprocals in
// fixed point (16 bytes a mode and frequency, 8 bytes an unknown read from
// HBM); computing them would take FP64 operations.  Measured at 255^2 x 256:
// 200 us, where the floating-point pass takes 1042 us (187 us with one exponent for
// all frequencies of a tile, which lost up to 22 bits of the factors).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "bec_fx_tiles.cuh"
#include "bec_internal.h"
#include "bec_passes.cuh"

namespace bec {
namespace {

using namespace fx;

constexpr int fxt_blocks(int threads) { return 512 / threads > 16 ? 16 : 512 / threads > 0 ? 512 / threads : 1; }

template <typename Tile>
__global__ void __launch_bounds__(Tile::THREADS, fxt_blocks(Tile::THREADS)) time_fx_kernel(TimeArgs g) {
  extern __shared__ __align__(16) unsigned char fx_smem[];
  const int tid = threadIdx.x;
  typename Tile::Ctx c;
  typename Tile::Reg r;
  Tile::init(c, g, fx_smem, tid, blockIdx.x);
  Tile::load(c, r, g);
  Tile::factors(c, g);
  __syncthreads();
  Tile::measure(c, r);
  __syncthreads();
  Tile::first(c, r, g);
#pragma unroll 1
  for (int dir = 0; dir < 2; ++dir) {
    if (dir == 1) Tile::read0(c, r);
    Tile::pass0(c, r, g);
    if constexpr (Tile::G::NP > 1) {
      __syncthreads();
      Tile::template pass<1>(c, r, g);
    }
    if constexpr (Tile::G::NP > 2) {
      __syncthreads();
      Tile::template pass<2>(c, r, g);
    }
    if (dir == 1) break;
    __syncthreads();
    Tile::natural(c, r);
    __syncthreads();
    Tile::solve(c, r, g);
    __syncthreads();
    Tile::rescale(c, r);
    __syncthreads();
  }
  Tile::store(c, r, g);
}

template <int LOGN, int LPB>
bec_status fx_time_launch(bec_problem* p, const TimeArgs& g) {
  using Tile = TimeTile<LOGN, LPB>;
  auto k = time_fx_kernel<Tile>;
  if (Tile::SMEM > 48 * 1024)
    BEC_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile::SMEM));
  BEC_LAUNCH_BEGIN(p);
  k<<<(unsigned)(p->J / p->m * fx_xg(p)), Tile::THREADS, Tile::SMEM, p->stream>>>(g);
  BEC_LAUNCH_CHECK(p, "time_fx_kernel");
  return BEC_OK;
}
template <int LOGN>
bec_status fx_time_w(bec_problem* p, const TimeArgs& g) {
  return p->fx.lpb == 8 ? fx_time_launch<LOGN, 8>(p, g) : fx_time_launch<LOGN, 16>(p, g);
}

// The multigrid route's time transforms (FP64).  The floating-point kernels
// (bec_time.cu) are bound by the FP64 pipe: at 127^2 x 64 (1M unknowns) 83 us
// forward and 80 back, where these take 16, a good part of it launch and
// latency (16.5 MB of traffic are 2.4 us of HBM).
template <typename Tile, bool INV>
__global__ void __launch_bounds__(Tile::THREADS, fxt_blocks(Tile::THREADS)) time_spec_fx_kernel(SpecArgs g) {
  extern __shared__ __align__(16) unsigned char fx_smem[];
  typename Tile::Ctx c;
  typename Tile::Reg r;
  Tile::init(c, g, fx_smem, threadIdx.x, blockIdx.x);
  if constexpr (INV) Tile::load_spec(c, r, g);
  else Tile::load(c, r, g);
  Tile::max_in(c, r);
  __syncthreads();
  if constexpr (INV) Tile::measure_spec(c, r);
  else Tile::measure(c, r);
  __syncthreads();
  if constexpr (INV) {
    Tile::rescale(c, r);
    __syncthreads();
    Tile::read0(c, r);
  } else {
    Tile::first(c, r);
  }
  Tile::pass0(c, r, g);
  if constexpr (Tile::G::NP > 1) {
    __syncthreads();
    Tile::template pass<1>(c, r, g);
  }
  if constexpr (Tile::G::NP > 2) {
    __syncthreads();
    Tile::template pass<2>(c, r, g);
  }
  if constexpr (INV) {
    Tile::store_time(c, r, g);
  } else {
    __syncthreads();
    Tile::natural(c, r);
    __syncthreads();
    Tile::store(c, g);
  }
}

template <int LOGN, int LPB, bool INV>
bec_status fx_spec_launch(bec_problem* p, const SpecArgs& g) {
  using Tile = SpecTile<LOGN, LPB>;
  auto k = time_spec_fx_kernel<Tile, INV>;
  if (Tile::SMEM > 48 * 1024)
    BEC_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile::SMEM));
  BEC_LAUNCH_BEGIN(p);
  k<<<(unsigned)(p->J / p->m * fx_xg(p)), Tile::THREADS, Tile::SMEM, p->stream>>>(g);
  BEC_LAUNCH_CHECK(p, INV ? "time_inv_fx_kernel" : "time_fwd_fx_kernel");
  return BEC_OK;
}
template <bool INV>
bec_status fx_spec(bec_problem* p, const SpecArgs& g) {
  switch (p->tab.time.logn) {
    case 5: return fx_spec_launch<5, 16, INV>(p, g);
    case 6: return fx_spec_launch<6, 16, INV>(p, g);
    case 7: return fx_spec_launch<7, 16, INV>(p, g);
    case 8: return fx_spec_launch<8, 16, INV>(p, g);
    case 9: return fx_spec_launch<9, 8, INV>(p, g);
    default: break;
  }
  set_error("unsupported number of time steps");
  return BEC_EUNSUPPORTED;
}

// q[k][q] = scale conj(d) / |d|^2 with d = lambda'_k mu^M + tau mu^K, times
// 2^(63 - qe[k]): the largest |q| of the W modes of a tile (W lanes) at k sets
// qe[tile][k] so that |q| stays below 0.9.  With one exponent for all k, that of
// the smallest |d|, the factors of the high frequencies would keep only 63 -
// log2(|d_k| / |d_0|) bits: 41 at eps = 1 and a = 1e-5.
template <int W>
__global__ void fx_table_kernel(CW64* __restrict__ q, int* __restrict__ qe, long long rows, int xg,
                                long long J, int NK, int m, int dim, const double2* __restrict__ lamf,
                                ModeEigs<double> me, double tau, double scale) {
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long row = id / (xg * W);
  const int x = (int)(id - row * (xg * W));
  const bool in = row < rows && x < m;
  const long long i = in ? row * m + x : 0;
  double muM, muK;
  mode_eigs(i, J, m, m, dim, me, muM, muK);
  const bool fe = me.m != nullptr;
  int* tile_qe = qe + (row * xg + x / W) * NK;
  for (int k = 0; k < NK; ++k) {
    const double2 L = lamf[k];
    const double dr = fe ? fma(L.x, muM, tau * muK) : L.x + tau * muK, di = fe ? L.y * muM : L.y;
    const double s = scale / fma(dr, dr, di * di);
    // |q|^2 = scale s < 2^(E - 1022) with E its exponent field; / 0.81 in [1, 2)
    int e = (((int)(fx::d_bits(scale * s * (1.0 / 0.81)) >> 52) - 1022 + 1) >> 1);
    if (!in) e = -kFxNan;
#pragma unroll
    for (int o = 1; o < W; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if (!in) continue;
    if (x % W == 0) tile_qe[k] = e;
    auto fixed = [e](double v) {
      i64 w = d_to_fx(d_bits(v), e - 63);
      if ((int)w == (int)0x80000000) ++w;        // the low word can be negated
      return split64(w);
    };
    q[(long long)k * J + i] = CW64{fixed(dr * s), fixed(di * s)};
  }
}

const long double kPiL = 3.14159265358979323846264338327950288L;

i64 quantise(long double v, int bits) {
  i64 w = (i64)llroundl(ldexpl(v, bits));
  if ((int)w == (int)0x80000000) ++w;
  return w;
}

// the twiddle tables of a transform of length 2^LOGN (tw_first, tw_count)
template <int LOGN>
std::vector<CW64> fx_twiddles_n() {
  std::vector<CW64> t((size_t)tw_count(LOGN), CW64{{0, 0}, {0, 0}});
  for (int p = 0; p + 1 < npass(LOGN); ++p) {
    const int before = before_log(LOGN, p), lr = radix_log(LOGN, p), lm = LOGN - before - lr;
    for (int l = 0; l < (1 << lr); ++l)
      for (int i = 0; i < (1 << lm); ++i) {
        const long double a = 2 * kPiL * ((l * i) << before) / (1 << LOGN), c = cosl(a), s = sinl(a);
        for (int k = 0; k < kFxShifts; ++k)
          t[(size_t)tw_first(LOGN, p) + (k << (LOGN - before)) + (l << lm) + i] =
              CW64{split64(quantise(c, 62 - k)), split64(quantise(s, 62 - k))};
      }
  }
  return t;
}
std::vector<CW64> fx_twiddles(int logn) {
  switch (logn) {
    case 5: return fx_twiddles_n<5>();
    case 6: return fx_twiddles_n<6>();
    case 7: return fx_twiddles_n<7>();
    case 8: return fx_twiddles_n<8>();
    case 9: return fx_twiddles_n<9>();
    case 10: return fx_twiddles_n<10>();
    default: return std::vector<CW64>(1, CW64{{0, 0}, {0, 0}});   // one pass: no twiddles
  }
}

}  // namespace

void fx_free(bec_problem* p) {
  if (p->fx.tables) cudaFree(p->fx.tables);
  if (p->fx.q) cudaFree(p->fx.q);
  p->fx = FxTables{};
}

// Lengths from 32: there the whole apply is faster at every size measured, from
// 44 against 71 us at 63 x 64 (1D) to 1.19 against 6.86 ms at 255^2 x 512;
// shorter transforms would leave a block less than a warp.
bool fx_wanted(const bec_problem_desc* d, int logn, int logt) {
  return d->precision == BEC_PC_FP64 && d->route == BEC_ROUTE_FST && logn >= 5 && logt >= 5;
}

bec_status fx_setup(bec_problem* p) {
  FxTables& t = p->fx;
  const int n = p->m + 1, N = p->N;
  // 16 line pairs a block (256-byte segments across the lines); 8 for the long
  // lines whose blocks would otherwise pass 512 threads, and where both passes
  // still have 64 threads a block with 8: more and smaller blocks overlap
  // better there (255^2 x 256: 596 against 621 us an apply), while shorter
  // lines lose (63^3 x 64: 743 against 682 us)
  t.lpb = p->tab.space.logn >= 9 || p->tab.time.logn >= 9 || (p->tab.space.logn == 8 && p->tab.time.logn >= 7)
              ? 8 : 16;
  // one exponent a tile: of rows, and of columns or modes
  const long long units = p->J / p->m, tiles = units * fx_xg(p);
  const long long ne = std::max((units * N + 2 * t.lpb - 1) / (2 * t.lpb),
                                p->dim == 1 ? 0 : tiles / p->m * N);
  std::vector<W64> sinw(n / 2, W64{0, 0});
  for (int j = 1; j < n / 2; ++j) sinw[j] = split64(quantise(2 * sinl(j * kPiL / n) - 1, 63));
  const std::vector<CW64> ts = fx_twiddles(p->tab.space.logn), tt = fx_twiddles(p->tab.time.logn);
  // one allocation: the constant tables first (one copy), then the work arrays
  size_t size = 0;
  auto place = [&size](size_t bytes) {
    const size_t at = size;
    size += (bytes + 15) & ~(size_t)15;
    return at;
  };
  const size_t o_ts = place(ts.size() * sizeof(CW64)), o_tt = place(tt.size() * sizeof(CW64));
  const size_t o_sin = place(sinw.size() * sizeof(W64)), fixed = size;
  const size_t o_esm = place(N * sizeof(W64)), o_ese = place(N * sizeof(int));
  const size_t o_x = place(N * sizeof(int)), o_qe = place(tiles * (N / 2 + 1) * sizeof(int));
  const size_t o_em = place(tiles * sizeof(int)), o_e0 = place(ne * sizeof(int)), o_e1 = place(ne * sizeof(int));
  cudaError_t e = cudaMalloc(&t.tables, size);
  if (e == cudaSuccess) e = cudaMalloc(&t.q, (size_t)p->J * (N / 2 + 1) * sizeof(CW64));
  if (e == cudaSuccess) {
    std::vector<unsigned char> host(fixed);
    std::memcpy(host.data() + o_ts, ts.data(), ts.size() * sizeof(CW64));
    std::memcpy(host.data() + o_tt, tt.data(), tt.size() * sizeof(CW64));
    std::memcpy(host.data() + o_sin, sinw.data(), sinw.size() * sizeof(W64));
    e = cudaMemcpy(t.tables, host.data(), fixed, cudaMemcpyHostToDevice);
  }
  if (e != cudaSuccess) {
    fx_free(p);
    cudaGetLastError();
    set_error(std::string("fixed-point tables: ") + cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? BEC_ENOMEM : BEC_ECUDA;
  }
  unsigned char* base = static_cast<unsigned char*>(t.tables);
  t.tw_space = base + o_ts;
  t.tw_time = base + o_tt;
  t.sinw = base + o_sin;
  t.esm = base + o_esm;
  auto ints = [base](size_t at) { return reinterpret_cast<int*>(base + at); };
  t.ese = ints(o_ese);
  t.xadd = ints(o_x);
  t.qe = ints(o_qe);
  t.em = ints(o_em);
  t.e0 = ints(o_e0);
  t.e1 = ints(o_e1);
  return BEC_OK;
}

void fx_alloc_spare(bec_problem* p) {
  const int logt = p->tab.time.logn;
  if (p->desc.precision != BEC_PC_FP64 || p->desc.route == BEC_ROUTE_FST || logt < 5 || logt > 9) return;
  const std::vector<CW64> tt = fx_twiddles(logt);
  const size_t bytes = tt.size() * sizeof(CW64);
  FxTables& t = p->fx;
  if (cudaMalloc(&t.tables, bytes) != cudaSuccess ||
      cudaMemcpy(t.tables, tt.data(), bytes, cudaMemcpyHostToDevice) != cudaSuccess) {
    fx_free(p);
    cudaGetLastError();
    return;
  }
  t.tw_time = t.tables;
  t.lpb = logt >= 9 ? 8 : 16;
}

bec_status launch_fx_spec(bec_problem* p, const double* y, double* z, void* spec, const double* scale_dev) {
  SpecArgs g{};
  g.data = reinterpret_cast<i64*>(y != nullptr ? const_cast<double*>(y) : z);
  g.spec = static_cast<double2*>(spec);
  g.J = p->J;
  g.m = p->m;
  g.w = y != nullptr ? p->tab.es64 : p->tab.eis64;
  g.scale = y != nullptr ? 1.0 : 1.0 / p->N;
  g.scale_dev = scale_dev;
  g.tw = static_cast<const CW64*>(p->fx.tw_time);
  return y != nullptr ? fx_spec<false>(p, g) : fx_spec<true>(p, g);
}

bec_status fx_set_eps(bec_problem* p, const std::vector<double>& es) {
  FxTables& t = p->fx;
  std::vector<W64> m(es.size());
  std::vector<int> x(es.size());
  for (size_t j = 0; j < es.size(); ++j) m[j] = mant_of(es[j], x[j]);
  BEC_CUDA_TRY(cudaMemcpyAsync(t.esm, m.data(), m.size() * sizeof(W64), cudaMemcpyHostToDevice, p->stream));
  BEC_CUDA_TRY(cudaMemcpyAsync(t.ese, x.data(), x.size() * sizeof(int), cudaMemcpyHostToDevice, p->stream));
  const int NK = p->N / 2 + 1;
  BEC_LAUNCH_BEGIN(p);
  const long long rows = p->J / p->m, n = rows * fx_xg(p) * 2 * t.lpb;
  auto k = t.lpb == 8 ? fx_table_kernel<16> : fx_table_kernel<32>;
  k<<<(unsigned)((n + 127) / 128), 128, 0, p->stream>>>(
      static_cast<CW64*>(t.q), t.qe, rows, fx_xg(p), p->J, NK, p->m, p->dim, p->tab.lamf64,
      ModeEigs<double>{p->tab.mu64, p->tab.mum64}, p->tau, pinv_scale(p));
  BEC_LAUNCH_CHECK(p, "fx_table_kernel");
  BEC_CUDA_TRY(cudaStreamSynchronize(p->stream));
  return BEC_OK;
}

bec_status launch_fx_time(bec_problem* p, double* data, const double* scale_dev) {
  const FxTables& t = p->fx;
  TimeArgs g{};
  g.data = reinterpret_cast<i64*>(data);
  g.J = p->J;
  g.m = p->m;
  g.dim = p->dim;
  g.ein = p->dim == 2 ? t.e1 : t.e0;
  g.eout = t.em;
  g.xadd = t.xadd;
  g.esm = static_cast<const W64*>(t.esm);
  g.ese = t.ese;
  g.eis = p->tab.eis64;
  g.scale_dev = scale_dev;
  g.q = static_cast<const CW64*>(t.q);
  g.qe = t.qe;
  g.tw = static_cast<const CW64*>(t.tw_time);
  switch (p->tab.time.logn) {
    case 5: return fx_time_w<5>(p, g);
    case 6: return fx_time_w<6>(p, g);
    case 7: return fx_time_w<7>(p, g);
    case 8: return fx_time_w<8>(p, g);
    case 9: return fx_time_w<9>(p, g);
    case 10: return fx_time_w<10>(p, g);
    default: break;
  }
  set_error("unsupported number of time steps");
  return BEC_EUNSUPPORTED;
}

}  // namespace bec
