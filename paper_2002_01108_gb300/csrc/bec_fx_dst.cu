// Row and column DST passes of the fixed-point P_eps^{-1} (bec_fx_tiles.cuh).
//
// One block transforms 2 LPB lines, 16 complex values a thread, in two or
// three radix passes through shared memory.  What bounds a pass: about 100
// integer instructions an element at 16 warps an SM (128 registers a thread),
// next to 16 bytes an element of HBM traffic.  Measured at 255^2 x 256 (16.6M
// unknowns): y-DST 93 us, x-DST 105 us, where the floating-point passes take
// 550 us (17 FP64 instructions an element at 2 a clock and SM).
#include <cuda_runtime.h>

#include "bec_fx_tiles.cuh"
#include "bec_internal.h"

namespace bec {
namespace {

using namespace fx;

// 128 registers a thread: 512 threads an SM
constexpr int fx_blocks(int threads) { return 512 / threads > 16 ? 16 : 512 / threads > 0 ? 512 / threads : 1; }

template <typename Tile, bool ROWS>
__global__ void __launch_bounds__(Tile::THREADS, fx_blocks(Tile::THREADS)) dst_fx_kernel(DstArgs g) {
  extern __shared__ __align__(16) unsigned char fx_smem[];
  const int tid = threadIdx.x;
  const long long blk = blockIdx.x;
  typename Tile::Ctx c;
  typename Tile::Reg r;
  Tile::init(c, g, fx_smem, tid, blk);
  Tile::load(c, r, g);
  if constexpr (!(Tile::kInD && Tile::Join::LOCAL)) __syncthreads();
  Tile::measure(c, r);
  if constexpr (!Tile::Join::LOCAL) __syncthreads();
  Tile::prepass(c, r, g);
  __syncthreads();
  Tile::template pass<0>(c, r, g);
  if constexpr (Tile::G::NP > 1) {
    __syncthreads();
    Tile::template pass<1>(c, r, g);
  }
  if constexpr (Tile::G::NP > 2) {
    __syncthreads();
    Tile::template pass<2>(c, r, g);
  }
  __syncthreads();
  Tile::natural(c, r);
  __syncthreads();
  Tile::chunk(c, r);
  __syncthreads();
  if constexpr (Tile::GROUPS) {
    Tile::chunk_group(c);
    __syncthreads();
  }
  Tile::store(c, r, g);
  Tile::store_exp(c, g, blk);
  if constexpr (ROWS) {
    __syncthreads();
    Tile::store_rows(c, g, fx_smem, blk);
  }
}

template <int LOGN, int LPB, bool ROWS, bool IN_D, bool OUT_D>
bec_status fx_dst_launch(bec_problem* p, const DstArgs& g, long long units) {
  using Tile = DstTile<LOGN, LPB, ROWS, IN_D, OUT_D>;
  auto k = dst_fx_kernel<Tile, ROWS>;
  if (Tile::SMEM > 48 * 1024)
    BEC_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile::SMEM));
  const long long blocks = ROWS ? (g.rows + Tile::W - 1) / Tile::W : units * Tile::XG;
  BEC_LAUNCH_BEGIN(p);
  k<<<(unsigned)blocks, Tile::THREADS, Tile::SMEM, p->stream>>>(g);
  BEC_LAUNCH_CHECK(p, ROWS ? "dst_rows_fx_kernel" : "dst_cols_fx_kernel");
  return BEC_OK;
}
template <int LOGN, bool ROWS, bool IN_D, bool OUT_D>
bec_status fx_dst_w(bec_problem* p, const DstArgs& g, long long units) {
  return p->fx.lpb == 8 ? fx_dst_launch<LOGN, 8, ROWS, IN_D, OUT_D>(p, g, units)
                        : fx_dst_launch<LOGN, 16, ROWS, IN_D, OUT_D>(p, g, units);
}

template <bool ROWS, bool IN_D, bool OUT_D>
bec_status fx_dst(bec_problem* p, const DstArgs& g, long long units) {
  switch (p->tab.space.logn) {
    case 5: return fx_dst_w<5, ROWS, IN_D, OUT_D>(p, g, units);
    case 6: return fx_dst_w<6, ROWS, IN_D, OUT_D>(p, g, units);
    case 7: return fx_dst_w<7, ROWS, IN_D, OUT_D>(p, g, units);
    case 8: return fx_dst_w<8, ROWS, IN_D, OUT_D>(p, g, units);
    case 9: return fx_dst_w<9, ROWS, IN_D, OUT_D>(p, g, units);
    case 10: return fx_dst_w<10, ROWS, IN_D, OUT_D>(p, g, units);
    default: break;
  }
  set_error("unsupported spatial transform length");
  return BEC_EUNSUPPORTED;
}

DstArgs fx_args(const bec_problem* p, const void* in, void* out, int kind) {
  const FxTables& t = p->fx;
  DstArgs g{};
  g.in = in;
  g.out = out;
  g.m = p->m;
  g.dim = p->dim;
  g.kind = kind;
  g.J = p->J;
  g.rows = p->J / p->m * p->N;
  g.xadd = t.xadd;
  g.sinw = static_cast<const W64*>(t.sinw);
  g.tw = static_cast<const CW64*>(t.tw_space);
  return g;
}

}  // namespace

// The exponents of the tiles alternate between e0 and e1; the time pass's are
// em: forward rows -> e0, y -> e1, z -> e0; back y -> e0, z -> e1.
bec_status launch_fx_rows(bec_problem* p, const double* in, double* out, bool forward) {
  const FxTables& t = p->fx;
  DstArgs g = fx_args(p, in, out, forward ? kRowsFwd : kRowsBack);
  if (forward) {
    g.eout = t.e0;
    return fx_dst<true, true, false>(p, g, 0);
  }
  g.ein = p->dim == 1 ? t.em : p->dim == 2 ? t.e0 : t.e1;
  return fx_dst<true, false, true>(p, g, 0);
}

bec_status launch_fx_cols(bec_problem* p, double* data, bool forward) {
  const FxTables& t = p->fx;
  const long long units = (long long)p->N * (p->dim == 3 ? p->m : 1);
  DstArgs g = fx_args(p, data, data, forward ? kColsY : kColsYBack);
  g.ein = forward ? t.e0 : t.em;
  g.eout = forward ? t.e1 : t.e0;
  bec_status s = fx_dst<false, false, false>(p, g, units);
  if (s != BEC_OK || p->dim == 2) return s;
  g.kind = kColsZ;
  g.ein = g.eout;
  g.eout = forward ? t.e0 : t.e1;
  return fx_dst<false, false, false>(p, g, units);
}

}  // namespace bec
