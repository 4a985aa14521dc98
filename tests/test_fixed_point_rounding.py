"""The rounding errors of the forward sine transforms of the fixed-point passes
have no mean over rows or time steps: the time pass amplifies frequency 0 of the
lowest modes most, and a mean adds up there.  The tiles run on the host, thread
by thread, against long double."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "bec_fx_tiles.cuh"
using namespace bec::fx;
typedef long double ld;
static const ld kPi = 3.14159265358979323846264338327950288L;
constexpr int LOGN = 6, LPB = 16, n = 1 << LOGN, m = n - 1, N = 512, W = 2 * LPB, XG = n / W;

static i64 quantise(ld v, int bits) {
  i64 w = (i64)llroundl(ldexpl(v, bits));
  if ((int)w == (int)0x80000000) ++w;
  return w;
}
static std::vector<CW64> twiddles() {
  std::vector<CW64> t(tw_count(LOGN), CW64{{0, 0}, {0, 0}});
  for (int p = 0; p + 1 < npass(LOGN); ++p) {
    const int before = before_log(LOGN, p), lr = radix_log(LOGN, p), lm = LOGN - before - lr;
    for (int l = 0; l < (1 << lr); ++l)
      for (int i = 0; i < (1 << lm); ++i)
        for (int k = 0; k < kFxShifts; ++k) {
          const ld a = 2 * kPi * ((l * i) << before) / n;
          t[tw_first(LOGN, p) + (k << (LOGN - before)) + (l << lm) + i] =
              CW64{split64(quantise(cosl(a), 62 - k)), split64(quantise(sinl(a), 62 - k))};
        }
  }
  return t;
}

#define ALL(call) for (int t = 0; t < Tile::THREADS; ++t) call
template <typename Tile, bool ROWS>
void pass(const DstArgs& g, long long blocks) {
  std::vector<unsigned char> buf(Tile::SMEM + 64);
  unsigned char* sm = reinterpret_cast<unsigned char*>(((size_t)buf.data() + 15) & ~(size_t)15);
  std::vector<typename Tile::Ctx> c(Tile::THREADS);
  std::vector<typename Tile::Reg> r(Tile::THREADS);
  for (long long b = 0; b < blocks; ++b) {
    ALL(Tile::init(c[t], g, sm, t, b));
    ALL(Tile::load(c[t], r[t], g));
    ALL(Tile::measure(c[t], r[t]));
    ALL(Tile::prepass(c[t], r[t], g));
    ALL(Tile::template pass<0>(c[t], r[t], g));
    ALL(Tile::template pass<1>(c[t], r[t], g));
    ALL(Tile::natural(c[t], r[t]));
    ALL(Tile::chunk(c[t], r[t]));
    ALL(Tile::store(c[t], r[t], g));
    ALL(Tile::store_exp(c[t], g, b));
    if (ROWS) ALL(Tile::store_rows(c[t], g, sm, b));
  }
}

int main() {
  const long long J = m * m, U = J * N;
  std::vector<double> y(U);
  unsigned long long s = 1;
  for (double& v : y) {
    s = s * 6364136223846793005ULL + 1442695040888963407ULL;
    v = (double)(long long)(s >> 11) * 0x1p-52 - 1.0;
  }
  ld sn[n][n];
  for (int j = 0; j < n; ++j)
    for (int k = 0; k < n; ++k) sn[j][k] = 4 * sinl(kPi * (j * k % (2 * n)) / n);
  const std::vector<CW64> tw = twiddles();
  std::vector<W64> sinw(n / 2, W64{0, 0});
  for (int j = 1; j < n / 2; ++j) sinw[j] = split64(quantise(2 * sinl(j * kPi / n) - 1, 63));
  std::vector<i64> d(U);
  std::vector<int> e0(m * N / W + 1), e1(N * XG), xadd(N, 0);
  DstArgs g{};
  g.in = y.data();
  g.out = d.data();
  g.m = m;
  g.dim = 2;
  g.xg = XG;
  g.J = J;
  g.rows = (long long)m * N;
  g.xadd = xadd.data();
  g.sinw = sinw.data();
  g.tw = tw.data();
  g.kind = kRowsFwd;
  g.eout = e0.data();
  pass<DstTile<LOGN, LPB, true, true, false>, true>(g, (g.rows + W - 1) / W);
  std::vector<ld> v(U, 0);
  // rows: errors in the tile's units, by mode
  std::vector<double> mean(m, 0), var(m, 0);
  for (long long r = 0; r < g.rows; ++r)
    for (int k = 0; k < m; ++k) {
      ld a = 0;
      for (int j = 0; j < m; ++j) a += sn[j + 1][k + 1] * y[r * m + j];
      v[r * m + k] = a;
      const double e = (double)((ld)d[r * m + k] - ldexpl(a, -e0[r / W]));
      mean[k] += e;
      var[k] += e * e;
    }
  double rows = 0;
  for (int k = 0; k < m; ++k) {
    const double mu = mean[k] / g.rows, se = sqrt(var[k] / g.rows) / sqrt((double)g.rows);
    rows = fmax(rows, fabs(mu) / (6 * se + 0.02));
  }
  g.kind = kColsY;
  g.in = d.data();
  g.ein = e0.data();
  g.eout = e1.data();
  pass<DstTile<LOGN, LPB, false, false, false>, false>(g, (long long)N * XG);
  // columns: mean over the steps, by mode, against the rms value
  std::vector<double> mc(J, 0);
  double sq = 0;
  for (int t = 0; t < N; ++t)
    for (int k = 0; k < m; ++k)
      for (int i = 0; i < m; ++i) {
        ld a = 0;
        for (int j = 0; j < m; ++j) a += sn[j + 1][k + 1] * v[t * J + j * m + i];
        mc[k * m + i] += (double)(ldexpl((ld)d[t * J + k * m + i], e1[t * XG + i / W]) - a) / N;
        sq += (double)(a * a);
      }
  double cols = 0;
  for (double x : mc) cols = fmax(cols, fabs(x));
  std::printf("%g %g\n", rows, cols / sqrt(sq / U) * 0x1p53);
}
"""


def test_errors_have_no_mean(tmp_path):
    """Rows, 32256 of them: each mode's mean error is within 6 standard errors plus
    1/50 of a unit.  Columns: each mode's mean over 512 steps stays below half of
    2^-53 of the rms value, the least that one rounding in FP64 would add."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "rounding.cu"
    src.write_text(_PROGRAM)
    exe = tmp_path / "rounding"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2002_01108_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert float(out[0]) <= 1.0
    assert float(out[1]) <= 0.5
