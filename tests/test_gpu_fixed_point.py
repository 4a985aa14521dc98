"""The fixed-point passes of the FP64 sine-transform P_eps^{-1}: every length of
the spatial and the time transform against the oracle, in one, two and three
dimensions and for every discretisation; the exponents between the passes
(scaling by a power of two changes nothing else; zeros, spikes, slices of very
different size); non-finite values; in-place and 8-byte aligned vectors."""
import math

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


def apply(p, y):
    import torch
    z = p.apply_Pinv(torch.from_numpy(np.ascontiguousarray(y)).cuda())
    torch.cuda.synchronize()
    return z.cpu().numpy()


def problem(dim, m, N, eps, **kw):
    from paper_2002_01108_gb300 import Problem
    p = Problem(dim, m, N, max_restart=2, **kw)
    p.set_eps(eps)
    return p


def tol(dim, m, N, eps):
    """The bound of the floating-point passes: O(log2(N n^dim)) transform stages,
    each within a few roundings of max|z|, and the unscaling by at most 1/eps."""
    return 16 * U64 * math.log2(N * (m + 1) ** dim) / eps


# every space length with the shortest and the longest time transform, and the
# reverse; line counts that leave the last tile of a row or of all rows ragged
_SIZES = [(1, 31, 32), (1, 63, 1024), (1, 127, 64), (1, 255, 128), (1, 511, 512), (1, 1023, 32),
          (1, 1023, 1024), (2, 31, 32), (2, 31, 1024), (2, 63, 256), (2, 127, 32), (2, 255, 64),
          (2, 511, 32), (3, 31, 32)]


@pytest.mark.parametrize("dim,m,N", _SIZES)
@pytest.mark.parametrize("kind", ["flat", "spike", "first"])
def test_matches_oracle(dim, m, N, kind):
    """Flat random data, one spike, and data in the first time step only (the
    right-hand side of an initial value without a source)."""
    eps = 0.05
    rng = np.random.default_rng(m + N)
    y = rng.uniform(-1, 1, (N,) + (m,) * dim)
    if kind == "spike":
        v = np.zeros_like(y)
        v[(N // 3,) + (m // 2,) * dim] = 1.7
        y = v
    elif kind == "first":
        y[1:] = 0.0
    with problem(dim, m, N, eps) as p:
        z = apply(p, y)
    ref = O.apply_Pinv_fst(y, dim, 1.0, 1.0 / N, eps)
    assert np.max(np.abs(z - ref)) <= tol(dim, m, N, eps) * np.max(np.abs(ref))


@pytest.mark.parametrize("space,scheme,dim", [("q1", "bdf1", 1), ("q1", "bdf1", 2), ("fd", "bdf2", 2),
                                              ("q1", "bdf2", 2)])
def test_inverts_P_for_every_discretisation(space, scheme, dim):
    """P_eps (P_eps^{-1} y) = y through the stencils: the relative residual is
    within the error bound of z times cond(P) <= ||P|| ||z|| / ||y||."""
    import torch
    m, N, eps = 63, 64, 0.1
    y = np.random.default_rng(8).uniform(-1, 1, (N,) + (m,) * dim)
    with problem(dim, m, N, eps, space=space, scheme=scheme, a=1e-2) as p:
        yd = torch.from_numpy(y).cuda()
        z = p.apply_Pinv(yd)
        r = p.apply_P(z) - yd
        # ||P|| <= 4 (largest time coefficient sum) + tau times the largest eigenvalue
        norm = 4.0 + 1e-2 * 8.0 * dim * (m + 1) ** 2 / N
        if space == "q1":                       # element matrices scale with h^dim (h^(dim-2))
            norm = (4.0 + 1e-2 * 24.0 * (m + 1) ** 2 / N) / (m + 1) ** dim
        bound = tol(dim, m, N, eps) * norm * float(z.abs().max()) * math.sqrt(y.size)
        assert float(r.norm()) <= bound


def test_power_of_two_scaling_is_exact():
    """The lines' exponents carry any common scale: z(2^k y) = 2^k z(y) bit for bit."""
    dim, m, N = 2, 63, 64
    y = np.random.default_rng(9).standard_normal((N, m, m))
    with problem(dim, m, N, 0.02) as p:
        z = apply(p, y)
        for k in (-600, -37, 1, 500):
            assert np.array_equal(apply(p, np.ldexp(y, k)), np.ldexp(z, k))


def test_zero_and_tiny_and_huge_vectors():
    dim, m, N, eps = 2, 31, 32, 0.1
    rng = np.random.default_rng(10)
    y = rng.uniform(-1, 1, (N, m, m))
    ref = O.apply_Pinv_fst(y, dim, 1.0, 1.0 / N, eps)
    with problem(dim, m, N, eps) as p:
        assert np.array_equal(apply(p, np.zeros_like(y)), np.zeros_like(y))
        # results in the subnormal range: within half a unit of the smallest number
        # per rounding on the way (16 covers the passes)
        z = apply(p, np.ldexp(y, -1060))
        assert np.max(np.abs(z - np.ldexp(ref, -1060))) <= 16 * 2.0 ** -1010
        # the largest results overflow to infinity, never to a finite wrong number
        big = apply(p, np.ldexp(y, 1023))
        with np.errstate(over="ignore"):
            want = np.ldexp(ref, 1023)
        fin = np.isfinite(big) & np.isfinite(want)
        assert np.all(np.isfinite(big) | (np.abs(ref) > 0.99))
        assert np.max(np.abs(np.ldexp(big[fin], -1023) - ref[fin])) <= tol(dim, m, N, eps) * np.max(np.abs(ref))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("dim,m,N", [(1, 31, 32), (2, 31, 32), (2, 63, 64), (3, 31, 32)])
def test_non_finite_input_gives_nan(dim, m, N, bad):
    """Every output depends on every input, so one non-finite value leaves none finite."""
    y = np.random.default_rng(11).uniform(-1, 1, (N,) + (m,) * dim)
    y.reshape(-1)[y.size // 2 + 3] = bad
    with problem(dim, m, N, 0.1) as p:
        assert not np.isfinite(apply(p, y)).any()
        y = np.nan_to_num(y, nan=0.0, posinf=0.0, neginf=0.0)      # the next apply is clean
        ref = O.apply_Pinv_fst(y, dim, 1.0, 1.0 / N, 0.1)
        assert np.max(np.abs(apply(p, y) - ref)) <= tol(dim, m, N, 0.1) * np.max(np.abs(ref))


def test_slices_of_very_different_size():
    """Time slices and modes that span 30 decades: the error is bounded by the
    largest ones."""
    dim, m, N, eps = 2, 63, 64, 0.1
    rng = np.random.default_rng(12)
    y = rng.uniform(-1, 1, (N, m, m)) * 10.0 ** rng.uniform(-30, 0, (N, 1, 1))
    ref = O.apply_Pinv_fst(y, dim, 1.0, 1.0 / N, eps)
    with problem(dim, m, N, eps) as p:
        z = apply(p, y)
    assert np.max(np.abs(z - ref)) <= tol(dim, m, N, eps) * np.max(np.abs(ref))


def test_in_place_and_eight_byte_aligned():
    import torch
    dim, m, N = 2, 63, 64
    y = np.random.default_rng(13).uniform(-1, 1, (N, m, m))
    with problem(dim, m, N, 0.1) as p:
        z = apply(p, y)
        buf = torch.zeros(2 * y.size + 3, dtype=torch.float64, device="cuda")
        a, b = buf[1:1 + y.size], buf[2 + y.size:2 + 2 * y.size]      # 8- but not 16-byte aligned
        a.copy_(torch.from_numpy(y).cuda().reshape(-1))
        p.apply_Pinv(a, b)
        torch.cuda.synchronize()
        assert np.array_equal(b.cpu().numpy().reshape(y.shape), z)
        assert float(buf[0]) == 0.0 and float(buf[1 + y.size]) == 0.0 and float(buf[-1]) == 0.0
        p.apply_Pinv(a, a)
        torch.cuda.synchronize()
        assert np.array_equal(a.cpu().numpy().reshape(y.shape), z)
