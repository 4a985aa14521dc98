"""P_eps^{-1} of vectors next to and below the smallest normal number, 2^-1022, in
the fixed-point passes: no bits are lost but those that the numbers themselves
do not have."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


def vectors(dim, m, N):
    """Values in [1/2, 1) of either sign, and a slice of zeros."""
    rng = np.random.default_rng(m + N + dim)
    y = rng.uniform(0.5, 1.0, (N,) + (m,) * dim) * rng.choice([-1.0, 1.0], (N,) + (m,) * dim)
    y[N // 2] = 0.0
    return y


def apply(p, y):
    import torch
    z = p.apply_Pinv(torch.from_numpy(y).cuda())
    torch.cuda.synchronize()
    return z.cpu().numpy()


@pytest.mark.parametrize("dim,m,N", [(1, 63, 64), (2, 31, 32), (2, 63, 64), (3, 31, 32)])
@pytest.mark.parametrize("k", [-940, -1000, -1021])
def test_scaling_by_a_power_of_two(dim, m, N, k):
    """The inputs are normal numbers, exactly 2^k times others: the results are 2^k
    times theirs, to the last bit where they are normal, else to one subnormal
    number (they are rounded to a double before they are rounded to that)."""
    from paper_2002_01108_gb300 import Problem
    y = vectors(dim, m, N)
    with Problem(dim, m, N, max_restart=2) as p:
        p.set_eps(0.05)
        z, t = apply(p, y), apply(p, np.ldexp(y, k))
    want = np.ldexp(z, k)
    normal = np.abs(want) >= 2.0 ** -1022
    assert np.array_equal(t[normal], want[normal])
    assert np.all(np.abs(t - want) <= 2.0 ** -1074)


@pytest.mark.parametrize("dim,m,N", [(1, 63, 64), (2, 31, 32), (3, 31, 32)])
def test_subnormal_numbers(dim, m, N):
    """Inputs below 2^-1040, of at most 34 bits: against the oracle on 2^1040 times
    them; each result is within one subnormal number and the passes' own error."""
    from paper_2002_01108_gb300 import Problem
    y = np.ldexp(vectors(dim, m, N), -1040)
    with Problem(dim, m, N, max_restart=2) as p:
        p.set_eps(0.05)
        z = apply(p, y)
    ref = O.apply_Pinv_fst(np.ldexp(y, 1040), dim, 1.0, 1.0 / N, 0.05)
    assert np.max(np.abs(np.ldexp(z, 1040) - ref)) <= 2.0 ** -34 + 1e-13 * np.max(np.abs(ref))


def test_multigrid_route():
    """Its time transforms: an FP64 cycle lies between them, whose own rounding to
    subnormal numbers is below 2^-80 of these values; 4 units of the largest."""
    from paper_2002_01108_gb300 import Problem
    m, N = 31, 64
    a = np.exp(np.random.default_rng(75).uniform(-1, 1, (m + 2, m + 2)))
    y = vectors(2, m, N)
    with Problem(2, m, N, a_nodes=a, route="mg", precision="fp64", flexible=True) as p:
        p.set_eps(0.05)
        z, t = apply(p, y), apply(p, np.ldexp(y, -985))
    assert np.max(np.abs(np.ldexp(t, 985) - z)) <= 4 * U64 * np.max(np.abs(z))
