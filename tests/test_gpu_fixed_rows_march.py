"""The fixed-point rows of L along a chunk of time steps: sizes at which a warp
walks 8 or 16 steps, with steps of very different size one after the other,
steps out of the fixed-point range, and values that are not finite.  Every row
is held to a bound on its own operands' steps, |v^n| and those before it that
the row takes, not on the whole vector."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53
STEPS = 40                     # rows compared (two and a half chunks or more)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


def chunk(dim, m, N):
    """Steps a warp walks: 16, halved until the card's 3648 warps all have a tile."""
    per = (m + 31) // 32 * ((m + 3) // 4) * (m if dim == 3 else 1)
    c = 16
    while c > 1 and per * ((N + c - 1) // c) < 3648:
        c //= 2
    return c


def fd_rows(v, dim, m, N, a, bdf2):
    v = v.astype(np.longdouble)
    c = np.longdouble(a) / N * (m + 1) ** 2
    p = np.pad(v, [(0, 0)] + [(1, 1)] * dim)
    inner = (slice(None),) + (slice(1, -1),) * dim
    lap = 2 * dim * v
    for d in range(1, dim + 1):
        for s in (slice(None, -2), slice(2, None)):
            k = list(inner)
            k[d] = s
            lap = lap - p[tuple(k)]
    y = c * lap + (1.5 * v if bdf2 else v)
    y[1:] -= (2 if bdf2 else 1) * v[:-1]
    if bdf2:
        y[2:] += 0.5 * v[:-2]
    return y


def q1_weights(m, N, a):
    h, tau = 1.0 / (m + 1), 1.0 / N
    M = [16.0 * h * h / 36.0, 4.0 * h * h / 36.0, h * h / 36.0]
    K = [8.0 * a / 3.0, -a / 3.0, -a / 3.0]
    return [x + tau * k for x, k in zip(M, K)], M


def q1_rows(v, m, N, a):
    A, M = q1_weights(m, N, a)
    p = np.pad(v.astype(np.longdouble), [(0, 0), (1, 1), (1, 1)])

    def form(w):
        edge = p[:, :-2, 1:-1] + p[:, 2:, 1:-1] + p[:, 1:-1, :-2] + p[:, 1:-1, 2:]
        corner = p[:, :-2, :-2] + p[:, :-2, 2:] + p[:, 2:, :-2] + p[:, 2:, 2:]
        return np.longdouble(w[0]) * p[:, 1:-1, 1:-1] + np.longdouble(w[1]) * edge + np.longdouble(w[2]) * corner
    y, mv = form(A), form(M)
    y[1:] -= mv[:-1]
    return y


KINDS = {"fd": (2, 255, 128, 1.0, 16), "bdf2": (2, 255, 64, 1e-3, 8), "3d": (3, 31, 128, 0.1, 8),
         "q1": (2, 255, 64, 1e-2, 8)}


def sizes_of(steps):
    """The bound's unit per row: the largest of the steps it takes, per step."""
    return np.array([np.max(np.abs(s[np.isfinite(s)])) for s in steps])


def case(form, v):
    """(y, reference, bound per row) of the first STEPS rows of L v."""
    import torch
    from paper_2002_01108_gb300 import Problem
    dim, m, N, a, want = KINDS[form]
    assert chunk(dim, m, N) == want
    kw = {"bdf2": dict(scheme="bdf2"), "q1": dict(space="q1")}.get(form, {})
    with Problem(dim, m, N, a=a, max_restart=1, **kw) as p:
        y = p.apply_A(torch.from_numpy(v).cuda())[:STEPS].cpu().numpy()
    with np.errstate(all="ignore"):
        ref = q1_rows(v[:STEPS], m, N, a) if form == "q1" else fd_rows(v[:STEPS], dim, m, N, a, form == "bdf2")
    big = sizes_of(v[:STEPS])
    top = big.copy()
    top[1:] = np.maximum(top[1:], big[:-1])
    if form == "bdf2":
        top[2:] = np.maximum(top[2:], big[:-2])
    if form == "q1":
        A, M = q1_weights(m, N, a)
        size = 16 * sum(abs(w[0]) + 4 * abs(w[1]) + 4 * abs(w[2]) for w in (A, M))
    else:
        size = 8 * ((3 if form == "bdf2" else 1) + 2 * dim * a / N * (m + 1) ** 2)
    return y, ref, (U64 * size * top).reshape((-1,) + (1,) * dim)


def data(form):
    dim, m, N = KINDS[form][:3]
    return np.random.default_rng(m + N).uniform(-1, 1, (N,) + (m,) * dim)


_SIZES = {
    # each step 2^-20 of the one before, back to 1 every 12
    "falling": lambda n: 2.0 ** (-20 * (n % 12)),
    "rising": lambda n: 2.0 ** (20 * (n % 12)),
    # ordinary steps after one that is much larger, at every place in a chunk
    "single 1e18": lambda n: 1e18 if n % 7 == 2 else 1.0 + n / 8,
    "single 1e-3": lambda n: 1e-3 if n % 5 == 3 else 1.0,
    # a step whose rows are out of the fixed-point range
    "single 1e300": lambda n: 1e300 if n % 7 == 2 else 1.25,
    "zero steps": lambda n: 0.0 if n % 4 in (1, 2) else 3.0,
}


@pytest.mark.parametrize("form", list(KINDS))
@pytest.mark.parametrize("sizes", list(_SIZES))
def test_rows_after_steps_of_another_size(form, sizes):
    v = data(form)
    v *= np.array([_SIZES[sizes](n) for n in range(len(v))]).reshape((-1,) + (1,) * (v.ndim - 1))
    y, ref, bound = case(form, v)
    assert np.all(np.abs(y - ref) <= bound)


@pytest.mark.parametrize("form", list(KINDS))
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("step", [0, 2, 6, 17])
def test_rows_after_a_step_that_is_not_finite(form, bad, step):
    """The rows that do not take the value are those of the finite formula."""
    v = data(form)
    at = (step,) + (min(v.shape[1] // 2, 127),) * (v.ndim - 1)
    v[at] = bad
    y, ref, bound = case(form, v)
    hit = ~np.isfinite(ref)
    assert hit.any() and not np.isfinite(y[hit]).any()
    assert np.all(np.abs(y[~hit] - ref[~hit]) <= np.broadcast_to(bound, y.shape)[~hit])


@pytest.mark.parametrize("form", list(KINDS))
def test_residual_after_a_large_step(form):
    """RES of a vector with one large step: f is L u in extended precision, rounded, so
    that RES is the rows' and f's rounding alone, dominated by the large step's; with
    the large step's two rows taken out by f = 0 there the others still have to agree."""
    import torch
    from paper_2002_01108_gb300 import Problem
    dim, m, N, a, _ = KINDS[form]
    v = np.zeros_like(data(form))
    v[:STEPS] = data(form)[:STEPS]
    v[3] *= 2.0 ** 40
    _, ref, bound = case(form, v)
    f = np.zeros_like(v)
    f[:STEPS] = ref.astype(np.float64)
    kw = {"bdf2": dict(scheme="bdf2"), "q1": dict(space="q1")}.get(form, {})
    with Problem(dim, m, N, a=a, max_restart=1, **kw) as p:
        u = torch.from_numpy(v).cuda()
        y = p.apply_A(u)
        f[STEPS:] = y[STEPS:].cpu().numpy()
        res = p.true_relres(torch.from_numpy(f).cuda(), u)
    per = v[0].size
    top = float(np.sqrt(per * np.sum(bound.astype(np.float64) ** 2)))
    assert res * float(np.linalg.norm(f)) <= top
