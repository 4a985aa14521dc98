"""The fixed-point rows of L where a tile's values span many binades: every row is
held to a bound on its own operands, sum |coefficient| |value|, as an FP64 row
would be, down to subnormal numbers.

Tolerance, in units of 2^-53 times that sum: a row in fixed point has its largest
operand within 6 bits of the tile's largest or goes through FP64, so that the
roundings of its operands to the unit, at most 12 of them (3D), of its products
and of the step difference stay below 24; an FP64 row takes at most 12."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


FORMS = {"fd": (2, 255, 1.0), "fd small c": (2, 255, 1e-5), "bdf2": (2, 255, 1.0), "bdf2 small c": (2, 255, 1e-5),
         "3d": (3, 31, 0.1), "3d small c": (3, 31, 1e-4), "q1": (2, 255, 1e-2), "q1 small a": (2, 255, 1e-5)}
N = 16


def sums(v, dim):
    """(the 2 dim nearest neighbours, 2D: the 4 corners), zeros outside."""
    p = np.pad(v, [(0, 0)] + [(1, 1)] * dim)
    inner = (slice(None),) + (slice(1, -1),) * dim
    near, corner = np.zeros_like(v), None
    for d in range(1, dim + 1):
        for s in (slice(None, -2), slice(2, None)):
            k = list(inner)
            k[d] = s
            near = near + p[tuple(k)]
    if dim == 2:
        corner = p[:, :-2, :-2] + p[:, :-2, 2:] + p[:, 2:, :-2] + p[:, 2:, 2:]
    return near, corner


def rows(form, v):
    """(L v, sum |coefficient| |value|) in extended precision."""
    dim, m, a = FORMS[form]
    v = v.astype(np.longdouble)
    out = []
    for w, sign in ((v, -1), (np.abs(v), 1)):
        near, corner = sums(w, dim)
        if form.startswith("q1"):
            h = 1.0 / (m + 1)
            M = [np.longdouble(x) * h * h / 36 for x in (16, 4, 1)]
            K = [np.longdouble(a) * 8 / 3, -np.longdouble(a) / 3, -np.longdouble(a) / 3]
            A = [x + k / N for x, k in zip(M, K)]
            if sign > 0:
                A = [abs(x) for x in A]
            y = A[0] * w + A[1] * near + A[2] * corner
            y[1:] += sign * (M[0] * w + M[1] * near + M[2] * corner)[:-1]
        else:
            c = np.longdouble(a) / N * (m + 1) ** 2
            y = c * (2 * dim * w + sign * near) + (1.5 if form.startswith("bdf2") else 1.0) * w
            if form.startswith("bdf2"):
                y[1:] += sign * 2 * w[:-1]
                y[2:] += 0.5 * w[:-2]
            else:
                y[1:] += sign * w[:-1]
        out.append(y)
    return out


def steep(v, dim):
    return v * (10.0 ** (-14.0 * np.arange(v.shape[-1]) / v.shape[-1]))


def spikes(v, dim):
    r = np.random.default_rng(3).uniform(0, 1, v.shape)
    return np.where(r < 0.01, 1e9 * v, np.where(r < 0.2, 1e-7 * v, v))


def islands(v, dim):
    """Blocks of zeros among blocks of very different size."""
    b = -(-v.shape[-1] // 8)
    e = np.random.default_rng(4).choice([0.0, 1.0, 1e-12, 1e-3], (v.shape[0],) + (b,) * dim)
    for d in range(1, dim + 1):
        e = np.repeat(e, 8, axis=d)
    return v * e[(slice(None),) + (slice(0, v.shape[-1]),) * dim]


VALUES = {"steep": steep, "spikes": spikes, "islands": islands,
          "tiny": lambda v, dim: np.ldexp(steep(v, dim), -960), "subnormal": lambda v, dim: np.ldexp(v, -1050)}


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("values", list(VALUES))
def test_every_row_to_its_own_operands(form, values):
    import torch
    from paper_2002_01108_gb300 import Problem
    dim, m, a = FORMS[form]
    v = VALUES[values](np.random.default_rng(m).uniform(-1, 1, (N,) + (m,) * dim), dim)
    kw = {"bdf2": dict(scheme="bdf2"), "q1": dict(space="q1")}.get(form.split()[0], {})
    with Problem(dim, m, N, a=a, max_restart=1, **kw) as p:
        y = p.apply_A(torch.from_numpy(v).cuda()).cpu().numpy()
    ref, size = rows(form, v)
    # the smallest subnormal for each of the 24 roundings
    assert np.all(np.abs(y - ref) <= 24 * (U64 * size + np.longdouble(2.0) ** -1074 * (1 + FORMS[form][2] * m * m)))


@pytest.mark.parametrize("form", list(FORMS))
def test_zeros(form):
    import torch
    from paper_2002_01108_gb300 import Problem
    dim, m, a = FORMS[form]
    kw = {"bdf2": dict(scheme="bdf2"), "q1": dict(space="q1")}.get(form.split()[0], {})
    with Problem(dim, m, N, a=a, max_restart=1, **kw) as p:
        y = p.apply_A(torch.zeros((N,) + (m,) * dim, dtype=torch.float64, device="cuda"))
    assert float(y.abs().max()) == 0.0
