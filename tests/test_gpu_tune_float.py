"""Block widths of the FP64 floating-point passes, which sides or step counts below
32 still run: every width gives the same result bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


@pytest.mark.parametrize("m,N,tiles", [(63, 16, [(4, 4, 0), (16, 16, 0), (4, 16, 0)]),
                                       (15, 64, [(0, 0, 4), (0, 0, 16), (0, 0, 8)])])
def test_every_block_width_gives_the_same_result(m, N, tiles):
    import torch
    from paper_2002_01108_gb300 import Problem
    y = torch.from_numpy(np.random.default_rng(5).uniform(-1, 1, (N, m, m))).cuda()
    with Problem(2, m, N, precision="fp64") as p:
        p.set_eps(0.05)
        ref = p.apply_Pinv(y).clone()
        for t in tiles:
            p.set_tiles(*t)
            z = p.apply_Pinv(y)
            torch.cuda.synchronize()
            assert torch.equal(z, ref), t
