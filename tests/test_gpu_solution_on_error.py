"""A solve that ends with an error before its first update leaves u = 0, as a
solve without a first guess starts from."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


def test_persistent_batch_whose_wait_runs_out():
    """The withheld launch (bec_inject_fault on the host; the wait is bounded, about
    0.2 s) is the first Arnoldi step's; the next solve is as usual."""
    import torch
    from paper_2002_01108_gb300 import Batch, BecError, bec
    lib = bec.load()
    specs = [dict(dim=2, nx=m, N=N, eps=0.05, precision="fp32", max_restart=10) for m, N in ((31, 32), (63, 32))]
    rng = np.random.default_rng(21)
    fs = [torch.from_numpy(rng.uniform(-1, 1, (s["N"], s["nx"], s["nx"]))).cuda() for s in specs]
    with Batch(specs, nstreams=2, mode="persistent") as b:
        us = [torch.full_like(f, 7.0) for f in fs]
        torch.cuda.synchronize()
        assert lib.bec_inject_fault(2) == 0
        with pytest.raises(BecError) as e:
            b.solve(fs, us, restart=10, rtol=1e-8)
        assert e.value.status == 6
        assert all(not u.any() for u in us)
        assert all(i["converged"] for i in b.solve(fs, us, restart=10, rtol=1e-8))
