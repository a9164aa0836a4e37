"""Plans that share kernels: a batch that was planned keeps running after another one, of smaller systems, was."""
import numpy as np
import pytest
import torch

from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def make(cgp, nt, precision):
    m = cgp.Mesh(*inputs.ogrid(nt, nt // 2))
    b = torch.as_tensor(np.random.default_rng(nt).standard_normal(m.n_c), device=DEV)
    b -= b.mean()
    x = torch.zeros_like(b)
    return m, cgp.Batch([m], [b], [x], precision=precision), x


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("tuning", [(0, 0, 0, 0), (512, 1, 1, 0), (512, 1, 1, 8), (512, 1, 1, 4), (256, 1, 1, 8)])
def test_batch_solves_after_a_smaller_one_was_planned(precision, tuning):
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    big, B, x = make(cgp, 400, precision)
    B.set_tuning(*tuning)
    B.solve()
    assert B.info()[0][0]["status"] == cgp.CGP_OK and B.query()["resident"] == 1
    ref = x.clone()
    small, S, _ = make(cgp, 40, precision)
    S.set_tuning(*tuning)
    x.zero_()
    B.solve()
    assert B.info()[0][0]["status"] == cgp.CGP_OK
    assert torch.equal(x, ref)
    for o in (B, S, big, small):
        o.close()
