"""The self-test of the solvers' grid-wide waits: every kind passes with all blocks present and runs out of time, with
the context usable afterwards, when some never arrive."""
import time

import numpy as np
import pytest
import torch

from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nblk", [1, 8, 33, 152, 600])
def test_waits_with_every_block_present(nblk):
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    assert cgp.cgp_barrier_selftest(nblk, 0, 1_000_000_000) == cgp.CGP_OK


@pytest.mark.parametrize("nblk,absent", [(2, 1), (8, 1), (40, 8), (152, 151), (600, 1)])
def test_waits_run_out(nblk, absent):
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    cgp.cgp_barrier_selftest(2, 0, 1_000_000_000)
    t0 = time.perf_counter()
    assert cgp.cgp_barrier_selftest(nblk, absent, 10_000_000) == cgp.CGP_ERR_TIMEOUT
    assert time.perf_counter() - t0 < 5.0
    m = cgp.Mesh(*inputs.ogrid(24, 10))
    b = torch.as_tensor(np.random.default_rng(0).standard_normal(m.n_c), device="cuda:0")
    assert cgp.cgp_poisson_solve(m.handle, b - b.mean(), torch.zeros_like(b))["status"] == cgp.CGP_OK
    m.close()
