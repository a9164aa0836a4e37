"""Launch shapes of the dataflow iterations at their limits, each shown to have run (resident, with the blocks asked
for): blocks of a single row, several passes of polled blocks, every warp of a block polling."""
import numpy as np
import pytest
import torch

from oracle import cgp_oracle as O
from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, r):
    return float(np.linalg.norm(a - r) / np.linalg.norm(r))


@pytest.fixture(scope="module")
def lib():
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    return cgp


# (n_theta, n_r, threads, blocks): single rows; 32, 33 and 152 blocks; more blocks than SMs where two share one
SHAPES = [(12, 8, 256, 108), (12, 8, 512, 108), (12, 10, 256, 132), (64, 32, 256, 32), (64, 32, 512, 33), (129, 67, 288, 152),
          (129, 67, 256, 304), (257, 100, 256, 304)]


@pytest.mark.parametrize("nt,nr,block,blocks", SHAPES)
@pytest.mark.parametrize("flags", [8, 12, 40])
def test_fp64_shapes(lib, nt, nr, block, blocks, flags):
    """Tolerances as of the other FP64 forms: 1e-10 in x at tol 1e-12."""
    m, om = lib.Mesh(*inputs.ogrid(nt, nr)), O.OracleMesh(*inputs.ogrid(nt, nr))
    lib.cgp_mesh_set_ogrid(m.handle, nt, nr)
    b = np.random.default_rng(7).standard_normal(m.n_c)
    b -= b.mean()
    ref = O.pcg(om.K, om.d, b, tol=1e-12)
    lib.cgp_set_tuning(m.handle, lib.CGP_TUNE_SOLVE_FP64, block, 1, blocks, flags)
    x = torch.zeros(m.n_c, dtype=torch.float64, device=DEV)
    info = lib.cgp_poisson_solve(m.handle, torch.as_tensor(b, device=DEV), x, tol=1e-12)
    ran = lib.cgp_last_launch(m.handle)
    assert ran["resident"] == 1 and ran["blocks"] == blocks and ran["block"] == block
    assert info["status"] == lib.CGP_OK, info
    assert rel(x.cpu().numpy(), ref["x"]) <= 1e-10
    m.close()


@pytest.mark.parametrize("nt,nr,block,blocks", SHAPES)
@pytest.mark.parametrize("flags", [8, 12])
def test_mixed_shapes(lib, nt, nr, block, blocks, flags):
    """304 blocks of 256 threads: ten groups of 32 polled blocks on eight warps, so every warp polls and two of them
    twice, and the halo is fetched by polling threads."""
    m, om = lib.Mesh(*inputs.ogrid(nt, nr)), O.OracleMesh(*inputs.ogrid(nt, nr))
    b = np.random.default_rng(7).standard_normal(m.n_c)
    b -= b.mean()
    exact = O.pcg(om.K, om.d, b, tol=1e-14)["x"]
    ref = O.mixed_ir(om.K, om.d, b, tol=1e-8, inner_tol=1e-4)
    lib.cgp_set_tuning(m.handle, lib.CGP_TUNE_SOLVE_MIXED, block, 1, blocks, flags)
    x = torch.zeros(m.n_c, dtype=torch.float64, device=DEV)
    info = lib.cgp_poisson_solve(m.handle, torch.as_tensor(b, device=DEV), x, tol=1e-8, precision=lib.CGP_MIXED,
                                 inner_tol=1e-4)
    ran = lib.cgp_last_launch(m.handle, lib.CGP_MIXED)
    assert ran["resident"] == 1 and ran["blocks"] == blocks and ran["block"] == block
    assert info["status"] == lib.CGP_OK and info["rel_res_true"] <= 1e-8, info
    assert rel(x.cpu().numpy(), exact) <= max(10 * rel(ref["x"], exact), 1e-9)
    m.close()
