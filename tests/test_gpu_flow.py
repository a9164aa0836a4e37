"""The dataflow iterations of the resident solvers (tuning flag bit 3, blocks of at least 256 threads) at the
sizes where their roles and groups change: one block, one and several groups of 32 polled blocks, blocks with
a single row, rows in two register slots, more rows than register slots, and rows longer than the eight
entries kept in registers."""
import numpy as np
import pytest
import torch

from oracle import cgp_oracle as O
from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def fan(spokes, rings):
    """A disc: a centre of degree `spokes` and `rings` rings of nodes around it (rows of 4 to 7 entries, one long)."""
    th = 2.0 * np.pi * np.arange(spokes) / spokes
    xy = [np.zeros((1, 2))] + [np.stack([(j + 1) * np.cos(th), (j + 1) * np.sin(th)], axis=1) for j in range(rings)]
    tri = []
    for i in range(spokes):
        k = (i + 1) % spokes
        tri.append((0, 1 + i, 1 + k))
        for j in range(rings - 1):
            a, b, c, d = 1 + j * spokes + i, 1 + j * spokes + k, 1 + (j + 1) * spokes + i, 1 + (j + 1) * spokes + k
            tri += [(a, c, d), (a, d, b)]
    return np.concatenate(xy), np.array(tri, dtype=np.int32)


MESHES = {"ogrid-64x32": lambda: inputs.ogrid(64, 32), "ogrid-33x17": lambda: inputs.ogrid(33, 17),
          "fan-20x40": lambda: fan(20, 40)}


@pytest.fixture(scope="module", params=list(MESHES))
def system(request):
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    xy, tri = MESHES[request.param]()
    m, om = cgp.Mesh(xy, tri), O.OracleMesh(xy, tri)
    if request.param.startswith("ogrid"):
        cgp.cgp_mesh_set_ogrid(m.handle, *(int(t) for t in request.param[6:].split("x")))
    b = np.random.default_rng(5).standard_normal(m.n_c)
    b -= b.mean()
    yield cgp, m, om, b
    m.close()


def rel(a, r):
    return float(np.linalg.norm(a - r) / np.linalg.norm(r))


@pytest.mark.parametrize("block,blocks", [(256, 1), (512, 1), (512, 2), (512, 32), (256, 33), (512, 65), (288, 152), (512, 600)])
@pytest.mark.parametrize("flags", [8, 12, 40])
def test_fp64_dataflow_matches_the_oracle(system, block, blocks, flags):
    """Same tolerances as the other FP64 forms: 1e-10 in x at tol 1e-12."""
    cgp, m, om, b = system
    ref = O.pcg(om.K, om.d, b, tol=1e-12)
    cgp.cgp_set_tuning(m.handle, cgp.CGP_TUNE_SOLVE_FP64, block, 1, blocks, flags)
    x = torch.zeros(m.n_c, dtype=torch.float64, device=DEV)
    info = cgp.cgp_poisson_solve(m.handle, torch.as_tensor(b, device=DEV), x, tol=1e-12)
    cgp.cgp_set_tuning(m.handle, cgp.CGP_TUNE_SOLVE_FP64, 0, 0, 0, 0)
    assert info["status"] == cgp.CGP_OK, info
    assert abs(info["iterations"] - ref["iterations"]) <= 3 + info["outer_sweeps"] * max(10, ref["iterations"] // 5)
    assert rel(x.cpu().numpy(), ref["x"]) <= 1e-10


@pytest.mark.parametrize("block,blocks", [(256, 1), (512, 1), (512, 2), (512, 5), (256, 33), (512, 65), (288, 152)])
@pytest.mark.parametrize("flags", [8, 12])
def test_mixed_dataflow_reaches_the_fp64_answer(system, block, blocks, flags):
    cgp, m, om, b = system
    exact = O.pcg(om.K, om.d, b, tol=1e-14)["x"]
    ref = O.mixed_ir(om.K, om.d, b, tol=1e-8, inner_tol=1e-4)
    cgp.cgp_set_tuning(m.handle, cgp.CGP_TUNE_SOLVE_MIXED, block, 1, blocks, flags)
    x = torch.zeros(m.n_c, dtype=torch.float64, device=DEV)
    info = cgp.cgp_poisson_solve(m.handle, torch.as_tensor(b, device=DEV), x, tol=1e-8, precision=cgp.CGP_MIXED,
                                 inner_tol=1e-4)
    cgp.cgp_set_tuning(m.handle, cgp.CGP_TUNE_SOLVE_MIXED, 0, 0, 0, 0)
    assert info["status"] == cgp.CGP_OK and info["rel_res_true"] <= 1e-8, info
    assert rel(x.cpu().numpy(), exact) <= max(10 * rel(ref["x"], exact), 1e-9)
