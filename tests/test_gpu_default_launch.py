"""The launch of meshes that were never tuned: every route of the default rule (few rows, bisection order,
registered O-grid, far field, rows too many for shared memory) against a solve with an explicit shape."""
import numpy as np
import pytest
import torch

from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("nt,nr,ogrid,far", [(3, 1, False, 0), (24, 10, False, 0), (24, 10, True, 0), (129, 31, False, 1),
                                             (129, 31, True, 1), (161, 80, False, 0), (1024, 512, False, 0)])
@pytest.mark.parametrize("precision", [0, 1])
def test_default_launch_agrees_with_an_explicit_one(nt, nr, ogrid, far, precision):
    """Both meet tol 1e-11 on the true residual, so x differs by at most the system's condition number
    (about (n_theta / 2)^2) times that."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    m = cgp.Mesh(*inputs.ogrid(nt, nr))
    if ogrid:
        cgp.cgp_mesh_set_ogrid(m.handle, nt, nr)
    if far:
        cgp.cgp_set_far_field(m.handle, 1)
    b = np.random.default_rng(2).standard_normal(m.n_c)
    b = torch.as_tensor(b - b.mean(), device=DEV)
    out = []
    for shape in ((0, 0, 0, 0), (256, 1, 8, 1)):     # rows in global memory, untagged reductions
        cgp.cgp_set_tuning(m.handle, precision, *shape)
        x = torch.zeros_like(b)
        info = cgp.cgp_poisson_solve(m.handle, b, x, tol=1e-11, precision=precision)
        assert info["status"] == cgp.CGP_OK and info["rel_res_true"] <= 1.1e-11, info
        if shape[0] == 0:
            assert cgp.cgp_last_launch(m.handle, precision)["resident"] == (0 if m.n_c > 400000 else 1)
        out.append(x)
    d = float(torch.linalg.norm(out[0] - out[1]) / torch.linalg.norm(out[1]))
    assert d <= 2e-11 * max(10.0, (nt / 2.0) ** 2), d
    m.close()


@pytest.mark.parametrize("warm", [False, True])
def test_untuned_solve_under_stream_capture(warm):
    """A captured untuned solve replays to the same answer, whether or not a first solve has built its plan."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    m = cgp.Mesh(*inputs.ogrid(129, 40))     # more than 4096 rows: the bisection order when it can be built
    b = np.random.default_rng(3).standard_normal(m.n_c)
    b = torch.as_tensor(b - b.mean(), device=DEV)
    x, ref = torch.zeros_like(b), torch.zeros_like(b)
    if warm:
        cgp.cgp_poisson_solve(m.handle, b, x, tol=1e-11)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        cgp.cgp_poisson_solve_async(m.handle, b, x, tol=1e-11)
    x.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert cgp.cgp_last_launch(m.handle)["resident"] == int(warm)
    assert cgp.cgp_poisson_solve(m.handle, b, ref, tol=1e-11)["status"] == cgp.CGP_OK
    assert float(torch.linalg.norm(x - ref) / torch.linalg.norm(ref)) <= 2e-11 * (129 / 2.0) ** 2
    m.close()
