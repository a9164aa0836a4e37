"""Solves in the bisection order on a mesh with one very long row (sorted as a whole, not by insertion)."""
import numpy as np
import pytest
import torch

from oracle import cgp_oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("spokes", [31, 32, 300])    # 32, 33 and 301 entries in the centre's row
@pytest.mark.parametrize("flags", [4, 12])
def test_bisection_order_with_a_hub(spokes, flags):
    """As of the other FP64 forms: 1e-10 in x at tol 1e-12."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    th = 2.0 * np.pi * np.arange(spokes) / spokes
    ring = np.stack([np.cos(th), np.sin(th)], axis=1)
    xy = np.concatenate([np.zeros((1, 2)), ring, 2.0 * ring])
    tri = []
    for i in range(spokes):
        k = (i + 1) % spokes
        a, b, c, d = 1 + i, 1 + k, 1 + spokes + i, 1 + spokes + k
        tri += [(0, a, b), (a, c, d), (a, d, b)]
    tri = np.array(tri, dtype=np.int32)
    m, om = cgp.Mesh(xy, tri), O.OracleMesh(xy, tri)
    b = np.random.default_rng(spokes).standard_normal(m.n_c)
    b -= b.mean()
    ref = O.pcg(om.K, om.d, b, tol=1e-12)["x"]
    cgp.cgp_set_tuning(m.handle, 0, 256, 1, 5, flags)
    x = torch.zeros(m.n_c, dtype=torch.float64, device=DEV)
    assert cgp.cgp_poisson_solve(m.handle, torch.as_tensor(b, device=DEV), x, tol=1e-12)["status"] == cgp.CGP_OK
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)
    m.close()
