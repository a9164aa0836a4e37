"""The mapping kernels on a mesh with long rows: a fan whose centre has 20 neighbours (more than one batch of a
row's entries in the right-hand side and in the velocity correction's operator, slices of uneven rows)."""
import numpy as np
import pytest
import torch

from oracle import cgp_oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def T(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def rel(a, r):
    return float(np.linalg.norm(a - r) / np.linalg.norm(r))


@pytest.mark.parametrize("spokes,levels", [(20, 1), (20, 2), (9, 1), (33, 1)])
def test_maps_on_a_fan(spokes, levels):
    """Tolerances as on the other meshes: rounding of sums of up to 33 terms."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    th = 2.0 * np.pi * np.arange(spokes) / spokes
    xy = np.concatenate([np.zeros((1, 2)), np.stack([np.cos(th), np.sin(th)], axis=1)])
    tri = np.array([(0, 1 + i, 1 + (i + 1) % spokes) for i in range(spokes)], dtype=np.int32)
    m, om = cgp.Mesh(xy, tri, levels), O.OracleMesh(xy, tri, levels=levels)
    rng = np.random.default_rng(spokes)
    p, u, v = (rng.standard_normal(m.n_f) for _ in range(3))
    b = torch.empty(m.n_c, dtype=torch.float64, device=DEV)
    B = (0.2, -0.4, 1.3)
    for kind in (0, 1):
        cgp.cgp_restrict(m.handle, kind, B, 20.0, T(u), T(v), b)
        Fx, Fy = O.source_field(kind, om.restrict(u), om.restrict(v), B, 20.0)
        ref = O.rhs(om.Gx, om.Gy, Fx, Fy)
        scale = np.max(np.abs(np.concatenate([Fx, Fy]))) * np.max(np.abs(om.Gx.data) + np.abs(om.Gy.data)) * spokes
        assert np.max(np.abs(b.cpu().numpy() - ref)) <= 1e-14 * scale
    grad = torch.empty(2 * m.t_f, dtype=torch.float64, device=DEV)
    force = torch.empty_like(grad)
    cgp.cgp_lorentz(m.handle, T(p), T(u), T(v), B, 2.5, grad, force)
    g_ref, f_ref = O.lorentz(om.xy_f, om.tri_f, p, u, v, B, 2.5)
    assert rel(grad.cpu().numpy().reshape(2, -1).T, g_ref) <= 1e-13
    assert rel(force.cpu().numpy().reshape(2, -1).T, f_ref) <= 1e-13
    u1, v1 = torch.empty(m.n_f, dtype=torch.float64, device=DEV), torch.empty(m.n_f, dtype=torch.float64, device=DEV)
    cgp.cgp_velocity_correct(m.handle, T(p), T(u), T(v), 0.05, u1, v1)
    ref_u, ref_v = O.velocity_correct(om.xy_f, om.tri_f, p, u, v, 0.05)
    assert rel(u1.cpu().numpy() - u, ref_u - u) <= 1e-13
    assert rel(v1.cpu().numpy() - v, ref_v - v) <= 1e-13
    m.close()
