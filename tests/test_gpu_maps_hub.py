"""The velocity correction around a node of very many triangles (a fan of 1500 spokes)."""
import time

import numpy as np
import pytest
import torch

from oracle import cgp_oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def T(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("spokes", [32, 33, 1500])   # 64 entries a list (merged), 66 and 3000 (not merged)
def test_velocity_correction_around_a_hub(spokes):
    """Against the oracle, to the rounding of a sum of `spokes` terms of one size; and the first call, which builds
    the operator, does work linear in the number of triangles: well under 0.2 s (comparing every pair of a list of
    3000 entries in one thread takes 1 s)."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    th = 2.0 * np.pi * np.arange(spokes) / spokes
    xy = np.concatenate([np.zeros((1, 2)), np.stack([np.cos(th), np.sin(th)], axis=1)])
    tri = np.array([(0, 1 + i, 1 + (i + 1) % spokes) for i in range(spokes)], dtype=np.int32)
    m, om = cgp.Mesh(xy, tri), O.OracleMesh(xy, tri)
    rng = np.random.default_rng(spokes)
    p, u, v = (rng.standard_normal(m.n_f) for _ in range(3))
    args = T(p), T(u), T(v)
    out = [torch.empty(m.n_f, dtype=torch.float64, device=DEV) for _ in range(2)]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    cgp.cgp_velocity_correct(m.handle, *args, 0.05, *out)
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 0.2
    for got, old, ref in zip(out, (u, v), O.velocity_correct(om.xy_f, om.tri_f, p, u, v, 0.05)):
        assert np.linalg.norm(got.cpu().numpy() - ref) <= 3e-16 * spokes * np.linalg.norm(ref - old) + 1e-15 * np.linalg.norm(ref)
    m.close()


def test_first_corrections_of_several_threads():
    """Host threads that make the first velocity correction on one mesh at the same time, each on its own stream: one
    builds the operator, and all get the bits of a later call."""
    from concurrent.futures import ThreadPoolExecutor

    from paper_2003_00082_gb300 import build, cgp, inputs
    build.build()
    cgp.load()
    m = cgp.Mesh(*inputs.ogrid(129, 40))
    rng = np.random.default_rng(3)
    p, u, v = (T(rng.standard_normal(m.n_f)) for _ in range(3))
    jobs = [(torch.cuda.Stream(), torch.empty_like(u), torch.empty_like(v)) for _ in range(4)]
    torch.cuda.synchronize()
    with ThreadPoolExecutor(4) as ex:
        list(ex.map(lambda j: cgp.cgp_velocity_correct(m.handle, p, u, v, 0.05, j[1], j[2], stream=j[0]), jobs))
    torch.cuda.synchronize()
    ref = torch.empty_like(u), torch.empty_like(v)
    cgp.cgp_velocity_correct(m.handle, p, u, v, 0.05, *ref)
    torch.cuda.synchronize()
    for _, a, b in jobs:
        assert torch.equal(a, ref[0]) and torch.equal(b, ref[1])
    m.close()
