"""The totals of the FP64 dataflow iterations, bit for bit: one iteration from x = 0 with the far-field condition
(which projects nothing) leaves x = alpha u with alpha = (r,u) / (w,u), r = b, u = D^-1 r, w = K u, so x shows whether
the two sums were exact up to one rounding and whether the quotient was rounded correctly."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def one_step(rp, col, K, dinv, b):
    """x after one iteration with one row a thread: every product rounded once, the sums exact."""
    u = [float(d) * float(r) for d, r in zip(dinv, b)]
    gamma = delta = Fraction(0)
    for i in range(len(b)):
        w = 0.0
        for k in range(rp[i], rp[i + 1]):
            w = fma(float(K[k]), u[col[k]], w)
        gamma += Fraction(float(b[i]) * u[i])
        delta += Fraction(w * u[i])
    gamma, delta = float(gamma), float(delta)
    alpha = gamma / delta
    return np.array([alpha * ui for ui in u])


@pytest.mark.parametrize("block,blocks", [(256, 3), (256, 33), (512, 2), (512, 89), (0, 0)])
@pytest.mark.parametrize("spread", [0, 40])
def test_first_step_is_exact(block, blocks, spread):
    """Right-hand sides of one size, and of sizes down to 2^-40 of the largest (squares of them: a sum in 57-bit images
    loses their low bits); several seeds, so that a sum or a quotient off by a few units in the last place shows.
    Blocks of up to 128 or 256 rows (one a thread), one and three groups of polled blocks, and the default launch."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    m = cgp.Mesh(*inputs.ogrid(24, 10))
    cgp.cgp_set_far_field(m.handle, 1)
    q = m.matrices()
    rp, col, K = q["rowptr"], q["col"], q["K"].copy()
    fixed = np.zeros(m.n_c, bool)
    fixed[cgp.cgp_far_field_nodes(m.handle)] = True
    row = np.repeat(np.arange(m.n_c), np.diff(rp))
    K[(fixed[row] | fixed[col]) & (row != col)] = 0.0
    K[(row == col) & fixed[row]] = 1.0
    dinv = 1.0 / K[row == col]
    cgp.cgp_set_tuning(m.handle, 0, block, 1 if block else 0, blocks, 8 if block else 0)
    for seed in range(12):
        rng = np.random.default_rng(seed)
        b = rng.standard_normal(m.n_c) * np.exp2(-spread * rng.random(m.n_c))
        b[fixed] = 0.0
        x = torch.zeros(m.n_c, dtype=torch.float64, device=DEV)
        info = cgp.cgp_poisson_solve(m.handle, torch.as_tensor(b, device=DEV), x, tol=1e-12, max_it=1)
        assert info["iterations"] == 1 and cgp.cgp_last_launch(m.handle)["resident"] == 1
        np.testing.assert_array_equal(x.cpu().numpy(), one_step(rp, col, K, dinv, b))
    m.close()
