"""Which systems keep their rows in shared memory: the barrier forms need what their vectors, halo and slice take and
nothing else, and a system that fits them stays resident whatever form was asked for."""
import numpy as np
import pytest
import torch

from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
OPTIN = 232448            # shared memory a block may have (227 KB)
STATIC = 1024 + 3584      # the runtime's and the kernels' own


def sizes(rp, col, blocks):
    """(rows, entries, halo) of the largest block of a split into `blocks` chunks."""
    n = rp.size - 1
    chunk = -(-n // blocks)
    nnz = halo = 0
    for r0 in range(0, n, chunk):
        r1 = min(n, r0 + chunk)
        c = col[rp[r0]:rp[r1]]
        nnz = max(nnz, c.size)
        halo = max(halo, np.unique(c[(c < r0) | (c >= r1)]).size)
    return chunk, nnz, halo


def need(form, chunk, nnz, halo):
    ints = 4 * (chunk + 1 + nnz + halo)
    s = {"textbook": 8 * (7 * chunk + halo + nnz) + ints, "single": 8 * (10 * chunk + 5 * halo + nnz) + ints,
         "mixed": 4 * (9 * chunk + 6 * halo + 2 * nnz + 1)}[form]
    return -(-s // 16) * 16


@pytest.mark.parametrize("form,precision,flags", [("textbook", 0, 2), ("single", 0, 0), ("single", 0, 8), ("mixed", 1, 0),
                                                  ("mixed", 1, 8)])
def test_largest_resident_system(form, precision, flags):
    """The fewest blocks of a mesh whose barrier form fits: resident, in exactly that form's bytes."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    m = cgp.Mesh(*inputs.ogrid(*((512, 256) if precision == 0 else (600, 401))))
    q = m.matrices()
    lo, hi = 1, 152
    while lo < hi:                                   # need() falls with the number of blocks, up to a few rows of halo
        mid = (lo + hi) // 2
        if need(form, *sizes(q["rowptr"], q["col"], mid)) <= OPTIN - STATIC:
            hi = mid
        else:
            lo = mid + 1
    bytes_ = need(form, *sizes(q["rowptr"], q["col"], lo))
    assert OPTIN - STATIC - 4096 < bytes_ <= OPTIN - STATIC
    b = torch.as_tensor(np.random.default_rng(6).standard_normal(m.n_c), device=DEV)
    b -= b.mean()
    x = torch.zeros_like(b)
    cgp.cgp_set_tuning(m.handle, precision, 512, 1, lo, flags)
    info = cgp.cgp_poisson_solve(m.handle, b, x, precision=precision)
    assert info["status"] == cgp.CGP_OK
    ran = cgp.cgp_last_launch(m.handle, precision)
    assert ran["resident"] == 1 and ran["blocks"] == lo
    if not flags & 8:
        assert ran["smem"] == bytes_
    m.close()
