"""Systems whose rows fit in shared memory only without the dataflow iterations' additional few KB: an untuned solve
keeps the exact sums of the untagged form, bit for bit what that form gives when it is asked for."""
import numpy as np
import pytest
import torch

from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LIMIT = 232448 - 1024 - 3136      # shared memory a block may have, less the runtime's and the kernels' own


def barrier_bytes(q, blocks):
    """Shared memory of the largest block in the mesh's order (single-reduction form)."""
    rp, col = q["rowptr"], q["col"]
    n = rp.size - 1
    chunk = -(-n // blocks)
    nnz = halo = 0
    for r0 in range(0, n, chunk):
        r1 = min(n, r0 + chunk)
        c = col[rp[r0]:rp[r1]]
        nnz, halo = max(nnz, c.size), max(halo, np.unique(c[(c < r0) | (c >= r1)]).size)
    return chunk, 8 * (10 * chunk + 5 * halo + nnz) + 4 * (chunk + 1 + nnz + halo)


def test_untuned_batch_of_a_system_without_room_for_the_dataflow_state():
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    for nr in range(330, 300, -1):    # one more ring is about seven rows a block
        m = cgp.Mesh(*inputs.ogrid(512, nr))
        chunk, need = barrier_bytes(m.matrices(), 152)
        if LIMIT - 4000 - chunk < need <= LIMIT - 64:
            break
        m.close()
    assert LIMIT - 4000 - chunk < need <= LIMIT - 64
    b = np.random.default_rng(0).standard_normal(m.n_c)
    b = torch.as_tensor(b - b.mean(), device=DEV)
    out = []
    for tuning in ((0, 0, 0, 0), (512, 1, 1, 0)):
        x = torch.zeros_like(b)
        B = cgp.Batch([m], [b], [x], tol=1e-6)
        B.set_tuning(*tuning)
        assert B.query()["resident"] == 1 and B.query()["grid"] == 152
        B.solve()
        assert B.info()[0][0]["status"] == cgp.CGP_OK
        out.append(x)
        B.close()
    assert torch.equal(*out)
    m.close()
