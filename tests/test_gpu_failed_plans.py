"""The default launch when a form of it cannot be built: the solve takes the next one, nothing of the failure is left
for a later call to report, and it is not tried again."""
import numpy as np
import pytest
import torch

from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
MB = 1 << 20


def fill_device(leave):
    """Allocate the device's free memory down to about `leave` bytes; returns the tensors that hold it."""
    held = []
    while True:
        want = torch.cuda.mem_get_info()[0] - leave
        if want < 20 * MB:
            return held
        while want >= 10 * MB:
            try:
                held.append(torch.empty(want, dtype=torch.uint8, device=DEV))
                break
            except torch.OutOfMemoryError:
                want //= 2
        else:
            return held


def test_renumbered_system_that_does_not_fit_the_memory():
    """512x256 on a registered grid: the tiles and the bisection order need more than 20 MB on the device, the mesh's
    own order only the halo lists of about 5 MB."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    small = cgp.Mesh(*inputs.ogrid(129, 40))         # loads every kernel used below
    sb = torch.randn(small.n_c, dtype=torch.float64, device=DEV)
    for flags in (0, 8, 40):
        if flags == 40:
            cgp.cgp_mesh_set_ogrid(small.handle, 129, 40)
        cgp.cgp_set_tuning(small.handle, 0, 0, 0, 0, flags)
        cgp.cgp_poisson_solve(small.handle, sb - sb.mean(), torch.zeros_like(sb))
    sf = torch.empty(small.n_f, dtype=torch.float64, device=DEV)
    cgp.cgp_prolong(small.handle, sb, sf)

    m = cgp.Mesh(*inputs.ogrid(512, 256))
    cgp.cgp_mesh_set_ogrid(m.handle, 512, 256)
    b = torch.as_tensor(np.random.default_rng(1).standard_normal(m.n_c), device=DEV)
    b -= b.mean()
    x, x2, xf = torch.zeros_like(b), torch.zeros_like(b), torch.empty(m.n_f, dtype=torch.float64, device=DEV)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = fill_device(14 * MB)
    if torch.cuda.mem_get_info()[0] > 20 * MB:
        del held
        torch.cuda.empty_cache()
        pytest.skip("the device's memory could not be filled")
    info = cgp.cgp_poisson_solve(m.handle, b, x, tol=1e-10)
    cgp.cgp_prolong(m.handle, x, xf)                 # raises if it finds the failed allocation's error
    torch.cuda.synchronize()
    del held
    torch.cuda.empty_cache()
    assert info["status"] == cgp.CGP_OK and cgp.cgp_last_launch(m.handle)["resident"] == 1
    free = torch.cuda.mem_get_info()[0]
    assert cgp.cgp_poisson_solve(m.handle, b, x2, tol=1e-10)["status"] == cgp.CGP_OK
    assert torch.cuda.mem_get_info()[0] == free      # the forms that failed are not tried again
    assert torch.equal(x, x2)
    m.close()
    small.close()


@pytest.mark.parametrize("ogrid", [False, True])
@pytest.mark.parametrize("nt,nr", [(1024, 512), (690, 340), (676, 336), (640, 310), (634, 306)])
def test_systems_too_large_for_shared_memory_are_not_copied(nt, nr, ogrid):
    """Rows that cannot be resident (far beyond the limit, and a few percent around it, where only the halo decides):
    the first solve leaves no renumbered copy behind, at most the halo lists (4 bytes an entry and the lists)."""
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    m = cgp.Mesh(*inputs.ogrid(nt, nr))
    if ogrid:
        cgp.cgp_mesh_set_ogrid(m.handle, nt, nr)
    b = torch.as_tensor(np.random.default_rng(4).standard_normal(m.n_c), device=DEV)
    b -= b.mean()
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert cgp.cgp_poisson_solve(m.handle, b, x)["status"] == cgp.CGP_OK
    if not cgp.cgp_last_launch(m.handle)["resident"]:
        assert free - torch.cuda.mem_get_info()[0] <= 8 * m.nnz + 4 * MB
    else:
        assert m.n_c < 245000
    m.close()
