"""Device memory of small meshes: what a mesh keeps besides its own arrays is the solvers' scratch for every block that
can be resident (about 1.8 MB on 152 SMs), so that many small systems can be held at once."""
import pytest
import torch

from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_small_meshes_take_two_megabytes():
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    xy, tri = inputs.ogrid(24, 10)
    keep = [cgp.Mesh(xy, tri)]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    keep += [cgp.Mesh(xy, tri) for _ in range(40)]
    assert free - torch.cuda.mem_get_info()[0] <= 42 * (2 << 20)
    for m in keep:
        m.close()
