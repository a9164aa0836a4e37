"""The learned guess's gradients at the edges of the backward kernels' batches: row counts that four does not divide
(a warp takes four rows) and a node with more than 32 neighbours (out-edges come in batches of eight and 32)."""
import numpy as np
import pytest

from oracle import cgp_oracle as O
from oracle import gnn_oracle as G
from paper_2003_00082_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"
# Both sides round to BF16 at ten points of the forward pass, where a value near a rounding boundary may land one step
# (2^-7 of an element's magnitude) apart, and the backward runs on those values: twenty steps at most, twelve allowed.
BF16_STEPS = 24 * 2.0 ** -8


def fan(spokes):
    th = 2.0 * np.pi * np.arange(spokes) / spokes
    xy = np.concatenate([np.zeros((1, 2)), np.stack([np.cos(th), np.sin(th)], axis=1)])
    return xy, np.array([(0, 1 + i, 1 + (i + 1) % spokes) for i in range(spokes)], dtype=np.int32)


MESHES = {"ogrid-33x17": lambda: inputs.ogrid(33, 17), "fan-45": lambda: fan(45)}


@pytest.mark.parametrize("mesh,batch", [("ogrid-33x17", 1), ("ogrid-33x17", 3), ("fan-45", 1), ("fan-45", 3)])
def test_gradients_match_the_oracle_elementwise(mesh, batch):
    from paper_2003_00082_gb300 import build, cgp
    build.build()
    cgp.load()
    xy, tri = MESHES[mesh]()
    m, om = cgp.Mesh(xy, tri), O.OracleMesh(xy, tri)
    assert (m.n_c * batch) % 4 == 2        # a partial group of rows
    g = G.Graph(om.K, om.xy_c)
    rng = np.random.default_rng(batch)
    data = [tuple(rng.standard_normal(m.n_c) for _ in range(4)) for _ in range(batch)]
    shapes = G.param_shapes()
    p0 = G.init_params(5, zero_decoder=False)
    flat = np.concatenate([p0[k].reshape(-1) for k in shapes]).astype(np.float32)

    def unpack(v):
        out, o = {}, 0
        for k, shp in shapes.items():
            out[k] = np.asarray(v[o:o + int(np.prod(shp))], dtype=np.float64).reshape(shp)
            o += int(np.prod(shp))
        return out

    p = unpack(flat)                       # the FP32 values the GPU holds
    net = cgp.GNN(m, batch, flat)
    stacked = [torch.as_tensor(np.concatenate([d[k] for d in data]), dtype=torch.float64, device=DEV) for k in range(4)]
    grads, out, loss = net.gradients(batch, *stacked)
    samples = []
    for b, phi1, phi2, phit in data:
        f, s = G.features(g, om.K, b, phi1, phi2)
        samples.append((f, (phit - phi1) / s))
    mag_out, mag_grads = G.magnitudes(p, g, samples)
    for s, (f, _) in enumerate(samples):
        assert np.all(np.abs(out[s] - G.forward(p, g, f, bf16_storage=True)[0]) <= BF16_STEPS * mag_out[s])
    ref_loss, ref = G.loss_and_grad(p, g, samples, bf16_storage=True)
    assert abs(loss - ref_loss) <= 2e-2 * ref_loss
    got = unpack(grads)
    for k in ref:
        assert np.all(np.abs(got[k] - ref[k]) <= BF16_STEPS * mag_grads[k] + 1e-30), k
    net.close()
    m.close()
