"""The preparation's paths by size and data, bit for bit against the CPU oracle:
nearest neighbours that all fall to one lane of the warp that looks for them
(its kept keys run out and the row is searched again), and T_NN with one, four,
ten and twenty nodes per thread and with its nodes in memory."""
import numpy as np
import pytest

from helpers import atsp, euclid, params
from paper_2601_19041_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hac():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_19041_gb300 import build, heataco
    build.build()
    return heataco


def _one_lane(n, seed=1):
    # node u belongs to cluster u % 32: a node's neighbours share its lane
    rng = np.random.default_rng(seed)
    centre = np.stack(np.meshgrid(np.arange(8), np.arange(4)), -1).reshape(-1, 2)
    return (centre[np.arange(n) % 32] + 0.05 * rng.random((n, 2))).astype(np.float32)


@pytest.mark.parametrize("n,k", [(640, 20), (640, 5), (90, 32), (333, 7)])
@pytest.mark.parametrize("kind", [0, 1])
def test_neighbours_of_one_lane(hac, orc, n, k, kind):
    pts = _one_lane(n).astype(np.float64)
    if kind == 0:
        inst, kw = euclid(pts), dict(local_search=1, ls_k=min(k, 32))
    else:
        inst = atsp(np.sqrt(((pts[:, None] - pts[None]) ** 2).sum(-1)).astype(np.float32))
        kw = dict(degree_target=1)
    p = params(m=4, k=k, iterations=1, rho=0.2, seed=3, **kw)
    o = orc.Oracle(inst, p).iterate(1)
    with hac.Batch([inst], [p]) as bt:
        bt.run().sync()
        for f, of in (("CAND", "cand"), ("CDIST", "cdist"), ("NN_TOUR", "nn_tour"), ("TOURS", "tours")):
            assert np.array_equal(bt.read(0, f), o.get(of)), f


@pytest.mark.parametrize("n", [4, 129, 512, 513, 2049, 5121, 10300])
def test_nearest_neighbour_tour(hac, orc, n):
    inst = synth.euclid_instance(n, n, K=min(6, n - 1))
    p = params(m=1, k=4, iterations=0, rho=0.2, seed=1)
    o = orc.Oracle(inst, p)
    with hac.Batch([inst], [p]) as bt:
        bt.sync()
        assert np.array_equal(bt.read(0, "NN_TOUR"), o.get("nn_tour"))
        assert bt.scalars(0)["L_nn"] == o.scalars()["L_nn"]
