"""The preparation at the limits of its paths, bit for bit against the CPU
oracle: squared distances at the end of the FP32 range, T_NN of a cost matrix with
one to twenty nodes per thread and from memory, costs below zero and ties."""
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


def _same(hac, orc, inst, p, fields=("CAND", "CDIST", "NN_TOUR")):
    o = orc.Oracle(inst, p)
    with hac.Batch([inst], [p]) as bt:
        bt.sync()
        for f in fields:
            assert np.array_equal(bt.read(0, f), o.get(f.lower())), f
        return o


@pytest.mark.parametrize("n,k", [(40, 1), (40, 2), (200, 2)])
def test_a_nearer_node_whose_fp32_key_overflows(hac, orc, n, k):
    """Node 9 is nearer to node 0 than node 5 in FP64, but its FP32 squared distance
    rounds up past the largest number and node 5's does not."""
    pts = np.full((n, 2), 1e20, np.float32)
    pts[:, 0] += np.arange(n, dtype=np.float32) * np.float32(1e18)
    pts[0] = 0.0
    pts[5] = (float.fromhex("0x1.ffe9620000000p+63"), float.fromhex("0x1.305ae40000000p+58"))
    pts[9] = (float.fromhex("0x1.b159940000000p+63"), float.fromhex("0x1.10ace20000000p+63"))
    if k == 2:
        pts[2] = (1.0, 1.0)
    o = _same(hac, orc, euclid(pts), params(m=1, k=k, iterations=0, rho=0.2), ("CAND", "CDIST"))
    assert o.get("cand").reshape(n, -1)[0, k - 1] == 9


@pytest.mark.parametrize("n", [4, 129, 513, 2048, 2049, 5121, 10300])
def test_nearest_neighbour_tour_of_a_cost_matrix(hac, orc, n):
    # 1000 different costs: equal smallest costs fall to nodes of different threads
    cost = np.random.default_rng(n).integers(1, 1001, (n, n)).astype(np.float32)
    np.fill_diagonal(cost, 0.0)
    rng = np.random.default_rng(1)
    nbr = np.stack([rng.choice(n - 1, 3, replace=False) for _ in range(n)])
    nbr += nbr >= np.arange(n)[:, None]
    nbr.sort(axis=1)
    inst = synth.Instance(n=n, kind=1, coords=None, cost=cost, rowptr=np.arange(0, 3 * n + 1, 3, dtype=np.int32),
                          col=nbr.ravel().astype(np.int32), val=np.full(3 * n, 0.25, np.float32), symmetrize=0)
    p = params(m=1, k=3, iterations=0, rho=0.2, degree_target=1)
    o = orc.Oracle(inst, p)
    with hac.Batch([inst], [p]) as bt:
        bt.sync()
        assert np.array_equal(bt.read(0, "NN_TOUR"), o.get("nn_tour"))
        assert bt.scalars(0)["L_nn"] == o.scalars()["L_nn"]


@pytest.mark.parametrize("n", [50, 640])
@pytest.mark.parametrize("k", [1, 7, 32])
@pytest.mark.parametrize("levels", [3, 1000])
def test_costs_below_zero(hac, orc, n, k, levels):
    # the cheapest nodes of a row share a lane (its kept keys run out), many costs are equal
    rng = np.random.default_rng(n + levels)
    cost = rng.integers(0, levels, (n, n)).astype(np.float32) - np.float32(levels + 5)
    cost[:, np.arange(n) % 32 == 3] -= np.float32(levels)
    cost[:, np.arange(n) % 32 == 4] = 0.0
    np.fill_diagonal(cost, 0.0)
    _same(hac, orc, atsp(cost), params(m=1, k=k, iterations=0, rho=0.2, degree_target=1))
