"""Nearest-unvisited steps with the lookup list where a candidate's choice value
underflows to zero, bit for bit against the CPU oracle: such a candidate is never
chosen by the roulette but may be the nearest unvisited node, so the list must hold
it.  With one candidate per node the pheromone's lower bound is infinite and its
upper bound is the smallest value that the pheromone takes."""
import numpy as np
import pytest

from helpers import euclid, params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hac():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_19041_gb300 import build, heataco
    build.build()
    return heataco


@pytest.mark.parametrize("k", [1, 2, 8])
@pytest.mark.parametrize("n,scale,beta", [(50, 1e18, 2.0), (97, 3e19, 2.0), (120, 1e5, 8.0), (5, 1e18, 2.0)])
def test_choice_values_that_underflow(hac, orc, n, scale, beta, k):
    inst = euclid((np.random.default_rng(n).random((n, 2)) * scale).astype(np.float32))
    p = params(m=9, k=k, iterations=3, rho=0.2, seed=n, beta=beta, logw_clip=80.0)
    o = orc.Oracle(inst, p).iterate(3)
    for kw in (dict(fallback_list=32), dict(fused=1, fallback_list=32), dict(fused=1, ants_per_warp=16, fallback_list=32)):
        with hac.Batch([inst], [p], hac.make_exec(**kw)) as bt:
            bt.run().sync()
            assert np.array_equal(bt.read(0, "TOURS"), o.get("tours")), kw
            assert np.array_equal(bt.read(0, "TAU"), o.get("tau")), kw
