"""The 3-opt's FP32 scan and its helper warps (csrc/threeopt.cuh), bit for bit
against the CPU oracle's FP64 search: gains that are exactly zero (lattice,
duplicate points), more pairs than lanes (long neighbour lists), lists that are
no multiple of four, middle rewrites long enough to be shared, and the search
of every ant's tour (one warp, no helpers)."""
import numpy as np
import pytest

from helpers import euclid
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


def _lattice(side, scale):
    return np.stack(np.meshgrid(np.arange(side), np.arange(side)), -1).reshape(-1, 2) * scale


CASES = {
    "n7": lambda: (synth.euclid_instance(1, 7, K=5), dict(ls_k=4)),
    "n900_k8": lambda: (synth.euclid_instance(2, 900, K=10), dict(ls_k=8)),
    "n700_k32": lambda: (synth.euclid_instance(3, 700, K=10, family="gmm"), dict(ls_k=32)),
    "n401_k5": lambda: (synth.euclid_instance(4, 401, K=10, family="grid"), dict(ls_k=5)),
    "lattice": lambda: (euclid(_lattice(20, 1.0 / 16)), dict(ls_k=11)),
    "duplicates": lambda: (euclid(np.repeat(np.random.default_rng(5).random((60, 2)), 3, axis=0)), dict(ls_k=17)),
    "large_scale": lambda: (euclid(np.random.default_rng(6).random((150, 2)) * 1e18), dict(ls_k=10)),
    "tiny_scale": lambda: (euclid(np.random.default_rng(7).random((150, 2)) * 1e-9), dict(ls_k=10)),
}


@pytest.mark.parametrize("mode", [3, 4])
@pytest.mark.parametrize("name", sorted(CASES))
def test_equals_oracle(hac, orc, name, mode):
    inst, kw = CASES[name]()
    p = synth.Params(m=5, k=10, iterations=2, rho=0.2, seed=9, local_search=mode, **kw)
    o = orc.Oracle(inst, p).iterate(p.iterations)
    for ex in (hac.make_exec(fallback_list=32), hac.make_exec(fused=1)):
        with hac.Batch([inst], [p], ex) as bt:
            bt.run().sync()
            assert np.array_equal(bt.read(0, "NN_TOUR"), o.get("nn_tour"))
            assert np.array_equal(bt.read(0, "IB_TOUR"), o.get("ib_tour"))
            assert np.array_equal(bt.read(0, "TOURS"), o.get("tours"))
            assert bt.scalars(0)["L_gb"] == o.scalars()["L_gb"]

