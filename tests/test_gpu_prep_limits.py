"""The preparation at the limits of its paths, bit for bit against the CPU
oracle: squared distances at the end of the FP32 range."""
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
