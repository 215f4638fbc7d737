"""One ant per lane quad (csrc/ant_quad.cuh) at the sizes where it can go wrong,
bit for bit against the CPU oracle: tours shorter than, equal to and just past
the 16-step window, visited masks at word boundaries, every number of slot
groups (one or two per lane, the split fifth group, lanes without a group),
warps whose quads are not all taken, and every count of ants per warp."""
import numpy as np
import pytest

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


def _batch():
    ins, ps = [], []
    for n in (3, 15, 16, 17, 31, 32, 33, 48, 64, 65, 97):
        for k, m in ((1, 3), (4, 8), (9, 9), (13, 1), (17, 7), (20, 17), (21, 5), (29, 8), (32, 11)):
            s = 100 * n + k
            ins.append(synth.euclid_instance(s, n, K=min(n - 1, 12)))
            ps.append(synth.Params(m=m, k=k, iterations=3, rho=0.2, seed=s))
    return ins, ps


@pytest.fixture(scope="module")
def expected(orc):
    ins, ps = _batch()
    return [orc.Oracle(i, p).iterate(p.iterations) for i, p in zip(ins, ps)]


@pytest.mark.parametrize("cfg", [dict(), dict(fallback_list=32), dict(ants_per_warp=2, fallback_list=32, warps_per_block=3),
                                 dict(ants_per_warp=4), dict(fused=1, fallback_list=32), dict(fused=1),
                                 dict(fused=1, fallback_list=32, cluster_log2=1), dict(fused=1, ants_per_warp=2, cluster_log2=2),
                                 dict(fused=1, ants_per_warp=4, fallback_list=32)],
                         ids=lambda c: "_".join(f"{k}{v}" for k, v in c.items()) or "default")
def test_edges(hac, expected, cfg):
    ins, ps = _batch()
    with hac.Batch(ins, ps, hac.make_exec(**cfg)) as bt:
        bt.run().sync()
        for b, o in enumerate(expected):
            what = (ins[b].n, ps[b].k, ps[b].m)
            assert np.array_equal(bt.read(b, "TOURS"), o.get("tours")), what
            assert np.array_equal(bt.read(b, "LENS"), o.get("lens")), what
            assert np.array_equal(bt.read(b, "TAU"), o.get("tau")), what
            assert bt.scalars(b)["n_fallback"] == o.ints()["n_fallback"], what


@pytest.mark.parametrize("m", [64, 250, 1000])
def test_ants_per_warp_left_open(hac, orc, m):
    # 40 instances: the per-step kernels take 3, 8 and 8 (capped) ants per warp
    ins = [synth.euclid_instance(7, 40, K=12)] * 40
    ps = [synth.Params(m=m, k=20, iterations=2, rho=0.2, seed=b % 2) for b in range(40)]
    ref = [orc.Oracle(ins[0], ps[b]).iterate(2) for b in range(2)]
    with hac.Batch(ins, ps, hac.make_exec(fallback_list=32)) as bt:
        bt.run().sync()
        for b in (0, 1, 20, 39):
            assert np.array_equal(bt.read(b, "TOURS"), ref[b % 2].get("tours"))
