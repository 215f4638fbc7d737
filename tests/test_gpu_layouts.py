"""Layouts of the cluster kernel beyond one SM per instance, bit for bit against
the CPU oracle: instances whose many ants are spread over a cluster, the ants
per warp that follow from it, blocks narrower than an SM, and groups with and
without local search."""
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


def _check(hac, orc, ins, ps, ex):
    ref = {}
    with hac.Batch(ins, ps, ex) as bt:
        bt.run().sync()
        for b, (i, p) in enumerate(zip(ins, ps)):
            key = (i.seed, p.seed)
            if key not in ref:
                ref[key] = orc.Oracle(i, p).iterate(p.iterations)
            o = ref[key]
            for f, of in (("TOURS", "tours"), ("LENS", "lens"), ("TAU", "tau"), ("GB_TOUR", "gb_tour")):
                assert np.array_equal(bt.read(b, f), o.get(of)), (b, f)
            assert bt.scalars(b)["n_fallback"] == o.ints()["n_fallback"], b


def _instances(n, m, count, iterations=3, k=20, **kw):
    ins = [synth.euclid_instance(n, n, K=min(n - 1, 12))] * count
    return ins, [synth.Params(m=m, k=k, iterations=iterations, rho=0.2, seed=b % 2, **kw) for b in range(count)]


@pytest.mark.parametrize("n,m,count", [
    (40, 65, 1), (97, 127, 15), (65, 128, 16), (333, 100, 36), (64, 300, 37), (40, 1000, 2), (33, 66, 76), (40, 65, 77),
])
def test_many_ants(hac, orc, n, m, count):
    _check(hac, orc, *_instances(n, m, count), hac.make_exec(fused=1, fallback_list=32))


@pytest.mark.parametrize("clog,m,count", [(1, 16, 3), (1, 30, 160), (2, 33, 80), (3, 9, 40), (3, 64, 16), (3, 5, 130)])
def test_clusters(hac, orc, clog, m, count):
    _check(hac, orc, *_instances(70, m, count, k=29), hac.make_exec(fused=1, fallback_list=32, cluster_log2=clog))


@pytest.mark.parametrize("apw", [0, 2, 4, 16, 32])
@pytest.mark.parametrize("clog", [0, 1])
def test_groups_with_and_without_local_search(hac, orc, apw, clog):
    ins, ps = _instances(90, 20, 4)
    ins2, ps2 = _instances(61, 9, 4, local_search=1, ls_k=8)
    _check(hac, orc, ins + ins2, ps + ps2, hac.make_exec(apw, fused=1, fallback_list=32, cluster_log2=clog))
