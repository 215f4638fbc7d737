"""The block-wide 2-opt and 3-opt of T_NN and T_ib where their arrays do not all fit
in shared memory.  A launch's shared memory follows from its batch's largest
instance (220 KB hold every array of n = 10727, all but the coordinates of
n = 17329), so a larger companion moves the arrays of an instance beside it to
global memory: the small ones equal the CPU oracle, the larger one equals the
same instance decoded alone, bit for bit."""
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


def _companion(n):
    inst = synth.Instance(n=n, kind=0, coords=np.random.default_rng(n).random((n, 2)).astype(np.float32), cost=None,
                          rowptr=np.zeros(n + 1, np.int32), col=np.zeros(0, np.int32), val=np.zeros(0, np.float32), symmetrize=1)
    return inst, synth.Params(m=1, k=4, iterations=1, rho=0.2, seed=1)


FIELDS = (("NN_TOUR", "nn_tour"), ("IB_TOUR", "ib_tour"), ("GB_TOUR", "gb_tour"))


@pytest.mark.parametrize("mode", [1, 3])
def test_every_array_in_global_memory(hac, orc, mode):
    big, pbig = _companion(17330)
    ins, ps = [big], [pbig]
    for n, k in ((7, 4), (200, 10), (901, 8), (1500, 17)):
        ins.append(synth.euclid_instance(n, n, K=min(n - 1, 10), family="gmm" if n == 901 else "uniform"))
        ps.append(synth.Params(m=4, k=min(n - 1, 10), iterations=2, rho=0.2, seed=n, local_search=mode, ls_k=k))
    with hac.Batch(ins, ps, hac.make_exec(fallback_list=32)) as bt:
        bt.run().sync()
        for b in range(1, len(ins)):
            o = orc.Oracle(ins[b], ps[b]).iterate(2)
            for f, of in FIELDS:
                assert np.array_equal(bt.read(b, f), o.get(of)), (ins[b].n, f)


@pytest.mark.parametrize("mode", [1, 3])
def test_coordinates_in_global_memory(hac, mode):
    # 13 bytes a node of the companion are fewer than the 21 of this instance
    big, pbig = _companion(10728)
    inst = synth.euclid_instance(8000, 8000, K=8)
    p = synth.Params(m=4, k=8, iterations=2, rho=0.2, seed=8, local_search=mode, ls_k=8)
    got = []
    for ins, ps in (([inst], [p]), ([big, inst], [pbig, p])):
        with hac.Batch(ins, ps, hac.make_exec(fallback_list=32)) as bt:
            bt.run().sync()
            got.append([bt.read(len(ins) - 1, f) for f, _ in FIELDS] + [bt.scalars(len(ins) - 1)["L_gb"]])
    for x, y in zip(*got):
        assert np.array_equal(x, y)
