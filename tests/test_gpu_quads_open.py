"""Every number of ants per warp that the per-step kernels take when it is left
open (csrc/host.h: as few as keep 8 warps on each of 152 SMs), bit for bit against
the CPU oracle."""
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


@pytest.mark.parametrize("m", [30, 60, 91, 121, 152, 182, 212, 243])   # 1 to 8 ants per warp, the last warp not full
def test_ants_per_warp(hac, orc, m):
    ins = [synth.euclid_instance(7, 45, K=12)] * 40
    ps = [synth.Params(m=m, k=20, iterations=2, rho=0.2, seed=b % 2) for b in range(40)]
    ref = [orc.Oracle(ins[0], ps[b]).iterate(2) for b in range(2)]
    with hac.Batch(ins, ps, hac.make_exec(fallback_list=32)) as bt:
        bt.run().sync()
        for b in (0, 1, 20, 39):
            assert np.array_equal(bt.read(b, "TOURS"), ref[b % 2].get("tours"))
            assert np.array_equal(bt.read(b, "TAU"), ref[b % 2].get("tau"))
