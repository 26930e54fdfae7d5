"""Which point masses prepare their next candidates beside the selection: at the
edges of the rule (Akima up to 3 axes, else up to 2^21 candidate elements), the same
results with and without the preparation."""
import numpy as np
import pytest

from paper_2505_01059_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def mtp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_01059_gb300 import _build, mtp as m
    _build.build_library()
    m.load_library()
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("spec,mode", [
    (W.pointmass(k=3, B=300, H=33, interp="akima", M=6), 2),
    (W.pointmass(k=4, B=300, H=33, interp="akima", M=6), 0),
    (W.pointmass(k=8, B=2048, H=128), 2),  # 2^21 elements
    (W.pointmass(k=8, B=2049, H=128), 0),
])
def test_rule(mtp, spec, mode):
    outs = []
    for flags in (0, mtp.FLAG_NO_PIPELINE):
        h = mtp.mtp_create(dict(spec, flags=flags))
        assert h.sizes["pipelined"] == (0 if flags else mode)
        u = torch.empty(spec["n"], device=DEV)
        x0 = torch.tensor(spec["x0"], dtype=torch.float32, device=DEV)
        for iters in (1, 3):
            mtp.mtp_plan_step(h, x0, iters, u)
        torch.cuda.synchronize()
        mu, sg, it = mtp.mtp_get_state(h)
        outs.append((mu, sg, it, u.cpu().numpy()))
        mtp.mtp_destroy(h)
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
