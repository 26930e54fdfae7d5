"""Batched updates on 16 and 8 lanes per element, the counts between a small
batch's 32 and a large one's 4: mean and spread are the bits that each instance
gets alone, with elite counts around a round of 32."""
import numpy as np
import pytest

from paper_2505_01059_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SHAPES = [(2, 33, 31), (3, 100, 32), (5, 50, 33), (12, 37, 65), (1, 1, 1), (4, 60, 130)]  # (axes, steps, elites)


@pytest.fixture(scope="module")
def mtp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_01059_gb300 import _build, mtp as m
    _build.build_library()
    m.load_library()
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("lanes", [16, 8])
@pytest.mark.parametrize("rule", ["softmax", "plain_cem"])
def test_batched_updates_are_each_instance_alone(mtp, lanes, rule):
    # the fewest copies whose elements reach 256 threads per SM with that many lanes
    elements = sum(k * H for k, H, _ in SHAPES)
    threads = 256 * torch.cuda.get_device_properties(0).multi_processor_count
    copies = -(-threads // (lanes * elements))
    assert copies * elements * lanes // 2 < threads <= copies * elements * lanes
    specs = [W.pointmass(seed=7 * c + i, k=k, H=H, B=200, E=E, M=4, N=8, degree=2, alpha=0.3, update_rule=rule)
             for c in range(copies) for i, (k, H, E) in enumerate(SHAPES)]
    x0 = torch.zeros(sum(s["d"] for s in specs), device=DEV)
    hs = [mtp.mtp_create(s) for s in specs]
    b = mtp.mtp_batch_create(hs)
    mtp.mtp_batch_plan_step(b, x0, 2, torch.empty(b.ustar_offset[-1], device=DEV))
    for s, h in zip(specs[:12], hs):
        twin = mtp.mtp_create(s)
        mtp.mtp_plan_step(twin, x0[:s["d"]], 2, torch.empty(s["n"], device=DEV))
        for got, want in zip(mtp.mtp_get_state(h), mtp.mtp_get_state(twin)):
            assert np.array_equal(got, want), (s["n"], s["H"], s["E"])
        mtp.mtp_destroy(twin)
    mtp.mtp_batch_destroy(b)
    for h in hs:
        mtp.mtp_destroy(h)
