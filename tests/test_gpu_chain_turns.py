"""A link angle's whole turns come from rintf or from an addition off the SFU,
whichever is faster for the link count: the same bits from both, for chains that
diverge past 2^22 turns too (lone chains of five links take one, batches the
other), and the short chains are not slower than longer ones' share.  Times of
rollout launches, the best of several: one link does less than half of two links'
work, five links less than six."""
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


def test_same_bits_past_2_to_the_22_turns(mtp):
    # torques and a start far beyond what the step length takes: some candidates diverge
    specs = [W.chain(seed=s, links=5, H=60, B=500, E=8, M=4, N=8, tau_max=40.0, dt=0.02) for s in range(3)]
    x0 = np.zeros(10, np.float32)
    x0[:5] = [3e6, -2e7, 5e7, 1.0, -0.5]
    x0[5:] = 30.0
    hs = [mtp.mtp_create(s) for s in specs]
    b = mtp.mtp_batch_create(hs)
    mtp.mtp_batch_plan_step(b, torch.tensor(np.tile(x0, 3), device=DEV), 1, torch.empty(15, device=DEV))
    for s, h in zip(specs, hs):
        twin = mtp.mtp_create(s)
        mtp.mtp_plan_step(twin, torch.tensor(x0, device=DEV), 1, torch.empty(5, device=DEV))
        got, want = (torch.as_tensor(mtp.mtp_get_buffers(q)["cost"], device=DEV) for q in (h, twin))
        assert torch.equal(got, want)
        mtp.mtp_destroy(twin)
    mtp.mtp_batch_destroy(b)
    for h in hs:
        mtp.mtp_destroy(h)


def _batch_time(mtp, links):
    hs = [mtp.mtp_create(W.chain(seed=i, links=links, H=101, B=600, E=8, M=4)) for i in range(2)]
    b = mtp.mtp_batch_create(hs)
    mtp.mtp_batch_plan_step(b, torch.zeros(b.x0_offset[-1], device=DEV), 1, torch.empty(b.ustar_offset[-1], device=DEV))
    ms = min(mtp.mtp_batch_rollout_times(b, 20)[0]["ms"] for _ in range(5))
    mtp.mtp_batch_destroy(b)
    for h in hs:
        mtp.mtp_destroy(h)
    return ms


def _lone_time(mtp, links):
    spec = W.chain(links=links, H=128, B=2048, E=1)
    h = mtp.mtp_create(spec)
    U = torch.zeros(2048, 128, links, device=DEV)
    x0 = torch.zeros(2 * links, device=DEV)
    cost = torch.empty(2048, device=DEV)
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    mtp.mtp_rollout_cost(h, 2, x0, U, cost)
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        for _ in range(20):
            mtp.mtp_rollout_cost(h, 2, x0, U, cost, stream=s.cuda_stream)
    times = []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    mtp.mtp_destroy(h)
    return min(times[1:])


def test_one_link_in_a_batch(mtp):
    assert _batch_time(mtp, 1) < 0.6 * _batch_time(mtp, 2)


def test_five_links_alone(mtp):
    assert _lone_time(mtp, 5) < 0.9 * _lone_time(mtp, 6)
