"""Chain rollouts with staged controls at the edges of their chunks of 8 (4 from
9 links on) steps: horizons below, at and past a chunk, candidate counts around a
warp's, shared models (each model stages the rows again), and rows that cannot be
staged (H n not a multiple of 4, unaligned).  Costs against the FP64 oracle at the
stated FP32 target (1e-4 relative); staged and direct loads give the same bits."""
import numpy as np
import pytest

import oracle as orc
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


CASES = [(1, 33, 4, {}), (2, 31, 10, {}), (3, 100, 8, {}), (3, 65, 36, dict(dr_mode="shared", R=3)), (3, 40, 33, {}),
         (10, 64, 6, {}), (12, 35, 17, {}), (7, 14700, 12, {})]


@pytest.mark.parametrize("links,B,H,extra", CASES)
def test_lone_rollouts(mtp, links, B, H, extra):
    spec = W.chain(seed=links, links=links, B=B, H=H, E=1, M=4, N=8, **extra)
    h = mtp.mtp_create(spec)
    rng = np.random.default_rng(B + H)
    U = rng.uniform(-2.0, 2.0, size=(B, H, links)).astype(np.float32)
    x0 = rng.uniform(-0.2, 0.2, size=2 * links).astype(np.float32)
    cost = torch.empty(B, device=DEV)
    mtp.mtp_rollout_cost(h, 2, torch.tensor(x0, device=DEV), torch.tensor(U, device=DEV), cost)
    rows = min(B, 512)  # the oracle's share of the large case
    ref = np.asarray(orc.rollout_costs(spec, 2, x0.astype(np.float64), U[:rows].astype(np.float64)))
    got = cost.cpu().numpy().astype(np.float64)
    assert (np.abs(got[:rows] - ref) / np.maximum(np.abs(ref), 1.0)).max() < 1e-4
    # rows that start 4 bytes past a 16-byte boundary are loaded directly
    buf = torch.empty(U.size + 1, device=DEV)
    buf[1:] = torch.tensor(U, device=DEV).reshape(-1)
    direct = torch.empty(B, device=DEV)
    mtp.mtp_rollout_cost(h, 2, torch.tensor(x0, device=DEV), buf[1:].view(B, H, links), direct)
    assert torch.equal(direct, cost)
    mtp.mtp_destroy(h)


def test_batched_rollouts_are_the_lone_ones_bits(mtp):
    shapes = [(1, 33, 4), (3, 100, 8), (5, 70, 20), (8, 40, 33), (8, 40, 12), (9, 33, 9), (9, 64, 8)]
    specs = [W.chain(seed=i, links=k, B=B, H=H, E=1, M=4, N=8, **(dict(dr_mode="shared", R=2) if i == 2 else {}))
             for i, (k, B, H) in enumerate(shapes)]
    alone = []
    for s in specs:
        h = mtp.mtp_create(s)
        mtp.mtp_plan_step(h, torch.zeros(s["d"], device=DEV), 1, torch.empty(s["n"], device=DEV))
        alone.append(torch.as_tensor(mtp.mtp_get_buffers(h)["cost"], device=DEV).clone())
        mtp.mtp_destroy(h)
    for mode in (mtp.BATCH_ROLLOUT_GROUPS, mtp.BATCH_ROLLOUT_PERSISTENT_STAGED, mtp.BATCH_ROLLOUT_PERSISTENT_DIRECT):
        hs = [mtp.mtp_create(s) for s in specs]
        b = mtp.mtp_batch_create(hs)
        mtp.mtp_batch_set_rollout_mode(b, mode)
        x0 = torch.zeros(b.x0_offset[-1], device=DEV)
        mtp.mtp_batch_plan_step(b, x0, 1, torch.empty(b.ustar_offset[-1], device=DEV))
        for h, c, s in zip(hs, alone, specs):
            assert torch.equal(torch.as_tensor(mtp.mtp_get_buffers(h)["cost"], device=DEV), c), (mode, s["n"], s["H"])
        mtp.mtp_batch_destroy(b)
        for h in hs:
            mtp.mtp_destroy(h)
