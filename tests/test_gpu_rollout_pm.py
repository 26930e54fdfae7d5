"""Point-mass rollouts at the edges of their tiles: axis counts 1..16 (padded
rows at 8 and 16, odd ones by single floats), horizons around the chunk of 64
steps and the turn of 2 or 4, candidate counts around a warp's, rows that do
not start on 16 bytes, no obstacles and all eight, shared models, plain sums.
Costs against the FP64 oracle at the stated FP32 target (1e-4 relative, which
the oracle tests of the other rollouts hold); the batched rollouts (a lane per
candidate) bitwise against the lone ones (a warp per tile of candidates)."""
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


CASES = [
    # k, B, H, obstacles, extra
    (1, 1, 1, 0, {}),
    (1, 33, 65, 8, dict(dr_mode="per_sample", dr_lo=0.8, dr_hi=1.2)),
    (2, 5, 3, 5, {}),
    (2, 1900, 64, 5, {}),
    (2, 7400, 63, 1, {}),
    (3, 31, 33, 4, {}),
    (4, 100, 130, 8, dict(dr_mode="shared", R=3, dr_lo=0.9, dr_hi=1.1)),
    (5, 64, 37, 3, dict(flags=0x1)),
    (7, 2000, 20, 2, {}),
    (8, 130, 129, 5, dict(dr_mode="per_sample", dr_lo=0.8, dr_hi=1.2)),
    (9, 65, 31, 7, {}),
    (12, 1000, 66, 5, {}),
    (15, 40, 17, 5, {}),
    (16, 1900, 64, 8, dict(dr_mode="per_sample", dr_lo=0.8, dr_hi=1.2)),
]


def _spec(k, B, H, n_obs, extra):
    return W.pointmass(seed=k + H, k=k, B=B, H=H, E=1, M=4, N=8, degree=2, n_obstacles=n_obs, w_ctrl=0.01, **extra)


@pytest.mark.parametrize("k,B,H,n_obs,extra", CASES)
def test_costs_match_the_oracle(mtp, k, B, H, n_obs, extra):
    spec = _spec(k, B, H, n_obs, extra)
    h = mtp.mtp_create(spec)
    rng = np.random.default_rng(B + H)
    U = rng.uniform(-1.0, 1.0, size=(B, H, k)).astype(np.float32)
    x0 = rng.uniform(-0.2, 0.8, size=2 * k).astype(np.float32)
    cost = torch.full((B,), -1.0, device=DEV)
    Ud = torch.tensor(U, device=DEV)
    mtp.mtp_rollout_cost(h, 3, torch.tensor(x0, device=DEV), Ud, cost)
    ref = np.asarray(orc.rollout_costs(spec, 3, x0.astype(np.float64), U.astype(np.float64)))
    got = cost.cpu().numpy().astype(np.float64)
    assert (np.abs(got - ref) / np.maximum(np.abs(ref), 1.0)).max() < 1e-4
    # the same bits from rows that start 4 bytes past a 16-byte boundary, and from a part of the rows
    buf = torch.empty(U.size + 1, device=DEV)
    buf[1:] = Ud.reshape(-1)
    again = torch.empty(B, device=DEV)
    mtp.mtp_rollout_cost(h, 3, torch.tensor(x0, device=DEV), buf[1:].view(B, H, k), again)
    assert torch.equal(again, cost)
    row0 = B // 3
    part = torch.empty(B - row0, device=DEV)
    mtp.mtp_rollout_cost(h, 3, torch.tensor(x0, device=DEV), Ud[row0:].contiguous(), part, row0=row0)
    assert torch.equal(part, cost[row0:])
    mtp.mtp_destroy(h)


def test_batched_rollouts_are_the_lone_ones_bits(mtp):
    specs = [_spec(*c) for c in CASES]
    x0s = [np.random.default_rng(i).uniform(-0.2, 0.2, size=s["d"]).astype(np.float32) for i, s in enumerate(specs)]
    alone = []
    for s, x0 in zip(specs, x0s):
        h = mtp.mtp_create(s)
        u = torch.empty(s["n"], device=DEV)
        mtp.mtp_plan_step(h, torch.tensor(x0, device=DEV), 1, u)
        alone.append(torch.as_tensor(mtp.mtp_get_buffers(h)["cost"], device=DEV).clone())
        mtp.mtp_destroy(h)
    for mode in (mtp.BATCH_ROLLOUT_GROUPS, mtp.BATCH_ROLLOUT_PERSISTENT_STAGED, mtp.BATCH_ROLLOUT_PERSISTENT_DIRECT):
        hs = [mtp.mtp_create(s) for s in specs]
        b = mtp.mtp_batch_create(hs)
        mtp.mtp_batch_set_rollout_mode(b, mode)
        us = torch.empty(b.ustar_offset[-1], device=DEV)
        mtp.mtp_batch_plan_step(b, torch.tensor(np.concatenate(x0s), device=DEV), 1, us)
        for h, c, s in zip(hs, alone, specs):
            assert torch.equal(torch.as_tensor(mtp.mtp_get_buffers(h)["cost"], device=DEV), c), (mode, s["n"], s["H"])
        mtp.mtp_batch_destroy(b)
        for h in hs:
            mtp.mtp_destroy(h)
