"""Point masses of a batch whose rows are not whole 16-byte pieces (H n not a
multiple of 4) are loaded directly, the next steps while the current ones' costs
are evaluated: a step takes about what it takes for rows that are staged (copied
into shared memory float by float it took 1.2 to 1.7 times as long).  Times of the
rollout launches alone, the best of several averages; 10 % covers one step in 100
and the noise of launches of 30 us."""
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


def _times(mtp, k, H):
    specs = [W.pointmass(seed=i, k=k, B=600, H=H, E=8, M=4, degree=2) for i in range(2)]
    hs = [mtp.mtp_create(s) for s in specs]
    b = mtp.mtp_batch_create(hs)
    mtp.mtp_batch_plan_step(b, torch.zeros(b.x0_offset[-1], device=DEV), 1, torch.empty(b.ustar_offset[-1], device=DEV))
    groups = min(sum(g["ms"] for g in mtp.mtp_batch_rollout_times(b, 20)) for _ in range(5))
    mtp.mtp_batch_set_rollout_mode(b, mtp.BATCH_ROLLOUT_PERSISTENT_STAGED)
    persistent = min(mtp.mtp_batch_persistent_time(b, 20)[0] for _ in range(5))
    mtp.mtp_batch_destroy(b)
    for h in hs:
        mtp.mtp_destroy(h)
    return groups, persistent


@pytest.mark.parametrize("k", [5, 7, 9])
def test_rows_that_cannot_be_staged(mtp, k):
    for odd, whole in zip(_times(mtp, k, 101), _times(mtp, k, 100)):
        assert odd < 1.1 * whole
