"""Lone chain rollouts of so many candidates that their angles' whole turns are taken
on the SFU: the bits that the same rows give in calls of few candidates, which take
them off it, for chains that diverge past 2^22 turns too."""
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


@pytest.mark.parametrize("dr", ["per_sample", "shared"])
@pytest.mark.parametrize("links", [1, 2, 3, 6, 7, 9, 12])
def test_same_bits_as_few_at_a_time(mtp, links, dr):
    H, few = 11, 3000
    B = 192 * torch.cuda.get_device_properties(0).multi_processor_count + 77  # just past the line, a ragged last warp
    spec = W.chain(links=links, B=B, H=H, E=1, tau_max=40.0, dt=0.05)
    spec.update(dr_mode=dr, R=2 if dr == "shared" else 1)
    gen = torch.Generator(device=DEV).manual_seed(links)
    U = 40.0 * (2.0 * torch.rand(B, H, links, generator=gen, device=DEV) - 1.0)
    U[::5] *= 1e7  # their angles leave the range where a float holds whole turns
    x0 = torch.tensor(np.linspace(-0.5, 0.5, 2 * links), dtype=torch.float32, device=DEV)
    h = mtp.mtp_create(spec)
    many, parts = torch.empty(B, device=DEV), torch.empty(B, device=DEV)
    mtp.mtp_rollout_cost(h, 3, x0, U, many)
    for r in range(0, B, few):
        n = min(few, B - r)
        mtp.mtp_rollout_cost(h, 3, x0, U[r:r + n].contiguous(), parts[r:r + n], r, n)
    assert torch.equal(many, parts)
    mtp.mtp_destroy(h)
