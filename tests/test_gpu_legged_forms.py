"""Legged rollouts keep a step's vectors in registers or in shared memory, by link
count and by how many candidates there are: the same bits for each candidate in calls
of many candidates and of few, with shared models too."""
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
@pytest.mark.parametrize("links", [3, 5, 13, 14, 15, 16])
def test_same_bits_in_both_forms(mtp, links, dr):
    H, few = 7, 9000
    B = 256 * torch.cuda.get_device_properties(0).multi_processor_count + 77  # just past the line, a ragged last warp
    spec = W.legged(links=links, B=B, H=H, E=1, interp="akima")
    spec.update(dr_mode=dr, R=2 if dr == "shared" else 1)
    gen = torch.Generator(device=DEV).manual_seed(links)
    U = 5.0 * (2.0 * torch.rand(B, H, links - 1, generator=gen, device=DEV) - 1.0)
    U[::5] *= 1e9  # some diverge
    x0 = torch.tensor(np.linspace(-0.1, 0.1, 2 * (links + 2)), dtype=torch.float32, device=DEV)
    h = mtp.mtp_create(spec)
    many, parts = torch.empty(B, device=DEV), torch.empty(B, device=DEV)
    mtp.mtp_rollout_cost(h, 3, x0, U, many)
    for r in range(0, B, few):
        n = min(few, B - r)
        mtp.mtp_rollout_cost(h, 3, x0, U[r:r + n].contiguous(), parts[r:r + n], r, n)
    assert torch.equal(many, parts)
    mtp.mtp_destroy(h)
