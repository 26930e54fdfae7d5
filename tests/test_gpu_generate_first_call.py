"""The first mtp_generate_candidates of a handle whose graph rows go to the tensor
cores makes no side stream (it may be the only call): it takes no longer than that
of a handle which has its stream, from a capture, already.  First calls of new
handles, in turn, by the host's clock; a stream and its events take 10 us or more."""
import time

import pytest

from paper_2505_01059_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
HANDLES = 40  # of each kind


@pytest.fixture(scope="module")
def mtp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_01059_gb300 import _build, mtp as m
    _build.build_library()
    m.load_library()
    torch.cuda.set_device(0)
    return m


def test_a_first_call_makes_no_stream(mtp):
    B, H, n = 300, 24, 5
    U = torch.empty(B, H, n, device=DEV)
    s = torch.cuda.Stream()
    took = {False: [], True: []}
    for i in range(2 * HANDLES):
        h = mtp.mtp_create(W.pointmass(seed=i, k=n, M=8, N=16, H=H, B=B, E=1, flags=0x4))
        has_stream = i % 2 == 1
        if has_stream:
            with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=s):
                mtp.mtp_generate_candidates(h, 3, U, s.cuda_stream)
        torch.cuda.synchronize()
        t = time.perf_counter()
        mtp.mtp_generate_candidates(h, 3, U, s.cuda_stream)
        s.synchronize()
        took[has_stream].append(time.perf_counter() - t)
        mtp.mtp_destroy(h)
    median = {k: sorted(v)[len(v) // 2] for k, v in took.items()}
    assert median[False] < median[True] + 6e-6, median
