"""Candidates whose graph rows are contracted on the tensor cores beside the local
rows: the same bits whether the first call is eager or captured, on the caller's
own stream with the result read there at once, and local and mean rows equal to
those made by themselves."""
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


# one path; fewer tiles than SMs; a ragged last tile; more than two CTAs' tiles per SM
@pytest.mark.parametrize("n,H,B,beta", [(2, 64, 16, 0.1), (5, 200, 300, 0.5), (7, 33, 1001, 0.9), (15, 256, 6000, 0.6)])
def test_same_bits_eager_and_captured(mtp, n, H, B, beta):
    spec = W.pointmass(k=n, M=8, N=16, H=H, B=B, E=1, beta=beta, u_min=[-2.0] * n, u_max=[3.0] * n, flags=0x4)
    eager, captured = mtp.mtp_create(spec), mtp.mtp_create(spec)
    U = [torch.full((B, H, n), float("nan"), device=DEV) for _ in range(3)]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):  # the captured handle's first call
        mtp.mtp_generate_candidates(captured, 3, U[1], s.cuda_stream)
    with torch.cuda.stream(s):
        for _ in range(3):
            mtp.mtp_generate_candidates(eager, 3, U[0], s.cuda_stream)
            first = U[0].clone()
            U[0].fill_(float("nan"))
        g.replay()
        replayed = U[1].clone()
        mtp.mtp_sample_local(eager, 3, U[2], s.cuda_stream)
    s.synchronize()
    assert torch.isfinite(first).all()
    assert torch.equal(first, replayed)
    L = eager.sizes["L"]
    assert torch.equal(first[:L], U[2][:L]) and torch.equal(first[-1], U[2][-1])
    mtp.mtp_destroy(eager)
    mtp.mtp_destroy(captured)
