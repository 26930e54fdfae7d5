"""The tensor-core contraction's accumulator is read 16 steps at a time by two
groups of warps, each on one half of a 128-step slice.  Its reads are
asynchronous: a register of tcgen05.ld holds the value only after
tcgen05.wait::ld, so both are one statement of the source (checked as text; no
run can show that a compiler keeps two apart statements apart).  Graph rows
around the edges of a chunk, a half and a slice, and with several tiles per CTA,
against the oracle's BF16-operand mode at the other contraction tests' FP32
summation tolerance (2e-6 of the largest value)."""
import os
import re

import numpy as np
import pytest

import oracle as orc
from paper_2505_01059_gb300 import workloads as W

torch = pytest.importorskip("torch")
DEV = "cuda:0"
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_01059_gb300", "csrc")


def test_every_accumulator_read_is_awaited_in_its_statement():
    reads = 0
    for name in os.listdir(CSRC):
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for asm in re.findall(r"asm\s+volatile\s*\((.*?)\)\s*;", text, re.S):
            if "tcgen05.ld" in asm:
                reads += 1
                assert "tcgen05.wait::ld" in asm.split("tcgen05.ld", 1)[1], name
    assert reads > 0


@pytest.fixture(scope="module")
def mtp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_01059_gb300 import _build, mtp as m
    _build.build_library()
    m.load_library()
    torch.cuda.set_device(0)
    return m


@pytest.mark.gpu
@pytest.mark.parametrize("n,H,P", [(3, 1, 50), (3, 16, 50), (2, 17, 150), (6, 64, 50), (6, 65, 50), (4, 80, 33),
                                   (1, 128, 300), (5, 129, 70), (7, 192, 40), (15, 193, 30), (16, 255, 3000)])
def test_rows_at_the_edges_of_chunks_and_halves(mtp, n, H, P):
    spec = W.pointmass(k=n, M=9, N=8, H=H, B=P + 1, E=1, beta=1.0, degree=2,
                       u_min=[-2.0] * n, u_max=[3.0] * n, flags=0x4)
    h = mtp.mtp_create(spec)
    C = np.random.default_rng(H).uniform(-2.0, 3.0, size=(P, 9, n)).astype(np.float32)
    U = torch.full((P, H, n), float("nan"), device=DEV)
    mtp.mtp_interpolate(h, torch.tensor(C, device=DEV), U)
    ref = np.clip(orc.interpolate(spec, C.astype(np.float64)), -2.0, 3.0)
    assert np.abs(U.cpu().numpy().astype(np.float64) - ref).max() <= 2e-6 * np.abs(ref).max()
    mtp.mtp_destroy(h)
