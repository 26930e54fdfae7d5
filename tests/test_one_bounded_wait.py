"""The wait that the self-test makes run out is the one that the tensor-core
contraction waits with: the sources hold one bounded mbarrier wait, and both
call it."""
import pathlib

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2505_01059_gb300" / "csrc"


def test_the_contraction_and_the_self_test_share_one_bounded_wait():
    text = {p.name: p.read_text() for p in sorted(CSRC.iterdir()) if p.suffix in (".cu", ".cuh")}
    assert [n for n, s in text.items() for _ in range(s.count("mbarrier.try_wait"))] == ["mtp_device.cuh"]
    assert {n for n, s in text.items() if "mbar_wait_bounded(&" in s} == {"bspline_tc.cu", "selftest.cu"}
