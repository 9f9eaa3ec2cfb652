"""Choices of the plan autotuner recorded for other kernels are not applied."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qb(qwlib):
    from paper_1603_06442_gb300 import binding
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return binding


def test_a_choice_recorded_for_other_kernels_is_measured_again(qb, tmp_path):
    path = tmp_path / "tune.txt"
    name = torch.cuda.get_device_name().replace(" ", "_")
    line = "plan %s dim=2 N=64 dtype=c64 | 5 4 64 16 1 123\n"  # a line without a generation: FUSED
    path.write_text(line + line.replace("dim=2", "kernels=1 dim=2"))
    qb.qw_set_autotune_cache(str(path))
    try:
        plan = qb.Plan(2, 64, 0.2, "c64")
        assert plan.autotune() != 123.0
        plan.close()
        assert len(path.read_text().splitlines()) == 3
    finally:
        qb.qw_set_autotune_cache(None)
