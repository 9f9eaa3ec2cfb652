"""The plan autotuner times runs of many steps, and choices recorded for other kernels are not applied."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qb(qwlib):
    from paper_1603_06442_gb300 import binding
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return binding


def rate(plan, x, t):
    plan.step(x, t)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = 0.0
    for _ in range(5):
        a.record()
        plan.step(x, t)
        b.record()
        b.synchronize()
        best = max(best, plan.sites * t / (a.elapsed_time(b) * 1e-3))
    return best


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


def test_a_long_chain_keeps_its_kernel_and_rate(qb):
    plan = qb.Plan(1, 20_000_003, 0.2, "c64")
    tuned = plan.autotune()
    assert plan.stencil == qb.STENCILS["plain"]
    x = torch.zeros(plan.elems, dtype=torch.complex64, device="cuda")
    assert tuned > 0.7 * rate(plan, x, 150)  # a run of 8 steps reaches half of it
    plan.close()
