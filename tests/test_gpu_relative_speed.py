"""Calls that must not fall behind another call on the same work: ratios of best-of-many device times, with bounds
between what the library reaches and what the faults named here cost."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qb(qwlib):
    from paper_1603_06442_gb300 import binding
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return binding


def best_ms(fn, calls=10, repeats=7):
    fn()
    best = float("inf")
    for _ in range(repeats):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(calls):
            fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / calls)
    return best


def test_overlapped_fp64_passes_do_not_crowd_sms(qb):
    """Half the chain takes 0.55 of the time; 0.84 where each launch's CTAs are placed while the one before runs."""
    ms = []
    for N in (1 << 17, 1 << 18):
        plan = qb.Plan(1, N, 0.1, "c128")
        x = torch.zeros(plan.elems, dtype=torch.complex128, device="cuda")
        plan.prepare_spectral()
        ms.append(best_ms(lambda: plan.evolve_spectral(x, 1000)))
        plan.close()
    assert ms[0] < 0.7 * ms[1], ms


def test_chains_of_a_batch_keep_their_threads(qb):
    """A batch's rounds update a long chain at the rate of the per-site kernel in launches of one step (1.5 of its
    time); 3.9 with a quarter of the threads per SM."""
    N, t = 4_000_000, 40
    x = torch.zeros((2, N), dtype=torch.complex64, device="cuda")
    batch = qb.Batch([(1, N, 0.1, t, x)])
    ms = best_ms(batch.run, 2)
    batch.sync()
    batch.close()
    assert ms < 2.5 * best_ms(lambda: qb.qw_step_static(1, N, 0.1, "c64", x, t), 2), ms


def test_a_single_step_of_a_large_box_is_as_fast_as_the_tma_kernel(qb):
    """1.27 of its time with the marching kernel's single step (a copy of the field included in both)."""
    plan = qb.Plan(3, 512, 0.1, "c64")
    x = torch.zeros(plan.elems, dtype=torch.complex64, device="cuda")
    ms = best_ms(lambda: plan.step(x, 1), 5)
    plan.set_stencil("tma")
    want = best_ms(lambda: plan.step(x, 1), 5)
    plan.close()
    assert ms < 1.1 * want, (ms, want)


def test_small_complex128_boxes_step_as_fast_as_a_thread_per_site(qb):
    """1.77 of its time with the marching kernel."""
    plan = qb.Plan(3, 48, 0.1, "c128")
    x = torch.zeros(plan.elems, dtype=torch.complex128, device="cuda")
    ms = best_ms(lambda: plan.step(x, 20))
    plan.close()
    want = best_ms(lambda: qb.qw_step_static(3, 48, 0.1, "c128", x, 20))
    assert ms < 1.2 * want, (ms, want)


def test_two_steps_of_a_complex128_chain_are_as_fast_as_a_thread_per_site(qb):
    """1.36 of its time where one launch of two steps and a copy of the field take the place of two launches."""
    N = 500_000
    plan = qb.Plan(1, N, 0.1, "c128")
    x = torch.zeros(plan.elems, dtype=torch.complex128, device="cuda")
    ms = best_ms(lambda: plan.step(x, 2))
    plan.close()
    want = best_ms(lambda: qb.qw_step_static(1, N, 0.1, "c128", x, 2))
    assert ms < 1.15 * want, (ms, want)
