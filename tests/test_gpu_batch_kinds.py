"""Which batches march (several steps per round in registers) and that marching launches keep a batch's contract:
odd and even round counts, a second run, and a bounded wait that gives up."""

import pytest

from paper_1603_06442_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qb(qwlib):
    from paper_1603_06442_gb300 import binding
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return binding


def field(dim, N):
    g = torch.Generator(device="cuda").manual_seed(1000 * dim + N)
    return torch.randn(inputs.field_shape(dim, N), dtype=torch.complex64, device="cuda", generator=g)


# work items: tiles of 2048 sites (whole rows) times a round per step, and the copy round of an odd count
@pytest.mark.parametrize("dim,N,t,tiles", [
    (3, 128, 50, 4 * 64), (3, 64, 61, 1 * 32), (2, 256, 50, 256 // 8), (2, 1024, 3, 512), (3, 320, 1, 27 * 160),
    (1, 10_000_000, 40, 4883)])
def test_small_and_short_batches_update_per_site(qb, dim, N, t, tiles):
    x = torch.zeros(inputs.field_shape(dim, N), dtype=torch.complex64, device="cuda")
    batch = qb.Batch([(dim, N, 0.1, t, x)])
    items = batch.tiling()[1]
    batch.close()
    assert items == (t + t % 2) * tiles


# a large walk makes the batch march; the small ones end their marching rounds at odd and even counts
WALKS = [(3, 256, 0.1, 48), (3, 66, 0.2, 10), (3, 26, 0.3, 9), (3, 8, 0.25, 5), (3, 42, 0.1, 1), (2, 130, 0.4, 11),
         (2, 61, 0.3, 8), (2, 300, 0.2, 5), (2, 9, 0.1, 4), (1, 301, 0.2, 7), (2, 64, 0.1, 0)]


def test_marching_rounds_of_two_runs_equal_steps(qb):
    fields = [field(d, N) for d, N, m, t in WALKS]
    batch = qb.Batch([(d, N, m, t, x) for (d, N, m, t), x in zip(WALKS, fields)])
    assert batch.tiling()[1] < 48 * 16 * 128  # the per-site rounds of the first walk alone
    for _ in range(2):
        batch.run()
    batch.sync()
    batch.close()
    for (d, N, m, t), got in zip(WALKS, fields):
        plan = qb.Plan(d, N, m, "c64")
        plan.set_stencil("plain")
        want = field(d, N)
        for _ in range(2):
            plan.step(want, t)
        plan.close()
        assert torch.equal(got, want), (d, N, t)


def test_stalled_marching_tile_times_out_and_the_batch_recovers(qb):
    fields = [field(d, N) for d, N, m, t in WALKS]
    batch = qb.Batch([(d, N, m, t, x) for (d, N, m, t), x in zip(WALKS, fields)])
    batch.debug_stall(1, spin_limit=4096)
    batch.run()
    with pytest.raises(qb.QwError) as error:
        batch.sync()
    assert error.value.status == qb.QW_ETIMEOUT
    batch.debug_stall(-1)
    for (d, N, m, t), x in zip(WALKS, fields):
        x.copy_(field(d, N))
    batch.run()
    batch.sync()
    batch.close()
    for (d, N, m, t), got in zip(WALKS, fields):
        plan = qb.Plan(d, N, m, "c64")
        plan.set_stencil("plain")
        want = field(d, N)
        plan.step(want, t)
        plan.close()
        assert torch.equal(got, want), (d, N, t)
