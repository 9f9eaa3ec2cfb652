"""The marching stencil kernels behind PLAIN (several steps per launch, the steps between held in
registers) at the sizes where their windows and tiles end: chains around the lengths of a window,
boxes around the tiles' widths, heights and chunks, and step counts that leave every remainder.

They apply the per-site update in the same order, so complex64 fields equal FUSED's (box tiles in
shared memory) bit for bit; complex128 has one per-site kernel, qw_step_static's.
"""

import numpy as np
import pytest

from oracle import walk
from paper_1603_06442_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qb(qwlib):
    from paper_1603_06442_gb300 import binding
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return binding


def field(dim, N, dtype):
    g = torch.Generator(device="cuda").manual_seed(1000 * dim + N)
    td = torch.complex64 if dtype == "c64" else torch.complex128
    return torch.randn(inputs.field_shape(dim, N), dtype=td, device="cuda", generator=g)


SIZES = [(1, n) for n in (2, 3, 31, 33, 63, 65, 127, 480, 481, 513, 1023, 20011)] + \
        [(2, n) for n in (2, 3, 27, 28, 29, 56, 57, 61, 64, 65, 130, 301)] + \
        [(3, n) for n in (2, 4, 18, 20, 26, 40, 42, 56, 58, 64, 66, 96, 130, 250)]


@pytest.mark.parametrize("dim,N", SIZES)
def test_c64_equals_fused_bit_for_bit(qb, dim, N):
    plan = qb.Plan(dim, N, 0.27, "c64")
    for t in (1, 2, 3, 4, 5, 9, 14, 67):
        got, want = field(dim, N, "c64"), field(dim, N, "c64")
        plan.set_stencil("plain")
        plan.step(got, t)
        plan.set_stencil("fused")
        plan.step(want, t)
        assert torch.equal(got, want), t
    plan.close()


@pytest.mark.parametrize("dim,N", [(d, n) for d, n in SIZES if n < 250 or d == 1])
def test_c128_equals_the_per_site_kernel_bit_for_bit(qb, dim, N):
    plan = qb.Plan(dim, N, 0.27, "c128")
    for t in (1, 2, 5, 14, 67):
        got, want = field(dim, N, "c128"), field(dim, N, "c128")
        plan.step(got, t)
        qb.qw_step_static(dim, N, 0.27, "c128", want, t)
        assert torch.equal(got, want), t
    plan.close()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("dim,N", [(1, 97), (2, 31), (3, 44)])
def test_marching_matches_the_oracle(qb, dtype, dim, N):
    m, t = 0.31, 23
    a = inputs.random_field(dim, N, seed=N)
    x = torch.from_numpy(np.ascontiguousarray(a.astype(np.complex64 if dtype == "c64" else np.complex128))).cuda()
    plan = qb.Plan(dim, N, m, dtype)
    plan.step(x, t)
    plan.close()
    exp = walk.to_device(dim, N, walk.step(dim, m, walk.from_device(dim, N, a), t))
    err = np.linalg.norm(x.cpu().numpy() - exp) / np.linalg.norm(exp)
    assert err <= (1e-5 if dtype == "c64" else 1e-11)


def test_batch_rounds_equal_plain_bit_for_bit(qb):
    """A batch's default rounds (marching tiles of every walk in one launch): walks around the tiles'
    sizes, step counts with every remainder."""
    spec = [(d, N, 0.05 * (i % 9), 5 + i) for i, (d, N) in enumerate(SIZES) if d > 1] + [(1, 300, 0.2, 9)]
    fields = [field(d, N, "c64") for d, N, m, t in spec]
    batch = qb.Batch([(d, N, m, t, x) for (d, N, m, t), x in zip(spec, fields)])
    batch.run()
    batch.sync()
    batch.close()
    for (d, N, m, t), got in zip(spec, fields):
        plan = qb.Plan(d, N, m, "c64")
        want = field(d, N, "c64")
        plan.step(want, t)
        plan.close()
        assert torch.equal(got, want), (d, N, t)
