"""Which kernels a run of qw_step is made of: single steps that take the TMA kernels (AUTO) or a thread per site, and
the instantiations of the marching kernels that only long chains and large boxes reach.  The marching, per-site and
FUSED kernels apply the same sums in the same order, so complex64 results are equal bit for bit; the TMA kernels round
differently, by less than 1.5e-7 of the norm a step.
"""

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


def field(dim, N, dtype="c64"):
    g = torch.Generator(device="cuda").manual_seed(1000 * dim + N)
    td = torch.complex64 if dtype == "c64" else torch.complex128
    return torch.randn(inputs.field_shape(dim, N), dtype=td, device="cuda", generator=g)


def rel(a, b):
    return float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))


@pytest.mark.parametrize("N", [384, 512])
@pytest.mark.parametrize("t", [1, 2, 3, 5, 7])
def test_auto_equals_plain_up_to_rounding(qb, N, t):
    plan = qb.Plan(3, N, 0.27, "c64")
    got, want = field(3, N), field(3, N)
    plan.step(got, t)
    plan.sync()
    plan.set_stencil("plain")
    plan.step(want, t)
    plan.close()
    assert rel(got, want) < 1.5e-7 * t


def test_auto_on_a_field_of_element_alignment_is_plain(qb):
    N = 384
    plan = qb.Plan(3, N, 0.27, "c64")
    buf = torch.empty(plan.elems + 1, dtype=torch.complex64, device="cuda")
    got, want = buf[1:].view(inputs.field_shape(3, N)), field(3, N)
    got.copy_(want)
    plan.step(got, 1)
    plan.set_stencil("plain")
    plan.step(want, 1)
    plan.close()
    assert torch.equal(got, want)


# chains of 16 sites a lane; boxes of one cell up to whole tiles per CTA; two steps on the square lattice
@pytest.mark.parametrize("dim,N,steps", [
    (1, 1_000_003, (150, 7, 1)), (1, 200_003, (150, 96)), (2, 1000, (2, 6)), (2, 2998, (1, 2, 3, 7)),
    (3, 2, (1, 3, 6, 13)), (3, 4, (2, 4, 10)), (3, 66, (1, 2, 5)), (3, 256, (1, 2, 3, 4)), (3, 300, (1, 5)), (3, 640, (3, 4))])
def test_c64_equals_fused_bit_for_bit(qb, dim, N, steps):
    plan = qb.Plan(dim, N, 0.27, "c64")
    for t in steps:
        got, want = field(dim, N), field(dim, N)
        plan.set_stencil("plain")
        plan.step(got, t)
        plan.set_stencil("fused")
        plan.step(want, t)
        assert torch.equal(got, want), t
    plan.close()


# chains of 4 and 8 sites a lane, boxes of both tiles and a thread per site
@pytest.mark.parametrize("dim,N,t", [(1, 100_003, 150), (1, 400_009, 64), (1, 1_000_003, 40), (1, 2_000_003, 3),
                                     (3, 48, 4), (3, 50, 3), (3, 66, 3), (3, 80, 5), (3, 112, 2), (3, 128, 4)])
def test_c128_equals_the_per_site_kernel_bit_for_bit(qb, dim, N, t):
    plan = qb.Plan(dim, N, 0.27, "c128")
    got, want = field(dim, N, "c128"), field(dim, N, "c128")
    plan.step(got, t)
    qb.qw_step_static(dim, N, 0.27, "c128", want, t)
    plan.close()
    assert torch.equal(got, want)


@pytest.mark.parametrize("dim,N,t", [(1, 3 ** 15, 5), (3, 384, 3), (3, 512, 3)])
def test_large_c128_runs_against_the_fourier_form(qb, dim, N, t):
    plan = qb.Plan(dim, N, 0.27, "c128")
    got, want = field(dim, N, "c128"), field(dim, N, "c128")
    plan.step(got, t)
    plan.evolve_spectral(want, t)
    plan.close()
    assert rel(got, want) < 1e-11
