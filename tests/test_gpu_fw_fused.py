"""The Foldy-Wouthuysen transform inside the fused x pass (complex64, 2D and BCC): lengths that are no power of two,
degenerate masses, in place, against the complex128 transform (held to 1e-11 of the oracle elsewhere).

The transforms' rounding is 1.8e-7 to 3.0e-7 of the norm at these sizes.  The coefficients add little to it:
1 - |vW| and 1 - vD come from wa^2 / r^2 and m^2 / den^2, so a small mass costs no digits (as differences they made
3.6e-7 to 4.4e-7 at m = 0.05).
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


@pytest.mark.parametrize("dim,N", [(2, 64), (2, 81), (2, 243), (2, 512), (3, 128), (3, 144), (3, 162), (3, 256), (3, 288)])
@pytest.mark.parametrize("m", [0.0, 0.05, 0.3, 1.0])
def test_fused_fw_against_complex128(qb, dim, N, m):
    g = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn(inputs.field_shape(dim, N), dtype=torch.complex64, device="cuda", generator=g)
    plan = qb.Plan(dim, N, m, "c64")
    got = plan.fw_transform(x)
    plan.fw_transform(x, out=x.clone())  # another output leaves the input as it is
    inplace = x.clone()
    plan.fw_transform(inplace, out=inplace)
    plan.close()
    assert torch.equal(inplace, got)
    plan = qb.Plan(dim, N, m, "c128")
    want = plan.fw_transform(x.to(torch.complex128))
    plan.close()
    err = float(torch.linalg.vector_norm(got - want) / torch.linalg.vector_norm(want))
    assert err < 3.5e-7, err
