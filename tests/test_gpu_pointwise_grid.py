"""The pointwise spectral kernels (D_k^t and the Foldy-Wouthuysen coefficients outside the fused x pass) take a grid
over rows where the rows fill their CTAs, else the box's positions in one row of CTAs: both forms at the sides where
one gives way to the other (7/8 of a multiple of the CTA), chains, and small boxes.  Tolerances as elsewhere for the
Fourier path: relative L2 1e-11 (complex128), 1e-5 (complex64).
"""

import numpy as np
import pytest

from oracle import observables, spectral, walk
from paper_1603_06442_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = {"c64": 1e-5, "c128": 1e-11}


@pytest.fixture(scope="module")
def qb(qwlib):
    from paper_1603_06442_gb300 import binding
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return binding


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("dim,N,dtype", [
    (1, 2, "c64"), (1, 128, "c128"), (1, 3 ** 8, "c64"), (1, 3 ** 8, "c128"),
    (2, 2, "c64"), (2, 54, "c64"), (2, 81, "c128"), (2, 108, "c128"), (2, 128, "c128"), (2, 144, "c128"),
    (2, 192, "c128"), (2, 216, "c128"), (2, 243, "c128"), (2, 486, "c64"),
    (3, 2, "c64"), (3, 2, "c128"), (3, 24, "c64"), (3, 54, "c128")])
def test_evolution_and_fw_against_the_oracle(qb, dim, N, dtype):
    m, t = 0.23, 6
    a = inputs.random_field(dim, N, seed=N + dim).astype(np.complex64 if dtype == "c64" else np.complex128)
    psi = walk.from_device(dim, N, a.astype(np.complex128))
    plan = qb.Plan(dim, N, m, dtype)
    x = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    fw = plan.fw_transform(x).cpu().numpy().astype(np.complex128)
    plan.evolve_spectral(x, t)
    got = x.cpu().numpy().astype(np.complex128)
    plan.close()
    assert rel_l2(got, walk.to_device(dim, N, spectral.evolve(dim, m, psi, t))) <= TOL[dtype]
    assert rel_l2(walk.from_device(dim, N, fw), observables.fw_field(dim, m, psi)) <= TOL[dtype]


def test_bcc_rows_against_steps(qb):
    """BCC rows of 243 cells (the smallest that fill a CTA of 256): the Fourier form against two steps."""
    N, t = 486, 2
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(inputs.field_shape(3, N), dtype=torch.complex128, device="cuda", generator=g)
    y = x.clone()
    plan = qb.Plan(3, N, 0.23, "c128")
    plan.evolve_spectral(x, t)
    plan.step(y, t)
    plan.close()
    assert float(torch.linalg.vector_norm(x - y) / torch.linalg.vector_norm(y)) <= TOL["c128"]
