"""The complex64 packet and the served pipeline built on it.

The packet kernel takes positions as whole numbers, the phase in fixed point and the envelope in FP32 pieces;
a CTA takes groups of rows that may straddle the BCC cosets.  Compared with the packet in 64 bits: one rounding
of the phase (within +-pi), one of the exponent, the functions and two complex products, each below 2.5e-7 of
the value, so 1e-6 of the norm (the tolerance of the packet elsewhere).
"""

import time

import numpy as np
import pytest

from paper_1603_06442_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHI = {1: [0.6, 0.8j], 2: [0.5, 0.5j, 0.5, -0.5j], 3: [0.6, 0.0, 0.0, 0.8j]}


@pytest.fixture(scope="module")
def qb(qwlib):
    from paper_1603_06442_gb300 import binding
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return binding


# lengths below a row of threads, odd, several tiles and groups; centres on and between sites, outside the box,
# and half a box from a site
@pytest.mark.parametrize("dim,N", [(1, 2), (1, 5), (1, 2048), (1, 100003), (2, 3), (2, 37), (2, 300), (3, 4),
                                   (3, 34), (3, 2 * 129)])
@pytest.mark.parametrize("where", [0.0, 0.5, 0.37, -1.25, 3.6])
def test_packet_against_64_bits(qb, dim, N, where):
    x0 = [where * N + 0.125 * j for j in range(dim)]
    sigma, k0 = max(0.7, N / 9), [0.45, -3.0, 1.7][:dim]
    want = inputs.gaussian_packet(dim, N, x0, sigma, k0, CHI[dim])
    with_plan = qb.Plan(dim, N, 0.1, "c64")
    x = torch.full((with_plan.elems,), float("nan"), dtype=torch.complex64, device="cuda")
    with_plan.prepare_packet(x, x0, sigma, k0, CHI[dim])
    got = x.cpu().numpy().reshape(want.shape).astype(np.complex128)
    got /= np.sqrt(np.sum(np.abs(got) ** 2))
    assert np.linalg.norm(got - want) < 1e-6


# Parameters outside the fixed-point range take the FP64 form: same values where both can be compared.
@pytest.mark.parametrize("k0,sigma", [(2.0e6, 20.0), (0.3, 5e-7)])
def test_packet_outside_the_fixed_point_range(qb, k0, sigma):
    N, x0 = 256, [100.0]
    want = inputs.gaussian_packet(1, N, x0, sigma, [k0], CHI[1])
    plan = qb.Plan(1, N, 0.1, "c64")
    x = torch.zeros(plan.elems, dtype=torch.complex64, device="cuda")
    plan.prepare_packet(x, x0, sigma, [k0], CHI[1])
    got = x.cpu().numpy().reshape(want.shape).astype(np.complex128)
    got /= np.sqrt(np.sum(np.abs(got) ** 2))
    assert np.linalg.norm(got - want) < 1e-6


# The weights summed while evolving (several rounds of the resident CTAs with a remainder) against the plan's own packet, evolution and observables; the tolerances are those
# of a served request against the oracle.
@pytest.mark.parametrize("dim,N", [(1, 3 ** 14), (2, 2187), (2, 288), (3, 2 * 81), (3, 2 * 54), (3, 2 * 216)])
@pytest.mark.parametrize("t", [0, 1, 4321])
def test_served_weights_against_plan(qb, dim, N, t):
    mass, x0, sigma, k0 = 0.21, [0.4 * N + 0.3] * dim, N / 16, [0.3, 0.1, -0.2][:dim]
    srv = qb.qw_server_create(2 << 30, slots=2, max_pending=8)
    tk = qb.qw_submit(srv, qb.make_request(dim, N, mass, t, x0=x0, sigma=sigma, k0=k0, chi=CHI[dim]))
    plan = qb.Plan(dim, N, mass, "c64")
    x = torch.zeros(plan.elems, dtype=torch.complex64, device="cuda")
    plan.prepare_packet(x, x0, sigma, k0, CHI[dim])
    plan.evolve_spectral(x, t)
    want = plan.observables(x)
    done, t0 = False, time.time()
    while not done:
        done, got, _ = qb.qw_poll(srv, tk)
        assert time.time() - t0 < 60
    qb.qw_server_destroy(srv)
    assert abs(got["norm"] - 1.0) < 2e-5
    for j in range(dim):
        assert abs(got["x_mean"][j] - want["x_mean"][j]) < 2e-5 * N
    assert abs(got["w_particle"] - want["w_particle"]) < 2e-5
    assert abs(got["w_antiparticle"] - want["w_antiparticle"]) < 2e-5
