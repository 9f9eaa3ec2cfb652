"""Performance cases of the quantum-walk library: what its users have it do, through its public binding.

A case is one call (or the short sequence of calls that belong together) on fields that live on the GPU: stencil
steps, the Fourier evolution, the observables of a snapshot, the readout of a particle state, a batch of uneven
walks, a burst of served requests.  ``listed`` gives the fixed cases and ``draw`` more of the same ranges.  Inputs
are random-phase Gaussian packets (width N/16, |k0| <= 0.5) with random spinors; ``exact`` evolves the same inputs
in 64 bits with plain torch, in the Fourier form with the closed-form power of the walk's symbol.
"""

import math
import time

import numpy as np
import torch

from paper_1603_06442_gb300 import binding as qb


def listed():
    return [
        # the 1D run of a single packet in double precision, step by step: the smallest field, 512 short steps
        {"name": "chain_step_c128_1024", "kind": "step", "dim": 1, "N": 1024, "mass": 0.1, "dtype": "c128", "t": 512},
        # the same run in one Fourier evolution: the smallest call there is
        {"name": "chain_spectral_c128_1024", "kind": "spectral", "dim": 1, "N": 1024, "mass": 0.1, "dtype": "c128",
         "t": 512},
        # a long chain of odd length over the 150 steps of the 1D jitter run
        {"name": "chain_step_c64_20m", "kind": "step", "dim": 1, "N": 20_000_003, "mass": 0.15, "dtype": "c64", "t": 150},
        # a square lattice larger than L2 with a ragged side
        {"name": "square_step_c64_2998", "kind": "step", "dim": 2, "N": 2998, "mass": 0.1, "dtype": "c64", "t": 150},
        # the BCC jitter run: a field that stays in L2, a thousand steps
        {"name": "bcc_step_c64_128", "kind": "step", "dim": 3, "N": 128, "mass": 0.05, "dtype": "c64", "t": 1000},
        # a BCC box of a side that is no multiple of anything large (odd number of cells per axis)
        {"name": "bcc_step_c64_250", "kind": "step", "dim": 3, "N": 250, "mass": 0.3, "dtype": "c64", "t": 150},
        # the headline run: 100 steps of the largest box, then the observables of the snapshot
        {"name": "bcc_snapshot_c64_512", "kind": "snapshot", "dim": 3, "N": 512, "mass": 0.1, "dtype": "c64", "t": 100},
        # the double-precision reference run of the jitter box
        {"name": "bcc_step_c128_128", "kind": "step", "dim": 3, "N": 128, "mass": 0.05, "dtype": "c128", "t": 100},
        # the long-time run of the largest box in the Fourier form
        {"name": "bcc_spectral_c64_512", "kind": "spectral", "dim": 3, "N": 512, "mass": 0.1, "dtype": "c64",
         "t": 10_000},
        # reading a particle state: moments, projections, the Newton-Wigner field and its moments
        {"name": "bcc_readout_c64_288", "kind": "readout", "dim": 3, "N": 288, "mass": 0.3, "dtype": "c64"},
        # 256 uneven square-lattice and BCC walks in one launch (a fifth of the 100..5000 steps of the full mix)
        {"name": "batch_256", "kind": "batch", "walks": 256, "mix": 0, "t_lo": 20, "t_hi": 1000},
        # a burst of requests of every lattice and size, submitted at once and polled until all are done
        {"name": "served_48", "kind": "served", "requests": 48, "mix": 0, "sites_lo": 10_000, "sites_hi": 100_000_000},
    ]


_MAX_SITE_STEPS = {"c64": 2.0e9, "c128": 1.0e8}  # bounds on a drawn stencil run


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sites(dim, N):
    return N if dim == 1 else N * N if dim == 2 else N ** 3 // 4


def _smooth(v):
    """The size 2^a 3^b nearest to v (in log distance), at least 2."""
    best = 2
    for b in range(0, 18):
        for a in range(0, 28):
            c = 2 ** a * 3 ** b
            if 2 <= c <= 2 * v and abs(math.log(c / v)) < abs(math.log(best / v)):
                best = c
    return best


def draw(rng):
    what = rng.random()
    mass = round(rng.uniform(0.0, 0.5), 4)
    if what < 0.50:  # stencil runs and snapshots of any size
        dim = rng.choice([1, 2, 3])
        dtype = rng.choice(["c64", "c64", "c64", "c128"])
        kind = "snapshot" if rng.random() < 0.25 else "step"
        N = {1: lambda: _log_int(rng, 1000, 1 << 26), 2: lambda: _log_int(rng, 64, 8192),
             3: lambda: 2 * _log_int(rng, 16, 256)}[dim]()
        if dtype == "c128":  # the double-precision runs are the smaller ones
            N = {1: min(N, 1 << 22), 2: min(N, 2048), 3: min(N, 256)}[dim]
        most = _MAX_SITE_STEPS[dtype] / _sites(dim, N)
        return {"kind": kind, "dim": dim, "N": N, "mass": mass, "dtype": dtype,
                "t": max(1, int(min(_log_int(rng, 10, 1000), most)))}
    if what < 0.72:  # Fourier evolutions: axis lengths 2^a 3^b
        dim = rng.choice([1, 2, 3])
        dtype = rng.choice(["c64", "c64", "c128"])
        N = {1: lambda: _smooth(_log_int(rng, 1000, 1 << 26)), 2: lambda: _smooth(_log_int(rng, 64, 4096)),
             3: lambda: 2 * _smooth(_log_int(rng, 16, 256))}[dim]()
        if dtype == "c128":
            N = {1: min(N, 1 << 22), 2: min(N, 2048), 3: min(N, 256)}[dim]
        return {"kind": "spectral", "dim": dim, "N": N, "mass": mass, "dtype": dtype, "t": _log_int(rng, 10, 1_000_000)}
    if what < 0.82:
        dim = rng.choice([2, 3])
        N = _smooth(_log_int(rng, 64, 4096)) if dim == 2 else 2 * _smooth(_log_int(rng, 16, 192))
        return {"kind": "readout", "dim": dim, "N": N, "mass": mass, "dtype": "c64"}
    if what < 0.92:
        return {"kind": "batch", "walks": _log_int(rng, 16, 160), "mix": rng.randrange(1 << 20), "t_lo": 10,
                "t_hi": _log_int(rng, 50, 600)}
    return {"kind": "served", "requests": rng.randrange(8, 32), "mix": rng.randrange(1 << 20), "sites_lo": 10_000,
            "sites_hi": _log_int(rng, 1_000_000, 100_000_000)}


# ---------------------------------------------------------------- inputs


def _shape(dim, N):
    return (2, N) if dim == 1 else (4, N, N) if dim == 2 else (2, 4, N // 2, N // 2, N // 2)


def _packet(dim, N, x0, sigma, k0, chi, dtype):
    """Gaussian packet on the periodic box in the device layout (components planar, x fastest, BCC as two cosets)."""
    axis = torch.arange(N, dtype=torch.float64, device="cuda")

    def factor(pos, j):
        d = (pos - x0[j] + N / 2.0) % N - N / 2.0
        return torch.polar(torch.exp(-d * d / (4.0 * sigma * sigma)), k0[j] * d).to(dtype)

    spin = torch.tensor([complex(c) for c in chi], dtype=dtype, device="cuda")
    if dim == 1:
        return spin[:, None] * factor(axis, 0)
    if dim == 2:
        return spin[:, None, None] * (factor(axis, 1)[:, None] * factor(axis, 0))
    cosets = []
    for c in (0, 1):
        pos = 2.0 * axis[: N // 2] + c
        fx, fy, fz = (factor(pos, j) for j in range(3))
        cosets.append(spin[:, None, None, None] * (fz[:, None, None] * (fy[:, None] * fx)))
    return torch.stack(cosets)


def _spinor(g, dim):
    c = g.normal(size=2 if dim == 1 else 4) + 1j * g.normal(size=2 if dim == 1 else 4)
    return c / np.linalg.norm(c)


def _direction(g, dim):
    d = g.normal(size=dim)
    return d / np.linalg.norm(d)


def _field(dim, N, dtype, g, packets):
    """Normalised superposition of random-phase packets."""
    td = torch.complex64 if dtype == "c64" else torch.complex128
    psi = None
    chi = _spinor(g, dim)
    for _ in range(packets):
        x0 = g.uniform(0, N, size=dim)
        k0 = _direction(g, dim) * g.uniform(0.0, 0.5)
        part = _packet(dim, N, x0, N / 16.0, k0, chi * np.exp(2j * np.pi * g.uniform()), td)
        psi = part if psi is None else psi.add_(part)
    norm = torch.linalg.vector_norm(torch.view_as_real(psi).reshape(-1, 1 << 6 if psi.numel() % 32 == 0 else 2),
                                    dim=1).double().square().sum().sqrt()
    return psi.mul_((1.0 / norm).to(psi.real.dtype)).contiguous()


def _walks(case):
    """The batch's walks: square lattices of side 64..1024 and BCC boxes of side 32..128, log-uniform."""
    g = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["walks"]):
        if g.random() < 0.5:
            dim, N = 2, int(round(math.exp(g.uniform(math.log(64), math.log(1024)))))
        else:
            dim, N = 3, 2 * int(round(math.exp(g.uniform(math.log(32), math.log(128))) / 2))
        out.append((dim, N, float(g.uniform(0.0, 0.5)), int(g.integers(case["t_lo"], case["t_hi"] + 1))))
    return out


def _requests(case, seed):
    """The burst's requests: the sizes come from the case, the packets from the seed."""
    g = np.random.default_rng(case["mix"])
    p = np.random.default_rng(seed)
    out = []
    for _ in range(case["requests"]):
        dim = int(g.integers(1, 4))
        sites = math.exp(g.uniform(math.log(case["sites_lo"]), math.log(case["sites_hi"])))
        if dim == 1:
            N = _smooth(sites)
        elif dim == 2:
            N = _smooth(math.sqrt(sites))
        else:
            N = 2 * _smooth((sites / 2.0) ** (1.0 / 3.0))
        mass, t = float(g.uniform(0.0, 0.5)), int(round(math.exp(g.uniform(math.log(10), math.log(1e5)))))
        out.append({"dim": dim, "N": N, "mass": mass, "t": t, "x0": list(N * p.uniform(0.3, 0.7, size=dim)),
                    "sigma": N / 16.0, "k0": list(_direction(p, dim) * p.uniform(0.0, 0.5)), "chi": _spinor(p, dim)})
    return out


class _Server:
    def __init__(self, pool_bytes):
        self.handle = qb.qw_server_create(pool_bytes, slots=8, max_pending=4096)

    def __del__(self):
        if getattr(self, "handle", None):
            qb.qw_server_destroy(self.handle)
            self.handle = None


def prepare(case, seed):
    g = np.random.default_rng(seed)
    if case["kind"] == "batch":
        # one buffer holds every walk's field
        walks = _walks(case)
        elems = [math.prod(_shape(dim, N)) for dim, N, _, _ in walks]
        fields = torch.empty(sum(elems), dtype=torch.complex64, device="cuda")
        args, at = [], 0
        for (dim, N, mass, t), n in zip(walks, elems):
            own = fields[at: at + n]
            own.copy_(_field(dim, N, "c64", g, 1).reshape(-1))
            args.append((dim, N, mass, t, own))
            at += n
        return {"kind": "batch", "fields": fields, "batch": qb.Batch(args)}
    if case["kind"] == "served":
        return {"kind": "served", "server": _Server(16 << 30),
                "requests": [qb.make_request(**r) for r in _requests(case, seed)]}
    dim, N = case["dim"], case["N"]
    plan = qb.Plan(dim, N, case["mass"], case["dtype"])
    state = {"kind": case["kind"], "plan": plan, "psi": _field(dim, N, case["dtype"], g, 4), "t": case.get("t", 0)}
    if case["kind"] in ("spectral", "readout"):
        plan.prepare_spectral()
    return state


# ---------------------------------------------------------------- one pass


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].run()
        return state["fields"]
    if kind == "served":
        return _serve(state["server"].handle, state["requests"])
    plan, psi = state["plan"], state["psi"]
    if kind == "spectral":
        plan.evolve_spectral(psi, state["t"])
        return psi
    if kind == "readout":
        # projections onto the x axis and the (x, y) plane, the density's moments, the Newton-Wigner position
        moments = plan.position_moments(psi)
        out = {"line": plan.projection(psi, (0,)), "plane": plan.projection(psi, (0, 1)),
               "fw": plan.fw_transform(psi)}
        nw = plan.position_moments(out["fw"])
        for name, m in (("x", moments), ("nw", nw)):
            out[name + "_norm"] = m["norm"]
            out[name + "_mean"] = torch.tensor(m["mean"], dtype=torch.float32)
            out[name + "_cov"] = torch.tensor(m["cov"], dtype=torch.float32)
        return out
    plan.step(psi, state["t"])
    if kind == "snapshot":
        return {"psi": psi, **plan.observables(psi)}
    return psi


def _serve(server, requests):
    tickets = [qb.qw_submit(server, r) for r in requests]
    got, left = {}, list(tickets)
    while left:
        waiting = []
        for t in left:
            done, obs, _ = qb.qw_poll(server, t)
            if done:
                got[t] = obs
            else:
                waiting.append(t)
        left = waiting
        if left:
            time.sleep(0.0002)
    return _served_results([got[t] for t in tickets])


def _served_results(obs):
    # the fields are complex64: the results carry single precision
    return {k: torch.tensor([o[k] for o in obs], dtype=torch.float32)
            for k in ("norm", "x_mean", "w_particle", "w_antiparticle")}


# ---------------------------------------------------------------- the work of one pass


def _elem_bytes(case):
    return 8 if case.get("dtype", "c64") == "c64" else 16


def _field_bytes(dim, N, eb):
    return math.prod(_shape(dim, N)) * eb


# real operations of one site and step: the Weyl part factored into one addition per hop and component pair, and
# the coupling n W psi + i m psi (two products and one sum for each real number)
_STEP_FLOPS = {1: 12, 2: 64, 3: 64}


def _fft_flops(dim, N):
    shape = _shape(dim, N)
    vol = math.prod(shape[-dim:]) if dim != 3 else (N // 2) ** 3
    planes = math.prod(shape) // vol
    return planes * 5.0 * vol * math.log2(vol)


def work(case):
    eb = _elem_bytes(case)
    if case["kind"] == "batch":
        b = f = 0.0
        for dim, N, _, t in _walks(case):
            b += 2.0 * _field_bytes(dim, N, 8)
            f += float(_STEP_FLOPS[dim]) * _sites(dim, N) * t
        return {"bytes": b, "flops": f}
    if case["kind"] == "served":
        # the packet is built on the device, so nothing has to be read: one transform there and one back
        f = 0.0
        b = 0.0
        for r in _requests(case, 0):
            f += 2.0 * _fft_flops(r["dim"], r["N"]) + 60.0 * _sites(r["dim"], r["N"])
            b += _field_bytes(r["dim"], r["N"], 8)
        return {"bytes": b, "flops": f}
    dim, N = case["dim"], case["N"]
    fb, sites = _field_bytes(dim, N, eb), _sites(dim, N)
    if case["kind"] == "spectral":
        return {"bytes": 2.0 * fb, "flops": 2.0 * _fft_flops(dim, N) + 60.0 * sites}
    if case["kind"] == "readout":
        return {"bytes": 2.0 * fb + 8.0 * N + 8.0 * N * N, "flops": 2.0 * _fft_flops(dim, N) + 150.0 * sites}
    w = {"bytes": 2.0 * fb, "flops": float(_STEP_FLOPS[dim]) * sites * case["t"]}
    if case["kind"] == "snapshot":
        w["flops"] += _fft_flops(dim, N) + 60.0 * sites
    return w


# ---------------------------------------------------------------- the same in 64 bits, with plain torch


def _halves(dim, N, mass, psi):
    """The spectrum as a list of (components, u, (nx, ny, nz)) with u, n~ the Weyl walk's symbol (1D: the chain's)."""
    k = 2.0 * math.pi * torch.arange(N if dim < 3 else N // 2, dtype=torch.float64, device="cuda") / \
        (N if dim < 3 else N // 2)
    if dim == 1:
        return [(torch.fft.fft(psi, dim=1), torch.cos(k), (None, None, torch.sin(k)))]
    if dim == 2:
        kx, ky = 0.5 * (k[None, :] + k[:, None]), 0.5 * (k[None, :] - k[:, None])
        cx, cy, sx, sy = kx.cos(), ky.cos(), kx.sin(), ky.sin()
        return [(torch.fft.fft2(psi), cx * cy, (sx * cy, cx * sy, sx * sy))]
    spec = torch.fft.fftn(psi, dim=(2, 3, 4))
    a = _coset_phase(k)
    out = []
    for half in (0, 1):  # q = kappa/2, and the same with pi added to its x component
        c = torch.stack([(spec[0, i] + (1 - 2 * half) * a.conj() * spec[1, i]) * 0.5 for i in range(4)])
        qx, qy, qz = (0.5 * k + math.pi * half)[None, None, :], 0.5 * k[None, :, None], 0.5 * k[:, None, None]
        cx, cy, cz, sx, sy, sz = qx.cos(), qy.cos(), qz.cos(), qx.sin(), qy.sin(), qz.sin()
        out.append((c, cx * cy * cz + sx * sy * sz,
                    (sx * cy * cz - cx * sy * sz, cx * sy * cz + sx * cy * sz, cx * cy * sz - sx * sy * cz)))
    return out


def _coset_phase(k):
    return torch.polar(torch.ones((), dtype=torch.float64, device="cuda"),
                       0.5 * (k[:, None, None] + k[None, :, None] + k[None, None, :]))


def _back(dim, N, parts):
    """Components per half spectrum -> the field in position space."""
    if dim == 1:
        return torch.fft.ifft(parts[0], dim=1)
    if dim == 2:
        return torch.fft.ifft2(parts[0])
    a = _coset_phase(2.0 * math.pi * torch.arange(N // 2, dtype=torch.float64, device="cuda") / (N // 2))
    return torch.fft.ifftn(torch.stack([parts[0] + parts[1], a * (parts[0] - parts[1])]), dim=(2, 3, 4))


def _angle(dim, N, mass, u, nt):
    """cos and sin of omega, and omega, with n = sqrt(1 - m^2)."""
    n = math.sqrt(1.0 - mass * mass)
    r2 = sum(v * v for v in nt if v is not None)
    c, s = n * u, torch.sqrt(mass * mass + n * n * r2)
    return c, s, torch.atan2(s, c)


def _symbol_times(dim, mass, psi, u, nt):
    """D_k psi."""
    n, im = math.sqrt(1.0 - mass * mass), 1j * mass
    nx, ny, nz = nt
    if dim == 1:
        return torch.stack([n * torch.complex(u, -nz) * psi[0] + im * psi[1],
                            n * torch.complex(u, nz) * psi[1] + im * psi[0]])
    w00, w01, w10, w11 = torch.complex(u, -nz), torch.complex(-ny, -nx), torch.complex(ny, -nx), torch.complex(u, nz)
    return torch.stack([n * (w00 * psi[0] + w01 * psi[1]) + im * psi[2],
                        n * (w10 * psi[0] + w11 * psi[1]) + im * psi[3],
                        n * (w00.conj() * psi[2] + w10.conj() * psi[3]) + im * psi[0],
                        n * (w01.conj() * psi[2] + w11.conj() * psi[3]) + im * psi[1]])


def _evolved(dim, N, mass, psi, t):
    parts = []
    for c, u, nt in _halves(dim, N, mass, psi.to(torch.complex128)):
        co, si, om = _angle(dim, N, mass, u, nt)
        if dim == 1 and N <= 1 << 16:  # the phase of a small chain in extended precision
            x = np.arange(N).astype(np.longdouble) * (2 * np.arccos(np.longdouble(-1)) / N)
            m = np.longdouble(mass)
            n = np.sqrt(1 - m * m)
            ph = np.arctan2(np.sqrt(m * m + (n * np.sin(x)) ** 2), n * np.cos(x)) * t
            ct, st = (torch.from_numpy(f(ph).astype(np.float64)).cuda() for f in (np.cos, np.sin))
        else:
            ct, st = torch.cos(om * t), torch.sin(om * t)
        # D^t = cos(omega t) + sin(omega t) / sin(omega) (D - cos(omega))
        r = torch.where(si > 0, st / torch.where(si > 0, si, 1.0), 0.0)
        parts.append(ct * c + r * (_symbol_times(dim, mass, c, u, nt) - co * c))
    return _back(dim, N, parts)


def _moments(dim, N, psi):
    """Norm, mean and covariance of the density on the window [0, N)."""
    rho = psi.real.square().add_(psi.imag.square()).double()
    pos = torch.arange(N, dtype=torch.float64, device="cuda")
    if dim == 3:  # both cosets: marginal sums per axis and pair of axes
        parts = [(rho[c].sum(0), [2.0 * pos[: N // 2] + c] * 3) for c in (0, 1)]
    else:
        parts = [(rho.sum(0), [pos] * dim)]
    norm = float(sum(r.sum() for r, _ in parts))
    mean = [0.0] * 3
    for a in range(dim):
        mean[a] = float(sum((r.sum([d for d in range(dim) if d != dim - 1 - a]) if dim > 1 else r).mul(p[a]).sum()
                            for r, p in parts)) / norm
    cov = [[0.0] * 3 for _ in range(3)]
    for a in range(dim):
        for b in range(a, dim):
            s = 0.0
            for r, p in parts:
                m = r.sum([d for d in range(dim) if d not in (dim - 1 - a, dim - 1 - b)]) if dim > (1 if a == b else 2) \
                    else r
                if a == b:
                    s += float((m * (p[a] - mean[a]) ** 2).sum())
                else:  # axis b > a is the slower one
                    s += float((m * (p[b] - mean[b])[:, None] * (p[a] - mean[a])[None, :]).sum())
            cov[a][b] = cov[b][a] = s / norm
    return norm, mean, cov


def _weights(dim, N, mass, psi):
    tot = diff = 0.0
    for c, u, nt in _halves(dim, N, mass, psi.to(torch.complex128)):
        co, si, _ = _angle(dim, N, mass, u, nt)
        g = 1j * (_symbol_times(dim, mass, c, u, nt) - co * c)
        r = torch.where(si > 0, 1.0 / torch.where(si > 0, si, 1.0), 0.0)
        tot += float(c.abs().square().sum())
        diff += float(((c.conj() * g).real * r).sum())
    return 0.5 * (1 + diff / tot), 0.5 * (1 - diff / tot)


def _observables(dim, N, mass, psi):
    norm, mean, _ = _moments(dim, N, psi)
    wp, wm = _weights(dim, N, mass, psi)
    return {"norm": norm, "x_mean": mean, "w_particle": wp, "w_antiparticle": wm}


def _fw(dim, N, mass, psi):
    """The state on the eigenvectors of D_k (spin and energy sign (+,+), (+,-), (-,+), (-,-)), in position space."""
    n = math.sqrt(1.0 - mass * mass)
    parts = []
    for c, u, (nx, ny, nz) in _halves(dim, N, mass, psi.to(torch.complex128)):
        r = torch.sqrt(nx * nx + ny * ny + nz * nz)
        small = r < 1e-12
        vw = torch.where(small, 0.0, -nz / torch.where(small, 1.0, r)).clamp(-1, 1)
        w = torch.complex(ny, -nx)
        ep = torch.where(w.abs() > 1e-12, w * (-1j) / torch.where(w.abs() > 1e-12, w.abs(), 1.0), 1.0 + 0j)
        den = torch.sqrt(mass * mass + n * n * r * r)
        vd = torch.where(den > 1e-12, n * r / torch.where(den > 1e-12, den, 1.0), 0.0).clamp(-1, 1)
        out = []
        for s in (1, -1):
            for p in (1, -1):
                a, b = torch.sqrt(1 - p * vw), torch.sqrt(1 + p * vw)
                d, e = torch.sqrt(1 + s * p * vd), torch.sqrt(1 - s * p * vd)
                out.append(0.5 * (a * d * c[0] - p * b * d * ep.conj() * c[1] - s * a * e * c[2]
                                  + s * p * b * e * ep.conj() * c[3]))
        parts.append(torch.stack(out))
    return _back(dim, N, parts)


def _projections(dim, N, psi):
    """Density summed onto the x axis and onto the (x, y) plane of the physical grid."""
    rho = psi.real.double().square() + psi.imag.double().square()
    if dim == 2:
        rho = rho.sum(0)
        return rho.sum(0), rho
    line = torch.zeros(N, dtype=torch.float64, device="cuda")
    plane = torch.zeros(N, N, dtype=torch.float64, device="cuda")
    for c in (0, 1):
        m = rho[c].sum((0, 1))
        plane[c::2, c::2] = m
        line[c::2] = m.sum(0)
    return line, plane


def exact(case, seed):
    g = np.random.default_rng(seed)
    if case["kind"] == "batch":
        out = []
        for dim, N, mass, t in _walks(case):
            out.append(_evolved(dim, N, mass, _field(dim, N, "c64", g, 1), t).reshape(-1))
        return torch.cat(out)
    if case["kind"] == "served":
        obs = []
        for r in _requests(case, seed):
            psi = _packet(r["dim"], r["N"], r["x0"], r["sigma"], r["k0"], r["chi"], torch.complex128)
            psi /= torch.linalg.vector_norm(psi)
            psi = _evolved(r["dim"], r["N"], r["mass"], psi, r["t"])
            obs.append(_observables(r["dim"], r["N"], r["mass"], psi))
        return _served_results(obs)
    dim, N, mass = case["dim"], case["N"], case["mass"]
    psi = _field(dim, N, case["dtype"], g, 4)
    if case["kind"] == "readout":
        line, plane = _projections(dim, N, psi)
        fw = _fw(dim, N, mass, psi)
        out = {"line": line, "plane": plane, "fw": fw}
        for name, f in (("x", psi), ("nw", fw)):
            norm, mean, cov = _moments(dim, N, f.to(torch.complex128))
            out[name + "_norm"] = norm
            out[name + "_mean"] = torch.tensor(mean, dtype=torch.float64)
            out[name + "_cov"] = torch.tensor(cov, dtype=torch.float64)
        return out
    psi = _evolved(dim, N, mass, psi, case["t"])
    if case["kind"] == "snapshot":
        obs = _observables(dim, N, mass, psi)
        smooth = all(_smooth(v) == v for v in ([N] if dim < 3 else [N // 2]))
        if not smooth:  # the weights need the transform's axis lengths 2^a 3^b
            obs["w_particle"] = obs["w_antiparticle"] = None
        return {"psi": psi, **obs}
    return psi
