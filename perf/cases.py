"""Performance cases: the work a user of this library has it do.

Kinds of case (one pass = one ``run``):

  step       advance a device-resident ensemble by a few time steps and fetch
             the spectral state (what a run does between two snapshots)
  host       one step of an ensemble whose state lives in host memory
             (``ens_step_host``), state in and state out
  stats      one statistics snapshot of every member (gradient invariants,
             histograms, moments) and its counts and moments on the host
  mixture    lambda mixture of gathered member statistics (FP64)
  quadrature mixture of the learned interpolant over a fine lambda quadrature
  gradient   loss and gradient of the interpolant on the members' histograms

Sizes come from the workloads of ``ens_inputs.py`` and ``bench.py``: one
32^3 member (RK2, fixed step), 16 x 64^3, the uneven 128^3 / 256^3 / 384^3
batch, the 64 x 256^3 benchmark ensemble and the single 512^3 member.
Initial fields are seeded solenoidal random fields with a turbulence-like
spectrum whose dissipation equals the member's injection rate, so the
gradients fill the histogram ranges as in a running simulation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2506_23712_gb300 import ens as E

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
_STEP = {"kind": "step", "nu": 0.0, "band_lo": 6.0, "band_hi": 8.0, "lam_lo": -2.0, "lam_hi": 2.0, "rk": 3,
         "dt": -1.0, "stored_tuning": False}
_STATS = {"kind": "stats", "nu": 0.0, "lam_lo": -2.0, "lam_hi": 2.0, "qr_bins": 64, "tail_bins": 256, "grad_bins": 0}


def listed():
    return [
        # the smallest run: one 32^3 member, RK2, fixed step (latency and launches)
        dict(_STEP, name="step_1x32", sizes="32x1", steps=10, nu=0.02, band_lo=1.0, band_hi=2.0, lam_lo=0.0,
             lam_hi=0.0, rk=2, dt=0.01),
        # a small ensemble between two snapshots of a long run (every 10 steps)
        dict(_STEP, name="step_16x64", sizes="64x16", steps=10, nu=0.01, band_lo=3.0, band_hi=5.0, lam_lo=-3.0,
             lam_hi=3.0),
        # the 128^3 members of the uneven batch on their own
        dict(_STEP, name="step_24x128", sizes="128x24", steps=3),
        # a quarter of the uneven batch: three grid sizes in one ensemble
        dict(_STEP, name="step_uneven", sizes="128x6,256x3,384x1", steps=3),
        # the benchmark ensemble, launch variants as a stored autotuning has them
        dict(_STEP, name="step_64x256", sizes="256x64", steps=2, nu=0.005, lam_lo=-5.1, lam_hi=5.8,
             stored_tuning=True),
        # the single large reference run
        dict(_STEP, name="step_1x512", sizes="512x1", steps=2, nu=0.0015, band_lo=1.0, band_hi=2.0, lam_lo=0.0,
             lam_hi=0.0),
        # state in host memory, streamed through the device once per step
        dict(_STEP, kind="host", name="host_16x256", sizes="256x16", steps=1, nu=0.005, lam_lo=-5.1, lam_hi=5.8),
        # statistics snapshots: the long small-ensemble run and the benchmark ensemble
        dict(_STATS, name="stats_16x64", sizes="64x16", nu=0.01, lam_lo=-3.0, lam_hi=3.0, grad_bins=128),
        dict(_STATS, name="stats_64x256", sizes="256x64", nu=0.005, lam_lo=-5.1, lam_hi=5.8),
        # one prediction from the members' statistics
        {"kind": "mixture", "name": "mixture_64", "members": 64, "qr_bins": 64, "tail_bins": 256, "grad_bins": 0},
        # the learned interpolant: a fine quadrature, and one training step's gradient
        {"kind": "quadrature", "name": "quadrature_512", "points": 512, "qr_bins": 64, "tail_bins": 256},
        {"kind": "gradient", "name": "gradient_64", "members": 64, "qr_bins": 64, "tail_bins": 256},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# most members of a grid size in a drawn case (at most half the listed 64 x 256^3)
_MOST = {16: 64, 32: 64, 64: 64, 128: 48, 256: 24, 384: 6, 512: 2}


def draw(rng):
    kind = rng.choice(["step", "step", "step", "host", "stats", "stats", "mixture", "quadrature", "gradient"])
    if kind in ("step", "host", "stats"):
        n1 = rng.choice([16, 32, 64, 64, 128, 128, 256, 256, 384, 512])
        sizes = [(n1, _log_int(rng, 1, _MOST[n1]))]
        if kind != "host" and rng.random() < 0.3:   # a second grid size
            n2 = rng.choice([n for n in _MOST if n != n1 and n <= 256])
            sizes.append((n2, _log_int(rng, 1, max(1, _MOST[n2] // 2))))
        text = ",".join("%dx%d" % s for s in sorted(sizes))
        small = max(n for n, _ in sizes) <= 64
        spread = rng.uniform(0.5, 3.0)
        lams = {"lam_lo": round(-spread, 2), "lam_hi": round(spread, 2)}
        if kind == "stats":
            return dict(_STATS, sizes=text, qr_bins=rng.choice([31, 48, 64, 100]),
                        tail_bins=_log_int(rng, 65, 512), grad_bins=rng.choice([0, 0, 77, 128]), **lams)
        lo = min(n for n, _ in sizes)
        band = (1.0, 2.0) if lo <= 32 else (3.0, 5.0) if lo <= 64 else (6.0, 8.0)
        steps = 1 if kind == "host" else rng.choice([5, 10]) if small else rng.choice([1, 2])
        return dict(_STEP, kind=kind, sizes=text, steps=steps, band_lo=band[0], band_hi=band[1],
                    rk=rng.choice([2, 3, 3]), dt=rng.choice([-1.0, -1.0, 0.005]) if small else -1.0, **lams)
    bins = {"qr_bins": rng.choice([24, 33, 48, 64, 90]), "tail_bins": _log_int(rng, 48, 512)}
    if kind == "mixture":
        return dict(kind=kind, members=_log_int(rng, 3, 256), grad_bins=rng.choice([0, 0, 101]), **bins)
    if kind == "quadrature":
        return dict(kind=kind, points=_log_int(rng, 16, 512), **bins)
    return dict(kind=kind, members=_log_int(rng, 4, 64), **bins)


# ---------------------------------------------------------------------------
# members and fields
# ---------------------------------------------------------------------------
EPS_BAR = 0.1


def _sizes(case):
    return [tuple(int(v) for v in part.split("x")) for part in case["sizes"].split(",")]


def _members(case):
    """Member parameters, ascending grid size (the order of the state buffer)."""
    out = []
    for N, n in sorted(_sizes(case)):
        for lam in (np.linspace(case["lam_lo"], case["lam_hi"], n) if n > 1 else [0.5 * (case["lam_lo"] + case["lam_hi"])]):
            eps = EPS_BAR * math.exp(float(lam))
            # given viscosity, or k_max eta = 1.5 for every member
            nu = case["nu"] or (1.5 / (N / 3.0)) ** (4.0 / 3.0) * eps ** (1.0 / 3.0)
            k_hi = min(case.get("band_hi", 2.0), (N + 2) // 3 - 1)
            out.append(E.Member(N=N, nu=nu, lam=float(lam), eps_bar=EPS_BAR, k_lo=min(case.get("band_lo", 1.0), k_hi),
                                k_hi=k_hi, dt=case.get("dt", -1.0), cfl=0.2, dt_max=0.01 if N <= 64 else 0.0,
                                rk_order=case.get("rk", 3), seed=len(out), init_energy=0.5))
    return out


def _dims(N):
    kc = (N + 2) // 3 - 1
    return kc, 2 * kc + 1, kc + 1, (kc + 1 + 15) // 16 * 16


def _wave(N, dtype):
    """Integer wave numbers of the kept modes: kx [NK,1,1], ky [1,NK,1], kz [1,1,NZ], and kept row indices."""
    kc, NK, NZ, _ = _dims(N)
    k = torch.cat([torch.arange(0, kc + 1, device="cuda"), torch.arange(-kc, 0, device="cuda")])
    kz = torch.arange(NZ, device="cuda")
    return k.to(dtype).view(-1, 1, 1), k.to(dtype).view(1, -1, 1), kz.to(dtype).view(1, 1, -1), k % N


def _fields(members, seed):
    """Seeded FP32 states in the library's compact layout, one float tensor of
    the whole ensemble: per member [3][kx NK][ky NK][kz NZp] complex.  Random
    solenoidal fields, spectrum k^4 / (k^2 + k_f^2)^(17/6) exp(-5.2 k eta),
    scaled so that the dissipation equals the injection rate."""
    parts = []
    gen = torch.Generator(device="cuda")
    for i, m in enumerate(members):
        gen.manual_seed(1_000_003 * (seed % 1_000_003) + i)
        kc, NK, NZ, NZp = _dims(m.N)
        kx, ky, kz, rows = _wave(m.N, torch.float32)
        noise = torch.randn(3, m.N, m.N, m.N, generator=gen, device="cuda")
        u = torch.fft.rfftn(noise, dim=(1, 2, 3))[:, :, :, :NZ]
        del noise
        u = u[:, rows][:, :, rows]
        k2 = kx * kx + ky * ky + kz * kz
        k2[0, 0, 0] = 1.0
        u -= torch.stack([kx.expand_as(k2), ky.expand_as(k2), kz.expand_as(k2)]) * \
            ((kx * u[0] + ky * u[1] + kz * u[2]) / k2)
        eps = m.eps_bar * math.exp(m.lam)
        eta = (m.nu ** 3 / eps) ** 0.25
        k = k2.sqrt()
        amp2 = k2 / (k2 + m.k_hi ** 2) ** (17.0 / 6.0) * torch.exp(-5.2 * eta * k)   # E(k) / k^2
        u *= amp2.sqrt()
        u[:, 0, 0, 0] = 0
        wgt = torch.full((NZ,), 2.0, device="cuda")
        wgt[0] = 1.0
        diss = m.nu * float((k2 * wgt * (u.real.square() + u.imag.square()).sum(0)).sum(dtype=torch.float64))
        u *= math.sqrt(eps / diss)
        full = torch.zeros(3, NK, NK, NZp, dtype=torch.complex64, device="cuda")
        full[..., :NZ] = u
        parts.append(torch.view_as_real(full).reshape(-1))
    return torch.cat(parts)


def _hist(case, members):
    return E.hist_spec(qr_bins=case["qr_bins"], tail_bins=case["tail_bins"], eps_norm=EPS_BAR, nu_norm=members[0].nu,
                       grad_bins=case["grad_bins"])


def _pinned(n):
    return torch.empty(n, dtype=torch.float32, pin_memory=True)


def _prepare_ensemble(case, seed):
    members = _members(case)
    ens = E.Ensemble(members, hist=_hist(case, members) if case["kind"] == "stats" else None)
    if case.get("stored_tuning"):
        t = ens.tuning()
        for g in t["groups"]:
            if g["N"] == 256:
                g.update(tile_x=16, tile_y=16, plan_x=0, z_variant=2, z_ctas_per_sm=1, fx_split=1)
        ens.set_tuning(t)
    host = _pinned(ens.state_bytes() // 4)
    host.copy_(_fields(members, seed))
    if case["kind"] == "host":
        return {"case": case, "ens": ens, "in": host, "out": _pinned(host.numel())}
    E.ens_set_state(ens.ctx, host.data_ptr(), ens.state_bytes())
    ens.synchronize()
    return {"case": case, "ens": ens, "out": host}


# ---------------------------------------------------------------------------
# histograms and network parameters
# ---------------------------------------------------------------------------
def _counts(case, seed):
    """Member statistics with a smooth lambda dependence (Poisson counts of
    model densities): lambdas, counts in the library's layout, moments."""
    rng = np.random.Generator(np.random.Philox(key=seed))
    n, nq, nt, ng = case["members"], case["qr_bins"], case["tail_bins"], case.get("grad_bins", 0)
    lams = np.sort(np.clip(2.0 * rng.standard_normal(n), -5.1, 5.8))
    npoints = 256 ** 3
    c = (np.arange(nq) + 0.5) / nq * 2 - 1
    Q, R = np.meshgrid(c, c, indexing="ij")
    x = (np.arange(nt) + 0.5) / nt * 2 - 1
    g = (np.arange(ng) + 0.5) / max(ng, 1) * 2 - 1
    counts = np.zeros((n, nq * nq + 2 * nt + 8 + (2 * ng + 4 if ng else 0)), dtype=np.uint64)
    moments = np.zeros((n, 48))
    for i, lam in enumerate(lams):
        s = 0.25 * math.exp(lam / 8.0)
        ps = [np.exp(-(Q ** 2 + (R - 0.2 * Q) ** 2) / (2 * s * s)) * (1 + 0.3 * np.tanh(3 * (R + Q))),
              np.exp(-(x + 0.2 - 0.08 * lam) ** 2 / (2 * (0.15 * math.exp(lam / 10)) ** 2)),
              np.exp(-(x + 0.1 - 0.1 * lam) ** 2 / (2 * (0.18 * math.exp(lam / 10)) ** 2))]
        counts[i, :nq * nq + 2 * nt] = rng.poisson(np.concatenate([(p / p.sum()).ravel() for p in ps]) * npoints)
        off = nq * nq + 2 * nt
        counts[i, off + 6] = npoints
        for q in range(2 if ng else 0):
            p = np.exp(-g ** 2 / (2 * (0.1 * math.exp(lam / 6) * (1 + 0.4 * q)) ** 2))
            counts[i, off + 8 + q * ng:off + 8 + (q + 1) * ng] = rng.poisson(p / p.sum() * npoints * (3, 6)[q])
        sig2 = math.exp(2 * lam / 3)
        comp = np.array([1.0, 0.0, 3.5, 30.0])
        for a in range(9):
            lon = a % 4 == 0
            scale = sig2 * (1.0 if lon else 2.0) * (1 + 0.01 * rng.standard_normal(4))
            comp[1] = -0.5 if lon else 0.01 * rng.standard_normal()
            moments[i, 4 * a:4 * a + 4] = npoints * comp * scale ** np.array([1.0, 1.5, 2.0, 3.0])
        moments[i, 36:44] = npoints * sig2 * np.abs(rng.standard_normal(8))
    return lams, counts, moments


_HID, _IN, _FEAT = 256, 64, 31


def _params(seed):
    """He-uniform parameters in the surrogate's order W1 b1 W2 b2 W3 b3 w4 b4."""
    rng = np.random.Generator(np.random.Philox(key=seed + 17))

    def u(shape, scale):
        return (scale * (2.0 * rng.random(shape) - 1.0)).astype(np.float32).ravel()
    h = math.sqrt(6.0 / _HID)
    return np.concatenate([u((_HID, _IN), math.sqrt(6.0 / _FEAT)), u(_HID, 0.05), u((_HID, _HID), h), u(_HID, 0.05),
                           u((_HID, _HID), h), u(_HID, 0.05), u(_HID, math.sqrt(3.0 / _HID)), u(1, 0.05)])


_LAM_LO, _LAM_HI, _C, _Z = -5.1, 5.8, 0.023, 3.0   # quadrature range; scaling parameter and scale gap


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "host", "stats"):
        return _prepare_ensemble(case, seed)
    hist = E.hist_spec(qr_bins=case["qr_bins"], tail_bins=case["tail_bins"], eps_norm=EPS_BAR, nu_norm=0.005,
                       grad_bins=case.get("grad_bins", 0))
    state = {"case": case, "hist": hist}
    if kind in ("quadrature", "gradient"):
        state["net"] = E.Surrogate(seed=0)
        state["net"].set_params(_params(seed))
    if kind in ("mixture", "gradient"):
        state["lams"], state["counts"], state["moments"] = _counts(case, seed)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        state["ens"].step(case["steps"])
        E.ens_get_state(state["ens"].ctx, state["out"].data_ptr(), state["ens"].state_bytes())
        return state["out"]
    if kind == "host":
        E.ens_step_host(state["ens"].ctx, state["in"].data_ptr(), state["out"].data_ptr(), state["ens"].state_bytes())
        return state["out"]
    if kind == "stats":
        state["ens"].gradient_stats(accumulate=False)
        counts, moments = state["ens"].stats()
        return {"counts": counts.view(np.int64), "moments": moments}
    if kind == "mixture":
        m = E.ens_mixture_host(state["lams"], state["counts"], state["moments"], state["hist"], kind=E.W_GAUSS_PAPER,
                               c=_C, Z=_Z)
        return {k: m[k] for k in ("weights", "covered", "pdf_qr", "pdf_eps", "pdf_ens", "pdf_long", "pdf_trans",
                                  "moments", "ratios")}
    if kind == "quadrature":
        m = state["net"].mixture(state["hist"], _LAM_LO, _LAM_HI, nquad=case["points"], kind=E.W_GAUSS_PAPER, c=_C,
                                 Z=_Z)
        return {k: m[k] for k in ("pdf_qr", "pdf_eps", "pdf_ens")}
    loss, grad = state["net"].loss_grad(state["lams"], state["counts"], state["hist"])
    return {"loss": loss, "grad": grad}


def work(case):
    """Bytes: every input read once, every output written once.  Flops: 2.5
    N^3 log2 N^3 per real 3D transform (nine per RK stage, eight per
    snapshot), 2 per multiply-add of the network (three times that for a
    gradient), the additions of a mixture."""
    kind = case["kind"]
    if kind in ("step", "host", "stats"):
        bytes_, flops = 0.0, 0.0
        for N, n in _sizes(case):
            _, NK, NZ, _ = _dims(N)
            fft = 2.5 * N ** 3 * 3 * math.log2(N)
            state = 3 * NK * NK * NZ * 8
            if kind == "stats":
                bytes_ += n * (state + 8 * (case["qr_bins"] ** 2 + 2 * case["tail_bins"] + 2 * case["grad_bins"]))
                flops += n * (8 * fft + 150.0 * N ** 3)
            else:
                bytes_ += n * 2 * state
                flops += n * case["steps"] * case["rk"] * 9 * fft
        return {"bytes": bytes_, "flops": flops}
    bins = case["qr_bins"] ** 2 + 2 * case["tail_bins"]
    if kind == "mixture":
        L = bins + 2 * case["grad_bins"]
        return {"bytes": 8.0 * (case["members"] * (L + 48) + L), "flops": 3.0 * case["members"] * L}
    mac = (_IN + 2 * _HID + 1) * _HID
    weights = 4.0 * (mac + 3 * _HID + 1)
    if kind == "quadrature":
        return {"bytes": weights + 8.0 * bins, "flops": 2.0 * mac * bins * case["points"]}
    return {"bytes": 2 * weights + 8.0 * case["members"] * bins, "flops": 6.0 * mac * bins * case["members"]}


# ---------------------------------------------------------------------------
# the same in 64 bits with torch and numpy
# ---------------------------------------------------------------------------
_EXACT_MOST = 7.0e9   # point-stages of a step case that take well under 20 s


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "host"):
        points = sum(n * N ** 3 for N, n in _sizes(case)) * case["steps"] * case["rk"]
        return _exact_step(case, seed) if points <= _EXACT_MOST else None
    if kind == "stats":
        return {"counts": None, "moments": _exact_moments(case, seed)}
    if kind == "mixture":
        return _exact_mixture(case, seed)
    if kind == "quadrature":
        return _exact_quadrature(case, seed)
    return _exact_gradient(case, seed)


def _states64(case, seed):
    """(member, FP64 spectral field [3, NK, NK, NZ]) of the prepared states."""
    members = _members(case)
    flat = _fields(members, seed)
    off = 0
    for m in members:
        _, NK, NZ, NZp = _dims(m.N)
        size = 3 * NK * NK * NZp * 2
        u = torch.view_as_complex(flat[off:off + size].view(3, NK, NK, NZp, 2))[..., :NZ].to(torch.complex128)
        off += size
        yield m, u


def _to_physical(uh, N, rows):
    full = torch.zeros(uh.shape[0], N, N, N // 2 + 1, dtype=torch.complex128, device="cuda")
    full[:, rows.view(-1, 1), rows.view(1, -1), :uh.shape[-1]] = uh
    return torch.fft.irfftn(full, s=(N, N, N), dim=(1, 2, 3), norm="forward")


def _exact_step(case, seed):
    parts = []
    for m, un in _states64(case, seed):
        N = m.N
        _, NK, NZ, NZp = _dims(N)
        kx, ky, kz, rows = _wave(N, torch.float64)
        k2 = kx * kx + ky * ky + kz * kz
        inv = 1.0 / torch.where(k2 == 0, 1.0, k2)
        wgt = torch.full((NZ,), 2.0, dtype=torch.float64, device="cuda")
        wgt[0] = 1.0
        band = (k2 >= m.k_lo ** 2 - 1e-9) & (k2 <= m.k_hi ** 2 + 1e-9)
        eps = m.eps_bar * math.exp(m.lam)

        def rhs(u):
            energy = 0.5 * float((band * wgt * (u.real.square() + u.imag.square()).sum(0)).sum())
            om = 1j * torch.stack([ky * u[2] - kz * u[1], kz * u[0] - kx * u[2], kx * u[1] - ky * u[0]])
            v, w = _to_physical(u, N, rows), _to_physical(om, N, rows)
            umax = float(v.abs().max())
            n = []
            for a, b in ((1, 2), (2, 0), (0, 1)):
                f = torch.fft.rfftn(v[a] * w[b] - v[b] * w[a], dim=(0, 1, 2), norm="forward")
                n.append(f[rows.view(-1, 1), rows.view(1, -1), :NZ])
                del f
            n = torch.stack(n)
            p = (kx * n[0] + ky * n[1] + kz * n[2]) * inv
            n = torch.stack([n[0] - kx * p, n[1] - ky * p, n[2] - kz * p])
            n[:, 0, 0, 0] = 0
            return n + (eps / (2.0 * energy)) * band * u, umax

        for _ in range(case["steps"]):
            f, umax = rhs(un)
            dt = m.dt if m.dt > 0 else m.cfl * (2.0 * math.pi / N) / umax
            if m.dt <= 0 and m.dt_max > 0:
                dt = min(dt, m.dt_max)

            def decay(h):
                return torch.exp(-m.nu * k2 * h * dt)
            u1 = decay(1.0) * (un + dt * f)
            if m.rk_order == 2:
                f, _ = rhs(u1)
                un = 0.5 * decay(1.0) * un + 0.5 * (u1 + dt * f)
            else:
                f, _ = rhs(u1)
                u2 = 0.75 * decay(0.5) * un + 0.25 * decay(-0.5) * (u1 + dt * f)
                f, _ = rhs(u2)
                un = decay(1.0) * un / 3.0 + 2.0 / 3.0 * decay(0.5) * (u2 + dt * f)
        full = torch.zeros(3, NK, NK, NZp, dtype=torch.complex128, device="cuda")
        full[..., :NZ] = un
        parts.append(torch.view_as_real(full).reshape(-1))
    return torch.cat(parts)


def _exact_moments(case, seed):
    out = []
    for m, u in _states64(case, seed):
        kx, ky, kz, rows = _wave(m.N, torch.float64)
        A = [_to_physical(1j * k * u[i:i + 1], m.N, rows)[0] for i in range(3) for k in (kx, ky, kz)]
        row = [float((a ** p).sum()) for a in A for p in (2, 3, 4, 6)]
        tr2 = sum(A[3 * i + j] * A[3 * j + i] for i in range(3) for j in range(3))
        det = (A[0] * (A[4] * A[8] - A[5] * A[7]) - A[1] * (A[3] * A[8] - A[5] * A[6])
               + A[2] * (A[3] * A[7] - A[4] * A[6]))
        ss = sum((0.5 * (A[3 * i + j] + A[3 * j + i])).square() for i in range(3) for j in range(3))
        om2 = (A[7] - A[5]).square() + (A[2] - A[6]).square() + (A[3] - A[1]).square()
        inv = [-0.5 * tr2, -det, 2.0 * m.nu * ss, om2]
        out.append(row + [float(v.sum()) for v in inv] + [float(v.square().sum()) for v in inv] + [0.0] * 4)
    return np.array(out)


def _normal_masses(lo, hi, mu, sigma):
    """Mass of a Gaussian in the cells [lo, hi] (FP64)."""
    r = math.sqrt(0.5)
    out = []
    for a, b in zip(lo, hi):
        za, zb = (a - mu) / sigma, (b - mu) / sigma
        out.append(0.5 * (math.erfc(za * r) - math.erfc(zb * r)) if za >= 0
                   else 0.5 * (math.erfc(-zb * r) - math.erfc(-za * r)))
    return np.array(out)


def _exact_mixture(case, seed):
    lams, counts, moments = _counts(case, seed)
    nq, nt, ng = case["qr_bins"], case["tail_bins"], case["grad_bins"]
    values = np.unique(lams)
    mid = 0.5 * (values[1:] + values[:-1])
    lo = np.concatenate([[values[0] - (mid[0] - values[0])], mid])
    hi = np.concatenate([mid, [values[-1] + (values[-1] - mid[-1])]])
    at = np.searchsorted(values, lams)
    w = (_normal_masses(lo, hi, -4.5 * _C * _Z, math.sqrt(9.0 * _C * _Z)) / np.bincount(at))[at]
    covered = w.sum()
    w = w / covered
    off = nq * nq + 2 * nt
    wn = w / counts[:, off + 6].astype(np.float64)
    pdf = wn @ counts.astype(np.float64)
    dq, dt = 20.0 / nq, 16.0 / nt
    mom = wn @ moments
    lon, tra = [0, 4, 8], [1, 2, 3, 5, 6, 7]
    a = [mom[[4 * c + q for c in lon]].mean() for q in range(4)]
    b = [mom[[4 * c + q for c in tra]].mean() for q in range(4)]
    out = {"weights": w, "covered": covered, "pdf_qr": (pdf[:nq * nq] / dq ** 2).reshape(nq, nq),
           "pdf_eps": pdf[nq * nq:nq * nq + nt] / dt, "pdf_ens": pdf[nq * nq + nt:off] / dt, "pdf_long": None,
           "pdf_trans": None, "moments": mom,
           "ratios": {"S_long": a[1] / a[0] ** 1.5, "F_long": a[2] / a[0] ** 2, "F_trans": b[2] / b[0] ** 2,
                      "H_long": a[3] / a[0] ** 3, "H_trans": b[3] / b[0] ** 3}}
    if ng:
        dg = 80.0 / ng
        out["pdf_long"] = pdf[off + 8:off + 8 + ng] / (3.0 * dg)
        out["pdf_trans"] = pdf[off + 8 + ng:off + 8 + 2 * ng] / (6.0 * dg)
    return out


def _features64(case, lams):
    """Network inputs [len(lams) * bins, 64] in FP64."""
    nq, nt = case["qr_bins"], case["tail_bins"]
    c = (torch.arange(nq, dtype=torch.float64, device="cuda") + 0.5) / nq * 2 - 1
    x = (torch.arange(nt, dtype=torch.float64, device="cuda") + 0.5) / nt * 2 - 1
    bins = nq * nq + 2 * nt
    f = torch.zeros(bins, _IN, dtype=torch.float64, device="cuda")
    f[:nq * nq, 0] = c.repeat_interleave(nq)
    f[:nq * nq, 1] = c.repeat(nq)
    f[nq * nq:, 3] = x.repeat(2)
    f[:nq * nq, 4] = 1
    f[nq * nq:nq * nq + nt, 5] = 1
    f[nq * nq + nt:, 6] = 1
    o = 7
    for s in (f[:, 0].clone(), f[:, 1].clone(), f[:, 3].clone()):
        for k in range(1, 5):
            f[:, o] = torch.sin(math.pi * k * s)
            f[:, o + 1] = torch.cos(math.pi * k * s)
            o += 2
    f = f.repeat(len(lams), 1)
    f[:, 2] = torch.as_tensor(lams, dtype=torch.float64, device="cuda").repeat_interleave(bins) / 5.0
    return f


def _net64(p, f):
    """Logits of the network with parameters p (FP64 vector, differentiable)."""
    o, h = 0, f
    for width in (_IN, _HID, _HID):
        W = p[o:o + _HID * width].view(_HID, width)
        b = p[o + _HID * width:o + _HID * width + _HID]
        o += _HID * width + _HID
        h = torch.nn.functional.silu(h @ W.T + b)
    return h @ p[o:o + _HID] + p[o + _HID]


def _kinds(case):
    nq2, nt = case["qr_bins"] ** 2, case["tail_bins"]
    return (slice(0, nq2), slice(nq2, nq2 + nt), slice(nq2 + nt, nq2 + 2 * nt))


def _exact_quadrature(case, seed):
    n, nq, nt = case["points"], case["qr_bins"], case["tail_bins"]
    d = (_LAM_HI - _LAM_LO) / n
    lo = _LAM_LO + d * np.arange(n)
    w = _normal_masses(lo, lo + d, -4.5 * _C * _Z, math.sqrt(9.0 * _C * _Z))
    w = w / w.sum()
    p = torch.as_tensor(_params(seed), dtype=torch.float64, device="cuda")
    pdf = torch.zeros(nq * nq + 2 * nt, dtype=torch.float64, device="cuda")
    for s in range(0, n, 32):
        z = _net64(p, _features64(case, lo[s:s + 32] + 0.5 * d)).view(-1, nq * nq + 2 * nt)
        q = torch.cat([torch.softmax(z[:, k], 1) for k in _kinds(case)], 1)
        pdf += torch.as_tensor(w[s:s + 32], device="cuda") @ q
    a, b, c = (pdf[k].cpu().numpy() for k in _kinds(case))
    return {"pdf_qr": (a / (20.0 / nq) ** 2).reshape(nq, nq), "pdf_eps": b / (16.0 / nt), "pdf_ens": c / (16.0 / nt)}


def _exact_gradient(case, seed):
    lams, counts, _ = _counts(case, seed)
    n, bins = len(lams), case["qr_bins"] ** 2 + 2 * case["tail_bins"]
    t = torch.as_tensor(counts[:, :bins].astype(np.float64), device="cuda")
    for k in _kinds(case):
        t[:, k] /= t[:, k].sum(1, keepdim=True)
    p = torch.as_tensor(_params(seed), dtype=torch.float64, device="cuda").requires_grad_(True)
    total, grad = 0.0, torch.zeros_like(p)
    for s in range(0, n, 16):   # a few members at a time
        z = _net64(p, _features64(case, lams[s:s + 16])).view(-1, bins)
        loss = sum(-(t[s:s + 16, k] * torch.log_softmax(z[:, k], 1)).sum() for k in _kinds(case)) / (3.0 * n)
        grad += torch.autograd.grad(loss, p)[0]
        total += float(loss)
    return {"loss": total, "grad": grad.detach().cpu().numpy()}
