"""Performance cases of the library: what a user's program calls, over the
sizes, precisions and options it calls them with.

listed() are the cases, draw(rng) one more of the same ranges, prepare(case,
seed) what a program has in hand before the call, run(state) one pass through
the public entry points, work(case) the bytes and operations one pass cannot do
without, and exact(case, seed) the pass's outputs from a plain FP64 direct sum
in torch (no code of the package).
"""
import math

import numpy as np
import torch

import paper_2106_11143_gb300 as nb
from paper_2106_11143_gb300 import workloads as W

SPECIES_U = (40.0, 24.0)  # the two species' masses (u)
CHUNK_PAIRS = 1 << 28     # pairs per block of the plain direct sum


def _steps(n):
    """Steps of one call: 100 for small systems, fewer as n^2 grows."""
    return int(max(1, min(100, 2_000_000_000 // (n * n))))


def _step(name, n, precision, trap="harmonic", species=False):
    return dict(name=name, kind="step", n=n, precision=precision, trap=trap, species=species, nsteps=_steps(n))


def listed():
    return [
        # the 16-ion chain in the RF trap, FP64: the smallest runs, all latency
        _step("chain-16-fp64", 16, "fp64", trap="rf"),
        # the 1024-ion cloud in the pseudopotential, FP64, 100 steps
        _step("cloud-1024-fp64", 1024, "fp64"),
        # a few thousand ions in the fast mixed form: a mid-size run, ragged
        _step("cloud-3001-split", 3001, "mixed_split"),
        # sympathetic cooling: two species with charges and masses of their own
        _step("species-5003-df64", 5003, "df64", trap="rf", species=True),
        # the 16384-ion cloud in the RF trap with friction, FP64
        _step("rf-16384-fp64", 16384, "fp64", trap="rf"),
        # the literal mixed form at an odd size
        _step("cloud-50021-mixed", 50021, "mixed"),
        # the large cloud: forces and a step in FP64 and in the split mixed form
        _step("cloud-100000-fp64", 100000, "fp64"),
        _step("cloud-100000-split", 100000, "mixed_split"),
        # the diagnostics of a large run: forces, per-ion potentials and energies
        dict(name="energy-65537", kind="energy", n=65537, precision="fp64", trap="harmonic", species=False),
        # 512 quench realisations of uneven size in one launch
        dict(name="quench-512-fp64", kind="ensemble", n_inst=512, n_min=32, n_max=4096, precision="fp64",
             each=False, nsteps=2),
        # the force Jacobian product (implicit methods, sensitivities)
        dict(name="vjp-20000", kind="vjp", n=20000, precision="fp64", trap="harmonic", species=False),
        # loss and gradient of a trajectory, forward and backward
        dict(name="adjoint-4096", kind="adjoint", n=4096, precision="fp64", nsteps=20, every=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "step", "energy", "ensemble", "vjp", "adjoint"])
    if kind == "step":
        n = _log_int(rng, 10, 100000)
        c = _step("", n, rng.choice(["fp64", "fp64", "df64", "mixed", "mixed_split", "mixed_split_rsq"]),
                  trap=rng.choice(["harmonic", "rf"]), species=rng.random() < 0.25)
    elif kind == "energy":
        c = dict(kind=kind, n=_log_int(rng, 500, 65537), precision="fp64", trap=rng.choice(["harmonic", "rf"]),
                 species=rng.random() < 0.25)
    elif kind == "vjp":
        c = dict(kind=kind, n=_log_int(rng, 500, 60000), precision=rng.choice(["fp64", "df64"]), trap="harmonic",
                 species=rng.random() < 0.25)
    elif kind == "ensemble":
        n_max = _log_int(rng, 200, 4096)
        c = dict(kind=kind, n_inst=_log_int(rng, 16, 512), n_min=rng.randint(16, 64), n_max=n_max,
                 precision=rng.choice(["fp64", "df64"]), each=rng.random() < 0.5,
                 nsteps=max(2, min(10, 32_000_000 // (n_max * n_max))))
    else:
        n = _log_int(rng, 300, 4096)
        c = dict(kind=kind, n=n, precision=rng.choice(["fp64", "df64"]), nsteps=rng.randint(10, 20),
                 every=rng.choice([5, 10]))
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# Inputs.


def _rng(case, seed):
    return np.random.default_rng([int(seed), case.get("n", case.get("n_inst", 0))])


def _phys(case):
    """Trap and time step: the pseudopotential (dt = 1 ns), or the RF trap with
    laser-cooling friction (dt = 2 ns)."""
    if case.get("trap") == "rf":
        return W.phys(trap="rf", q_mathieu=0.3, omega_rf=W.TWO_PI * 10e6, omega=(0.0, 0.0, W.TWO_PI * 200e3),
                      gamma=1e-20, dt=2e-9)
    n = case["n"]
    if n >= 40000:
        om = W.cold_fluid_omegas(100000, 200e-6, 1000e-6)
    else:
        om = (W.TWO_PI * 1e6, W.TWO_PI * 1e6, W.TWO_PI * 200e3)
    return W.phys(omega=om, dt=1e-9)


def _ions(case, seed):
    """Positions, velocities (3, n) and, with two species, charges and masses.
    Below 33 ions a chain, else a uniform ellipsoid at the density the trap
    holds; 10 mK velocities."""
    rng = _rng(case, seed)
    n = case["n"]
    if n <= 32:
        pos = np.zeros((3, n))
        pos[2] = W.chain_positions(n, W.TWO_PI * 200e3)
        pos += 0.05e-6 * rng.standard_normal((3, n))
    elif n >= 40000:
        pos = W.ellipsoid_uniform(n, (200e-6, 200e-6, 1000e-6), rng)
    else:
        a = 20e-6 * (n / 1024.0) ** (1.0 / 3.0)
        pos = W.ellipsoid_uniform(n, (a, a, 5 * a), rng)
    vel = W.thermal_velocities(n, 10e-3, W.MASS_40U, rng)
    q = m = None
    if case.get("species"):
        other = rng.random(n) < 0.4
        m = np.where(other, SPECIES_U[1], SPECIES_U[0]) * W.AMU
        q = np.where(other, 2.0, 1.0) * W.E_CHARGE
    return pos, vel, q, m


def _quench_sizes(case):
    r = np.random.default_rng([case["n_inst"], case["n_min"], case["n_max"]])
    return r.integers(case["n_min"], case["n_max"] + 1, size=case["n_inst"])


def _quench(case, seed):
    """The quench ensemble: chains at the continuum density's quantiles with
    thermal transverse spread, Doppler velocities, the radial trap ramped; one
    ramp rate for all instances or a decade of them (`each`)."""
    rng = _rng(case, seed)
    sizes = _quench_sizes(case)
    off = np.zeros(len(sizes) + 1, dtype=np.int64)
    off[1:] = np.cumsum(sizes)
    total = int(off[-1])
    wz, temp = W.TWO_PI * 100e3, 0.5e-3
    w0, w1, dt, steps = W.TWO_PI * 1.2e6, W.TWO_PI * 0.6e6, 5e-9, 20000
    rate = (w1 - w0) / (steps * dt)
    ell = W.chain_length_scale(wz)
    pos = rng.standard_normal((3, total)) * (math.sqrt(W.K_B * temp / W.MASS_40U) / w0)
    for k, nk in enumerate(sizes):
        u = (np.arange(nk) + 0.5) / nk
        length = ell * (3.0 * nk * math.log(max(nk, 2))) ** (1.0 / 3.0)
        pos[2, off[k]:off[k + 1]] += length * 2.0 * np.sin(np.arcsin(2.0 * u - 1.0) / 3.0)
    vel = W.thermal_velocities(total, temp, W.MASS_40U, rng)
    base = W.phys(omega=(w0, w0, wz), omega_rate=(rate, rate, 0.0), gamma=1e-20, dt=dt, noise_T=temp, seed=4)
    per = []
    for k in range(len(sizes)):
        p = dict(base)
        if case["each"]:
            r = rate / 10.0 ** (k / max(len(sizes) - 1, 1))
            wr = 0.5 * (w0 + w1) - r * 0.5 * steps * dt
            p["omega"], p["omega_rate"] = (wr, wr, wz), (r, r, 0.0)
        p["instance"] = k
        per.append(p)
    return sizes, off, pos, vel, base, per


def _dev(a):
    return None if a is None else torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    kind, prec = case["kind"], case["precision"]
    if kind == "ensemble":
        sizes, off, pos, vel, base, per = _quench(case, seed)
        x, v = _dev(pos), _dev(vel)
        acc = torch.empty_like(x)  # the state resumed from: x, v and the acceleration at it
        for k in range(len(sizes)):
            s = slice(int(off[k]), int(off[k + 1]))
            acc[:, s] = _total(per[k], 0.0, x[:, s], v[:, s])
        sysm = nb.System(x, v)
        sysm.state[6:9, :sysm.n].copy_(acc)
        pars = [nb.Params.from_phys(p, precision=prec) for p in per] if case["each"] \
            else nb.Params.from_phys(base, precision=prec)
        return dict(case=case, sys=sysm, par=pars, off=off, state0=sysm.state.clone())
    if kind == "adjoint":
        w = W.adjoint_cloud(n=case["n"], seed=int(seed) + 17)
        return dict(case=case, par=nb.Params.from_phys(w["phys"], precision=prec), x0=_dev(w["pos"]),
                    v0=_dev(w["vel"]), omega=_dev(np.array(w["phys"]["omega"])), target=_dev(w["target"]))
    pos, vel, q, m = _ions(case, seed)
    par = nb.Params.from_phys(_phys(case), precision=prec)
    sysm = nb.System(pos, vel, q=q, m=m)
    st = dict(case=case, sys=sysm, par=par)
    if kind == "vjp":
        st["lam"] = _dev(_lam(case, seed))
    if kind == "step":
        st["state0"] = sysm.state.clone()
    return st


def _lam(case, seed):
    return np.random.default_rng([int(seed), 77, case["n"]]).standard_normal((3, case["n"]))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "adjoint":
        x0 = state["x0"].detach().requires_grad_(True)
        v0 = state["v0"].detach().requires_grad_(True)
        om = state["omega"].detach().requires_grad_(True)
        loss = nb.trajectory_loss(x0, v0, om, state["par"], case["nsteps"], case["every"], state["target"])
        gx, gv, gw = torch.autograd.grad(loss, (x0, v0, om))
        return {"loss": loss.detach(), "gx0": gx, "gv0": gv, "gomega": gw}
    sysm = state["sys"]
    if kind == "energy":
        phi = nb.forces(state["par"], sysm, want_phi=True)
        return {"acc": sysm.state[6:9, :sysm.n], "phi": phi, "energy": nb.energy(state["par"], sysm)}
    if kind == "vjp":
        return {"g": nb.forces_vjp(state["par"], sysm, state["lam"], total=True)}
    # a run from the saved initial state: load it, then advance
    sysm.state.copy_(state["state0"])
    sysm.step = 0
    if kind == "ensemble":
        fn = nb.step_batched_each if case["each"] else nb.step_batched
        fn(state["par"], sysm, state["off"], case["nsteps"])
    else:
        nb.forces(state["par"], sysm, total=True)
        nb.step(state["par"], sysm, case["nsteps"])
    n = sysm.n
    return {"pos": sysm.state[0:3, :n], "vel": sysm.state[3:6, :n], "acc": sysm.state[6:9, :n]}


def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: 20 per
    unordered pair of a force evaluation (3 differences, 5 for r^2, 1/sqrt, 2
    for its cube, 3 products, 6 adds into both ions), 12 for the potential
    (no vector sums), 48 for the Jacobian product."""
    kind = case["kind"]
    if kind == "ensemble":
        s = _quench_sizes(case).astype(np.float64)
        pairs = float(np.sum(s * (s - 1)) / 2) * case["nsteps"]
        return {"bytes": 2 * 72.0 * float(s.sum()), "flops": 20.0 * pairs}
    n = float(case["n"])
    pairs = n * (n - 1) / 2
    if kind == "step":
        return {"bytes": (48 + 72 + (16 if case["species"] else 0)) * n, "flops": 20 * pairs * (case["nsteps"] + 1)}
    if kind == "energy":
        return {"bytes": (48 + 32) * n + 32, "flops": (20 + 12 + 12) * pairs}
    if kind == "vjp":
        return {"bytes": 72 * n, "flops": 48 * pairs}
    t = case["nsteps"]
    # forward: t + 1 forces and the loss; backward: t recomputed forces, t + 1 products
    return {"bytes": (72 + 48) * n, "flops": pairs * (20 * (2 * t + 1) + 12 + 48 * (t + 1))}


# ---------------------------------------------------------------------------
# The same outputs from a plain FP64 direct sum.


def _blocks(n):
    rows = max(1, min(n, CHUNK_PAIRS // max(n, 1)))
    return [(i, min(n, i + rows)) for i in range(0, n, rows)]


def _pair_rows(x, i0, i1):
    """Displacements d (3, rows, n) and 1/r (0 for the ion itself)."""
    d = x[:, i0:i1, None] - x[:, None, :]
    inv = torch.rsqrt((d * d).sum(0))
    rows = torch.arange(i0, i1, device=x.device)
    inv[rows - i0, rows] = 0.0
    return d, inv


def _coulomb(x, w):
    """sum_j w_j (x_i - x_j) / r^3."""
    out = torch.empty_like(x)
    for i0, i1 in _blocks(x.shape[1]):
        d, inv = _pair_rows(x, i0, i1)
        s = inv * inv * inv
        if w is not None:
            s = s * w
        out[:, i0:i1] = (d * s).sum(2)
    return out


def _trap(ph, t, x):
    om = [ph["omega"][k] + ph["omega_rate"][k] * t for k in range(3)]
    if ph["trap"] == "rf":
        c = 0.5 * ph["q_mathieu"] * ph["omega_rf"] ** 2 * math.cos(ph["omega_rf"] * t + ph["rf_phase"])
        return torch.stack([-c * x[0], c * x[1], -om[2] ** 2 * x[2]])
    return torch.stack([-om[k] ** 2 * x[k] for k in range(3)])


def _conservative(ph, t, x, q=None, m=None):
    kc, mass, ch = ph["k_coulomb"], ph["mass"], ph["charge"]
    if q is None:
        return kc * ch * ch / mass * _coulomb(x, None) + _trap(ph, t, x)
    return kc * q / m * _coulomb(x, q) + (q / m) / (ch / mass) * _trap(ph, t, x)


def _total(ph, t, x, v, q=None, m=None):
    return _conservative(ph, t, x, q, m) - ph["gamma"] / (ph["mass"] if m is None else m) * v


def _normals(seed, instance, step, n):
    """The Langevin draws: Philox4x32-10 (Salmon et al., SC'11) on the counter
    (ion, step, step >> 32, instance) and Box-Muller."""
    c = [np.arange(n, dtype=np.uint64), np.full(n, step & 0xffffffff, np.uint64),
         np.full(n, step >> 32, np.uint64), np.full(n, instance, np.uint64)]
    k0, k1, low = seed & 0xffffffff, seed >> 32, np.uint64(0xffffffff)
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & low,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xffffffff, (k1 + 0xBB67AE85) & 0xffffffff
    u = [(a.astype(np.float64) + 0.5) * 2.0 ** -32 for a in c]
    r0, r1 = np.sqrt(-2.0 * np.log(u[0])), np.sqrt(-2.0 * np.log(u[2]))
    return np.stack([r0 * np.cos(2 * np.pi * u[1]), r0 * np.sin(2 * np.pi * u[1]), r1 * np.cos(2 * np.pi * u[3])])


def _verlet(ph, x, v, a, nsteps, q=None, m=None):
    dt, gamma = ph["dt"], ph["gamma"]
    mass = ph["mass"] if m is None else m
    for s in range(1, nsteps + 1):
        t = ph["t0"] + s * dt
        x = x + v * dt + 0.5 * dt * dt * a
        u = _conservative(ph, t, x, q, m)
        v = (v + 0.5 * dt * (a + u)) / (1.0 + gamma * dt / (2.0 * mass))
        if ph["noise_T"] > 0:
            v = v + math.sqrt(2.0 * gamma * W.K_B * ph["noise_T"] * dt) / mass * _dev(
                _normals(ph["seed"], ph.get("instance", 0), s, x.shape[1]))
        a = u - gamma / mass * v
    return x, v, a


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        sizes, off, pos, vel, _, per = _quench(case, seed)
        x, v = _dev(pos), _dev(vel)
        out = [torch.empty_like(x) for _ in range(3)]
        for k in range(len(sizes)):
            s = slice(int(off[k]), int(off[k + 1]))
            a = _total(per[k], 0.0, x[:, s], v[:, s])
            for o, r in zip(out, _verlet(per[k], x[:, s], v[:, s], a, case["nsteps"])):
                o[:, s] = r
        return {"pos": out[0], "vel": out[1], "acc": out[2]}
    if kind == "adjoint":
        return _exact_adjoint(case, seed)
    pos, vel, q, m = _ions(case, seed)
    ph = _phys(case)
    x, v, q, m = _dev(pos), _dev(vel), _dev(q), _dev(m)
    if kind == "step":
        r = _verlet(ph, x, v, _total(ph, 0.0, x, v, q, m), case["nsteps"], q, m)
        return dict(zip(("pos", "vel", "acc"), r))
    mass = torch.full_like(x[0], ph["mass"]) if m is None else m
    qq = torch.full_like(x[0], ph["charge"]) if q is None else q
    if kind == "energy":
        phi = torch.cat([(_pair_rows(x, i0, i1)[1] * qq).sum(1) for i0, i1 in _blocks(case["n"])])
        kin = float((0.5 * mass * (v * v).sum(0)).sum())
        # the trap's potential energy is -(m/2) x . a_trap (the trap is linear)
        ts = (qq / mass) / (ph["charge"] / ph["mass"])
        trap = float((-0.5 * mass * ts * (x * _trap(ph, 0.0, x)).sum(0)).sum())
        cou = float((0.5 * ph["k_coulomb"] * qq * phi).sum())
        acc = ph["k_coulomb"] * qq / mass * (_coulomb(x, None) * ph["charge"] if q is None else _coulomb(x, q))
        return {"acc": acc, "phi": phi, "energy": np.array([kin, trap, cou, kin + trap + cou])}
    lam = _dev(_lam(case, seed))
    g = torch.empty_like(x)
    for i0, i1 in _blocks(case["n"]):
        d, inv = _pair_rows(x, i0, i1)
        dl = lam[:, i0:i1, None] - lam[:, None, :]
        s3 = qq * inv ** 3
        g[:, i0:i1] = (dl * s3 - d * (3.0 * (d * dl).sum(0) * s3 * inv * inv)).sum(2)
    ts = (qq / mass) / (ph["charge"] / ph["mass"])
    return {"g": ph["k_coulomb"] * qq / mass * g + ts * _trap(ph, 0.0, lam)}


def _exact_adjoint(case, seed):
    """The trajectory loss and its gradient by the discrete adjoint of the
    Verlet map, with the plain products above."""
    w = W.adjoint_cloud(n=case["n"], seed=int(seed) + 17)
    ph = w["phys"]
    n, dt, mass = case["n"], ph["dt"], ph["mass"]
    om = _dev(np.array(ph["omega"]))[:, None]
    pref = ph["k_coulomb"] * ph["charge"] ** 2 / mass
    x, v, tgt = _dev(w["pos"]), _dev(w["vel"]), _dev(w["target"])

    def accel(y):
        return pref * _coulomb(y, None) - om * om * y

    def product(y, lam):
        g = torch.empty_like(y)
        for i0, i1 in _blocks(n):
            d, inv = _pair_rows(y, i0, i1)
            dl = lam[:, i0:i1, None] - lam[:, None, :]
            s3 = inv ** 3
            g[:, i0:i1] = (dl * s3 - d * (3.0 * (d * dl).sum(0) * s3 * inv * inv)).sum(2)
        return pref * g - om * om * lam

    xs, a = [x], accel(x)
    for _ in range(case["nsteps"]):
        y = xs[-1] + dt * v + 0.5 * dt * dt * a
        an = accel(y)
        v = v + 0.5 * dt * (a + an)
        a = an
        xs.append(y)
    xt = xs[-1]
    phi = torch.cat([_pair_rows(xt, i0, i1)[1].sum(1) for i0, i1 in _blocks(n)])
    loss = (0.5 * ph["k_coulomb"] * ph["charge"] ** 2 * phi).sum() + (0.5 * mass * om * om * xt * xt).sum() \
        + ((xt - tgt) ** 2).sum()
    xb = -mass * a + 2.0 * (xt - tgt)
    vb, ab, wb = torch.zeros_like(x), torch.zeros_like(x), (mass * om * xt * xt).sum(1)
    for k in range(case["nsteps"], 0, -1):
        ab = ab + 0.5 * dt * vb
        xb = xb + product(xs[k], ab)
        wb = wb + (ab * (-2.0 * om * xs[k])).sum(1)
        vb, ab = vb + dt * xb, 0.5 * dt * vb + 0.5 * dt * dt * xb
    xb = xb + product(xs[0], ab)
    wb = wb + (ab * (-2.0 * om * xs[0])).sum(1)
    return {"loss": loss, "gx0": xb, "gv0": vb, "gomega": wb}
