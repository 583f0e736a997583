"""The half-pair kernels without FP64 in the pair loop (csrc/nb_tri.cu): sizes
where the block size, ragged tiles and output mode change, and the inputs that
send a tile or an item back to FP64 arithmetic.  Gates: the conditioned error of
the precision's contract, 1e-12 (fp64, df64) and 1e-6 (mixed)."""
import numpy as np
import pytest

from paper_2106_11143_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "df64": 1e-12, "mixed": 1e-6}


@pytest.fixture(scope="module")
def nb():
    import torch
    assert torch.cuda.is_available()
    import paper_2106_11143_gb300 as m
    return m


def check(nb, orc, pos, q=None, precision="fp64", sample=None, soft2=0.0):
    phys = W.phys(soft2=soft2)
    s = nb.System(pos, q=q)
    nb.forces(nb.Params.from_phys(phys, precision=precision), s)
    nb.sync_status()
    g = s.acc().cpu().numpy()
    assert np.all(np.isfinite(g))
    p = orc.make_params(**phys)
    idx = np.arange(pos.shape[1]) if sample is None else sample
    ref, cond = np.empty((3, len(idx))), np.empty(len(idx))
    if sample is None:
        ax, ay, az, _, cond = orc.coulomb(p, *pos, q=q, want_absf=True)
        ref = np.stack([ax, ay, az])
    else:
        for k, i in enumerate(idx):
            ax, ay, az, _, absf = orc.coulomb(p, *pos, q=q, i0=int(i), i1=int(i) + 1, want_absf=True)
            ref[:, k], cond[k] = (ax[0], ay[0], az[0]), absf[0]
    err = np.sqrt(np.sum((g[:, idx] - ref) ** 2, axis=0))
    assert np.all(err[cond == 0.0] == 0.0)  # ions without charge
    worst = np.max(err[cond > 0.0] / cond[cond > 0.0])
    print("n=%d %s: max conditioned error %.3g" % (pos.shape[1], precision, worst))
    assert worst <= TOL[precision]
    return g


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("charges", [False, True])
@pytest.mark.parametrize("n", [1500, 1537, 2799, 2800, 2817, 6145, 12160, 12161, 12289, 24577])
def test_sizes_at_the_edges(nb, orc, n, charges, precision):
    """One ion past a tile, a block and a P-tile; the last size of each block
    size and the first of the next; partials and the in-place output."""
    pos, _ = W.random_cloud(n, seed=n)
    rng = np.random.default_rng(n)
    q = W.E_CHARGE * rng.choice([-1.0, 1.0, 2.0, 0.0], size=n) if charges else None
    sample = None if n < 7000 else np.unique(np.concatenate([np.arange(16), np.arange(n - 16, n),
                                                             rng.integers(0, n, 64)]))
    a = check(nb, orc, pos, q, precision, sample)
    s = nb.System(pos, q=q)
    again = "df64" if precision == "fp64" and n >= 2000 else precision  # one kernel serves both
    nb.forces(nb.Params.from_phys(W.phys(), precision=again), s)
    assert np.array_equal(a, s.acc().cpu().numpy())


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("block", [64, 128, 256, 512, 1024])
@pytest.mark.parametrize("case", ["close", "coincident", "offset", "outlier", "zero", "weights", "tiny", "huge"])
def test_inputs_that_leave_the_fp32_path(nb, orc, case, block, precision):
    """Pairs closer than 2^-20 of the cloud (in one block, in one tile and
    across blocks), coincident ions, a cloud far off the origin, an ion a
    kilometre away, coordinates that are exactly zero, weights spread over 60
    decades, and length units far from one: the FP64 form of a tile or of the
    whole item, next to tiles that stay on the FP32 pipe."""
    n = 2100
    pos, _ = W.random_cloud(n, seed=77)
    rng = np.random.default_rng(block)
    q = None
    scale = 1.0
    if case == "close":
        for a, b, d in ((3, 4, 1e-11), (40, 100, 3e-12), (5, 2050, 2e-11)):
            pos[:, b] = pos[:, a] + np.array([d, -d, 0.0])
    elif case == "coincident":
        # the kernels' rule: coincident ions exert no force on each other
        pos[:, 9] = pos[:, 8]
        pos[:, 2060] = pos[:, 8]
        one = nb.System(pos)
        nb.set_tuning("symmetric", precision, 0, 1 << 40, block, R=0)
        try:
            nb.forces(nb.Params.from_phys(W.phys(), precision=precision), one)
            nb.set_tuning("force", "fp64", 0, 0, 0)
            nb.set_tuning("symmetric", precision, 0, 1 << 40, block, R=1)
            two = nb.System(pos)
            nb.forces(nb.Params.from_phys(W.phys(), precision=precision), two)
        finally:
            nb.set_tuning("force", "fp64", 0, 0, 0)
        a, b = one.acc().cpu().numpy(), two.acc().cpu().numpy()
        assert np.all(np.isfinite(b)) and np.max(np.abs(a - b)) <= TOL[precision] * np.max(np.abs(a))
        return
    elif case == "offset":
        pos = pos + np.array([[0.1], [-0.05], [0.3]])
        pos[:, 1] = pos[:, 0] + np.array([1e-8, 0.0, 0.0])
    elif case == "outlier":
        pos[:, 1234] = 1e3
        pos[:, 7] = pos[:, 6] + np.array([0.0, 1e-9, 0.0])
    elif case == "zero":
        pos[0:2] = 0.0
        pos[2] = np.sort(pos[2])
    elif case == "weights":
        q = W.E_CHARGE * rng.choice([-1.0, 1.0], size=n) * 10.0 ** rng.uniform(-30, 30, size=n)
    elif case == "tiny":
        scale = 2.0 ** -220
    elif case == "huge":
        scale = 2.0 ** 230
    try:
        nb.set_tuning("symmetric", precision, 0, 1 << 40, block, R=1)
        if scale == 1.0:
            check(nb, orc, pos, q, precision)
        else:
            # a power of two in the length unit scales every term exactly
            par = nb.Params.from_phys(W.phys(), k_coulomb=1.0, charge=1.0, mass=1.0, precision=precision)
            s, t = nb.System(pos), nb.System(pos * scale)
            nb.forces(par, s)
            nb.forces(par, t)
            a, b = s.acc().cpu().numpy(), t.acc().cpu().numpy() * scale ** 2
            assert np.max(np.abs(a - b)) <= TOL[precision] * np.max(np.abs(a))
    finally:
        nb.set_tuning("force", "fp64", 0, 0, 0)


@pytest.mark.parametrize("charges", [False, True])
@pytest.mark.parametrize("soft", [1e-20, 3e-7, 2e-5, 1.0])
@pytest.mark.parametrize("n", [1537, 3001, 12289])
def test_softened_sums(nb, orc, n, soft, charges):
    """A softening length far below the spacing, near it, near the cloud's size
    and far above it (where the item leaves the FP32 path), with a coincident
    and a close pair."""
    pos, _ = W.random_cloud(n, seed=n + 1)
    pos[:, 9] = pos[:, 8] + np.array([1e-12, 0.0, 0.0])
    pos[:, 700] = pos[:, 701]
    if soft < 1e-10:  # the oracle's own limit for coincident ions
        pos[:, 700] += 1e-7
    q = W.E_CHARGE * np.random.default_rng(n).choice([-1.0, 1.0, 2.0], size=n) if charges else None
    sample = None if n < 7000 else np.arange(0, n, 97)
    check(nb, orc, pos, q, "fp64", sample, soft2=soft * soft)


# ---------------------------------------------------------------------------
# The potential (csrc/nb_phi.cu) and the Jacobian product (csrc/nb_vjp.cu).


@pytest.mark.parametrize("case", ["plain", "charges", "soft", "close", "tiny-weights"])
@pytest.mark.parametrize("n", [1999, 2000, 2049, 9999, 10001, 16385, 31489])
def test_potential(nb, orc, n, case):
    """phi_i = sum_j q_j / s_ij at the edges of blocks, of the block sizes and of
    the output mode (in place from 1e6 partials), against the oracle: relative to
    sum_j |q_j| / s_ij within 1e-13 (FP64 rounding of n terms is 2^-52 sqrt(n),
    1/r itself 2^-46)."""
    pos, _ = W.random_cloud(n, seed=n + 5)
    rng = np.random.default_rng(n)
    q, soft2 = None, 0.0
    if case == "charges":
        q = W.E_CHARGE * rng.choice([-1.0, 1.0, 2.0, 0.0], size=n)
    elif case == "tiny-weights":
        q = W.E_CHARGE * 10.0 ** rng.uniform(-30, 30, size=n)
    elif case == "soft":
        soft2 = (1e-6) ** 2
    elif case == "close":
        pos[:, 40] = pos[:, 41] + np.array([1e-11, 0.0, 0.0])
        pos[:, n - 1] = pos[:, 3] + np.array([0.0, 3e-12, 0.0])
    phys = W.phys(soft2=soft2)
    phi = nb.forces(nb.Params.from_phys(phys), nb.System(pos, q=q), want_phi=True).cpu().numpy()
    nb.sync_status()
    p = orc.make_params(**phys)
    idx = np.unique(np.concatenate([np.arange(48), np.arange(n - 16, n), rng.integers(0, n, 64)]))
    qq = np.full(n, W.E_CHARGE) if q is None else q
    for i in idx:
        ref = orc.coulomb(p, *pos, q=q, i0=int(i), i1=int(i) + 1, want_phi=True)[3][0]
        mag = np.abs(qq) @ np.where(np.arange(n) == i, 0.0, 1.0 / np.sqrt(
            np.maximum(np.sum((pos - pos[:, [i]]) ** 2, axis=0) + soft2, 1e-300)))
        assert abs(phi[i] - ref) <= 1e-13 * mag, (n, case, i)


def vjp_bound(pos, lam, q, i):
    d = pos[:, [i]] - pos
    r = np.sqrt(np.sum(d * d, axis=0))
    dl = np.sqrt(np.sum((lam[:, [i]] - lam) ** 2, axis=0))
    with np.errstate(divide="ignore", invalid="ignore"):
        return np.sum(np.where(r > 0, 4.0 * np.abs(q) * dl / r ** 3, 0.0))


@pytest.mark.parametrize("case", ["plain", "charges", "soft", "zero", "uniform", "local", "decades", "close"])
@pytest.mark.parametrize("n", [2500, 2561, 4100, 16385])
def test_jacobian_product(nb, orc, n, case):
    """Edges of blocks and the two block sizes; cotangents that vanish, that are
    one constant plus a part 2^-30 of it, that decay over six decades across the
    cloud and that spread over twelve decades; close pairs.  Gate per ion: 1e-12
    of a bound on the sum of its term magnitudes (|T| <= 4 |dl| r^-3)."""
    pos, _ = W.random_cloud(n, seed=n + 9)
    rng = np.random.default_rng(n)
    lam = rng.standard_normal((3, n))
    q, soft2 = None, 0.0
    if case == "charges":
        q = W.E_CHARGE * rng.choice([-1.0, 1.0, 2.0], size=n)
    elif case == "soft":
        soft2 = (2e-6) ** 2
    elif case == "zero":
        lam[:] = 0.0
    elif case == "uniform":
        lam = np.array([[1.0], [-2.0], [0.0]]) + 2.0 ** -30 * lam
    elif case == "local":
        lam *= np.exp(-14.0 * np.abs(pos[2]) / np.max(np.abs(pos[2])))
    elif case == "decades":
        lam *= 10.0 ** rng.uniform(-6, 6, size=n)
    elif case == "close":
        pos[:, 40] = pos[:, 41] + np.array([1e-11, 0.0, 0.0])
        pos[:, n - 1] = pos[:, 3] + np.array([0.0, 3e-10, 0.0])
    phys = W.phys(soft2=soft2)
    g = nb.forces_vjp(nb.Params.from_phys(phys), nb.System(pos, q=q), lam).cpu().numpy()
    nb.sync_status()
    ref = np.stack(orc.forces_vjp(orc.make_params(**phys), 0.0, *pos, *lam, q=q))
    qq = np.full(n, W.E_CHARGE) if q is None else q
    idx = np.unique(np.concatenate([np.arange(48), np.arange(n - 16, n), rng.integers(0, n, 100)]))
    for i in idx:
        bound = W.K_COULOMB * abs(qq[i]) / W.MASS_40U * vjp_bound(pos, lam, qq, i)
        assert np.linalg.norm(g[:, i] - ref[:, i]) <= 1e-12 * bound, (n, case, i)


# ---------------------------------------------------------------------------
# The ensemble kernel's force phase (csrc/nb_batched.cu).


def ensemble(nb, sizes, seed, threads=512, one_sided=False, soft2=0.0, q=None, precision="fp64"):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pos, vel = W.random_cloud(int(off[-1]), seed=seed)
    par = nb.Params.from_phys(W.phys(omega=(6e6, 5e6, 1.2e6), soft2=soft2), precision=precision)
    nb.set_tuning("ensemble", precision, 0, 1 << 40, threads, R=0 if one_sided else 1)
    try:
        s = nb.System(pos, vel, q=q)
        nb.step_batched(par, s, off, 2)
        nb.sync_status()
    finally:
        nb.set_tuning("ensemble", precision, 0, 0, 0)
    return s.state[:, :s.n].cpu().numpy()


SIZES = [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 160, 192, 193, 256, 257, 320, 321, 383, 385, 513, 641, 1025]


@pytest.mark.parametrize("case", ["plain", "charges", "soft", "weights", "close"])
def test_ensemble_tiles_and_rounds(nb, case):
    """Instances at the edges of tiles, half and whole super-tiles and of odd
    and even round counts, against the one-sided phase (FP64 pair terms), and
    bitwise the same for 1, 3, 4 and 16 warps: accelerations within 1e-12 of the
    largest of the instance."""
    off = np.concatenate([[0], np.cumsum(SIZES)])
    n = int(off[-1])
    rng = np.random.default_rng(5)
    kw = {}
    if case == "charges":
        kw["q"] = W.E_CHARGE * rng.choice([-1.0, 1.0, 2.0, 0.0], size=n)
    elif case == "soft":
        kw["soft2"] = (2e-6) ** 2
    elif case == "weights":  # outside the FP32 path's range of weights
        kw["q"] = W.E_CHARGE * 10.0 ** rng.uniform(-20, 20, size=n)
    seed = 21 if case != "close" else 22
    if case == "close":  # a softening below 2^-20 of the cloud: close pairs' own rule
        kw["soft2"] = 1e-26
    a = ensemble(nb, SIZES, seed, **kw)
    ref = ensemble(nb, SIZES, seed, one_sided=True, **kw)
    for k in range(len(SIZES)):
        x, y = a[6:9, off[k]:off[k + 1]], ref[6:9, off[k]:off[k + 1]]
        assert np.max(np.abs(x - y)) <= 1e-12 * np.max(np.abs(y)), (case, SIZES[k])
    for threads in (32, 96, 128):
        assert np.array_equal(a, ensemble(nb, SIZES, seed, threads=threads, **kw)), (case, threads)
