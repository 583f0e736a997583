"""The FP64-class half-pair kernel on the FP32 pipe (csrc/nb_tri.cu): sizes
where its block size, ragged tiles and output mode change, and the inputs that
send a tile or an item back to FP64 arithmetic.  Gate: the FP64 contract's
conditioned error, 1e-12 (measured 2^-45 to 2^-46 on these clouds)."""
import numpy as np
import pytest

from paper_2106_11143_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def nb():
    import torch
    assert torch.cuda.is_available()
    import paper_2106_11143_gb300 as m
    return m


def check(nb, orc, pos, q=None, precision="fp64", sample=None):
    phys = W.phys()
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
    assert worst <= TOL
    return g


@pytest.mark.parametrize("charges", [False, True])
@pytest.mark.parametrize("n", [1500, 1537, 2799, 2800, 2817, 6145, 12160, 12161, 12289, 24577])
def test_sizes_at_the_edges(nb, orc, n, charges):
    """One ion past a tile, a block and a P-tile; the last size of each block
    size and the first of the next; partials and the in-place output."""
    pos, _ = W.random_cloud(n, seed=n)
    rng = np.random.default_rng(n)
    q = W.E_CHARGE * rng.choice([-1.0, 1.0, 2.0, 0.0], size=n) if charges else None
    sample = None if n < 7000 else np.unique(np.concatenate([np.arange(16), np.arange(n - 16, n),
                                                             rng.integers(0, n, 64)]))
    a = check(nb, orc, pos, q, "fp64", sample)
    s = nb.System(pos, q=q)
    nb.forces(nb.Params.from_phys(W.phys(), precision="df64" if n >= 2000 else "fp64"), s)
    assert np.array_equal(a, s.acc().cpu().numpy())  # one kernel serves both, bitwise reproducible


@pytest.mark.parametrize("block", [64, 128, 256, 512, 1024])
@pytest.mark.parametrize("case", ["close", "coincident", "offset", "outlier", "zero", "weights", "tiny", "huge"])
def test_inputs_that_leave_the_fp32_path(nb, orc, case, block):
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
        nb.set_tuning("symmetric", "fp64", 0, 1 << 40, block, R=0)
        try:
            nb.forces(nb.Params.from_phys(W.phys()), one)
            nb.set_tuning("force", "fp64", 0, 0, 0)
            nb.set_tuning("symmetric", "fp64", 0, 1 << 40, block, R=1)
            two = nb.System(pos)
            nb.forces(nb.Params.from_phys(W.phys()), two)
        finally:
            nb.set_tuning("force", "fp64", 0, 0, 0)
        a, b = one.acc().cpu().numpy(), two.acc().cpu().numpy()
        assert np.all(np.isfinite(b)) and np.max(np.abs(a - b)) <= TOL * np.max(np.abs(a))
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
        nb.set_tuning("symmetric", "fp64", 0, 1 << 40, block, R=1)
        if scale == 1.0:
            check(nb, orc, pos, q)
        else:
            # a power of two in the length unit scales every term exactly
            par = nb.Params.from_phys(W.phys(), k_coulomb=1.0, charge=1.0, mass=1.0)
            s, t = nb.System(pos), nb.System(pos * scale)
            nb.forces(par, s)
            nb.forces(par, t)
            a, b = s.acc().cpu().numpy(), t.acc().cpu().numpy() * scale ** 2
            assert np.max(np.abs(a - b)) <= TOL * np.max(np.abs(a))
    finally:
        nb.set_tuning("force", "fp64", 0, 0, 0)
