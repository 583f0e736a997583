"""The one-sided FP64-class sums on the FP32 pipe (csrc/nb_one.cu): the edges of
its range and of its tiles, ranges of ions against the full call, and the inputs
that send an ion's chunk or the whole call back to FP64.  Gate: the conditioned
error of the fp64 and df64 contracts, 1e-12."""
import numpy as np
import pytest

from paper_2106_11143_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nb():
    import torch
    assert torch.cuda.is_available()
    import paper_2106_11143_gb300 as m
    return m


def check(nb, orc, pos, q=None, precision="fp64", soft2=0.0):
    phys = W.phys(soft2=soft2)
    par = nb.Params.from_phys(phys, precision=precision)
    s = nb.System(pos, q=q)
    nb.forces(par, s)
    nb.sync_status()
    g = s.acc().cpu().numpy()
    ax, ay, az, _, cond = orc.coulomb(orc.make_params(**phys), *pos, q=q, want_absf=True)
    err = np.sqrt(np.sum((g - np.stack([ax, ay, az])) ** 2, axis=0))
    assert np.all(err[cond == 0.0] == 0.0)  # ions without charge
    assert np.max(err[cond > 0.0] / cond[cond > 0.0]) <= 1e-12
    n = pos.shape[1]
    parts = nb.System(pos, q=q)  # ranges that start anywhere in a block of threads
    for a, b in ((0, 1), (1, 130), (130, n - 3), (n - 3, n)):
        nb.forces_range(par, parts, a, b)
    nb.sync_status()
    if not nb.plan_info("force", precision, n)["symmetric"]:
        assert np.array_equal(g, parts.acc().cpu().numpy())


@pytest.mark.parametrize("precision", ["fp64", "df64"])
@pytest.mark.parametrize("form", ["plain", "charges", "soft", "charges+soft"])
@pytest.mark.parametrize("n", [512, 513, 641, 1023, 1499, 1999, 4096])
def test_sizes_at_the_edges(nb, orc, n, form, precision):
    pos, _ = W.random_cloud(n, seed=n)
    q = W.E_CHARGE * np.random.default_rng(n).choice([-1.0, 1.0, 2.0, 0.0], size=n) if "charges" in form else None
    check(nb, orc, pos, q, precision, 1e-14 if "soft" in form else 0.0)


@pytest.mark.parametrize("case", ["close", "coincident", "offset", "outlier", "zero", "weights", "tiny", "huge"])
def test_inputs_that_leave_the_fp32_path(nb, orc, case):
    n = 700
    pos, _ = W.random_cloud(n, seed=7)
    q = None
    if case == "close":
        for i, j in ((3, 9), (20, 650), (699, 130)):
            pos[:, i] = pos[:, j] + 2e-12
    elif case == "offset":
        pos += 0.1
    elif case == "outlier":
        pos[0, 5] = 1e3
    elif case == "zero":
        pos[2] = 0.0
    elif case == "weights":
        q = W.E_CHARGE * 10.0 ** np.random.default_rng(1).uniform(-30, 30, n)
    if case not in ("coincident", "tiny", "huge"):
        check(nb, orc, pos, q)
        return
    # against the FP64 kernel, which a tuned launch shape selects; a power of two
    # in the length unit scales every term exactly
    if case == "coincident":  # the kernels' rule: coincident ions exert no force on each other
        pos[:, 10] = pos[:, 11]
        pos[:, 600] = pos[:, 11]
    scale = {"coincident": 1.0, "tiny": 2.0 ** -220, "huge": 2.0 ** 230}[case]
    par = nb.Params.from_phys(W.phys(), k_coulomb=1.0, charge=1.0, mass=1.0, precision="fp64")
    s, t = nb.System(pos), nb.System(pos * scale)
    nb.forces(par, t)
    nb.set_tuning("force", "fp64", 0, 1 << 40, 32, R=1)
    try:
        nb.forces(par, s)
    finally:
        nb.set_tuning("force", "fp64", 0, 0, 0)
    nb.sync_status()
    a, b = s.acc().cpu().numpy(), t.acc().cpu().numpy() * scale ** 2
    assert np.all(np.isfinite(b)) and np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(a))
