"""One ion far outside the cloud (ejected from the trap) sets no other ion's units:
the one-sided and the ensemble force phases leave its own terms to FP64 and no
others, so that a step takes little longer.  The gates are well above what was
measured (1.2 for both) and well below the cost of sending every close pair to
FP64 (3.4 and 14)."""
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


def shortest(f, runs=9):
    import torch
    t = []
    for k in range(runs + 3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return min(t[3:])


@pytest.mark.parametrize("precision", ["fp64", "df64"])
def test_one_sided_steps(nb, precision):
    n, t = 1499, []
    for far in (None, 5.0):
        pos, _ = W.random_cloud(n, seed=n)
        if far:
            pos[:, 7] = far
        par = nb.Params.from_phys(W.phys(), k_coulomb=1e-30, precision=precision)
        s = nb.System(pos, np.zeros((3, n)))
        nb.forces(par, s, total=True)
        t.append(shortest(lambda: nb.step(par, s, 100)))
    nb.sync_status()
    assert t[1] <= 2.0 * t[0], t


def test_ensemble_steps(nb):
    sizes = np.random.default_rng(3).integers(64, 2049, 152)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    t = []
    for far in (None, 5.0):
        pos, _ = W.random_cloud(int(off[-1]), seed=1)
        if far:
            pos[:, off[:-1] + 3] = far
        par = nb.Params.from_phys(W.phys(), k_coulomb=1e-30)
        s = nb.System(pos, np.zeros_like(pos))
        t.append(shortest(lambda: nb.step_batched(par, s, off, 2)))
    nb.sync_status()
    assert t[1] <= 3.0 * t[0], t


@pytest.mark.parametrize("soft2", [0.0, 1e-14])
@pytest.mark.parametrize("charges", [False, True])
@pytest.mark.parametrize("n,far", [(513, [5]), (700, [5, 140]), (1024, [0, 1, 2, 3]), (1024, [0, 1, 2, 3, 4, 5, 6, 7, 8, 9]),
                                   (1499, [127, 128, 1400, 1498]), (640, list(range(128, 256)))])
def test_forces_on_and_of_far_ions(nb, orc, n, far, charges, soft2):
    """Some ions of a group, of a chunk and of both, up to and beyond the number a
    block leaves out of its unit, and a whole group: conditioned error 1e-12, and
    the bits of ranges of ions those of the full call."""
    pos, _ = W.random_cloud(n, seed=n)
    rng = np.random.default_rng(n)
    pos[:, far] = rng.uniform(0.5, 5.0, (3, len(far))) * rng.choice([-1.0, 1.0], (3, len(far)))
    q = W.E_CHARGE * rng.choice([-1.0, 1.0, 2.0, 0.0], size=n) if charges else None
    phys = W.phys(soft2=soft2)
    par = nb.Params.from_phys(phys, precision="df64")
    s, parts = nb.System(pos, q=q), nb.System(pos, q=q)
    nb.forces(par, s)
    for a, b in ((0, 3), (3, 129), (129, 300), (300, n)):
        nb.forces_range(par, parts, a, b)
    nb.sync_status()
    g = s.acc().cpu().numpy()
    assert np.array_equal(g, parts.acc().cpu().numpy())
    ax, ay, az, _, cond = orc.coulomb(orc.make_params(**phys), *pos, q=q, want_absf=True)
    err = np.sqrt(np.sum((g - np.stack([ax, ay, az])) ** 2, axis=0))
    assert np.all(err[cond == 0.0] == 0.0)
    assert np.max(err[cond > 0.0] / cond[cond > 0.0]) <= 1e-12
