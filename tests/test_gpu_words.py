"""Coordinates as three FP32 words (csrc/nb_tri.cuh): inputs whose small
components or low bits the words could lose, componentwise where that matters,
against plain FP64 sums on the host."""
import numpy as np
import pytest

from paper_2106_11143_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# k = q = m = 1: an acceleration is the bare pair sum
UNIT = dict(k_coulomb=1.0, charge=1.0, mass=1.0)


@pytest.fixture(scope="module")
def nb():
    import torch
    assert torch.cuda.is_available()
    import paper_2106_11143_gb300 as m
    return m


def pair_sums(pos, idx):
    """Of the ions idx: F_c = sum_j d_c r^-3, the sum of |d_c| r^-3 per component,
    and phi = sum_j 1/r."""
    f, a, phi = np.empty((3, len(idx))), np.empty((3, len(idx))), np.empty(len(idx))
    for k in range(0, len(idx), 128):
        d = pos[:, idx[k:k + 128], None] - pos[:, None, :]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        with np.errstate(divide="ignore"):
            y = np.where(r2 > 0.0, 1.0 / np.sqrt(r2), 0.0)
        t = d * (y * y * y)
        f[:, k:k + 128], a[:, k:k + 128], phi[k:k + 128] = t.sum(-1), np.abs(t).sum(-1), y.sum(-1)
    return f, a, phi


def grid_with_a_trace(n):
    """A cloud on the grid 2^-30 (no l word anywhere) with two ions 2^-35 apart, one
    of which is off the grid by 1.9 2^-70 in that direction: no word shows it."""
    rng = np.random.default_rng(n)
    pos = rng.integers(-2 ** 30, 2 ** 30, size=(3, n)) * 2.0 ** -30
    pos[:, 41] = pos[:, 40]
    pos[0, 40] = 0.0
    pos[0, 41] = 2.0 ** -35 + 1.9 * 2.0 ** -70
    return pos


@pytest.mark.parametrize("n", [700, 2100, 13000])
def test_bits_below_the_words_of_a_grid(nb, n):
    pos = grid_with_a_trace(n)
    s = nb.System(pos)
    phi = nb.forces(nb.Params.from_phys(W.phys(**UNIT)), s, want_phi=True).cpu().numpy()
    nb.sync_status()
    g = s.acc().cpu().numpy()
    idx = np.array([40, 41])
    f, _, ref = pair_sums(pos, idx)  # that pair's term is all but the whole sum: 1e21 against 1e5
    assert np.all(np.linalg.norm(g[:, idx] - f, axis=0) <= 1e-12 * np.linalg.norm(f, axis=0))
    assert np.all(np.abs(phi[idx] - ref) <= 1e-13 * ref)


# ---------------------------------------------------------------------------
# Flat and offset clouds: every component within 1e-12 (mixed: 1e-6) of the sum of
# its own terms' magnitudes, |d_c| r^-3.  The pair term is right to 2^-43 of itself
# in FP64 arithmetic and to 2^-46 on the FP32 pipe, the host's sum to 2^-49.


def flat(n, form, amp, seed=0):
    """A chain along z, 6e-4 long, with a transverse amplitude: `plane` in x alone,
    `spread` over 20 decades (most coordinates cut), `offset` on x = 1e-4, `seed`
    one displaced ion, its neighbours following with the cube of the distance."""
    rng = np.random.default_rng([n, seed])
    pos = np.zeros((3, n))
    pos[2] = np.sort(rng.uniform(-3e-4, 3e-4, n))
    if form == "plane":
        pos[0] = amp * rng.standard_normal(n)
    elif form == "spread":
        pos[:2] = amp * 10.0 ** rng.uniform(-20, 0, (2, n)) * rng.choice([-1.0, 1.0], (2, n))
    elif form == "offset":
        pos[0] = 1e-4 + amp * rng.standard_normal(n)
        pos[1] = amp * rng.standard_normal(n)
    else:
        pos[1] = amp / np.maximum(1.0, np.abs(np.arange(n) - n // 3)) ** 3
    return pos


def sample(n):
    rng = np.random.default_rng(n)
    return np.unique(np.concatenate([np.arange(min(n, 40)), np.arange(n - 8, n), rng.integers(0, n, 200)]))


def check_components(acc, pos, tol):
    idx = sample(pos.shape[1])
    f, a, _ = pair_sums(pos, idx)
    err = np.abs(acc[:, idx] - f)
    assert np.all(err <= tol * a), float(np.max(err[a > 0] / a[a > 0]))


FORMS = [("plane", 1e-8), ("plane", 1e-12), ("plane", 1e-15), ("plane", 1e-18), ("plane", 1e-21), ("plane", 1e-24),
         ("spread", 1e-9), ("offset", 1e-11), ("offset", 1e-15), ("seed", 1e-9), ("seed", 1e-20)]


@pytest.mark.parametrize("form,amp", FORMS)
@pytest.mark.parametrize("precision,n", [("fp64", 600), ("df64", 1900), ("fp64", 1600), ("df64", 2900), ("fp64", 12500),
                                         ("mixed", 2100), ("mixed", 13000)])
def test_components_of_a_flat_cloud(nb, precision, n, form, amp):
    pos = flat(n, form, amp)
    s = nb.System(pos)
    nb.forces(nb.Params.from_phys(W.phys(**UNIT), precision=precision), s)
    nb.sync_status()
    check_components(s.acc().cpu().numpy(), pos, 1e-6 if precision == "mixed" else 1e-12)


@pytest.mark.parametrize("form,amp", FORMS)
@pytest.mark.parametrize("precision", ["fp64", "df64"])
def test_components_of_a_flat_ensemble(nb, precision, form, amp):
    """One step from rest without a trap: the acceleration is the pair sum at the
    start's positions."""
    sizes = [40, 129, 600, 1100]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    parts = [flat(n, form, amp, seed=k) for k, n in enumerate(sizes)]
    s = nb.System(np.concatenate(parts, axis=1), np.zeros((3, off[-1])))
    nb.step_batched(nb.Params.from_phys(W.phys(**UNIT), precision=precision), s, off, 1)
    nb.sync_status()
    acc = s.acc().cpu().numpy()
    for k, pos in enumerate(parts):
        check_components(acc[:, off[k]:off[k + 1]], pos, 1e-12)


@pytest.mark.parametrize("form,amp", FORMS)
@pytest.mark.parametrize("lam_form,lam_amp", [("plane", 1e-15), ("spread", 1.0), ("offset", 1e-9)])
@pytest.mark.parametrize("n", [2500, 16500])
def test_components_of_a_flat_jacobian_product(nb, n, lam_form, lam_amp, form, amp):
    """g_c = sum_j (dl_c - 3 r^-2 (d . dl) d_c) r^-3, against the magnitudes |dl_c| r^-3
    and 3 |d| |dl| |d_c| r^-5."""
    pos, lam = flat(n, form, amp), flat(n, lam_form, lam_amp, seed=9)
    g = nb.forces_vjp(nb.Params.from_phys(W.phys(**UNIT)), nb.System(pos), lam).cpu().numpy()
    nb.sync_status()
    idx = sample(n)
    for k in range(0, len(idx), 64):
        i = idx[k:k + 64]
        d = pos[:, i, None] - pos[:, None, :]
        dl = lam[:, i, None] - lam[:, None, :]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        with np.errstate(divide="ignore"):
            y = np.where(r2 > 0.0, 1.0 / np.sqrt(r2), 0.0)
        y3 = y * y * y
        t = y3 * (dl - 3.0 * (y * y) * (d * dl).sum(0) * d)
        mag = y3 * (np.abs(dl) + 3.0 * y * np.sqrt((dl * dl).sum(0)) * np.abs(d))
        assert np.all(np.abs(g[:, i] - t.sum(-1)) <= 1e-12 * mag.sum(-1))


# ---------------------------------------------------------------------------
# The ensemble's tasks left to FP64 (btri_task_fp64): every kind of pair of ions a
# task can hold, in instances of one, two and more super-tiles of 128 ions.


def ensemble_once(nb, pos, off, q, soft2, threads, precision):
    """One step from rest without a trap: the pair sums at pos."""
    nb.set_tuning("ensemble", precision, 0, 1 << 40, threads, R=1)
    try:
        s = nb.System(pos, np.zeros_like(pos), q=q)
        nb.step_batched(nb.Params.from_phys(W.phys(soft2=soft2, **UNIT), precision=precision), s, off, 1)
        nb.sync_status()
    finally:
        nb.set_tuning("ensemble", precision, 0, 0, 0)
    return s.acc().cpu().numpy()


@pytest.mark.parametrize("precision", ["fp64", "df64"])
@pytest.mark.parametrize("soft", [0.0, 2e-6])
@pytest.mark.parametrize("charges", [False, True])
@pytest.mark.parametrize("kind", ["close", "coincident", "cut"])
def test_ensemble_tasks_left_to_fp64(nb, kind, charges, soft, precision):
    """Pairs at 2^-42 of the cloud or at no distance, and pairs with a coordinate of
    2^-40 of it: in one 32-ion tile, in one super-tile, across two and three, and in
    an instance of at most 64 ions.  Conditioned error of every ion 1e-12, and the
    bits of 1, 3 and 16 warps."""
    sizes = [20, 64, 128, 200, 300, 513]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    rng = np.random.default_rng(8)
    pos = rng.uniform(-1e-4, 1e-4, (3, off[-1]))
    pos[:, off[:-1] + 1] = 1e-4  # so that every task of super-tile 0 has L > 1e-4
    for k, n in enumerate(sizes):
        for a, b in ((2, 9), (3, 40), (5, 127), (7, 130), (33, 199), (150, 299), (140, 260), (400, 512), (4, 512)):
            if b >= n:
                continue
            i, j = off[k] + a, off[k] + b
            if kind == "cut":
                pos[0, i], pos[0, j] = rng.uniform(1.0, 2.0, 2) * 1e-4 * 2.0 ** -40
            else:
                pos[:, j] = pos[:, i]
                if kind == "close":
                    pos[:, j] += 1e-4 * 2.0 ** -42 * np.array([1.0, -1.0, 0.5])
    q = rng.choice([-1.0, 1.0, 2.0, 0.0], size=off[-1]) if charges else None
    acc = ensemble_once(nb, pos, off, q, soft * soft, 512, precision)
    for threads in (32, 96):
        assert np.array_equal(acc, ensemble_once(nb, pos, off, q, soft * soft, threads, precision))
    for k, n in enumerate(sizes):
        p = pos[:, off[k]:off[k + 1]]
        w = np.ones(n) if q is None else q[off[k]:off[k + 1]]
        d = p[:, :, None] - p[:, None, :]
        r2 = (d * d).sum(0) + soft * soft
        same = np.all(d == 0.0, axis=0)  # coincident ions exert no force on each other
        y = np.where(same, 0.0, 1.0 / np.sqrt(np.where(same, 1.0, r2)))
        t = w * w[:, None] * y ** 3 * d if q is not None else y ** 3 * d
        ref, cond = t.sum(-1), np.sqrt((t * t).sum(0)).sum(-1)
        err = np.sqrt(((acc[:, off[k]:off[k + 1]] - ref) ** 2).sum(0))
        assert np.all(err <= 1e-12 * cond), (n, float(np.max(err / np.maximum(cond, 1e-300))))


# ---------------------------------------------------------------------------
# Residues: a few pairs of cut coordinates in tiles that keep to their words.


def few_cut(n):
    """A chain whose x is zero but for one ion at each end of the index range and six
    close pairs at the edges of tiles and blocks, with x some 2^-40 of theirs; the
    pairs are 3e-9 apart, so that their own x terms lead."""
    rng = np.random.default_rng(n)
    pos = np.zeros((3, n))
    pos[2] = np.sort(rng.uniform(-3e-4, 3e-4, n))
    pos[0, [0, n - 1, n // 2]] = 1e-6, -1.3e-6, 0.9e-6
    pairs = [(5, 40), (31, 32), (63, 64), (100, n - 5), (n - 2, 127), (128, 129)]
    for a, b in pairs:
        pos[2, b] = pos[2, a] + 3e-9
        pos[0, a], pos[0, b] = rng.uniform(1.0, 2.0, 2) * 1e-6 * 2.0 ** -40
    return pos, np.unique(np.array(pairs))


@pytest.mark.parametrize("charges", [False, True])
@pytest.mark.parametrize("precision,n", [("fp64", 700), ("fp64", 1600), ("df64", 2900), ("fp64", 12500), ("mixed", 13000)])
def test_residues_of_a_few_pairs(nb, precision, n, charges):
    pos, idx = few_cut(n)
    q = np.random.default_rng(n).choice([1.0, 2.0, -1.0], size=n) if charges else None
    s = nb.System(pos, q=q)
    nb.forces(nb.Params.from_phys(W.phys(**UNIT), precision=precision), s)
    nb.sync_status()
    g = s.acc().cpu().numpy()
    w = np.ones(n) if q is None else q
    for i in idx:
        d = pos[:, [i]] - pos
        r2 = (d * d).sum(0)
        y = np.where(r2 > 0.0, 1.0 / np.sqrt(np.where(r2 > 0.0, r2, 1.0)), 0.0)
        t = w[i] * w * y ** 3 * d
        tol = 1e-6 if precision == "mixed" else 1e-12
        assert np.all(np.abs(g[:, i] - t.sum(-1)) <= tol * np.abs(t).sum(-1)), i


@pytest.mark.parametrize("charges", [False, True])
@pytest.mark.parametrize("n", [2500, 16500])
def test_residues_of_a_few_pairs_in_the_jacobian_product(nb, n, charges):
    pos, idx = few_cut(n)
    lam, _ = few_cut(n)
    lam[2] = 1e-6 * np.random.default_rng(n).standard_normal(n)
    lam[0] *= 1.7
    q = np.random.default_rng(n).choice([1.0, 2.0, -1.0], size=n) if charges else None
    g = nb.forces_vjp(nb.Params.from_phys(W.phys(**UNIT)), nb.System(pos, q=q), lam).cpu().numpy()
    nb.sync_status()
    w = np.ones(n) if q is None else q
    for i in idx:
        d, dl = pos[:, [i]] - pos, lam[:, [i]] - lam
        r2 = (d * d).sum(0)
        y = np.where(r2 > 0.0, 1.0 / np.sqrt(np.where(r2 > 0.0, r2, 1.0)), 0.0)
        y3 = y * y * y
        t = w[i] * w * y3 * (dl - 3.0 * (y * y) * (d * dl).sum(0) * d)
        mag = np.abs(w[i] * w) * y3 * (np.abs(dl) + 3.0 * y * np.sqrt((dl * dl).sum(0)) * np.abs(d))
        assert np.all(np.abs(g[:, i] - t.sum(-1)) <= 1e-12 * mag.sum(-1)), i


# Coordinates of unlike sign: their l words' difference has 25 bits, one more than
# FP32.  The transverse terms lead where a pair is this close.


def crossing(n, gap):
    """A chain with pairs, gap apart, that straddle x = 0 at 2^-43 of the largest x; no
    other ion is near x = 0."""
    rng = np.random.default_rng([n, 1])
    pos = np.zeros((3, n))
    pos[2] = np.sort(rng.uniform(-3e-4, 3e-4, n))
    pos[0] = rng.uniform(0.5, 1.0, n) * 1e-6 * rng.choice([-1.0, 1.0], n)
    pairs = np.array([(5, 40), (31, 32), (63, 64), (100, n - 5), (n - 2, 127), (128, 129)])
    pos[2, pairs[:, 1]] = pos[2, pairs[:, 0]] + gap
    pos[0, pairs] = rng.uniform(1.0, 2.0, (6, 2)) * 1e-6 * 2.0 ** -43 * [1.0, -1.0]
    return pos, np.unique(pairs)


@pytest.mark.parametrize("charges", [False, True])
@pytest.mark.parametrize("precision,n", [("fp64", 700), ("df64", 2900), ("fp64", 12500), ("ensemble", 700)])
def test_pairs_across_an_axis(nb, precision, n, charges):
    pos, idx = crossing(n, 4e-15)
    q = np.random.default_rng(n).choice([1.0, 2.0, -1.0], size=n) if charges else None
    if precision == "ensemble":
        g = ensemble_once(nb, pos, np.array([0, n]), q, 0.0, 512, "fp64")
    else:
        s = nb.System(pos, q=q)
        nb.forces(nb.Params.from_phys(W.phys(**UNIT), precision=precision), s)
        nb.sync_status()
        g = s.acc().cpu().numpy()
    w = np.ones(n) if q is None else q
    for i in idx:
        d = pos[:, [i]] - pos
        r2 = (d * d).sum(0)
        y = np.where(r2 > 0.0, 1.0 / np.sqrt(np.where(r2 > 0.0, r2, 1.0)), 0.0)
        t = w[i] * w * y ** 3 * d
        assert np.all(np.abs(g[:, i] - t.sum(-1)) <= 1e-12 * np.abs(t).sum(-1)), i


def test_pairs_across_an_axis_of_the_jacobian_product(nb):
    n = 2500
    pos, idx = crossing(n, 1e-10)
    lam = pos * [[1.7], [0.0], [1.0]]
    g = nb.forces_vjp(nb.Params.from_phys(W.phys(**UNIT)), nb.System(pos), lam).cpu().numpy()
    nb.sync_status()
    for i in idx:
        d, dl = pos[:, [i]] - pos, lam[:, [i]] - lam
        r2 = (d * d).sum(0)
        y = np.where(r2 > 0.0, 1.0 / np.sqrt(np.where(r2 > 0.0, r2, 1.0)), 0.0)
        y3 = y * y * y
        t = y3 * (dl - 3.0 * (y * y) * (d * dl).sum(0) * d)
        mag = y3 * (np.abs(dl) + 3.0 * y * np.sqrt((dl * dl).sum(0)) * np.abs(d))
        assert np.all(np.abs(g[:, i] - t.sum(-1)) <= 1e-12 * mag.sum(-1)), i
