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
