"""FP64 products on the tensor cores by exact splitting (csrc/k_oz.cu), through
the two entry points that use them, at the sizes where tiles, K blocks and
chunks end.

Bound of every element, from the scheme: an operand entry is rounded at 2^-56
of 2^e with 2^e at most twice its row's largest magnitude (four times for the
phase-rotated Bloch functions), and the digit products dropped are at most
6.03 per K element of the same size, so

    |error| <= K * 8.03 * 2^-56 * 2^ea * 2^eb <= K * 2^-51 * max|a| * max|b|,

doubled for the comparison's own FP64 sums (and once more for the rotated operand).
"""
import numpy as np
import pytest

from oracle import bse_oracle as O
from paper_1601_07728_gb300 import bse, synth as S

pytestmark = pytest.mark.gpu


def _screening(psi, eps, mu, t, w):
    chi, g = bse.screening_chi0(psi, eps, mu, t, w, want_green=True)
    return chi, g, O.screening_green(psi, eps, mu, t)


def _row_max(m):
    return np.maximum(np.abs(m.real), np.abs(m.imag)).max(axis=-1)


# rows at and around the 128-row tile, states at and around the 64-element K
# block (32 complex states) and the 128-element chunk, one to three frequencies
@pytest.mark.parametrize("shape", [(128, 256, 1), (129, 287, 3), (255, 65, 2), (127, 289, 2), (900, 33, 1),
                                   (65, 1024, 1), (33, 4001, 3)])
def test_green_functions_within_the_bound(shape):
    nr, ns, nt = shape
    assert float(nr) * nr * ns * nt >= 1 << 22
    psi, eps = S.screening_grid_states(nr, ns, seed=7 * nr + ns)
    t, w = np.linspace(0.3, 5.0, nt), np.full(nt, 0.7)
    chi, g, ref = _screening(psi, eps, 0.1234, t, w)
    b = _row_max(psi)
    for j in range(nt):
        a = _row_max(psi / (0.1234 + 1j * t[j] - eps))
        assert np.all(np.abs(g[j] - ref[j]) <= 2 * 2 * ns * 2.0 ** -51 * a[:, None] * b[None, :])
    e = O.screening_chi0(psi, eps, 0.1234, t, w)
    assert np.abs(chi - e).max() <= 1e-12 * np.abs(e).max()


def test_full_digits_do_not_overflow_the_accumulators():
    """Every entry at the largest digit pattern (1 - 2^-53 and its negative):
    the FP32 sums reach their bound, and stay exact."""
    nr, ns = 130, 520
    psi = np.full((nr, ns), (1 - 2.0 ** -53) * (1 + 1j))
    psi[1::2] *= -1
    eps = np.full(ns, -1.0)
    chi, g, ref = _screening(psi, eps, 0.0, np.array([0.0]), np.array([1.0]))   # d = 1
    np.testing.assert_allclose(g, ref, rtol=1e-14, atol=0)


@pytest.mark.parametrize("ns", [63, 64, 65, 128, 255, 256, 520])
def test_accumulators_kept_over_several_chunks_stay_exact(ns):
    """Digits (128, -128, -128, ...): the products of every order reach the
    largest magnitude, and those of order one 2^24 after four chunks."""
    nr = 260
    v = 1 - sum(2.0 ** (-8 * i) for i in range(1, 7))
    psi = np.full((nr, ns), v * (1 + 1j))
    psi[1::2] *= -1
    chi, g, ref = _screening(psi, np.full(ns, -1.0), 0.0, np.array([0.0]), np.array([1.0]))
    np.testing.assert_allclose(g, ref, rtol=1e-14, atol=0)


def test_rows_of_any_scale_and_rows_of_zeros():
    nr, ns = 150, 300
    psi, eps = S.screening_grid_states(nr, ns, seed=3)
    psi *= 2.0 ** np.linspace(-300, 300, nr)[:, None]
    psi[17] = 0
    t, w = np.array([0.8]), np.array([1.0])
    chi, g, ref = _screening(psi, eps, 0.2, t, w)
    a, b = _row_max(psi / (0.2 + 0.8j - eps)), _row_max(psi)
    assert np.all(np.abs(g[0] - ref[0]) <= 4 * ns * 2.0 ** -51 * a[:, None] * b[None, :])
    assert np.all(g[0][17] == 0) and np.all(g[0][:, 17] == 0)


@pytest.mark.parametrize("value", [1e250, np.inf, np.nan])
def test_values_outside_the_scheme_take_the_fp64_kernel(value):
    nr, ns = 140, 260
    psi, eps = S.screening_grid_states(nr, ns, seed=4)
    psi[5, 9] = value
    t, w = np.array([1.5]), np.array([1.0])
    chi, g = bse.screening_chi0(psi, eps, 0.2, t, w, want_green=True)
    hit = np.zeros((nr, nr), bool)
    hit[5, :] = hit[:, 5] = True
    psi[5, 9] = 0
    ref = O.screening_green(psi, eps, 0.2, t)[0]
    assert np.all(np.isfinite(g[0][~hit]))
    assert np.abs(g[0] - ref)[~hit].max() <= 1e-12 * np.abs(ref).max()
    if np.isfinite(value):
        assert np.abs(g[0][hit]).max() > 1e200
    else:
        assert not np.any(np.isfinite(g[0][hit]))


# bands around the 64-column tile, projectors around the 128-row tile (two rows
# each), grids that do not fill a K block, a shifted and a non-cubic mesh
@pytest.mark.parametrize("shape", [((2, 2, 2), (9, 9, 9), 64, 64, (0.0, 0.0, 0.0)),
                                   ((3, 1, 2), (11, 8, 7), 65, 65, (0.25, 0.5, 0.0)),
                                   ((5, 4, 4), (5, 7, 6), 33, 16, (0.0, 0.0, 0.25)),
                                   ((1, 1, 1), (16, 16, 16), 130, 9, (0.0, 0.0, 0.0)),
                                   ((8, 8, 8), (5, 5, 5), 9, 9, (0.0, 0.5, 0.0))])
def test_projection_within_the_bound(shape):
    nk, nx, nb, npj, ks = shape
    assert np.prod(nk) * np.prod(nx) * nb * npj >= 1 << 22
    rng = np.random.default_rng(npj * nb)
    u = S.orthonormal_bloch(rng, int(np.prod(nk)), int(np.prod(nx)), nb)
    f = S.complex_normal(rng, (npj, int(np.prod(nx))))
    a = bse.local_projection(u, nk, nx, f, 0.37, ks)
    ref = O.local_projection(u, nk, nx, f, 0.37, ks)
    um = np.maximum(np.abs(u.real), np.abs(u.imag)).max(axis=1)   # [k][n]
    bound = 4 * 2 * np.prod(nx) * 2.0 ** -51 * 0.37 * _row_max(f)[:, None, None] * um[None]
    assert np.all(np.abs(a - ref) <= bound)
    assert np.linalg.norm(a - ref) <= 1e-14 * np.sqrt(np.prod(nx)) * np.linalg.norm(ref)


def test_projection_with_nan_takes_the_fp64_kernel():
    nk, nx, nb, npj = (2, 2, 2), (9, 9, 9), 40, 20
    rng = np.random.default_rng(8)
    u = S.complex_normal(rng, (8, 729, nb))
    f = S.complex_normal(rng, (npj, 729))
    ref = O.local_projection(u, nk, nx, f, 1.0)
    u[3, 100, 7] = np.nan
    a = bse.local_projection(u, nk, nx, f, 1.0)
    assert not np.any(np.isfinite(a[:, 3, 7]))
    a[:, 3, 7] = ref[:, 3, 7]
    assert np.abs(a - ref).max() <= 1e-12 * np.abs(ref).max()


def test_projection_in_several_passes():
    """More k points than one pass's phases hold; an odd number of blocks a tile."""
    nk, nx = (10, 8, 8), (32, 31, 29)
    rng = np.random.default_rng(12)
    u = rng.standard_normal((640, 32 * 31 * 29, 1)) + 1j * rng.standard_normal((640, 32 * 31 * 29, 1))
    f = S.complex_normal(rng, (1, 32 * 31 * 29))
    a = bse.local_projection(u, nk, nx, f, 0.11, (0.5, 0.0, 0.25))
    ref = O.local_projection(u, nk, nx, f, 0.11, (0.5, 0.0, 0.25))
    um = np.maximum(np.abs(u.real), np.abs(u.imag)).max(axis=1)
    assert np.all(np.abs(a - ref) <= 4 * 2 * np.prod(nx) * 2.0 ** -51 * 0.11 * _row_max(f)[:, None, None] * um[None])
