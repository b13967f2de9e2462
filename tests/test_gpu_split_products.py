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
