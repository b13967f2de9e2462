"""GMRES's Gram-Schmidt kernels: few systems (sums, norm and second-pass test
inside the two kernels) and many (kernels of their own), systems that finish
at different iterations, and more basis vectors than are staged at a time.
Bound: FP64 recurrences keep the reported residual within 1e-9 |b| of the true
one."""
import numpy as np
import pytest

from oracle import bse_oracle as O
from paper_1601_07728_gb300 import bse, synth as S

pytestmark = pytest.mark.gpu


def system(nk, nx, nb, na):
    return S.make_system_from(dict(id=972, n_alpha=na, nk=nk, n_bands=nb, nx=nx, cell=7.4, eps=5.0, n_proj=4,
                                   so_split=5.7, m_scale=0.5, kshift=(0.0, 0.1, 0.0)), 6)


def residuals(s, b, z, x):
    return np.array([np.linalg.norm(O.apply_h(s, x[j]) - z[j] * x[j] - b) / np.linalg.norm(b) for j in range(len(z))])


# N = 257 and 768 to 12,288 elements; 1 to 64 systems: up to 608 / systems blocks of 256 threads
@pytest.mark.parametrize("shape,n_z", [(((1, 1, 1), (7, 7, 7), 257, 1), 1), (((2, 2, 2), (4, 4, 4), 16, 6), 1),
                                       (((2, 2, 2), (4, 4, 4), 16, 6), 64), (((4, 4, 4), (4, 4, 4), 32, 6), 3),
                                       (((4, 4, 4), (4, 4, 4), 32, 6), 13), (((4, 4, 4), (4, 4, 4), 32, 6), 24)])
def test_shifts_on_both_routes(shape, n_z):
    s = system(*shape)
    b = S.make_start_vectors(s, 1)[0]
    z = np.linspace(-2.0, 12.0, n_z) + 1j * np.geomspace(0.5, 4.0, n_z)
    x, it, rel, st = bse.System(s, precision="fp64", max_vec=min(n_z, 16)).gmres(b, z, rtol=1e-7, restart=25)
    assert st == bse.BSE_OK and np.all(rel <= 1e-7)
    assert np.abs(residuals(s, b, z, x) - rel).max() <= 1e-9


def test_basis_longer_than_the_staged_part():
    s = system((4, 2, 2), (4, 4, 4), 24, 6)
    b = S.make_start_vectors(s, 1)[0]
    z = np.array([6.0 + 1e-4j])
    x, it, rel, st = bse.System(s, precision="fp64").gmres(b, z, rtol=1e-14, restart=600, max_iter=600, precond="none")
    assert it[0] == 600 or rel[0] <= 1e-14
    assert np.abs(residuals(s, b, z, x) - rel).max() <= 1e-9
