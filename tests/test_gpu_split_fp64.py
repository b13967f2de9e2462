"""The FP64 form's contractions: the split tensor-core kernels (csrc/k_ozh.cu)
and the FP64-pipe kernels for small problems against the oracle, at sizes
where their tiles end, and what they do with values outside the usual range.

Bound: 1e-13 relative to the largest element, from K <= 2^15 terms per sum at
2^-52 each with every term at the row maximum, would be 7e-12; random signs
leave sqrt(K): 181 * 2.2e-16 * 2 contractions < 1e-13.
"""
import numpy as np
import pytest

from oracle import bse_oracle as O
from paper_1601_07728_gb300 import bse, synth as S

pytestmark = pytest.mark.gpu


def system(nk, nx, nb, na, npj, ks=(0.0, 0.0, 0.0), seed=1):
    return S.make_system_from(dict(id=970, n_alpha=na, nk=nk, n_bands=nb, nx=nx, cell=7.4, eps=5.0, n_proj=npj,
                                   so_split=5.7, m_scale=0.5, kshift=ks), seed)


# grid rows around the 128-row tile and the 32-point block, bands around the
# 64-band tile, the 16-band block and one band, 1 to 20 columns (passes of 8),
# grids split over several blocks and K beyond one accumulator
@pytest.mark.parametrize("case", [
    ((2, 2, 2), (8, 4, 4), 16, 6, 4, 1), ((2, 2, 2), (3, 43, 1), 17, 6, 4, 1), ((2, 1, 2), (11, 9, 7), 64, 6, 9, 2),
    ((3, 2, 5), (11, 8, 13), 65, 4, 16, 2), ((1, 1, 1), (24, 24, 24), 130, 1, 0, 1), ((2, 2, 2), (12, 12, 12), 33, 7, 3, 1),
    ((4, 4, 4), (10, 10, 10), 1, 6, 9, 1), ((2, 2, 1), (29, 29, 29), 48, 9, 5, 1), ((1, 2, 1), (31, 5, 6), 80, 10, 4, 2),
    # FP64-pipe kernels: 1, 2, 3, 5, 7 and 9 columns on small grids
    ((2, 2, 2), (6, 6, 6), 16, 1, 0, 1), ((2, 2, 2), (4, 4, 3), 5, 2, 2, 1), ((2, 3, 1), (5, 5, 3), 70, 1, 0, 3),
    ((1, 1, 1), (4, 4, 3), 9, 5, 4, 1), ((2, 1, 1), (3, 3, 5), 3, 7, 2, 1), ((2, 2, 1), (3, 4, 3), 33, 3, 4, 3)])
def test_fp64_apply_matches_oracle(case):
    nk, nx, nb, na, npj, nv = case
    s = system(nk, nx, nb, na, npj, (0.1, 0.0, 0.2))
    psi = S.make_start_vectors(s, nv)
    psi *= np.logspace(-3, 3, nv)[:, None]
    out = bse.System(s, precision="fp64", max_vec=nv).apply_h(psi)
    for v in range(nv):
        ref = O.apply_h(s, psi[v])
        assert np.abs(out[v] - ref).max() <= 1e-13 * np.abs(ref).max()
        assert np.linalg.norm(out[v] - ref) <= 1e-14 * np.linalg.norm(ref)


@pytest.mark.parametrize("scale", [2.0 ** -900, 2.0 ** 900])
def test_vectors_of_extreme_scale(scale):
    s = system((2, 2, 2), (12, 12, 12), 32, 6, 9)
    psi = S.make_start_vectors(s, 1)
    h = bse.System(s, precision="fp64")
    ref = h.apply_h(psi)
    np.testing.assert_allclose(h.apply_h(psi * scale) / scale, ref, rtol=1e-12, atol=1e-14 * np.abs(ref).max())


def test_zero_and_non_finite_columns():
    s = system((2, 2, 2), (12, 12, 12), 32, 6, 9)
    h = bse.System(s, precision="fp64")
    assert np.all(h.apply_h(np.zeros((1, s.dim), complex)) == 0)
    psi = S.make_start_vectors(s, 1)
    psi[0, 7] = np.nan   # core state 0
    out = h.apply_h(psi)[0]
    assert np.all(np.isnan(out[: s.dim // 6].real))   # its whole column
    psi[0, 7] = np.inf
    assert not np.any(np.isfinite(h.apply_h(psi)[0][: s.dim // 6]))


def test_bloch_functions_outside_the_scheme_keep_the_fp64_kernels():
    s = system((2, 2, 2), (12, 12, 12), 32, 6, 0)
    psi = S.make_start_vectors(s, 1)
    ref = O.apply_h(s, psi[0])
    s.u[0, 0, 0] = 1e200
    out = bse.System(s, precision="fp64").apply_h(psi)[0]
    assert np.abs(out).max() > 1e150
    s.u[0, 0, 0] = np.nan
    assert not np.all(np.isfinite(bse.System(s, precision="fp64").apply_h(psi)[0]))
    assert np.all(np.isfinite(ref))


def test_haydock_in_graph_and_memory_cap(monkeypatch):
    """A captured recursion over the split kernels, and the same under a memory
    cap that leaves no room for their tables (the FP64 kernels)."""
    torch = pytest.importorskip("torch")
    s = system((4, 4, 2), (12, 12, 12), 32, 6, 9)
    b = S.make_start_vectors(s, 1)[0]
    st = torch.cuda.Stream()
    a, bc, n, _ = bse.System(s, precision="fp64", stream=st.cuda_stream).haydock(b, 10)
    u_bytes = s.u.size * 16
    phi = s.n_k * s.n_x * 6 * 16
    monkeypatch.setenv("BSE_DEVICE_BYTES_LIMIT", str(u_bytes + phi + 2_500_000))
    a2, bc2, n2, _ = bse.System(s, precision="fp64", stream=st.cuda_stream).haydock(b, 10)
    np.testing.assert_allclose(a, a2, rtol=1e-11, atol=1e-11)
    np.testing.assert_allclose(bc, bc2, rtol=1e-11)
    ao, bo, _, _ = O.haydock(lambda v: O.apply_h(s, v), b, 10)
    np.testing.assert_allclose(a[0], ao, rtol=1e-10, atol=1e-10)
