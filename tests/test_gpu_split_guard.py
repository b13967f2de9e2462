"""Sums over rows of wide range: where one operand's entries are large the
other's are small, so that what the sum consists of lies far below the rows'
largest entries.  The tensor-core forms hold every entry to 2^-56 of its row's
largest only; their results have to keep FP64's accuracy all the same.

Bound: a sum of n complex products in FP64, in any order, is off by at most
2 (n + 2) 2^-53 sum |a| |b|; chained sums add their factors.
"""
import numpy as np
import pytest

from oracle import bse_oracle as O
from paper_1601_07728_gb300 import bse, synth as S

pytestmark = pytest.mark.gpu
U64 = 2.0 ** -53


def graded_system(nk, nx, nb, na, npj, decades, ks=(0.0, 0.0, 0.0), seed=1, every=2):
    """Two groups of bands (each `every`-th one, the rest), each `decades` smaller on the other's half of the grid."""
    s = S.make_system_from(dict(id=971, n_alpha=na, nk=nk, n_bands=nb, nx=nx, cell=7.4, eps=5.0, n_proj=npj,
                                so_split=5.7, m_scale=0.5, kshift=ks), seed)
    s.chi = np.zeros_like(s.chi)   # no coupling that would lift the small entries
    if npj:
        s.a_proj = s.a_proj * 0.0
    half = np.arange(s.n_x) < s.n_x // 2
    group = np.arange(nb) % every == 0
    s.u = s.u * np.where(half[:, None] == group[None, :], 1.0, 10.0 ** -decades)
    return s, group


def apply_bound(s, psi):
    """(2 (n_b + 2) + 2 (n_x + 2) + 2 (n_k + 8)) 2^-53 |U|^H |W| |U| |psi|, the k sums from |phi| and |W|."""
    a = np.abs(s.u)
    p = np.abs(psi.reshape(s.n_alpha, s.n_k, s.n_bands))
    phi = np.einsum("kxn,akn->akx", a, p)
    conv = np.abs(s.w_rx).sum(0)[None, :] * phi.sum(1) / s.n_k
    out = np.einsum("kxn,ax->akn", a, conv) + np.abs(s.e_nk)[None] * p
    return (2 * (s.n_bands + s.n_x + s.n_k) + 40) * U64 * out.reshape(-1)


# one block of bands and several, the grid split over blocks and not, 1 to 12
# columns (two passes of eight), bands beyond one accumulator of 128 reals
@pytest.mark.parametrize("decades", [4, 12, 20])
@pytest.mark.parametrize("case", [((2, 1, 1), (16, 9, 11), 24, 6, 1), ((1, 1, 1), (16, 16, 16), 40, 1, 1),
                                  ((2, 2, 1), (13, 10, 10), 150, 6, 2)])
def test_graded_bands_keep_fp64_accuracy(case, decades):
    nk, nx, nb, na, nv = case
    s, group = graded_system(nk, nx, nb, na, 0, decades)
    rng = np.random.default_rng(decades)
    psi = S.complex_normal(rng, (nv, na, s.n_k, nb)) * group * 10.0 ** -(np.arange(nb) % 6.0)
    psi = psi.reshape(nv, -1)
    out = bse.System(s, precision="fp64", max_vec=nv).apply_h(psi)
    for v in range(nv):
        assert np.all(np.abs(out[v] - O.apply_h(s, psi[v])) <= 2 * apply_bound(s, psi[v]))


def test_few_graded_bands_keep_fp64_accuracy():
    """One band in 24: grid->band's sums are formed again one at a time, not by warps."""
    s, group = graded_system((2, 2, 1), (13, 10, 10), 150, 6, 0, 12, every=24)
    rng = np.random.default_rng(24)
    for part in (group, ~group):
        psi = (S.complex_normal(rng, (1, 6, s.n_k, 150)) * part).reshape(1, -1)
        out = bse.System(s, precision="fp64").apply_h(psi)[0]
        assert np.all(np.abs(out - O.apply_h(s, psi[0])) <= 2 * apply_bound(s, psi[0]))


def test_sparse_real_and_empty_columns():
    """Columns of one entry, of real entries (with real Bloch functions: no
    imaginary part at all) and of zeros, beside full ones."""
    s, _ = graded_system((1, 1, 1), (16, 16, 16), 32, 6, 0, 0)
    s.u = s.u.real.astype(complex)
    rng = np.random.default_rng(5)
    psi = S.complex_normal(rng, (6, 1, 32))
    psi[0] = 0
    psi[1] = 0
    psi[1, 0, 7] = 1e-5
    psi[2] = psi[2].real
    psi = psi.reshape(1, -1)
    h = bse.System(s, precision="fp64")
    out = h.apply_h(psi)[0]
    assert np.all(np.abs(out - O.apply_h(s, psi[0])) <= 2 * apply_bound(s, psi[0]))
    assert np.all(out[:32] == 0) and np.all(out[64:96].imag == 0)
    h.profile()
    h.apply_h(psi)
    assert h.profile_read()["prep"][0] == 2   # digits of psi and phi: the split kernels


@pytest.mark.parametrize("power", [-1000, -965, 1000])
def test_columns_of_extreme_scale_keep_fp64_accuracy(power):
    s, _ = graded_system((2, 1, 1), (16, 9, 11), 24, 6, 0, 3)
    psi = S.make_start_vectors(s, 1)
    scale = 2.0 ** power
    out = bse.System(s, precision="fp64").apply_h(psi * scale)[0]
    ref = O.apply_h(s, psi[0])
    # 2^-1074: what subnormal products and sums lose at the smallest scale
    assert np.all(np.abs(out / scale - ref) <= 2 * apply_bound(s, psi[0]) + 1e5 * 2.0 ** (-1074 - power))


def test_non_finite_entries_reach_what_they_reached_in_fp64():
    s, _ = graded_system((1, 1, 1), (16, 16, 16), 32, 6, 0, 0)
    psi = S.make_start_vectors(s, 1)
    h = bse.System(s, precision="fp64")
    ref = h.apply_h(psi)[0].reshape(6, 32)
    psi[0, 32 + 3] = np.inf   # core state 1, band 3
    out = h.apply_h(psi)[0].reshape(6, 32)
    assert not np.any(np.isfinite(out[1]))
    others = np.ix_([0, 2, 3, 4, 5], [n for n in range(32) if n != 3])   # 0 * inf of the spin-orbit term in band 3
    assert np.array_equal(out[others], ref[others])


# ---------------------------------------------------------------------------
# set-up projection (csrc/k_oz.cu)
# ---------------------------------------------------------------------------
def projection_bound(u, nk, f, dv):
    """2 (n_x + 16) 2^-53 dv |f| |u|: the sum's products, and the phases' three factors in each."""
    return 2 * (f.shape[1] + 16) * U64 * dv * np.einsum("px,kxn->pkn", np.abs(f), np.abs(u))


# some elements of the call (listed and formed again), most of them (the FP64
# kernel for all), a grid in several parts and one that ends inside a K block,
# more functions than one pass of the magnitudes takes
@pytest.mark.parametrize("decades", [10, 18])
@pytest.mark.parametrize("shape", [((3, 3, 3), (11, 11, 11), 64, 36, 10, 6), ((3, 3, 3), (11, 11, 11), 64, 36, 64, 36),
                                   ((2, 1, 1), (17, 16, 15), 130, 70, 6, 5), ((1, 1, 1), (24, 24, 24), 65, 16, 8, 1)])
def test_projection_of_graded_functions_keeps_fp64_accuracy(shape, decades):
    nk, nx, nb, npj, bands, functions = shape
    n, m = int(np.prod(nk)), int(np.prod(nx))
    rng = np.random.default_rng(m + bands)
    u, f = S.complex_normal(rng, (n, m, nb)), S.complex_normal(rng, (npj, m))
    rise = 10.0 ** (-decades * np.linspace(0, 1, m))
    u[:, :, :bands] *= rise[None, :, None]
    f[-functions:] *= rise[::-1]
    a = bse.local_projection(u, nk, nx, f, 0.3, (0.0, 0.25, 0.5))
    ref = O.local_projection(u, nk, nx, f, 0.3, (0.0, 0.25, 0.5))
    assert np.all(np.abs(a - ref) <= 2 * projection_bound(u, nk, f, 0.3))


def test_only_the_refused_elements_of_a_projection_leave_the_tensor_cores(monkeypatch):
    nk, nx, nb, npj = (3, 3, 3), (11, 11, 11), 64, 36
    rng = np.random.default_rng(3)
    u, f = S.complex_normal(rng, (27, 1331, nb)), S.complex_normal(rng, (npj, 1331))
    flat = bse.local_projection(u, nk, nx, f, 0.3)
    rise = 10.0 ** (-12 * np.linspace(0, 1, 1331))
    u[:, :, 5] *= rise[None, :]
    f[7] *= rise[::-1]
    f[9] = 0
    f[11, 700:] = 0
    u[:, :700, 40] = 0
    a = bse.local_projection(u, nk, nx, f, 0.3)
    monkeypatch.setenv("BSE_SPLIT_WAIT_NS", "1000")   # gives up: the FP64 kernel
    fp64 = bse.local_projection(u, nk, nx, f, 0.3)
    rows, cols = [p for p in range(npj) if p not in (7, 9, 11)], [n for n in range(nb) if n not in (5, 40)]
    same = np.ix_(rows, range(27), cols)
    assert np.array_equal(a[same], flat[same]) and np.mean(a[same] == fp64[same]) < 0.1
    assert np.all(a[9] == 0) and np.all(a[11, :, 40] == 0)
    bound = projection_bound(u, nk, f, 0.3)
    assert np.all(np.abs(a - O.local_projection(u, nk, nx, f, 0.3)) <= 2 * bound)


@pytest.mark.parametrize("power", [-390, -130, 130, 390])
def test_projection_of_functions_of_any_scale(power):
    """Magnitudes far outside FP32's range on either side, per column of u and row of f."""
    nk, nx, nb, npj = (3, 3, 3), (11, 11, 11), 64, 36
    rng = np.random.default_rng(power + 400)
    u, f = S.complex_normal(rng, (27, 1331, nb)), S.complex_normal(rng, (npj, 1331))
    a = bse.local_projection(u * 2.0 ** power, nk, nx, f * 2.0 ** -power, 0.3)
    assert np.array_equal(a, bse.local_projection(u, nk, nx, f, 0.3))


# ---------------------------------------------------------------------------
# Green's functions (csrc/k_oz.cu, csrc/k_screen.cu)
# ---------------------------------------------------------------------------
def green_case(nr, ns, nt, graded, decades, seed):
    """`graded` points where psi falls off over the states, as many where it rises."""
    psi, eps = S.screening_grid_states(nr, ns, seed=seed)
    rise = 10.0 ** (-decades * np.linspace(0, 1, ns))
    psi[:graded] *= rise
    psi[-graded:] *= rise[::-1]
    t = np.linspace(0.3, 5.0, nt)
    return psi, eps, t, np.full(nt, 0.7)


def green_bound(psi, eps, t):
    d = 1 / np.abs(0.1234 + 1j * t[:, None] - eps[None])
    return 2 * (psi.shape[1] + 16) * U64 * np.einsum("rs,js,qs->jrq", np.abs(psi), d, np.abs(psi), optimize=True)


# few elements, more than one in 32, rows at and past the 128-row tile (both
# sides of the diagonal), several K blocks and part of one
@pytest.mark.parametrize("decades", [10, 18])
@pytest.mark.parametrize("shape", [(129, 287, 3, 9), (256, 130, 1, 20), (300, 513, 2, 150), (140, 4001, 1, 5)])
def test_green_functions_of_graded_states_keep_fp64_accuracy(shape, decades):
    nr, ns, nt, graded = shape
    psi, eps, t, w = green_case(nr, ns, nt, graded, decades, nr)
    _, g = bse.screening_chi0(psi, eps, 0.1234, t, w, want_green=True)
    assert np.all(np.abs(g - O.screening_green(psi, eps, 0.1234, t)) <= 2 * green_bound(psi, eps, t))


def test_only_the_refused_green_functions_leave_the_tensor_cores(monkeypatch):
    psi, eps, t, w = green_case(300, 513, 2, 3, 0, 11)
    _, flat = bse.screening_chi0(psi, eps, 0.1234, t, w, want_green=True)
    psi, eps, t, w = green_case(300, 513, 2, 3, 14, 11)
    psi[50] = 0
    psi[60, :300] = 0
    psi[70, 300:] = 0
    _, g = bse.screening_chi0(psi, eps, 0.1234, t, w, want_green=True)
    monkeypatch.setenv("BSE_SPLIT_WAIT_NS", "1000")   # gives up: the FP64 kernel
    _, fp64 = bse.screening_chi0(psi, eps, 0.1234, t, w, want_green=True)
    rows = [r for r in range(3, 297) if r not in (50, 60, 70)]
    same = np.ix_(range(2), rows, rows)
    assert np.array_equal(g[same], flat[same]) and np.mean(g[same] == fp64[same]) < 0.1
    assert np.all(g[:, 50] == 0) and np.all(g[:, :, 50] == 0) and np.all(g[:, 60, 70] == 0)
    assert np.all(np.abs(g - O.screening_green(psi, eps, 0.1234, t)) <= 2 * green_bound(psi, eps, t))


def test_green_functions_of_states_that_the_first_look_misses(monkeypatch):
    """States with weight only where every fourth block of 32 is not: the look
    at part of the magnitudes refuses everything, the one at all of them nothing."""
    psi, eps, t, w = green_case(140, 2400, 1, 1, 0, 17)
    psi[:, np.arange(2400) // 32 % 4 == 0] = 0
    _, g = bse.screening_chi0(psi, eps, 0.1234, t, w, want_green=True)
    monkeypatch.setenv("BSE_SPLIT_WAIT_NS", "1000")   # gives up: the FP64 kernel
    _, fp64 = bse.screening_chi0(psi, eps, 0.1234, t, w, want_green=True)
    assert np.mean(g == fp64) < 0.1
    assert np.all(np.abs(g - O.screening_green(psi, eps, 0.1234, t)) <= 2 * green_bound(psi, eps, t))


def test_projection_of_device_arrays_waits_for_its_own_stream_only():
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(6)
    u = torch.from_numpy(S.complex_normal(rng, (27, 1331, 64))).cuda()
    f = torch.from_numpy(S.complex_normal(rng, (36, 1331))).cuda()
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    done = torch.cuda.Event()

    def call():
        return bse.local_projection(u, (3, 3, 3), (11, 11, 11), f, 0.3, stream=mine.cuda_stream)

    ref = call().clone()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(int(2e9))   # about a second
        done.record()
    out = call()
    assert not done.query()
    assert torch.equal(out, ref)
    torch.cuda.synchronize()


# ---------------------------------------------------------------------------
# the forms that calls take at the ends of the kernels' tiles
# ---------------------------------------------------------------------------
# grid rows at the 128-row tile, one short of it and one past it; enough k points
# and bands for the tensor-core form
@pytest.mark.parametrize("nx", [(127, 1, 1), (8, 4, 4), (3, 43, 1), (1, 5, 51), (4, 8, 8), (257, 1, 1)])
def test_split_contractions_at_the_ends_of_a_row_tile(nx):
    s = S.make_system_from(dict(id=972, n_alpha=6, nk=(5, 4, 4), n_bands=100, nx=nx, cell=7.4, eps=5.0, n_proj=4,
                                so_split=5.7, m_scale=0.5, kshift=(0.1, 0.0, 0.2)), 1)
    psi = S.make_start_vectors(s, 1)
    h = bse.System(s, precision="fp64")
    h.profile()
    out = h.apply_h(psi)[0]
    assert h.profile_read()["prep"][0] == 2   # digits of psi and phi: the split kernels
    ref = O.apply_h(s, psi[0])
    assert np.abs(out - ref).max() <= 1e-13 * np.abs(ref).max()
    assert np.linalg.norm(out - ref) <= 1e-14 * np.linalg.norm(ref)


# the shapes of test_gpu_split_products.py::test_projection_within_the_bound, and
# CTAs that own several whole tiles of more than one band and function
@pytest.mark.parametrize("shape", [((2, 2, 2), (9, 9, 9), 64, 64), ((3, 1, 2), (11, 8, 7), 65, 65),
                                   ((5, 4, 4), (5, 7, 6), 33, 16), ((1, 1, 1), (16, 16, 16), 130, 9),
                                   ((8, 8, 8), (5, 5, 5), 9, 9), ((8, 8, 8), (4, 5, 8), 17, 10)])
def test_projections_that_take_the_split_kernel(monkeypatch, shape):
    nk, nx, nb, npj = shape
    n, m = int(np.prod(nk)), int(np.prod(nx))
    rng = np.random.default_rng(npj * nb)
    u, f = S.complex_normal(rng, (n, m, nb)), S.complex_normal(rng, (npj, m))
    a = bse.local_projection(u, nk, nx, f, 0.37)
    ref = O.local_projection(u, nk, nx, f, 0.37)
    assert np.all(np.abs(a - ref) <= 2 * projection_bound(u, nk, f, 0.37))
    monkeypatch.setenv("BSE_SPLIT_WAIT_NS", "1000")   # gives up: the FP64 kernel
    assert np.mean(bse.local_projection(u, nk, nx, f, 0.37) == a) < 0.1
