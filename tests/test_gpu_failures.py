"""Failure detection on the GPU, made on purpose without faulting it.

* Bounded waits: every wait of the tensor-core pipeline is limited by
  %globaltimer.  With the limit set to 2 microseconds on a full-size L2,3
  launch (each 128-row tile takes several microseconds to stream), waits run
  out; the kernel then stops issuing, waits for its own copies and MMAs in
  flight, frees its tensor memory and returns, and the call reports
  BSE_ERR_TIMEOUT.  The next call on the same handle, with the limit back at
  2 s, must match the oracle.
* Out of memory: BSE_DEVICE_BYTES_LIMIT caps what bse_setup may allocate;
  caps below the handle's needs give BSE_ERR_OOM at different points of the
  set-up, and the device's free memory afterwards equals what it was before
  (nothing leaked).
"""
import numpy as np
import pytest

from oracle import bse_oracle as O
from paper_1601_07728_gb300 import bse, synth as S

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def l23():
    s = S.make_system("l23_multiplet")
    b = S.make_start_vectors(s, 1)
    return s, b, O.apply_h(s, b)


def test_tensor_core_wait_limit_times_out_and_handle_recovers(l23):
    s, b, ref = l23
    sysg = bse.System(s, precision="split_bf16", max_vec=1)
    sysg.set_wait_limit(2e-6)
    with pytest.raises(bse.BSEError) as e:
        sysg.apply_h(b)
    assert e.value.status == bse.BSE_ERR_TIMEOUT
    # the handle is still usable: normal limit, oracle-equal result, twice
    sysg.set_wait_limit(2.0)
    for _ in range(2):
        out = sysg.apply_h(b)
        assert rel(out[0], ref[0]) < 1e-5
        assert np.abs(out[0] - ref[0]).max() <= 1e-4 * np.abs(ref[0]).max()
    a, bc, steps, st = sysg.haydock(b[0], 5)
    assert st == bse.BSE_OK and steps[0] == 5
    sysg.close()


def test_wait_limit_range_checked():
    sysg = bse.System(S.tiny_system(3, n_alpha=1, nk=(2, 2, 2), n_bands=8, nx=(4, 4, 4)), precision="split_bf16")
    for bad in (0.0, 5e-7, 61.0, float("nan")):
        with pytest.raises(bse.BSEError) as e:
            sysg.set_wait_limit(bad)
        assert e.value.status == bse.BSE_ERR_INVALID_ARG
    sysg.close()


def test_device_memory_cap_gives_oom_without_leak(monkeypatch):
    torch = pytest.importorskip("torch")
    s = S.tiny_system(77, n_alpha=6, nk=(4, 4, 4), n_bands=64, nx=(16, 16, 16), n_proj=8)
    psi = S.make_start_vectors(s, 1)
    ref = O.apply_h(s, psi)
    monkeypatch.delenv("BSE_DEVICE_BYTES_LIMIT", raising=False)
    g = bse.System(s, precision="split_bf16")   # loads the device code once, outside the measurement
    g.close()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    # u_nk alone is 268 MB as complex128 staging; the split-bf16 copies another 268 MB
    for cap in (1, 4096, 10 ** 6, 100 * 10 ** 6, 300 * 10 ** 6, 500 * 10 ** 6):
        monkeypatch.setenv("BSE_DEVICE_BYTES_LIMIT", str(cap))
        with pytest.raises(bse.BSEError) as e:
            bse.System(s, precision="split_bf16")
        assert e.value.status == bse.BSE_ERR_OOM, cap
    monkeypatch.setenv("BSE_DEVICE_BYTES_LIMIT", "12x")
    with pytest.raises(bse.BSEError) as e:
        bse.System(s, precision="split_bf16")
    assert e.value.status == bse.BSE_ERR_INVALID_ARG
    monkeypatch.delenv("BSE_DEVICE_BYTES_LIMIT")
    torch.cuda.synchronize()
    free1 = torch.cuda.mem_get_info()[0]
    assert abs(free1 - free0) < 8 * 2 ** 20, (free0, free1)
    # a cap above the need lets the set-up through, with the same result
    monkeypatch.setenv("BSE_DEVICE_BYTES_LIMIT", str(4 * 10 ** 9))
    g = bse.System(s, precision="split_bf16")
    out = g.apply_h(psi)
    g.close()
    assert rel(out[0], ref[0]) < 1e-5


def _raises_timeout(f, *args, **kw):
    with pytest.raises(bse.BSEError) as e:
        f(*args, **kw)
    assert e.value.status == bse.BSE_ERR_TIMEOUT


@pytest.mark.parametrize("precision", ["fp64", "split_bf16"])
def test_every_call_over_h_reports_a_wait_that_gave_up(l23, precision):
    """The tensor-core kernels of the FP64 form and of the split-bf16 form, on a
    size where a tile takes longer than the limit of 2 microseconds: each entry
    point that applies H says BSE_ERR_TIMEOUT, and the call after it, with the
    normal limit, has nothing left to report."""
    torch = pytest.importorskip("torch")
    s, psi, ref = l23
    stream = torch.cuda.Stream()
    sysg = bse.System(s, precision=precision, max_vec=4, stream=stream.cuda_stream)
    net = bse.MLP(S.mlp_init(3))
    r = torch.from_numpy(psi).cuda()
    torch.cuda.synchronize()
    z = np.array([2.0 + 0.5j])
    calls = [lambda: sysg.apply_h(psi), lambda: sysg.haydock(psi[0], 4), lambda: bse.haydock_batch([sysg], [psi], 4),
             lambda: sysg.gmres(psi[0], z, rtol=1e-3, restart=4, max_iter=4),
             lambda: net.loss_grad(sysg, 2.0, 0.5, r, steps=0), lambda: net.loss_grad(sysg, 2.0, 0.5, r, steps=2),
             lambda: net.train([sysg], [psi[0]], z, epochs=1, batch=1, lr=1e-3, steps=1)]
    tol = 1e-13 if precision == "fp64" else 1e-5
    weights = net.params()
    for f in calls:
        sysg.set_wait_limit(2e-6)
        _raises_timeout(f)
        sysg.set_wait_limit(2.0)
        assert rel(sysg.apply_h(psi)[0], ref[0]) < tol
    assert np.array_equal(net.params(), weights)   # no step on a gradient that is none
    outs, sts = bse.haydock_batch([sysg], [psi], 4)
    assert list(sts) == [bse.BSE_OK] and outs[0][2][0] == 4
    sysg.close()


def _projection():
    rng = np.random.default_rng(4)
    u, f = S.complex_normal(rng, (27, 1331, 64)), S.complex_normal(rng, (36, 1331))
    args = (u, (3, 3, 3), (11, 11, 11), f, 0.3)
    return lambda: bse.local_projection(*args), O.local_projection(*args)


def _screening():
    psi, eps = S.screening_grid_states(260, 900, seed=2)
    args = (psi, eps, 0.1, np.array([0.4, 2.0]), np.array([1.0, 0.5]))
    return lambda: bse.screening_chi0(*args), O.screening_chi0(*args)


@pytest.mark.parametrize("case", [_projection, _screening])
def test_set_up_calls_finish_where_a_wait_gives_up(monkeypatch, case):
    """With 1 microsecond for each wait of the tensor-core kernel (a chunk of
    products takes several) it gives up, and the FP64 kernel does the work."""
    f, ref = case()
    monkeypatch.delenv("BSE_SPLIT_WAIT_NS", raising=False)
    split = f()
    monkeypatch.setenv("BSE_SPLIT_WAIT_NS", "1000")
    fp64 = f()
    assert not np.array_equal(split, fp64)   # other sums: it did give up
    monkeypatch.delenv("BSE_SPLIT_WAIT_NS")
    assert np.array_equal(f(), split)        # and left nothing behind
    for out in (split, fp64):
        assert np.abs(out - ref).max() <= 1e-13 * np.abs(ref).max()


def _short_of_memory(torch, leave):
    """All of the device's free memory but `leave` bytes, as an array that nothing touches."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def test_fp64_tables_make_room_for_a_krylov_basis():
    """The FP64 form's tables (64 MB here) are optional: a basis (97 MB) that fits
    the device's remaining 80 MB only without them is solved on the FP64 kernels."""
    torch = pytest.importorskip("torch")
    s = S.tiny_system(31, n_alpha=6, nk=(4, 4, 4), n_bands=64, nx=(16, 16, 16), n_proj=8)
    b = S.make_start_vectors(s, 1)[0]
    z = np.linspace(-3.0, 12.0, 8) + 1j
    stream = torch.cuda.Stream()
    h = bse.System(s, precision="fp64", max_vec=8, stream=stream.cuda_stream)
    x, iters, rel_res, _ = h.gmres(b, z, rtol=1e-8, restart=30, max_iter=30, precond="jacobi")
    a, bc, _, _ = h.haydock(b, 6)
    hold = _short_of_memory(torch, 80 << 20)
    try:
        x2, iters2, _, _ = h.gmres(b, z, rtol=1e-8, restart=30, max_iter=30, precond="jacobi")
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(iters, iters2) and np.abs(x2 - x).max() <= 1e-9 * np.abs(x).max()
    assert rel(h.apply_h(b[None])[0], O.apply_h(s, b)) < 1e-14
    a2, bc2, _, _ = h.haydock(b, 6)   # not the graph over the tables
    np.testing.assert_allclose(a2, a, rtol=1e-11)
    np.testing.assert_allclose(bc2, bc, rtol=1e-11)
    h.close()


def test_fp64_tables_of_a_callers_graph_stay():
    torch = pytest.importorskip("torch")
    s = S.tiny_system(31, n_alpha=6, nk=(4, 4, 4), n_bands=64, nx=(16, 16, 16), n_proj=8)
    psi = torch.from_numpy(S.make_start_vectors(s, 1)).cuda()
    stream = torch.cuda.Stream()
    h = bse.System(s, precision="fp64", max_vec=8, stream=stream.cuda_stream)
    ref, out = h.apply_h(psi, out=torch.empty_like(psi)), torch.empty_like(psi)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        h.apply_h(psi, out=out)
    hold = _short_of_memory(torch, 80 << 20)
    try:
        with pytest.raises(bse.BSEError) as e:
            h.gmres(psi[0].cpu().numpy(), np.linspace(-3.0, 12.0, 8) + 1j, rtol=1e-8, restart=30, max_iter=30)
        assert e.value.status == bse.BSE_ERR_OOM
    finally:
        del hold
        torch.cuda.empty_cache()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    h.close()


@pytest.mark.parametrize("precision", ["fp64", "split_bf16"])
def test_a_wait_that_gave_up_under_a_device_output_is_reported_by_the_next_call(l23, precision):
    torch = pytest.importorskip("torch")
    s, psi, ref = l23
    stream = torch.cuda.Stream()
    sysg = bse.System(s, precision=precision, stream=stream.cuda_stream)
    p = torch.from_numpy(psi).cuda()
    out = torch.empty_like(p)
    torch.cuda.synchronize()
    sysg.set_wait_limit(2e-6)
    sysg.apply_h(p, out=out)
    sysg.set_wait_limit(2.0)
    _raises_timeout(sysg.haydock, psi[0], 2)
    assert rel(sysg.apply_h(psi)[0], ref[0]) < (1e-13 if precision == "fp64" else 1e-5)
    sysg.close()
