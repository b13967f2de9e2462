"""Work that a user of the library has it do, as timed cases.

A case is a dict of plain values; its "kind" names the entry point:

  apply       System.apply_h             H psi on n_vec vectors (the solver's matrix-vector product)
  haydock     System.haydock             an absorption spectrum's recursion, one start vector per polarisation
  sites       haydock_batch              several absorbing sites of uneven size in one call
  gmres       System.gmres               (H - z) x = b for many shifts, with or without preconditioner
  rixs        rixs                       absorption resolvent, emission, final-state recursion
  mlp_grad    MLP.loss_grad              one training sample of the learned preconditioner (forward and backward)
  projection  local_projection           set-up: Bloch functions onto the local basis
  screening   screening_chi0             Green's functions on the imaginary axis and the static chi0

Systems are the seeded synthetic ones of ``synth``, with Bloch functions that
are drawn and orthonormalised on the GPU.  Every array that a program would
already hold on the device (start vectors, solutions) is a CUDA tensor; the
calls that return host arrays return them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1601_07728_gb300 import bse, synth as S

DEV = "cuda"
C128 = torch.complex128


def _shape(nk, nx, nb, na, n_proj, cell=7.4, eps=5.0, kshift=0.0):
    return {"nk0": nk[0], "nk1": nk[1], "nk2": nk[2], "nx0": nx[0], "nx1": nx[1], "nx2": nx[2], "nb": nb, "na": na,
            "n_proj": n_proj, "cell": cell, "eps": eps, "kshift": kshift}


K_EDGE = _shape((2, 2, 2), (8, 8, 8), 16, 1, 0)                       # 1s edge, N = 128
L23 = _shape((8, 8, 8), (16, 16, 16), 64, 6, 36)                      # L2,3 edge with multiplets, N = 196,608
L23R = _shape((4, 4, 4), (8, 8, 8), 32, 6, 36)                        # the same physics on a smaller mesh
SUPERCELL = _shape((2, 2, 2), (48, 48, 48), 1024, 6, 36, 29.5, 6.0)   # 4x4x4-like supercell, N = 49,152


def listed():
    return [
        # the smallest call: one H psi of a 1s edge inside somebody's own solver
        dict(K_EDGE, name="apply_k_edge_fp64", kind="apply", prec="fp64", n_vec=1),
        # the reference-accuracy form on the full L2,3 problem
        dict(L23, name="apply_l23_fp64", kind="apply", prec="fp64", n_vec=1),
        # a supercell: few k points, many bands, a large grid
        dict(SUPERCELL, name="apply_supercell", kind="apply", prec="split_bf16", n_vec=1),
        # the main use: the recursion of one L2,3 spectrum
        dict(L23, name="haydock_l23", kind="haydock", prec="split_bf16", n_vec=1, n_steps=40),
        # three polarisations of the same site advanced together
        dict(L23, name="haydock_l23_3pol", kind="haydock", prec="split_bf16", n_vec=3, n_steps=20),
        # averaging over absorbing sites of uneven size, one call
        dict(name="haydock_sites", kind="sites", prec="split_bf16", first=0, n_sites=4, n_vec=1, n_steps=20),
        # resolvent at many energies at once, two restart cycles
        dict(L23, name="gmres_l23", kind="gmres", prec="split_bf16", n_z=32, precond="none", rtol=1e-6, restart=30,
             max_iter=60),
        # the same to convergence with the learned preconditioner, on a mesh where launches count
        dict(L23R, name="gmres_reduced_mlp", kind="gmres", prec="split_bf16", n_z=16, precond="mlp", rtol=1e-4,
             restart=30, max_iter=600),
        # resonant inelastic scattering with a 3d-shell final state
        dict(L23R, name="rixs_reduced", kind="rixs", prec="split_bf16", n_z=3, n_v=10, n_steps=15, rtol=1e-4),
        # one training sample: four probes, ten Krylov steps, forward and backward
        dict(L23R, name="mlp_grad_reduced", kind="mlp_grad", prec="split_bf16", n_probes=4, steps=10),
        # set-up projection onto the 64 local functions, Bloch functions on the device
        dict(L23, name="projection_l23", kind="projection", n_f=64),
        # screening around the core hole: 36 x 25 grid points, 2^3 k x 512 bands, 16 frequencies
        dict(name="screening_900", kind="screening", n_r=900, n_states=4096, n_t=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_shape(rng, top):
    """A mesh, grid and band count of the range from the 1s edge to `top` reals of u_nk."""
    while True:
        n = rng.choice([2, 3, 4, 4, 5, 6, 7, 8, 8])
        nk = (n, n, n) if rng.random() < 0.75 else (n, rng.randint(1, 6), rng.randint(2, 6))
        m = rng.randint(6, 20)
        nx = (m, m, m) if rng.random() < 0.75 else (m, rng.randint(6, 17), rng.randint(6, 17))
        nb = _log(rng, 8, 200)
        size = 2 * math.prod(nk) * math.prod(nx) * nb
        if nb * 4 <= math.prod(nx) and 1 << 17 <= size <= top:
            break
    na = rng.choice([1, 6, 6, 6, 4])
    return _shape(nk, nx, nb, na, 0 if na == 1 else rng.choice([9, 16, 36, 36, 64]),
                  kshift=rng.choice([0.0, 0.0, 0.25]))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "haydock", "haydock", "sites", "gmres", "gmres", "rixs", "mlp_grad",
                       "projection", "screening"])
    if kind == "apply":
        # fp64 up to half of the L2,3 problem; the reduced forms up to the whole, on one to six vectors
        prec = rng.choice(["fp64", "fp64", "fp32", "split_bf16", "split_bf16"])
        return dict(_draw_shape(rng, 1.4e8 if prec != "split_bf16" else 2.7e8), kind=kind, prec=prec,
                    n_vec=rng.choice([1, 1, 2, 3, 6]))
    if kind == "haydock":
        prec = rng.choice(["fp64", "split_bf16", "split_bf16", "split_bf16"])
        return dict(_draw_shape(rng, 3e7 if prec == "fp64" else 2.7e8), kind=kind, prec=prec,
                    n_vec=rng.choice([1, 1, 1, 2, 3]), n_steps=rng.randint(8, 40))
    if kind == "sites":
        return dict(kind=kind, prec="split_bf16", first=rng.randint(1, 56), n_sites=rng.randint(2, 4), n_vec=1,
                    n_steps=rng.randint(8, 24))
    if kind == "gmres":
        small = rng.random() < 0.5
        pre = rng.choice(["none", "none", "jacobi", "mlp"])
        return dict(_draw_shape(rng, 1e7 if small else 1.4e8), kind=kind, prec=rng.choice(["split_bf16", "split_bf16", "fp32"])
                    if small else "split_bf16", n_z=_log(rng, 4, 40) if small else _log(rng, 3, 24), precond=pre,
                    rtol=1e-4, restart=rng.choice([20, 30]), max_iter=rng.randint(60, 200) if small else 45)
    if kind == "rixs":
        return dict(_draw_shape(rng, 1e7), na=6, n_proj=rng.choice([9, 36]), kind=kind, prec="split_bf16",
                    n_z=rng.randint(2, 6), n_v=rng.choice([4, 10]), n_steps=rng.randint(8, 20), rtol=1e-4)
    if kind == "mlp_grad":
        return dict(_draw_shape(rng, 4e7), kind=kind, prec="split_bf16", n_probes=rng.randint(1, 4),
                    steps=rng.choice([0, 4, 10]))
    if kind == "projection":
        return dict(_draw_shape(rng, 2.7e8), kind=kind, n_f=rng.choice([9, 16, 36, 64]))
    return dict(kind=kind, n_r=_log(rng, 60, 900), n_states=_log(rng, 300, 4096), n_t=rng.randint(6, 16))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 64 + stream) % (1 << 62))
    return g


def _bloch(nk, nx, nb, seed):
    """u_nk(x) [Nk][Nx][Nb] complex128, columns orthonormal per k: complex
    normal values, orthonormalised with the Cholesky factor of their FP32 Gram matrix."""
    g = _gen(seed, 1)
    u = torch.empty((nk, nx, nb), dtype=C128, device=DEV)
    chunk = max(1, int(1.5e8 // (nx * nb)))
    eye = torch.eye(nb, dtype=torch.complex64, device=DEV)
    for k0 in range(0, nk, chunk):
        k1 = min(nk, k0 + chunk)
        a = torch.randn((k1 - k0, nx, nb), dtype=torch.complex64, device=DEV, generator=g)
        r = torch.linalg.cholesky(a.mH @ a, upper=True)
        inv = torch.linalg.solve_triangular(r, eye.expand_as(r), upper=True)
        if nb <= 256:
            u[k0:k1] = a.to(C128) @ inv.to(C128)
        else:   # FP64 products of this size would dominate the drawing
            u[k0:k1] = a @ inv
    return u


def _system(case, seed):
    cfg = dict(id=2, n_alpha=case["na"], nk=(case["nk0"], case["nk1"], case["nk2"]), n_bands=case["nb"],
               nx=(case["nx0"], case["nx1"], case["nx2"]), cell=case["cell"], eps=case["eps"], n_proj=case["n_proj"],
               so_split=5.7, m_scale=0.5, kshift=(case["kshift"],) * 3)
    u = _bloch(math.prod(cfg["nk"]), math.prod(cfg["nx"]), cfg["n_bands"], seed)
    s = S.make_system_from(cfg, site=seed, u=u)
    torch.cuda.synchronize()
    return s


def _vectors(n, dim, seed, stream=2):
    b = torch.randn((n, dim), dtype=C128, device=DEV, generator=_gen(seed, stream))
    return b / torch.linalg.vector_norm(b, dim=1, keepdim=True)


def _site_cases(case):
    out = []
    for i in range(case["n_sites"]):
        c = S.batched_site_config(case["first"] + i)
        out.append(_shape(c["nk"], c["nx"], c["n_bands"], c["n_alpha"], c["n_proj"]))
    return out


def _shifts(case):
    return np.linspace(-5.0, 30.0, case["n_z"]) + 0.5j


def _params(seed):
    """Network weights as training leaves them: the seeded start with every layer in use."""
    p = S.mlp_init(int(seed) % 1000)
    rng = np.random.default_rng([7, int(seed)])
    w3 = p[-(128 * 34 + 34):-34].reshape(128, 34)
    w3 += (0.01 * rng.standard_normal((128, 34))).astype(np.float32)
    return p


def _valence(s, case, seed):
    val, d = S.valence_final_state(s, n_v=case["n_v"], seed=int(seed) % 1000)
    return val, d


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "screening":
        psi, eps = S.screening_grid_states(case["n_r"], case["n_states"], seed=seed)
        t, w = S.imag_axis_quadrature(case["n_t"])
        mu = 0.5 * (np.sort(eps)[case["n_states"] // 2 - 1] + np.sort(eps)[case["n_states"] // 2])
        st.update(psi=psi, eps=eps, mu=float(mu), t=t, w=w)
        return st
    if kind == "sites":
        st["systems"], st["bs"] = [], []
        for i, c in enumerate(_site_cases(case)):
            s = _system(c, 8 * seed + i)
            h = bse.System(s, precision=case["prec"], max_vec=case["n_vec"],
                           stream=st.setdefault("streams", [torch.cuda.Stream() for _ in range(case["n_sites"])])[i].cuda_stream)
            st["systems"].append(h)
            st["bs"].append(_vectors(case["n_vec"], h.dim, 8 * seed + i))
        return st
    if kind == "projection":
        nk, nx = (case["nk0"], case["nk1"], case["nk2"]), (case["nx0"], case["nx1"], case["nx2"])
        f = S.local_functions_on_grid(nx, case["cell"], 3.0, seed=seed % 1000)[:case["n_f"]]
        st.update(u=_bloch(math.prod(nk), math.prod(nx), case["nb"], seed), f=torch.from_numpy(f.copy()).to(DEV), nk=nk,
                  nx=nx, dv=case["cell"] ** 3 / math.prod(nx))
        return st
    s = _system(case, seed)
    st["stream"] = torch.cuda.Stream()
    stream = st["stream"].cuda_stream
    if kind == "rixs":
        val, d = _valence(s, case, seed)
        st["core"] = bse.System(s, precision=case["prec"], max_vec=case["n_z"], stream=stream)
        st["val"] = bse.System(val, precision=case["prec"], max_vec=case["n_z"], stream=stream)
        st.update(d=d, b=_vectors(1, s.dim, seed)[0].cpu().numpy(), z=np.linspace(2.0, 14.0, case["n_z"]) + 0.5j)
        return st
    columns = case.get("n_vec") or case.get("n_z") or case.get("n_probes")
    h = bse.System(s, precision=case["prec"], max_vec=columns, stream=stream)
    st["h"] = h
    if kind == "apply":
        st["psi"] = _vectors(case["n_vec"], h.dim, seed)
        st["out"] = torch.empty_like(st["psi"])
    elif kind == "haydock":
        st["b"] = _vectors(case["n_vec"], h.dim, seed)
    elif kind == "gmres":
        st["b"] = _vectors(1, h.dim, seed)[0]
        st["z"] = _shifts(case)
        st["x"] = torch.empty((case["n_z"], h.dim), dtype=C128, device=DEV)
        if case["precond"] == "mlp":
            st["net"] = bse.MLP(_params(seed))
            bse.attach_mlp(h, st["net"])
    elif kind == "mlp_grad":
        st["net"] = bse.MLP(_params(seed))
        st["r"] = _vectors(case["n_probes"], h.dim, seed)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "apply":
        return st["h"].apply_h(st["psi"], out=st["out"])
    if kind == "haydock":
        a, b, n, _ = st["h"].haydock(st["b"], case["n_steps"])
        return {"a": a, "b": b, "steps": n}
    if kind == "sites":
        outs, _ = bse.haydock_batch(st["systems"], st["bs"], case["n_steps"])
        return [{"a": a, "b": b, "steps": n} for a, b, n in outs]
    if kind == "gmres":
        x, iters, rel, _ = st["h"].gmres(st["b"], st["z"], rtol=case["rtol"], restart=case["restart"],
                                         max_iter=case["max_iter"], precond=case["precond"], x=st["x"])
        return {"x": x, "iters": iters, "rel": rel}
    if kind == "rixs":
        a, b, n, iters, rel, _ = bse.rixs(st["core"], st["val"], st["b"], st["z"], st["d"], case["n_steps"],
                                          rtol=case["rtol"])
        return {"a": a, "b": b, "steps": n, "iters": iters, "rel": rel}
    if kind == "mlp_grad":
        loss, g = st["net"].loss_grad(st["h"], 10.8, 0.5, st["r"], steps=case["steps"])
        return {"loss": loss, "grad": g}
    if kind == "projection":
        return bse.local_projection(st["u"], st["nk"], st["nx"], st["f"], st["dv"], kshift=(case["kshift"],) * 3)
    return bse.screening_chi0(st["psi"], st["eps"], st["mu"], st["t"], st["w"])


# ---------------------------------------------------------------------------
# bytes and operations that a pass cannot do without
# ---------------------------------------------------------------------------
def _apply_work(c, n_vec, prec):
    nk, nx = c["nk0"] * c["nk1"] * c["nk2"], c["nx0"] * c["nx1"] * c["nx2"]
    nb, na, npj = c["nb"], c["na"], c["n_proj"]
    cols = na * n_vec
    real = 8 if prec == "fp64" else 4
    u = 2 * real * nk * nx * nb
    small = real * nk * nx + 8 * nk * nb + 16 * na * na + 2 * real * npj * nk * nb + 16 * (na * npj) ** 2
    vec = 32 * cols * nk * nb
    flops = 16 * nk * nx * nb * cols + 10 * nk * max(1.0, math.log2(nk)) * nx * cols + 16 * npj * nk * nb * cols
    return u + small, vec, flops


def work(case):
    kind = case["kind"]
    if kind == "screening":
        r, k, t = case["n_r"], case["n_states"], case["n_t"]
        return {"bytes": 16 * r * k + 16 * r * r, "flops": 8 * r * r * k * t + 8 * r * r * t}
    if kind == "projection":
        nk, nx = case["nk0"] * case["nk1"] * case["nk2"], case["nx0"] * case["nx1"] * case["nx2"]
        return {"bytes": 16 * (nk * nx * case["nb"] + case["n_f"] * (nx + nk * case["nb"])),
                "flops": 8 * nk * nx * case["nb"] * case["n_f"]}
    if kind == "sites":
        b = f = 0
        for c in _site_cases(case):
            u, vec, fl = _apply_work(c, case["n_vec"], case["prec"])
            b += case["n_steps"] * (u + vec)
            f += case["n_steps"] * fl
        return {"bytes": b, "flops": f}
    if kind == "apply":
        u, vec, fl = _apply_work(case, case["n_vec"], case["prec"])
        return {"bytes": u + vec, "flops": fl}
    if kind == "haydock":
        u, vec, fl = _apply_work(case, case["n_vec"], case["prec"])
        return {"bytes": case["n_steps"] * (u + vec), "flops": case["n_steps"] * fl}
    n = case["na"] * case["nk0"] * case["nk1"] * case["nk2"] * case["nb"]
    if kind == "gmres":
        # max_iter H applications of every shift and one Gram-Schmidt pass over the basis of each step
        u, vec, fl = _apply_work(case, case["n_z"], case["prec"])
        it, m = case["max_iter"] if case["rtol"] < 1e-5 else min(60, case["max_iter"]), case["restart"]
        return {"bytes": it * (u + vec + 16 * case["n_z"] * n * (m + 1) / 2),
                "flops": it * (fl + 16 * case["n_z"] * n * (m + 1) / 2)}
    if kind == "rixs":
        u, vec, fl = _apply_work(case, case["n_z"], case["prec"])
        uv, vv, fv = _apply_work(dict(case, na=case["n_v"]), case["n_z"], case["prec"])
        return {"bytes": 60 * (u + vec) + case["n_steps"] * (uv + vv), "flops": 60 * fl + case["n_steps"] * fv}
    u, vec, fl = _apply_work(case, case["n_probes"], case["prec"])
    it = 2 * max(1, case["steps"])
    net = 12 * 128 + 128 * 128 + 128 * 34
    return {"bytes": it * (u + vec) + 4 * n * (12 + 34) * 3, "flops": it * fl + 6 * n * net}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------
class _Plain:
    """H in complex128 with torch matmul and FFT; vectors [V][N]."""

    def __init__(self, s):
        self.s = s
        dev = lambda a: torch.as_tensor(a).to(DEV)  # noqa: E731
        self.nk, self.nx, self.na, self.nb = s.nk, s.nx, s.n_alpha, s.n_bands
        j = np.stack(np.meshgrid(*[np.arange(n) for n in s.nx], indexing="ij"), -1).reshape(-1, 3) / np.asarray(s.nx)
        m = np.stack(np.meshgrid(*[np.arange(n) for n in s.nk], indexing="ij"), -1).reshape(-1, 3)
        k = (m + np.asarray(s.kshift)) / np.asarray(s.nk)
        self.u = dev(s.u) * torch.exp(2j * math.pi * dev(k @ j.T)).unsqueeze(-1)
        self.e, self.chi, self.w = dev(s.e_nk), dev(s.chi), dev(s.w_rx)
        self.a = None if s.a_proj is None else dev(s.a_proj).reshape(s.n_proj, -1)
        self.m = None if s.a_proj is None else dev(s.m_sr)

    def _conv(self, phi):
        """phi [Nk][Nx][C] -> R->k of W times k->R"""
        f = phi.reshape(*self.nk, *phi.shape[1:])
        f = torch.fft.ifftn(f, dim=(0, 1, 2), norm="forward")
        f = f * self.w.reshape(*self.nk, -1, 1)
        return torch.fft.fftn(f, dim=(0, 1, 2), norm="forward").reshape(phi.shape)

    def apply(self, psi):
        v = psi.shape[0]
        p = psi.reshape(v, self.na, len(self.e), self.nb)
        cols = p.permute(2, 3, 0, 1).reshape(len(self.e), self.nb, v * self.na)
        out = torch.empty_like(cols)
        step = max(1, int(2.5e8 // (self.u.shape[0] * self.u.shape[1])))
        for c in range(0, cols.shape[2], step):
            out[:, :, c:c + step] = self.u.mH @ self._conv(self.u @ cols[:, :, c:c + step])
        out = out.reshape(len(self.e), self.nb, v, self.na).permute(2, 3, 0, 1)
        out = out + self.e * p - torch.einsum("ab,vbkn->vakn", self.chi, p)
        if self.a is not None:
            c = torch.einsum("pi,vai->vap", self.a, p.reshape(v, self.na, -1)).reshape(v, -1) @ self.m.T
            out = out + torch.einsum("pi,vap->vai", self.a.conj(), c.reshape(v, self.na, -1)).reshape(p.shape)
        return out.reshape(psi.shape)

    def diag(self):
        lr = torch.einsum("kxn,x->kn", self.u.abs() ** 2, self.w.mean(0))
        d = (self.e + lr).unsqueeze(0) - torch.diagonal(self.chi).real.reshape(-1, 1, 1)
        if self.a is not None:
            np_ = self.a.shape[0]
            m = self.m.reshape(self.na, np_, self.na, np_)
            blk = torch.stack([m[a, :, a, :] for a in range(self.na)])
            d = d + torch.einsum("pi,apq,qi->ai", self.a.conj(), blk, self.a).real.reshape(d.shape)
        return d.reshape(-1)


def _lanczos(apply, b, steps):
    """Haydock coefficients of every row of b."""
    v = b.shape[0]
    a, bc = np.zeros((v, steps)), np.zeros((v, steps + 1))
    nrm = torch.linalg.vector_norm(b, dim=1)
    bc[:, 0] = nrm.cpu().numpy()
    cur, prev = b / nrm[:, None], torch.zeros_like(b)
    for i in range(steps):
        w = apply(cur)
        ai = (cur.conj() * w).sum(1).real
        w = w - ai[:, None] * cur - (nrm[:, None] * prev if i else 0.0)
        nrm = torch.linalg.vector_norm(w, dim=1)
        a[:, i], bc[:, i + 1] = ai.cpu().numpy(), nrm.cpu().numpy()
        prev, cur = cur, w / nrm[:, None]
    return a, bc


def _solve(apply, pre, b, z, rtol, restart=40, cycles=60):
    """x of (H - z) x = b for every z to rtol: restarted GMRES of all shifts together; None if it stalls."""
    z = torch.as_tensor(z, device=DEV)
    n = len(z)
    x = torch.zeros((n, b.numel()), dtype=C128, device=DEV)
    for _ in range(cycles):
        r = b - apply(x) + z[:, None] * x
        beta = torch.linalg.vector_norm(r, dim=1)
        if float(beta.max()) <= rtol * float(torch.linalg.vector_norm(b)):
            return x
        basis = torch.empty((n, restart + 1, b.numel()), dtype=C128, device=DEV)
        hess = torch.zeros((n, restart + 1, restart), dtype=C128, device=DEV)
        basis[:, 0] = r / beta[:, None]
        for j in range(restart):
            t = pre(basis[:, j])
            w = apply(t) - z[:, None] * t
            for _ in range(2):
                c = (basis[:, :j + 1].conj() @ w.unsqueeze(-1)).squeeze(-1)
                hess[:, :j + 1, j] += c
                w = w - (c.unsqueeze(1) @ basis[:, :j + 1]).squeeze(1)
            hn = torch.linalg.vector_norm(w, dim=1)
            hess[:, j + 1, j] = hn
            basis[:, j + 1] = w / hn[:, None].clamp_min(1e-300)
        rhs = torch.zeros((n, restart + 1, 1), dtype=C128, device=DEV)
        rhs[:, 0, 0] = beta
        q, rr = torch.linalg.qr(hess)
        y = torch.linalg.solve_triangular(rr, q.mH @ rhs, upper=True)
        x = x + pre((y.mT @ basis[:, :restart]).squeeze(1))
    return None


def _network(plain, params, omega, gamma):
    """(p, U, V) of the preconditioner at one shift, from leaf tensors of the FP16-rounded weights."""
    n = plain.na * plain.e.numel()
    d = plain.diag()
    ca = torch.diagonal(plain.chi).real
    x = torch.zeros((plain.na, plain.e.numel(), 12), dtype=torch.float64, device=DEV)
    e = plain.e.reshape(-1)
    for a in range(plain.na):
        da = d.reshape(plain.na, -1)[a]
        x[a, :, 0], x[a, :, 1], x[a, :, 2] = (da - omega) / 10, gamma, (e - omega) / 10
        x[a, :, 3], x[a, :, 4], x[a, :, 6 + min(a, 5)] = da - e + ca[a], ca[a] / 5, 1.0
        if plain.a is not None:
            x[a, :, 5] = torch.linalg.vector_norm(plain.a, dim=0)
    w1, b1, w2, b2, w3, b3 = params
    silu = torch.nn.functional.silu
    o = silu(silu(x.reshape(n, 12) @ w1 + b1) @ w2 + b2) @ w3 + b3
    sigma = 4.5j + 5.0 * torch.complex(o[:, 0], o[:, 1])
    return 1.0 / (d - complex(omega, gamma) - sigma), torch.complex(o[:, 2:10], o[:, 10:18]), \
        torch.complex(o[:, 18:26], o[:, 26:34])


def _unpack(flat):
    out, at = [], 0
    for shape in ((12, 128), (128,), (128, 128), (128,), (128, 34), (34,)):
        n = math.prod(shape)
        out.append(torch.as_tensor(flat[at:at + n].astype(np.float16).astype(np.float64)).to(DEV).reshape(shape))
        at += n
    return out


def _pfun(factors):
    """P on rows r [T][N] for one set of factors (p, U, V)."""
    p, u, v = factors
    return lambda r: p * r + ((r @ v.conj()) @ u.T) / r.shape[1]


def _loss_grad(plain, flat, r, steps):
    params = [q.requires_grad_() for q in _unpack(flat)]
    pre = _pfun(_network(plain, params, 10.8, 0.5))
    z = 10.8 + 0.5j
    r2 = (r.abs() ** 2).sum(1)
    if steps == 0:
        y = pre(r)
        res = plain.apply(y) - z * y - r
    else:
        ys, y = [], r
        for _ in range(steps):
            t = pre(y)
            y = plain.apply(t) - z * t
            ys.append(y)
        ys = torch.stack(ys, 1)
        with torch.no_grad():   # the optimal coefficients: their derivative does not contribute
            c = torch.linalg.lstsq(ys.mT.cpu(), r.unsqueeze(-1).cpu()).solution.to(DEV)
        res = r - (c.mT @ ys).squeeze(1)
    loss = ((res.abs() ** 2).sum(1) / r2).sum()
    loss.backward()
    return {"loss": float(loss), "grad": torch.cat([q.grad.reshape(-1) for q in params])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "screening":
        st = prepare(case, seed)
        psi, chi = torch.as_tensor(st["psi"]).to(DEV), 0.0
        eps = torch.as_tensor(st["eps"]).to(DEV)
        for t, w in zip(st["t"], st["w"]):
            g = (psi / (st["mu"] - eps + 1j * t)) @ psi.mH
            chi = chi + w / (2 * math.pi) * g * g.mT
        return chi
    if kind == "projection":
        st = prepare(case, seed)
        j = np.stack(np.meshgrid(*[np.arange(n) for n in st["nx"]], indexing="ij"), -1).reshape(-1, 3) / np.asarray(st["nx"])
        m = np.stack(np.meshgrid(*[np.arange(n) for n in st["nk"]], indexing="ij"), -1).reshape(-1, 3)
        k = (m + case["kshift"]) / np.asarray(st["nk"])
        out = torch.empty((case["n_f"], len(k), case["nb"]), dtype=C128, device=DEV)
        for i in range(len(k)):
            ph = torch.exp(2j * math.pi * torch.as_tensor(j @ k[i]).to(DEV))
            out[:, i] = st["dv"] * ((st["f"].conj() * ph) @ st["u"][i])
        return out
    if kind == "sites":
        out = []
        for i, c in enumerate(_site_cases(case)):
            plain = _Plain(_system(c, 8 * seed + i))
            n = plain.na * plain.e.numel()
            a, b = _lanczos(plain.apply, _vectors(case["n_vec"], n, 8 * seed + i), case["n_steps"])
            out.append({"a": a, "b": b, "steps": None})
        return out
    nk, nx = case["nk0"] * case["nk1"] * case["nk2"], case["nx0"] * case["nx1"] * case["nx2"]
    size = nk * nx * case["nb"]
    if kind in ("gmres", "rixs", "mlp_grad") and size > 4e6:
        return None   # minutes of FP64 products
    s = _system(case, seed)
    plain = _Plain(s)
    if kind == "apply":
        return plain.apply(_vectors(case["n_vec"], s.dim, seed))
    if kind == "haydock":
        a, b = _lanczos(plain.apply, _vectors(case["n_vec"], s.dim, seed), case["n_steps"])
        return {"a": a, "b": b, "steps": None}
    if kind == "mlp_grad":
        return _loss_grad(plain, _params(seed), _vectors(case["n_probes"], s.dim, seed), case["steps"])
    if kind == "gmres":
        # a solve that may stop at max_iter is compared with the other side's only
        if case["precond"] != "mlp" or case["max_iter"] < 400:
            return None
        z = _shifts(case)
        with torch.no_grad():
            f = [_network(plain, _unpack(_params(seed)), v.real, v.imag) for v in z]
        p, u, v = (torch.stack(q) for q in zip(*f))
        pre = lambda r: p * r + (u @ (v.mH @ r.unsqueeze(-1))).squeeze(-1) / r.shape[1]  # noqa: E731
        return {"x": _solve(plain.apply, pre, _vectors(1, s.dim, seed)[0], z, 1e-9), "iters": None, "rel": None}
    z = np.linspace(2.0, 14.0, case["n_z"]) + 0.5j
    x = _solve(plain.apply, lambda r: r, _vectors(1, s.dim, seed)[0], z, 1e-9)
    if x is None:
        return None
    val, d = _valence(s, case, seed)
    y = -torch.einsum("va,zai->zvi", torch.as_tensor(d).to(DEV), x.reshape(case["n_z"], case["na"], -1))
    a, b = _lanczos(_Plain(val).apply, y.reshape(case["n_z"], -1), case["n_steps"])
    return {"a": a, "b": b, "steps": None, "iters": None, "rel": None}
