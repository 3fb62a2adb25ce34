"""FP64 contractions by integer slices on rows of wide range: plane-wave coefficients that grow
by 10^6 with the kinetic energy against projectors that fall over 17 decades, states that
fall, spin blocks that do not meet, rows of one band each of these; every component of L x
against extended precision.

Without potentials and kernels, y = P_c [(kin - e) x + V_NL x] up to the sides' signs, and a
component's terms, taken by magnitude, are
  T = t + |U| |U|^T t,  t = |kin - e| |x| + |beta| |D| |beta|^T |x|.
A sum of n terms rounded at each step errs by some sqrt(n) roundings of its own magnitude; two
sums of at most 1320 terms in a row: 100 2^-53 T is more than twice sqrt(1320).  (Rows in
62-bit fixed point without regard to the products: 5000 2^-53 T for 25 falling states.)
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _falling(rng, kin, nb, scale, collinear):
    """nb orthonormal spinors that fall as exp(-kin / scale); collinear: of one spin each."""
    n = len(kin)
    v = rng.standard_normal((nb, 2, n)) + 1j * rng.standard_normal((nb, 2, n))
    v *= np.exp(-kin / scale)
    if collinear:
        v[: nb // 2, 1] = 0.0
        v[nb // 2:, 0] = 0.0
    v = v.reshape(nb, -1)
    for _ in range(2):
        v = np.linalg.solve(np.linalg.cholesky(v @ v.conj().T), v)
    return v.reshape(nb, 2, n)


def _system(cell, nocc, natom, nk, kind):
    import synth.configs as sc
    sc.CONFIGS["_range"] = dataclasses.replace(
        sc.CONFIGS[cell], name=cell, nocc=nocc, natom=natom, kgrid=(1, nk, 1), seed=71)
    try:
        gs = sc.make_ground_state("_range", solver="random", kernel_mask=0)
    finally:
        del sc.CONFIGS["_range"]
    rng = np.random.default_rng(73)
    bvec = 2.0 * np.pi * np.linalg.inv(gs.lattice).T
    ckq, beta = np.array(gs.coeff_kq), np.array(gs.beta_kq)
    x = np.zeros(gs.br_shape, dtype=np.complex128)
    kin = []
    for k in range(gs.nk):
        n = gs.npw_kq[k]
        e = 0.5 * np.sum((gs.kpts[k] + gs.q + gs.miller_kq[k, :n] @ bvec) ** 2, axis=1)
        kin.append(e)
        top = e.max()
        for i in range(beta.shape[1]):  # 17 decades over the sphere
            beta[k, i, :n] *= np.exp(-e / top * 39.0)
            beta[k, i] /= np.linalg.norm(beta[k, i])
        for s in range(2):
            if kind != "flat states":
                ckq[s, k, :, :, :n] = _falling(rng, e, nocc, top / 25.0, kind == "spins")
            v = rng.standard_normal((nocc, 2, n)) + 1j * rng.standard_normal((nocc, 2, n))
            grow = np.exp(e / top * 13.8)
            if kind == "bands":  # every third band grows, every third falls
                grow = np.exp(np.outer(np.arange(nocc) % 3 - 1, e / top * 13.8))[:, None, :]
            if kind == "spins":
                grow = np.ones(n)
                v[::2, 1] = 0.0
                v[1::2, 0] = 0.0
            x[s, k, :, :, :n] = v * grow
    nr = int(np.prod(gs.fft))
    return dataclasses.replace(gs, coeff_kq=ckq, beta_kq=beta, vloc=np.zeros(nr),
                               bfield=np.zeros((3, nr))), x, kin


def _reference(gs, x, kin):
    """y and T in extended precision."""
    ld, cl = np.longdouble, np.clongdouble
    y, big = np.zeros(x.shape, cl), np.zeros(x.shape, ld)
    d = gs.dnl.astype(cl)
    for s in range(2):
        for k in range(gs.nk):
            n = gs.npw_kq[k]
            xk = x[s, k, :, :, :n].astype(cl)
            b = gs.beta_kq[k, :, :n].astype(cl)
            e = kin[k].astype(ld)[None, None, :] - gs.evals[s, k].astype(ld)[:, None, None]

            def vnl(v, b, d):
                p = (v.reshape(-1, n) @ b.conj().T).reshape(gs.nocc, 2, -1)
                p = np.swapaxes(p, 1, 2).reshape(gs.nocc, -1) @ d.T
                return (np.swapaxes(p.reshape(gs.nocc, -1, 2), 1, 2).reshape(2 * gs.nocc, -1)
                        @ b).reshape(v.shape)

            h = (e * xk + vnl(xk, b, d)).reshape(gs.nocc, -1)
            t = np.abs(e) * np.abs(xk) + vnl(np.abs(xk), np.abs(b), np.abs(d))
            t = t.reshape(gs.nocc, -1)
            u = gs.coeff_kq[s, k, :, :, :n].reshape(gs.nocc, -1).astype(cl)
            h = h - (h @ u.conj().T) @ u
            t = t + (t @ np.abs(u).T) @ np.abs(u)
            y[s, k, :, :, :n] = (1 - 2 * s) * h.reshape(xk.shape)
            big[s, k, :, :, :n] = t.reshape(xk.shape)
    return y, big


@pytest.mark.parametrize("cell,nocc,natom,nk,kind", [
    ("C1", 25, 7, 24, "falling states"), ("C1", 25, 7, 24, "spins"), ("C1", 40, 10, 8, "bands"),
    ("C1", 49, 13, 6, "falling states"), ("C1", 130, 33, 2, "flat states"),
    ("C1", 130, 33, 2, "bands")])
def test_components(cell, nocc, natom, nk, kind, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_01120_gb300 import TDLZ_FP64, Context, build
    build()
    gs, x, kin = _system(cell, nocc, natom, nk, kind)
    ref, big = _reference(gs, x, kin)
    for tc in "10":
        monkeypatch.setenv("TDLZ_TC", tc)
        ctx = Context(0)
        try:
            q = ctx.load_ground_state(gs)
            xt = torch.as_tensor(x, device="cuda")
            yt = torch.empty_like(xt)
            torch.cuda.synchronize()
            ctx.apply_liouvillian(q, xt, yt, False, TDLZ_FP64)
            ctx.synchronize()
            err = np.abs(yt.cpu().numpy() - ref)
        finally:
            ctx.close()
        worst = float((err / np.where(big > 0, big, 1)).max() * 2.0 ** 53)
        print(kind, nocc, "slices" if tc == "1" else "pipe", f"{worst:.3g}")
        assert worst <= 100.0, (tc, worst)
