"""Workloads of the Liouville-Lanczos engine, with their inputs, one pass of each and its
exact results.

The sizes follow the repository's model crystals (the 16^3 Gamma cell, the 36x36x96 slab
with 40 bands, the 45x45x144 layer with 70 bands) and general cells between them.  The
occupied states are random orthonormal spinors that decay with the kinetic energy: L is
defined for any orthonormal occupied set, and its cost does not depend on the states.
The chains run the non-Hermitian recursion: on such states the J norm of the start vectors
all but vanishes, and the coefficients of a pseudo-Hermitian chain (the same kernels, half
the vectors) carry few exact digits.
"""

from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2203_01120_gb300 import TDLZ_FP64, TDLZ_MIXED, Context

HA_MEV = 27211.386245988
# FFT lengths of drawn cells: products of 2, 3 and 5
LENGTHS = (12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45)
LENGTHS_Z = LENGTHS + (48, 50, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128, 144)


def _cell(name, what, a, c, n1, n2, n3, ecut, k1, k2, nocc, natom, nchan, prec, **more):
    d = dict(name=name, what=what, a=a, c=c, hexagonal=more.pop("hexagonal", True), n1=n1, n2=n2,
             n3=n3, ecut=ecut, k1=k1, k2=k2, nocc=nocc, natom=natom, nchan=nchan, prec=prec,
             adjoint=False, nchain=1, ncomp=3, nq=1, steps=1)
    d.update(more)
    return d


def listed():
    slab = dict(a=13.0, c=30.0, n1=36, n2=36, n3=96, ecut=8.3, nocc=40, natom=8, nchan=8)
    layer = dict(a=13.0, c=38.0, n1=45, n2=45, n3=144, ecut=12.7, natom=8, nchan=8)
    gamma = dict(a=8.0, c=8.0, hexagonal=False, n1=16, n2=16, n3=16, ecut=5.3, k1=1, k2=1,
                 nocc=8, natom=2, nchan=2)
    return [
        # one product L x of a Gamma-point cell inside a user's own iterative solver: the
        # smallest call, all launches and latency
        _cell("gamma_apply_fp64", "apply", prec="fp64", **gamma),
        # the whole run of a small cell (load done): chain start, steps, coefficients on the host
        _cell("gamma_run_nh_fp64", "run", prec="fp64", steps=24, **gamma),
        # L^H x on a box whose lengths have no register plan and are not square
        _cell("ragged_adjoint_mixed", "apply", prec="mixed", adjoint=True, a=10.5, c=15.0,
              hexagonal=False, n1=30, n2=25, n3=40, ecut=6.0, k1=2, k2=1, nocc=11, natom=3,
              nchan=4),
        # the x, y, z columns of a medium cell in FP64 (reference spectra at full precision)
        _cell("medium_run_nh_fp64", "run", prec="fp64", nchain=3, steps=8, a=9.0,
              c=18.0, n1=24, n2=24, n3=48, ecut=6.5, k1=2, k2=2, nocc=18, natom=4, nchan=4),
        # one product of the slab's response vector (a user's own solver, mixed precision)
        _cell("slab_apply_mixed", "apply", prec="mixed", k1=4, k2=4, **slab),
        # the same product at full precision, on fewer k points (FP64 checks of mixed spectra)
        _cell("slab_apply_fp64", "apply", prec="fp64", k1=2, k2=2, **slab),
        # the benchmark's workload: three non-Hermitian chains of the slab, mixed precision
        _cell("slab_run_nh_mixed", "run", prec="mixed", nchain=3, steps=6, k1=4, k2=4, **slab),
        # chains of three q points, each with its own spheres, advancing together
        _cell("slab_multiq_nh_mixed", "run", prec="mixed", nq=3, nchain=2, steps=5, k1=2, k2=2,
              **slab),
        # the production form on the layer's cell: the longest lines, 70 bands, with the
        # charge as fourth left vector
        _cell("layer_run_nh_mixed", "run", prec="mixed", nchain=2, ncomp=4, steps=4, k1=4, k2=2,
              nocc=70, **layer),
        # the layer's product at full precision (few k points and bands)
        _cell("layer_apply_fp64", "apply", prec="fp64", k1=2, k2=1, nocc=24, **layer),
        # chi on 0-100 meV from three chains of 1500 coefficients
        dict(name="spectrum_full", what="spectrum", nchain=3, ncomp=3, steps=1500, itermax0=0,
             itermax=0, extrapolation="no", nomega=1001, eta=10.0),
        # a few hundred coefficients, extended by the bi-constant extrapolation
        dict(name="spectrum_osc", what="spectrum", nchain=1, ncomp=4, steps=400, itermax0=380,
             itermax=6000, extrapolation="osc", nomega=501, eta=5.0),
    ]


def draw(rng):
    what = rng.choice(("apply", "apply", "run", "run", "spectrum"))
    if what == "spectrum":
        steps = int(round(math.exp(rng.uniform(math.log(40), math.log(1500)))))
        ex = rng.choice(("no", "constant", "osc"))
        return dict(what=what, nchain=rng.randint(1, 3), ncomp=rng.choice((3, 4)), steps=steps,
                    itermax0=0 if ex == "no" else steps - rng.randint(0, 9),
                    itermax=0 if ex == "no" else rng.randint(2, 5) * steps, extrapolation=ex,
                    nomega=int(round(math.exp(rng.uniform(math.log(51), math.log(1001))))),
                    eta=rng.choice((5.0, 10.0, 20.0)))
    hexagonal = rng.random() < 0.7
    n1 = rng.choice(LENGTHS)
    n2 = n1 if rng.random() < 0.75 else rng.choice(LENGTHS)
    n3 = rng.choice([n for n in LENGTHS_Z if n >= n1])
    a = rng.uniform(6.0, 13.0)
    # the sphere reaches n1 / 4.4 reciprocal vectors, so products fit the box but for a
    # slight aliasing, and the height of the cell follows from n3
    b1 = 2.0 * math.pi / a * (2.0 / math.sqrt(3.0) if hexagonal else 1.0)
    gmax = min(n1, n2) / 4.4 * b1
    c = 2.0 * math.pi * (n3 / 4.6) / gmax
    omega = a * a * c * (math.sqrt(0.75) if hexagonal else 1.0)
    npw = omega * gmax ** 3 / (6.0 * math.pi ** 2)
    prec = rng.choice(("mixed", "mixed", "fp64"))
    natom, nchan = rng.randint(1, 8), rng.choice((2, 4, 8))
    nocc = int(round(math.exp(rng.uniform(math.log(2), math.log(70)))))
    nocc = max(1, min(nocc, int(npw / 8)))
    k1, k2 = rng.randint(1, 4), rng.randint(1, 4)
    nq, nchain, steps, adjoint, ncomp = 1, 1, 1, rng.random() < 0.3, 3
    if what == "run":
        adjoint = False
        nq, nchain, steps = rng.choice((1, 1, 1, 2)), rng.randint(1, 4), rng.randint(2, 6)
        ncomp = rng.choice((3, 3, 4))
    # at most the work of the largest listed case (FP64 costs about twenty times as much)
    cost = lambda: (k1 * k2 * nocc * n1 * n2 * n3 * nq * nchain * steps  # noqa: E731
                    * (2 if what == "run" else 1) * (20 if prec == "fp64" else 1))
    while cost() > 16 * 40 * 36 * 36 * 96 * 30 and k1 * k2 > 1:
        k1, k2 = (k1 - 1, k2) if k1 >= k2 else (k1, k2 - 1)
    while cost() > 16 * 40 * 36 * 36 * 96 * 30 and nocc > 2:
        nocc -= 1
    return {k: v for k, v in _cell("", what, a, c, n1, n2, n3, 0.5 * gmax * gmax, k1, k2, nocc,
                                   natom, nchan, prec, hexagonal=hexagonal, adjoint=adjoint,
                                   nchain=nchain, ncomp=ncomp, nq=nq, steps=steps).items() if k != "name"}


# ------------------------------------------------------------------------------ inputs
def _lattice(case):
    a, c = case["a"], case["c"]
    if case["hexagonal"]:
        return np.array([[a, 0, 0], [-0.5 * a, 0.5 * math.sqrt(3.0) * a, 0], [0, 0, c]])
    return np.diag([a, a, c])


def _sphere(p, bvec, ecut, fft):
    """Miller indices of |p + G|^2 / 2 <= ecut that fit the box, by kinetic energy."""
    m = np.stack(np.meshgrid(*[np.arange(-(n // 2), (n - 1) // 2 + 1) for n in fft],
                             indexing="ij"), axis=-1).reshape(-1, 3)
    kin = 0.5 * np.sum((p + m @ bvec) ** 2, axis=1)
    m, kin = m[kin <= ecut], kin[kin <= ecut]
    order = np.argsort(kin, kind="stable")
    return np.ascontiguousarray(m[order], dtype=np.int32), kin[order]


def _smooth_field(fft, bvec, gcut, rms, gen, ncomp):
    """ncomp random real grid fields with Fourier components up to gcut."""
    m = np.stack(np.meshgrid(*[np.fft.fftfreq(n, 1.0 / n) for n in fft], indexing="ij"), axis=-1)
    g = np.linalg.norm(m @ bvec, axis=-1)
    keep = torch.as_tensor((g > 0) & (g < gcut), device="cuda")
    f = torch.fft.fftn(torch.randn((ncomp,) + tuple(fft), generator=gen, device="cuda",
                                   dtype=torch.float64), dim=(1, 2, 3))
    f = torch.fft.ifftn(f * keep, dim=(1, 2, 3)).real.reshape(ncomp, -1)
    return f * (rms / f.square().mean(dim=1, keepdim=True).sqrt().clamp_min(1e-30))


def _ground_state(case, seed, iq):
    """Host bundle of q point iq: q = (iq + 1) / 8 (2 pi / a) along x, its own cutoff."""
    gen = torch.Generator(device="cuda").manual_seed(1000 * seed + iq)
    rng = np.random.default_rng([seed, iq])
    lat = _lattice(case)
    bvec = 2.0 * np.pi * np.linalg.inv(lat).T
    omega = abs(np.linalg.det(lat))
    fft = (case["n1"], case["n2"], case["n3"])
    nr = fft[0] * fft[1] * fft[2]
    ecut = case["ecut"] * (1.0 + 0.02 * iq)
    kpts = np.array([[i / case["k1"], j / case["k2"], 0.0] for i in range(case["k1"])
                     for j in range(case["k2"])]) @ bvec
    nk, nb = len(kpts), case["nocc"]
    q = np.array([0.125 * (iq + 1), 0.0, 0.0]) * 2.0 * np.pi / case["a"]
    sk = [_sphere(k, bvec, ecut, fft) for k in kpts]
    skq = [_sphere(k + q, bvec, ecut, fft) for k in kpts]
    npwx = max(m.shape[0] for m, _ in sk + skq)

    def states(spheres):
        c = torch.zeros((2, nk, nb, 2, npwx), dtype=torch.complex128, device="cuda")
        for ik, (m, kin) in enumerate(spheres):
            env = torch.as_tensor(np.exp(-kin / (0.3 + 0.1 * ecut)), device="cuda")
            v = torch.randn((2, nb, 2, len(kin)), generator=gen, device="cuda",
                            dtype=torch.complex128) * env
            v = v.reshape(2, nb, -1)
            for _ in range(2):  # Cholesky orthonormalisation, twice
                low = torch.linalg.cholesky(v.conj() @ v.transpose(1, 2))
                v = torch.linalg.solve_triangular(low.conj(), v, upper=False)
            c[:, ik, :, :, :len(kin)] = v.reshape(2, nb, 2, -1)
        return c

    ck, ckq = states(sk), states(skq)
    # ground densities of the X side's states at k
    n0, m0 = torch.zeros(nr, device="cuda", dtype=torch.float64), None
    m0 = torch.zeros((3, nr), device="cuda", dtype=torch.float64)
    for ik in range(nk):
        idx = torch.as_tensor(_grid_index(sk[ik][0], fft), device="cuda")
        for b0 in range(0, nb, 16):
            u = _to_grid(ck[0, ik, b0:b0 + 16, :, :len(idx)], idx, fft) / math.sqrt(omega)
            a, b = u[:, 0], u[:, 1]
            n0 += (a.abs().square() + b.abs().square()).sum(0) / nk
            ab = (a.conj() * b).sum(0)
            m0 += torch.stack([2 * ab.real, 2 * ab.imag,
                               (a.abs().square() - b.abs().square()).sum(0)]) / nk
    vloc = _smooth_field(fft, bvec, 3.0, 0.5, gen, 1)[0]
    b = _smooth_field(fft, bvec, 1.5, 0.1, gen, 3)
    b[2] += 0.2
    # Gaussian projectors of natom atoms, nchan channels each (s-like and p-like), coupled
    # within an atom by a Hermitian matrix with a spin part
    natom, nchan = case["natom"], case["nchan"]
    nproj = natom * nchan
    beta = np.zeros((nk, nproj, npwx), dtype=np.complex128)
    tau = rng.uniform(0.0, 1.0, (natom, 3)) @ lat
    for ik in range(nk):
        kg = kpts[ik] + q + skq[ik][0] @ bvec
        k2 = np.sum(kg * kg, axis=1)
        for at in range(natom):
            phase = np.exp(-1j * (kg @ tau[at]))
            for ch in range(nchan):
                rc = 0.7 + 0.15 * ch
                f = np.exp(-0.5 * k2 * rc * rc) * (1.0 if ch % 4 == 0 else kg[:, ch % 4 - 1])
                beta[ik, at * nchan + ch, :len(k2)] = f * phase
        beta[ik] /= np.linalg.norm(beta[ik], axis=1, keepdims=True)
    dnl = np.zeros((2 * nproj, 2 * nproj), dtype=np.complex128)
    for at in range(natom):
        w = 2 * nchan
        d = rng.standard_normal((w, w)) + 1j * rng.standard_normal((w, w))
        dnl[at * w:(at + 1) * w, at * w:(at + 1) * w] = 0.1 * (d + d.conj().T) + np.diag(
            np.linspace(1.0, -0.5, w))
    mk = np.zeros((nk, npwx, 3), dtype=np.int32)
    mkq = np.zeros((nk, npwx, 3), dtype=np.int32)
    for ik in range(nk):
        mk[ik, :len(sk[ik][1])] = sk[ik][0]
        mkq[ik, :len(skq[ik][1])] = skq[ik][0]
    host = lambda t: t.cpu().numpy()  # noqa: E731
    return SimpleNamespace(
        lattice=lat, fft=fft, ecutwfc=ecut, nk=nk, nocc=nb, npwx=npwx, nproj=nproj, kpts=kpts,
        q=q, wk=np.full(nk, 1.0 / nk), npw_k=np.array([len(k) for _, k in sk], np.int32),
        npw_kq=np.array([len(k) for _, k in skq], np.int32), miller_k=mk, miller_kq=mkq,
        evals=np.sort(rng.uniform(-1.0, 0.0, (2, nk, nb)), axis=-1), coeff_k=host(ck),
        coeff_kq=host(ckq), vloc=host(vloc), bfield=host(b), n0=host(n0), m0=host(m0),
        beta_kq=beta, dnl=dnl, kernel_mask=3)


def _vector(case, gs, seed):
    """A response vector in the layout [side][k][band][spin][plane wave], zero padding."""
    gen = torch.Generator(device="cuda").manual_seed(7 + seed)
    x = torch.randn((2, gs.nk, gs.nocc, 2, gs.npwx), generator=gen, device="cuda",
                    dtype=torch.complex128)
    for k in range(gs.nk):
        x[:, k, :, :, int(gs.npw_kq[k]):] = 0
    return x if case["prec"] == "fp64" else x.to(torch.complex64)


def _coefficients(case, seed):
    """Lanczos coefficients as chains give them: small alpha, beta around half the cutoff
    with the even-odd oscillation, z falling off."""
    rng = np.random.default_rng(seed)
    nc, m, nl = case["nchain"], case["steps"], case["ncomp"]
    cn = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    beta = 6.0 + 0.3 * (-1.0) ** np.arange(m) + 0.2 * rng.standard_normal((nc, m))
    z = cn(nc, nl, m) * np.exp(-np.arange(m) / (0.3 * m))
    return {"alpha": 0.02 * cn(nc, m), "beta": beta, "gamma": beta * (1.0 + 0.01 * cn(nc, m)),
            "z": z, "n0": rng.uniform(0.5, 1.5, nc), "wk": np.full(nc, 1.0 / 16),
            "steps_done": np.full(nc, m, np.int32), "status": np.zeros(nc, np.int32)}


_stream = None


def _context():
    """A context on the program's one stream (its q points and chains run in order on it)."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return Context(0, _stream.cuda_stream)


def prepare(case, seed):
    if case["what"] == "spectrum":
        return dict(case=case, ctx=_context(), coeffs=_coefficients(case, seed))
    ctx = _context()
    gss = [_ground_state(case, seed, iq) for iq in range(case["nq"])]
    slots = [ctx.load_ground_state(g) for g in gss]
    state = dict(case=case, ctx=ctx, slots=slots,
                 prec=TDLZ_FP64 if case["prec"] == "fp64" else TDLZ_MIXED)
    if case["what"] == "apply":
        state["x"] = _vector(case, gss[0], seed)
        state["y"] = torch.empty_like(state["x"])
    torch.cuda.synchronize()  # the inputs are there before the program's stream reads them
    torch.cuda.empty_cache()
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["what"] == "spectrum":
        return ctx.spectrum(state["coeffs"], 0.0, 100.0, 100.0 / (case["nomega"] - 1), case["eta"],
                            itermax0=case["itermax0"], itermax=case["itermax"],
                            extrapolation=case["extrapolation"])
    if case["what"] == "apply":
        ctx.apply_liouvillian(state["slots"][0], state["x"], state["y"], case["adjoint"],
                              state["prec"])
        return state["y"]
    qslots = [s for s in state["slots"] for _ in range(case["nchain"])]
    mus = [c for _ in state["slots"] for c in range(case["nchain"])]
    got = ctx.lanczos_run(qslots, mus, case["steps"], "nh", state["prec"], case["ncomp"])
    # the tridiagonal matrix by its three bands; a mixed chain's coefficients come from FP32
    # vectors, so single precision is what they carry
    ty, tr = (np.complex128, np.float64) if case["prec"] == "fp64" else (np.complex64, np.float32)
    return {"bands": _bands(got).astype(ty), "z": got["z"].astype(ty), "n0": got["n0"].astype(tr),
            "steps_done": got["steps_done"], "status": got["status"]}


def _bands(c):
    return np.stack([c["beta"].astype(complex), c["alpha"], c["gamma"]], axis=1)


def work(case):
    """Bytes and operations the method cannot do without (FFTs pruned to the sphere)."""
    if case["what"] == "spectrum":
        n = case["nchain"] * case["nomega"]
        tail = max(0, case["itermax"] - case["itermax0"]) if case["extrapolation"] != "no" else 0
        return {"bytes": case["nchain"] * case["steps"] * (40.0 + 16.0 * case["ncomp"])
                + 16.0 * n * case["ncomp"],
                "flops": float(n) * (case["steps"] * (60 + 8 * case["ncomp"]) + tail * 25)}
    lat = _lattice(case)
    npw = float(abs(np.linalg.det(lat))) * (2.0 * case["ecut"]) ** 1.5 / (6.0 * math.pi ** 2)
    nk, nb, nproj = case["k1"] * case["k2"], case["nocc"], case["natom"] * case["nchan"]
    nr = case["n1"] * case["n2"] * case["n3"]
    c = 16.0 if case["prec"] == "fp64" else 8.0
    vec = 4.0 * nk * nb * npw
    apply_flops = (2.0 * nk * nb * (4 * 5.0 * nr * math.log2(nr) * 0.56 + 110.0 * nr)
                   + 2.0 * nk * 16.0 * nb * 2.0 * npw * (nb + nproj))
    if case["what"] == "apply":
        return {"bytes": c * (4.0 * vec + nk * nproj * npw), "flops": apply_flops}
    m = case["nchain"]
    step_bytes = c * (m * 6.0 * vec + 2.0 * vec + nk * nproj * npw)
    return {"bytes": case["nq"] * case["steps"] * step_bytes,
            "flops": case["nq"] * case["steps"] * m * 2 * apply_flops}


# ----------------------------------------------------------------- exact, in 64 bits
def _grid_index(miller, fft):
    m = miller.astype(np.int64)
    return ((m[:, 0] % fft[0]) * fft[1] + m[:, 1] % fft[1]) * fft[2] + m[:, 2] % fft[2]


def _to_grid(c, idx, fft):
    g = torch.zeros(c.shape[:-1] + (fft[0] * fft[1] * fft[2],), dtype=c.dtype, device=c.device)
    g[..., idx] = c
    g = torch.fft.ifftn(g.reshape(c.shape[:-1] + tuple(fft)), dim=(-3, -2, -1), norm="forward")
    return g.reshape(c.shape[:-1] + (-1,))


class _Exact:
    """L and the recursions in plain complex128 torch."""

    def __init__(self, gs):
        self.gs = gs
        dev = lambda v: torch.as_tensor(v, device="cuda")  # noqa: E731
        self.ck, self.ckq = dev(gs.coeff_k), dev(gs.coeff_kq)
        self.beta, self.dnl = dev(gs.beta_kq), dev(gs.dnl)
        self.vloc, self.b, self.ev = dev(gs.vloc), dev(gs.bfield), dev(gs.evals)
        self.omega = abs(np.linalg.det(gs.lattice))
        bvec = 2.0 * np.pi * np.linalg.inv(gs.lattice).T
        self.ik = [dev(_grid_index(gs.miller_k[k, :gs.npw_k[k]], gs.fft)) for k in range(gs.nk)]
        mq = [gs.miller_kq[k, :gs.npw_kq[k]] for k in range(gs.nk)]
        self.iq = [dev(_grid_index(m, gs.fft)) for m in mq]
        self.kin = [dev(0.5 * np.sum((gs.kpts[k] + gs.q + m @ bvec) ** 2, axis=1))
                    for k, m in enumerate(mq)]
        m = np.stack(np.meshgrid(*[np.arange(n) - n * (np.arange(n) >= (n + 1) // 2)
                                   for n in gs.fft], indexing="ij"), axis=-1)
        g2 = np.sum((gs.q + m @ bvec) ** 2, axis=-1).reshape(-1)
        self.vh = dev(np.where(0.5 * g2 <= 4.0 * gs.ecutwfc, 4.0 * np.pi / g2, 0.0))
        self.f = dev(self._fxc())

    def _fxc(self):
        n, m = self.gs.n0, self.gs.m0
        c6 = (6.0 / np.pi) ** (1.0 / 3.0)
        ma = np.sqrt(np.sum(m * m, axis=0))
        up, dn = np.maximum(0.5 * (n + ma), 1e-4), np.maximum(0.5 * (n - ma), 1e-4)
        fu, fd = -(c6 / 3) * up ** (-2 / 3), -(c6 / 3) * dn ** (-2 / 3)
        small = ma < 1e-12 * n
        safe = np.where(small, 1.0, ma)
        h = np.where(small, np.array([[0.0], [0.0], [1.0]]), m / safe)
        half = np.maximum(0.5 * n, 1e-4)
        tr = np.where(small, 0.5 * (-(c6 / 3) * half ** (-2 / 3)),
                      -c6 * (up ** (1 / 3) - dn ** (1 / 3)) / (2 * safe))
        f = np.zeros((4, 4, len(n)))
        f[0, 0] = 0.25 * (fu + fd)
        for i in range(3):
            f[0, i + 1] = f[i + 1, 0] = 0.25 * (fu - fd) * h[i]
            for j in range(3):
                f[i + 1, j + 1] = f[0, 0] * h[i] * h[j] + tr * ((i == j) - h[i] * h[j])
        return f * (n >= 1e-10)

    def _bands(self):
        for side in range(2):
            for k in range(self.gs.nk):
                for b in range(0, self.gs.nocc, 16):
                    yield side, k, slice(b, b + 16)

    def _u(self, side, k, bs):
        return _to_grid(self.ck[side, k, bs, :, :len(self.ik[k])], self.ik[k],
                        self.gs.fft) / math.sqrt(self.omega)

    def apply(self, x):
        gs, rt = self.gs, math.sqrt(self.omega)
        nr = self.vloc.numel()
        rho = torch.zeros((4, nr), dtype=torch.complex128, device="cuda")
        for side, k, bs in self._bands():
            u = self._u(side, k, bs).conj()
            xr = _to_grid(x[side, k, bs, :, :len(self.iq[k])], self.iq[k], gs.fft) / rt
            w, t = gs.wk[k], 1.0 - 2.0 * side
            p = torch.einsum("nsr,ntr->str", u, xr) * w
            rho += torch.stack([p[0, 0] + p[1, 1], t * (p[0, 1] + p[1, 0]),
                                t * 1j * (p[1, 0] - p[0, 1]), t * (p[0, 0] - p[1, 1])])
        v = torch.einsum("abr,br->ar", self.f.to(rho.dtype), rho)
        v[0] += torch.fft.ifftn((torch.fft.fftn(rho[0].reshape(gs.fft)).reshape(-1)
                                 * self.vh).reshape(gs.fft)).reshape(-1)
        y = torch.zeros_like(x)
        for side, k, bs in self._bands():
            s, idx = 1.0 - 2.0 * side, self.iq[k]
            n = len(idx)
            u = self._u(side, k, bs)
            xk = x[side, k, bs, :, :n]
            xr = _to_grid(xk, idx, gs.fft) / rt
            bx, by, bz = s * self.b
            h = torch.stack([
                (self.vloc + bz) * xr[:, 0] + (bx - 1j * by) * xr[:, 1]
                + (v[0] + s * v[3]) * u[:, 0] + s * (v[1] - 1j * v[2]) * u[:, 1],
                (self.vloc - bz) * xr[:, 1] + (bx + 1j * by) * xr[:, 0]
                + s * (v[1] + 1j * v[2]) * u[:, 0] + (v[0] - s * v[3]) * u[:, 1]], dim=1)
            h = torch.fft.fftn(h.reshape(h.shape[:2] + tuple(gs.fft)), dim=(2, 3, 4))
            h = h.reshape(h.shape[:2] + (-1,))[..., idx] * (rt / nr)
            h = h + (self.kin[k] - self.ev[side, k, bs, None, None]) * xk
            pr = torch.einsum("ig,ntg->nit", self.beta[k, :, :n].conj(), xk)
            pr = (pr.reshape(pr.shape[0], -1) @ self.dnl.T).reshape(pr.shape)
            y[side, k, bs, :, :n] = h + torch.einsum("nit,ig->ntg", pr, self.beta[k, :, :n])
        for side in range(2):
            for k in range(gs.nk):
                self._project(y, side, k)
        y[1] *= -1
        return y

    def _project(self, y, side, k):
        o = self.ckq[side, k].reshape(self.gs.nocc, -1)
        h = y[side, k].reshape(self.gs.nocc, -1)
        y[side, k] = (h - (h @ o.conj().T) @ o).reshape(y[side, k].shape)

    def sigma_u(self, mu, ysign):
        """(sigma U, ysign sigma T U) on the k+q spheres; the charge has -ysign."""
        gs = self.gs
        out = torch.zeros_like(self.ckq)
        for k in range(gs.nk):
            where = torch.full((self.vloc.numel(),), -1, dtype=torch.int64, device="cuda")
            where[self.ik[k]] = torch.arange(len(self.ik[k]), device="cuda")
            src = where[self.iq[k]]
            c = self.ck[:, k][..., src.clamp_min(0)] * (src >= 0)
            a, b = c[:, :, 0], c[:, :, 1]
            o = [(b, a), (-1j * b, 1j * a), (a, -b), (a, b)][mu]
            out[:, k, :, :, :len(src)] = torch.stack(o, dim=2)
        out[1] *= -ysign if mu == 3 else ysign
        return out

    def start(self, mu):
        v = self.sigma_u(mu, 1.0)
        for side in range(2):
            for k in range(self.gs.nk):
                self._project(v, side, k)
        return v

    def chain(self, mu, steps, ncomp):
        dot = lambda a, b: complex(torch.vdot(a.reshape(-1), b.reshape(-1)))  # noqa: E731
        flip = lambda a: torch.stack([a[0], -a[1]])  # noqa: E731
        us = [self.sigma_u(l, -1.0) for l in range(ncomp)]
        v = self.start(mu)
        n0 = math.sqrt(dot(v, v).real)
        q, p = v / n0, v / n0
        qo, po, beta, gamma = torch.zeros_like(q), torch.zeros_like(q), 0.0, 0.0
        out = {"alpha": [], "beta": [], "gamma": [], "z": []}
        for _ in range(steps):
            a = self.apply(q)
            alpha = dot(p, a)
            out["z"].append([dot(q, u) for u in us])
            r = a - alpha * q - gamma * qo
            t = flip(self.apply(flip(p))) - np.conj(alpha) * p - beta * po
            c = dot(t, r)
            beta = math.sqrt(abs(c))
            gamma = c / beta
            qo, po, q, p = q, p, r / beta, t / np.conj(gamma)
            out["alpha"].append(alpha)
            out["beta"].append(beta)
            out["gamma"].append(gamma)
        return out, n0


def _exact_spectrum(case, co):
    """chi = w n0 sum conj(z) x, (omega + i eta - T) x = e_1, T extended explicitly with the
    window means; Gaussian elimination with partial pivoting, all frequencies at once."""
    om = (np.arange(case["nomega"]) * (100.0 / (case["nomega"] - 1)) + 1j * case["eta"]) / HA_MEV
    chi = np.zeros((case["nchain"], case["ncomp"], case["nomega"]), dtype=np.complex128)
    for c in range(case["nchain"]):
        al, be, ga = (co[k][c] for k in ("alpha", "beta", "gamma"))
        m = m0 = case["itermax0"] or case["steps"]
        if case["extrapolation"] != "no":
            m = case["itermax"]
            j = np.arange(m0 // 2, m0)
            tail = np.arange(m0, m)

            def extend(v):
                if case["extrapolation"] == "constant":
                    return np.concatenate([v[:m0], np.full(m - m0, v[j].mean())])
                par = [v[j[j % 2 == p]].mean() for p in (0, 1)]
                return np.concatenate([v[:m0], np.where(tail % 2, par[1], par[0])])

            al, be, ga = extend(al), extend(be), extend(ga)
        al, be, ga = al[:m], be[:m], ga[:m]
        # the part beyond m0 by its continued fraction from the far end (z = 0 there)
        g = 0.0
        for j in range(m - 1, m0 - 1, -1):
            g = 1.0 / (om - al[j] - (be[j] * ga[j] * g if j < m - 1 else 0.0))
        cut = be[m0 - 1] * ga[m0 - 1] * g if m > m0 else 0.0
        rows, x = [], np.zeros((m0 + 2, len(om)), dtype=np.complex128)
        d, du = om - al[0], np.full_like(om, -ga[0])
        b = np.ones_like(om)
        if m0 == 1:
            d, du = d - cut, 0.0 * du
        for i in range(m0 - 1):
            last = i + 2 == m0
            dn, dun = om - al[i + 1] - (cut if last else 0.0), (0.0 if last else -ga[i + 1]) + 0 * om
            dl = np.full_like(om, -be[i])
            swap = np.abs(d) < np.abs(dl)
            p = [np.where(swap, n, o) for o, n in ((d, dl), (du, dn), (0 * om, dun), (b, 0 * om))]
            o = [np.where(swap, n, o) for n, o in ((d, dl), (du, dn), (0 * om, dun), (b, 0 * om))]
            f = o[0] / p[0]
            rows.append(p)
            d, du, b = o[1] - f * p[1], o[2] - f * p[2], o[3] - f * p[3]
        rows.append([d, 0 * om, 0 * om, b])
        for i in range(m0 - 1, -1, -1):
            x[i] = (rows[i][3] - rows[i][1] * x[i + 1] - rows[i][2] * x[i + 2]) / rows[i][0]
        chi[c] = co["wk"][c] * co["n0"][c] * (co["z"][c][:, :m0].conj() @ x[:m0])
    return chi


def exact(case, seed):
    if case["what"] == "spectrum":
        return _exact_spectrum(case, _coefficients(case, seed))
    gss = [_ground_state(case, seed, iq) for iq in range(case["nq"])]
    if case["what"] == "apply":
        x = _vector(case, gss[0], seed).to(torch.complex128)
        if case["adjoint"]:
            x[1] *= -1
        y = _Exact(gss[0]).apply(x)
        if case["adjoint"]:
            y[1] *= -1
        return y
    # about twenty seconds of plain FP64 work: longer chains have no exact value here
    w = work(case)
    if w["flops"] > 6e12:
        return None
    got = {"alpha": [], "beta": [], "gamma": [], "z": [], "n0": []}
    for gs in gss:
        ex = _Exact(gs)
        for mu in range(case["nchain"]):
            c, n0 = ex.chain(mu, case["steps"], case["ncomp"])
            for k in ("alpha", "beta", "gamma"):
                got[k].append(np.array(c[k]))
            got["z"].append(np.array(c["z"]).T)
            got["n0"].append(n0)
    got = {k: np.array(v) for k, v in got.items()}
    return {"bands": _bands(got), "z": got["z"], "n0": got["n0"], "steps_done": None,
            "status": None}
