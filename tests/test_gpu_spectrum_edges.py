"""chi(omega) from given coefficients at the edges of the one-sweep solve: one to three
steps, pivots taken from both rows (alternating large and small sub-diagonals), tails of
one, two and many extrapolated steps, and grids that leave a partial last warp.

Oracle: the pivoted banded LAPACK solve of the (explicitly extended) system.  Both sides
are backward stable eliminations of well-separated systems (eta >= 0.3 of the couplings'
smallest scale), so they agree to a few hundred ulp times the step count: 1e-12 per
column.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_01120_gb300 import Context, build
    build()
    c = Context(0)
    yield c
    c.close()


def _coeffs(nc, m, nl, kind, seed):
    rng = np.random.default_rng(seed)
    cn = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    beta = 0.5 + rng.random((nc, m))
    if kind == "alternating":  # pivots from the pending row and from the next row in turn
        beta = beta * np.where(np.arange(m) % 2, 30.0, 0.05)
    alpha = cn(nc, m) * (20.0 if kind == "diagonal" else 0.1)
    return {"alpha": alpha, "beta": beta, "gamma": beta * np.exp(1j * rng.random((nc, m))),
            "z": cn(nc, nl, m), "n0": 0.5 + rng.random(nc), "wk": np.full(nc, 0.25),
            "steps_done": np.full(nc, m, np.int32)}


def _reference(co, om, eta, itermax0, itermax, ex):
    import dataclasses
    from oracle import spectrum as osp

    @dataclasses.dataclass
    class Coef:
        alpha: np.ndarray
        beta: np.ndarray
        gamma: np.ndarray
        z: np.ndarray
        n0: float
        steps: int

    out = []
    for c in range(len(co["n0"])):
        cf = Coef(co["alpha"][c], co["beta"][c], co["gamma"][c], co["z"][c], co["n0"][c],
                  int(co["steps_done"][c]))
        m = itermax0 or cf.steps
        cf = osp.extend_coefficients(cf, m, max(itermax, m), ex if itermax > m else "no")
        out.append(osp.chi_banded(cf, om, eta, co["wk"][c]))
    return np.array(out)


@pytest.mark.parametrize("m,nl,kind,itermax0,itermax,ex", [
    (1, 3, "plain", 0, 0, "no"), (2, 4, "plain", 0, 0, "no"), (3, 3, "alternating", 0, 0, "no"),
    (64, 4, "alternating", 0, 0, "no"), (65, 3, "diagonal", 0, 0, "no"),
    (200, 3, "plain", 150, 0, "no"), (40, 3, "alternating", 40, 41, "osc"),
    (40, 4, "plain", 39, 41, "osc"), (40, 3, "plain", 40, 57, "constant"),
    (41, 3, "alternating", 41, 700, "osc"), (30, 4, "plain", 30, 30, "osc"),
])
def test_edges(ctx, m, nl, kind, itermax0, itermax, ex):
    co = _coeffs(2, m, nl, kind, seed=m + nl)
    eta, nw = 0.3, 77
    om = np.arange(nw) * 0.05
    got = ctx.spectrum(co, 0.0, om[-1], 0.05, eta, units=0, itermax0=itermax0, itermax=itermax,
                       extrapolation=ex)
    ref = _reference(co, om, eta, itermax0, itermax, ex)
    assert got.shape == ref.shape
    err = np.linalg.norm(got - ref, axis=-1) / np.linalg.norm(ref, axis=-1)
    assert err.max() <= 1e-12, err


def test_noalloc_takes_the_same_solve(ctx):
    import torch
    co = _coeffs(3, 50, 4, "alternating", seed=9)
    ref = ctx.spectrum(co, 0.0, 1.0, 0.01, 0.3, units=0)
    dev = {k: torch.as_tensor(np.ascontiguousarray(v), device="cuda") for k, v in co.items()}
    chi = torch.full(ref.shape, float("nan"), dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    ctx.spectrum_noalloc(dev, 0.0, 1.0, 0.01, 0.3, 0, chi)
    ctx.synchronize()
    assert np.array_equal(chi.cpu().numpy(), ref)
