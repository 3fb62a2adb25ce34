"""L x on grids that run each register line length in the x, y and z passes, against the
oracle: relative L2 <= 1e-12 in FP64 and <= 2e-5 mixed (the parity suite's bars), forward
and adjoint.  A few bands on random orthonormal states; the sphere is cut so that it fits
the shortest axis.
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _ground_state(fft, nocc):
    import synth.configs as sc
    a = 8.0
    # the sphere reaches fft / 4.4 reciprocal vectors of the shortest axis
    gmax = 2 * np.pi / a * min(fft[0], fft[1]) / 4.4
    c = a * fft[2] / min(fft[0], fft[1])
    sc.CONFIGS["_line"] = dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", lattice=np.diag([a, a, c]), fft=fft, ecut=0.5 * gmax ** 2,
        kgrid=(1, 2, 1), nocc=nocc, alat=a, seed=77)
    try:
        return sc.make_ground_state("_line", solver="random")
    finally:
        del sc.CONFIGS["_line"]


@pytest.mark.parametrize("fft", [(24, 24, 36), (48, 48, 12), (12, 12, 24), (16, 16, 45),
                                 (45, 45, 16), (36, 36, 48), (12, 12, 96), (12, 12, 144),
                                 (16, 16, 192), (36, 24, 12), (16, 48, 45)])
def test_register_lines(fft):
    _check(fft, 3)


@pytest.mark.parametrize("fft", [(15, 18, 12), (18, 15, 20), (20, 25, 27), (25, 20, 16),
                                 (27, 30, 40), (30, 27, 12), (32, 40, 24), (40, 32, 30)])
@pytest.mark.parametrize("nocc", [1, 5])
def test_register_lines_between(fft, nocc):
    """The lengths between on both axes, with few bands (the reductions' K splits)."""
    _check(fft, nocc)


def _check(fft, nocc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_FP64, TDLZ_MIXED, Context, build
    from synth import random_br_vector
    build()
    gs = _ground_state(fft, nocc)
    x = random_br_vector(gs, seed=5)
    lv = Liouvillian(gs)
    flip = np.array([1.0, -1.0])[:, None, None, None, None]
    ref = lv.apply(x), flip * lv.apply(flip * x)
    ctx = Context(0)
    try:
        q = ctx.load_ground_state(gs)
        for prec, dt, tol in ((TDLZ_FP64, torch.complex128, 1e-12),
                              (TDLZ_MIXED, torch.complex64, 2e-5)):
            xt = torch.as_tensor(x, device="cuda").to(dt)
            yt = torch.empty_like(xt)
            torch.cuda.synchronize()
            for adj in (0, 1):
                ctx.apply_liouvillian(q, xt, yt, bool(adj), prec)
                ctx.synchronize()
                err = np.linalg.norm(yt.cpu().numpy() - ref[adj]) / np.linalg.norm(ref[adj])
                assert err <= tol, (fft, prec, adj, err)
    finally:
        ctx.close()
