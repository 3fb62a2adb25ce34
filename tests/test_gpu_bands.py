"""L x at band and projector counts around the kernels' tile edges: one band, counts that
leave remainders in the four-band product groups, the density's band-side slices and the
reduction and update tiles.  Against the oracle: relative L2 <= 1e-12 in FP64 and <= 2e-5
mixed (the parity suite's bars).  Random orthonormal states in a 12^3 cell, three k points.
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nocc,natom", [(1, 1), (2, 3), (5, 2), (9, 1), (17, 8), (23, 5), (33, 12),
                                        (50, 20)])
@pytest.mark.parametrize("tensor", [True, False])
def test_band_counts(nocc, natom, tensor, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth.configs as sc
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_FP64, TDLZ_MIXED, Context, build
    from synth import random_br_vector
    build()
    if not tensor:
        monkeypatch.setenv("TDLZ_TC", "0")
    monkeypatch.setitem(sc.CONFIGS, "_bands", dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", nocc=nocc, natom=natom, kgrid=(1, 3, 1), seed=31))
    gs = sc.make_ground_state("_bands", solver="random")
    x = random_br_vector(gs, seed=5)
    ref = Liouvillian(gs).apply(x)
    ctx = Context(0)
    try:
        q = ctx.load_ground_state(gs)
        precs = [(TDLZ_MIXED, torch.complex64, 2e-5)]
        if tensor:  # the FP64 path has one form
            precs.append((TDLZ_FP64, torch.complex128, 1e-12))
        for prec, dt, tol in precs:
            xt = torch.as_tensor(x, device="cuda").to(dt)
            yt = torch.empty_like(xt)
            torch.cuda.synchronize()
            ctx.apply_liouvillian(q, xt, yt, False, prec)
            ctx.synchronize()
            err = np.linalg.norm(yt.cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= tol, (nocc, natom, prec, err)
    finally:
        ctx.close()
