"""L x on 8192 k points with one band (2 x 8192 batches of 1 x 1 overlaps over 176 numbers, the
shape that wants most K splits per batch) against the oracle: relative L2 <= 1e-12 in FP64 and
<= 2e-5 mixed, the parity suite's bars."""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_many_k_points():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth.configs as sc
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_FP64, TDLZ_MIXED, Context, build
    from synth import random_br_vector
    build()
    sc.CONFIGS["_many_k"] = dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", kgrid=(32, 16, 16), ecut=3.75, nocc=1, seed=61)
    try:
        gs = sc.make_ground_state("_many_k", solver="random")
    finally:
        del sc.CONFIGS["_many_k"]
    x = random_br_vector(gs, seed=3)
    ref = Liouvillian(gs).apply(x)
    ctx = Context(0)
    try:
        q = ctx.load_ground_state(gs)
        for prec, dt, tol in ((TDLZ_FP64, torch.complex128, 1e-12),
                              (TDLZ_MIXED, torch.complex64, 2e-5)):
            xt = torch.as_tensor(x, device="cuda").to(dt)
            yt = torch.empty_like(xt)
            torch.cuda.synchronize()
            ctx.apply_liouvillian(q, xt, yt, False, prec)
            ctx.synchronize()
            err = np.linalg.norm(yt.cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= tol, (prec, err)
    finally:
        ctx.close()
