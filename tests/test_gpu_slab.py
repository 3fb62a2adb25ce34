"""The FP32 slab stages (square grids): group and sphere remainders, every kernel mask,
sub-batches and the adjoint.

Against the oracle: relative L2 <= 2e-5 (the parity suite's mixed bar) at band counts that
leave partial groups (groups of 4, 3 and 2 bands at up to 24, 36 and from 45 points).
Sub-batches of the stacked vectors change no result: bit for bit.
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_01120_gb300 import build
    build()
    return t


def _ground_state(n, n3, nocc, nk, mask=3):
    import synth.configs as sc
    a = 8.0
    gmax = 2 * np.pi / a * n / 4.4
    sc.CONFIGS["_slab"] = dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", lattice=np.diag([a, a, a * n3 / n]), fft=(n, n, n3),
        ecut=0.5 * gmax ** 2, kgrid=(1, nk, 1), nocc=nocc, alat=a, seed=91)
    try:
        return sc.make_ground_state("_slab", solver="random", kernel_mask=mask)
    finally:
        del sc.CONFIGS["_slab"]


@pytest.mark.parametrize("n,n3,nocc,nk,mask", [
    (12, 15, 7, 3, 3), (16, 12, 4, 2, 1), (24, 20, 5, 2, 2), (24, 24, 6, 3, 0), (36, 18, 5, 2, 3),
    (36, 12, 4, 3, 0), (45, 12, 5, 2, 3), (45, 16, 1, 1, 0), (48, 12, 3, 2, 3)])
def test_slab_apply(torch, n, n3, nocc, nk, mask):
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_MIXED, Context
    from synth import random_br_vector
    gs = _ground_state(n, n3, nocc, nk, mask)
    x = random_br_vector(gs, seed=8)
    lv = Liouvillian(gs)
    flip = np.array([1.0, -1.0])[:, None, None, None, None]
    ref = lv.apply(x), flip * lv.apply(flip * x)
    ctx = Context(0)
    try:
        q = ctx.load_ground_state(gs)
        xt = torch.as_tensor(x, device="cuda").to(torch.complex64)
        yt = torch.empty_like(xt)
        torch.cuda.synchronize()
        for adj in (0, 1):
            ctx.apply_liouvillian(q, xt, yt, bool(adj), TDLZ_MIXED)
            ctx.synchronize()
            err = np.linalg.norm(yt.cpu().numpy() - ref[adj]) / np.linalg.norm(ref[adj])
            assert err <= 2e-5, (adj, err)
    finally:
        ctx.close()


@pytest.mark.parametrize("n,n3,nocc,nk", [(24, 12, 6, 2), (36, 12, 5, 2)])
def test_sub_batches_change_no_result(torch, monkeypatch, n, n3, nocc, nk):
    from paper_2203_01120_gb300 import TDLZ_MIXED, Context
    gs = _ground_state(n, n3, nocc, nk)
    out = []
    for sub in (None, "1", "4"):
        if sub is None:
            monkeypatch.delenv("TDLZ_STAGED_SUB", raising=False)
        else:
            monkeypatch.setenv("TDLZ_STAGED_SUB", sub)
        c = Context(0)
        try:
            q = c.load_ground_state(gs)
            out.append(c.lanczos_run([q, q, q], [0, 1, 2], 6, "nh", TDLZ_MIXED))
        finally:
            c.close()
    for other in out[1:]:
        for key in ("alpha", "beta", "gamma", "z"):
            assert np.array_equal(out[0][key], other[key]), key
