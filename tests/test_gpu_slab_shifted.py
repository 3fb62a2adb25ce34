"""The FP32 slab stages on k+q spheres that a large q shifts along the first axis, so that their
planes are no run around index 0: all of them above it, some k points' above it and others'
around it, all below it.  L x and L^H x against the oracle (relative L2 <= 2e-5, the parity
suite's mixed bar), and the slab stages are what runs (no separate forward line pass).
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n3,nk,q", [
    (24, 20, 1, -6.2), (24, 20, 2, -5.9), (24, 12, 2, 6.1), (36, 12, 2, -8.8), (45, 12, 1, -11.5),
    (16, 12, 2, -4.2)])
def test_shifted_spheres(n, n3, nk, q):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth.configs as sc
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_MIXED, Context, build
    from synth import random_br_vector
    build()
    a = 8.0
    gmax = 2 * np.pi / a * n / 4.4
    sc.CONFIGS["_shift"] = dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", lattice=np.diag([a, a, a * n3 / n]), fft=(n, n, n3),
        ecut=0.5 * gmax ** 2, kgrid=(nk, 1, 1), nocc=5, alat=a, seed=91, q_2pi_a=(q, 0.0, 0.0))
    try:
        gs = sc.make_ground_state("_shift", solver="random")
    finally:
        del sc.CONFIGS["_shift"]
    first = gs.miller_kq[0, :gs.npw_kq[0], 0]
    assert first.min() > 0 if q < 0 else first.max() < 0
    x = random_br_vector(gs, seed=8)
    lv = Liouvillian(gs)
    flip = np.array([1.0, -1.0])[:, None, None, None, None]
    ref = lv.apply(x), flip * lv.apply(flip * x)
    ctx = Context(0)
    try:
        slot = ctx.load_ground_state(gs)
        xt = torch.as_tensor(x, device="cuda").to(torch.complex64)
        yt = torch.empty_like(xt)
        torch.cuda.synchronize()
        for adj in (0, 1):
            ctx.apply_liouvillian(slot, xt, yt, bool(adj), TDLZ_MIXED)
            ctx.synchronize()
            err = np.linalg.norm(yt.cpu().numpy() - ref[adj]) / np.linalg.norm(ref[adj])
            assert err <= 2e-5, (adj, err)
        ctx.profile(True)
        ctx.apply_liouvillian(slot, xt, yt, False, TDLZ_MIXED)
        ctx.synchronize()
        prof = ctx.profile_read()
        assert prof["product"]["ms"] > 0 and prof["fft_fwd"]["ms"] == 0
    finally:
        ctx.close()
