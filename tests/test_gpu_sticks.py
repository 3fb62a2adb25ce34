"""Z passes over spheres whose stick count leaves whole warps of the last block without a
stick (a block takes 32 sticks at 96 and 144 points, a warp eight): L x in mixed precision
against the oracle (relative L2 <= 2e-5, the parity suite's mixed bar), on square grids
(sticks transposed) and others, for one and for several k points of unequal spheres.
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fft,ecut,nk", [
    ((12, 12, 96), 0.45, 1), ((12, 12, 96), 1.1, 3), ((12, 12, 144), 1.7, 2),
    ((12, 16, 96), 0.45, 2), ((16, 12, 144), 1.1, 3), ((16, 16, 96), 6.5, 2)])
def test_warps_without_sticks(fft, ecut, nk):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth.configs as sc
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_MIXED, Context, build
    from synth import random_br_vector
    build()
    sc.CONFIGS["_sticks"] = dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", lattice=np.diag([6.0, 6.0, 24.0]), fft=fft, ecut=ecut,
        kgrid=(1, nk, 1), nocc=3, seed=53)
    try:
        gs = sc.make_ground_state("_sticks", solver="random")
    finally:
        del sc.CONFIGS["_sticks"]
    most = max(len({tuple(m[:2]) for m in gs.miller_kq[k][:gs.npw_kq[k]]}) for k in range(nk))
    assert most % 32 and most % 32 < 24, most  # the last block has warps beyond the table
    x = random_br_vector(gs, seed=5)
    ref = Liouvillian(gs).apply(x)
    ctx = Context(0)
    try:
        q = ctx.load_ground_state(gs)
        xt = torch.as_tensor(x, device="cuda").to(torch.complex64)
        yt = torch.empty_like(xt)
        torch.cuda.synchronize()
        ctx.apply_liouvillian(q, xt, yt, False, TDLZ_MIXED)
        ctx.synchronize()
        err = np.linalg.norm(yt.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= 2e-5, err
    finally:
        ctx.close()
