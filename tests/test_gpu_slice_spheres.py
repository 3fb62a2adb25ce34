"""FP64 X and Y lines by integer slices on larger spheres: largest Miller index h from 9 up to the
15 that the matrix image holds, on both axes (every index pair of a thread, the upper outputs of
the forward sum), h = 16 and spheres that reach half the line, which take another form.  L x
against the oracle (relative L2 <= 1e-12, the parity suite's bar) and against the FP64-pipe
forms (<= 1e-13, a few roundings); bits differ where the slices ran.
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,q", [
    ((45, 45), (10, 10), 0.1), ((48, 48), (15, 15), 0.1), ((40, 48), (9, 13), 0.1),
    ((32, 30), (15, 14), 0.1), ((36, 32), (14, 15), -0.1), ((48, 45), (16, 12), 0.1),
    ((45, 48), (12, 16), 0.1), ((30, 48), (14, 15), 0.5)])
def test_larger_spheres(n, h, q, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth.configs as sc
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_FP64, Context, build
    from synth import random_br_vector
    build()
    gmax = 4.0
    edge = [(m + 0.6) * 2.0 * np.pi / gmax for m in (*h, 2)]
    sc.CONFIGS["_sphere"] = dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", lattice=np.diag(edge), fft=(*n, 12), ecut=0.5 * gmax ** 2,
        kgrid=(1, 1, 2), nocc=19, alat=edge[0], q_2pi_a=(q, 0.0, 0.0), seed=67)
    try:
        gs = sc.make_ground_state("_sphere", solver="random")
    finally:
        del sc.CONFIGS["_sphere"]
    m = [gs.miller_kq[k, :gs.npw_kq[k]] for k in range(gs.nk)]
    reach = [max(int(np.abs(v[:, a]).max()) for v in m) for a in range(2)]
    assert reach == [h[0] + (abs(q) == 0.5), h[1]]
    # 64-line tiles of one vector, rows 4 nk nocc: the slices take 608 and more
    planes = max(len(set(v[:, 0].tolist())) for v in m)
    assert all(-(-12 * lines // 64) * 4 * gs.nk * 19 >= 608 for lines in (n[1], planes))
    x = random_br_vector(gs, seed=8)
    ref = Liouvillian(gs).apply(x)
    y = {}
    for tc in "01":
        monkeypatch.setenv("TDLZ_TC", tc)
        ctx = Context(0)
        try:
            slot = ctx.load_ground_state(gs)
            xt = torch.as_tensor(x, device="cuda")
            yt = torch.empty_like(xt)
            torch.cuda.synchronize()
            ctx.apply_liouvillian(slot, xt, yt, False, TDLZ_FP64)
            ctx.synchronize()
            y[tc] = yt.cpu().numpy()
        finally:
            ctx.close()
        err = np.linalg.norm(y[tc] - ref) / np.linalg.norm(ref)
        assert err <= 1e-12, (tc, err)
    assert not np.array_equal(y["0"], y["1"])
    assert np.linalg.norm(y["1"] - y["0"]) <= 1e-13 * np.linalg.norm(ref)
