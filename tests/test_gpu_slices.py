"""FP64 contractions by integer slices on the tensor cores: L x at band counts around the
tiles' edges (column tiles of 24 bands, row tiles of 128, the contraction's stages of 16 and
drains of 64 plane waves), against the oracle (relative L2 <= 1e-12, the parity suite's bar)
and against the FP64-pipe form (a few roundings: <= 1e-13; bits differ where the slices ran);
stacked chains against the FP64-pipe form; non-finite input stays non-finite.  Random
orthonormal states in 12^3 and 16^3 cells.
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cell,nocc,natom,nk", [
    ("C0", 24, 6, 6), ("C0", 25, 7, 6), ("C0", 40, 10, 3), ("C0", 49, 13, 3), ("C0", 64, 16, 2),
    ("C0", 130, 33, 1), ("C1", 24, 6, 24), ("C1", 25, 7, 24), ("C1", 40, 10, 8), ("C1", 49, 13, 6),
    ("C1", 70, 18, 4), ("C1", 130, 33, 2)])
def test_slices(cell, nocc, natom, nk, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth.configs as sc
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_FP64, Context, build
    from synth import random_br_vector
    build()
    monkeypatch.setitem(sc.CONFIGS, "_slices", dataclasses.replace(
        sc.CONFIGS[cell], name=cell, nocc=nocc, natom=natom, kgrid=(1, nk, 1), seed=37))
    gs = sc.make_ground_state("_slices", solver="random")
    x = random_br_vector(gs, seed=6)
    ref = Liouvillian(gs).apply(x)
    y, run = {}, {}
    for tc in "01":
        monkeypatch.setenv("TDLZ_TC", tc)
        ctx = Context(0)
        try:
            q = ctx.load_ground_state(gs)
            xt = torch.as_tensor(x, device="cuda")
            yt = torch.empty_like(xt)
            torch.cuda.synchronize()
            ctx.apply_liouvillian(q, xt, yt, False, TDLZ_FP64)
            ctx.synchronize()
            y[tc] = yt.cpu().numpy()
            err = np.linalg.norm(y[tc] - ref) / np.linalg.norm(ref)
            assert err <= 1e-12, (tc, err)
            run[tc] = ctx.lanczos_run([q, q], [0, 2], 2, "nh", TDLZ_FP64)
            xt.view(-1)[3] = complex(np.inf, 0.0)
            torch.cuda.synchronize()
            ctx.apply_liouvillian(q, xt, yt, False, TDLZ_FP64)
            ctx.synchronize()
            assert not torch.isfinite(torch.view_as_real(yt)).all()
        finally:
            ctx.close()
    if cell == "C1":  # 300 plane waves: the slices are the faster form
        assert not np.array_equal(y["0"], y["1"])
    assert np.linalg.norm(y["1"] - y["0"]) <= 1e-13 * np.linalg.norm(ref)
    for key in ("alpha", "beta", "gamma"):
        a, b = np.asarray(run["0"][key]), np.asarray(run["1"][key])
        assert np.allclose(a, b, rtol=1e-11, atol=1e-11 * np.abs(a).max()), key


@pytest.mark.parametrize("fft,ecut,nk,nocc", [
    ((15, 18, 20), 3.6, 4, 24), ((24, 25, 27), 12.0, 2, 20), ((32, 30, 36), 20.0, 2, 10),
    ((40, 45, 24), 12.0, 2, 20), ((48, 32, 32), 20.0, 1, 22), ((54, 48, 20), 12.0, 2, 30)])
def test_slice_lines(fft, ecut, nk, nocc, monkeypatch):
    """X and Y lines by slices: even and odd lengths up to 48, one and two halves of the
    forward sum, lengths without a register transform, ragged last tiles, and 54 (another line
    transform).  Same bars; scaled by 1e-290 (results near
    the end of the normal range) and zero."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth.configs as sc
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_FP64, Context, build
    from synth import random_br_vector
    build()
    monkeypatch.setitem(sc.CONFIGS, "_lines64", dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", fft=fft, ecut=ecut, nocc=nocc, kgrid=(1, nk, 1), seed=41))
    gs = sc.make_ground_state("_lines64", solver="random")
    x = random_br_vector(gs, seed=8)
    ref = Liouvillian(gs).apply(x)
    y = {}
    for tc in "01":
        monkeypatch.setenv("TDLZ_TC", tc)
        ctx = Context(0)
        try:
            q = ctx.load_ground_state(gs)
            for scale in (1.0, 1e-290, 0.0):
                xt = torch.as_tensor(x * scale, device="cuda")
                yt = torch.empty_like(xt)
                torch.cuda.synchronize()
                ctx.apply_liouvillian(q, xt, yt, False, TDLZ_FP64)
                ctx.synchronize()
                got = yt.cpu().numpy()
                if scale == 0.0:
                    assert not got.any()
                    continue
                err = np.linalg.norm(got / scale - ref) / np.linalg.norm(ref)
                assert err <= 1e-12, (tc, scale, err)
                y.setdefault(tc, got)
        finally:
            ctx.close()
    assert not np.array_equal(y["0"], y["1"])
    assert np.linalg.norm(y["1"] - y["0"]) <= 1e-13 * np.linalg.norm(ref)
