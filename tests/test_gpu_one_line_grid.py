"""Grids of one line (two axes of one point): stacked chains against the oracle's recursion
one chain at a time, FP64.  The Hartree filter's lines are then whole grids, one per stacked
vector.  Bars of the parity suite's coefficients: 1e-8 of the largest one, 5 steps.
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fft", [(24, 1, 1), (1, 20, 1), (1, 1, 18)])
def test_stacked_chains_on_one_line(fft):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth.configs as sc
    from oracle.lanczos import run_chain
    from oracle.liouvillian import Liouvillian
    from paper_2203_01120_gb300 import TDLZ_FP64, Context, build
    build()
    sc.CONFIGS["_line"] = dataclasses.replace(
        sc.CONFIGS["C0"], name="C0", lattice=np.diag([20.0 if n > 1 else 2.0 for n in fft]),
        fft=fft, ecut=2.0, kgrid=tuple(2 if n > 1 else 1 for n in fft), nocc=2,
        q_2pi_a=tuple(0.03 if n > 1 else 0.0 for n in fft), seed=59)
    try:
        gs = sc.make_ground_state("_line", solver="random")
    finally:
        del sc.CONFIGS["_line"]
    lv = Liouvillian(gs)
    ctx = Context(0)
    try:
        q = ctx.load_ground_state(gs)
        got = ctx.lanczos_run([q, q, q], [0, 1, 2], 5, "nh", TDLZ_FP64)
    finally:
        ctx.close()
    for mu in range(3):
        ref = run_chain(lv, mu, 5, "nh")
        for key in ("alpha", "beta", "gamma", "z"):
            want = np.asarray(getattr(ref, key))
            err = np.abs(np.asarray(got[key][mu]) - want).max() / np.abs(want).max()
            assert err <= 1e-8, (mu, key, err)
