"""Recorded steps after the q-slot's workspace was replaced: a chain set records its graph, a
larger set on the same q-slot grows the workspace, and the first set goes on.  Its
coefficients equal an uninterrupted run's (1e-9 of the largest in FP64; 2e-3 mixed, FP32
rounding carried through 13 steps), and memory that another owner has taken meanwhile (the
freed workspace's, among it) keeps its contents.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed", [False, True])
def test_graph_follows_a_replaced_workspace(mixed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from _cases import ground_state
    from paper_2203_01120_gb300 import TDLZ_FP64, TDLZ_MIXED, Context, build
    build()
    prec, tol = (TDLZ_MIXED, 2e-3) if mixed else (TDLZ_FP64, 1e-9)
    ctx = Context(0)
    try:
        q = ctx.load_ground_state(ground_state("C1"))
        a = ctx.chain_create([q], [0], 13, "nh", prec)
        a.advance(6)  # records the graph
        ctx.synchronize()
        b = ctx.chain_create([q] * 4, [0, 1, 2, 0], 6, "nh", prec)
        b.advance(6)  # a workspace for eight stacked vectors instead of two
        ctx.synchronize()
        held = [torch.full((n,), 7, dtype=torch.uint8, device="cuda")
                for n in [1 << 20] * 64 + [1 << 16] * 64]
        torch.cuda.synchronize()
        a.advance(7)
        got = a.read()
        for t in held:
            assert bool((t == 7).all())
        a.close()
        b.close()
        ref = ctx.lanczos_run([q], [0], 13, "nh", prec)
    finally:
        ctx.close()
    for key in ("alpha", "beta", "gamma", "z"):
        err = np.abs(got[key] - ref[key]).max() / np.abs(ref[key]).max()
        assert err <= tol, (key, err)
