"""Bounded waits that "expire" in the FP64 tensor-core kernels (integer slices of lines and
contractions), in a form that hangs nothing: the test hook TDLZ_TEST_INJECT_TC_TIMEOUT=n, read
when a context is created, makes the next n waits that complete report expiry.  The call that
synchronises next returns TDLZ_ERR_TIMEOUT, on the context that launched the work and on no
other, chain creation and saving included; a context made afterwards computes correctly.
"""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TDLZ_ERR_TIMEOUT = 7


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_01120_gb300 import build
    build()
    return t


@pytest.fixture(scope="module")
def system():
    """A cell whose FP64 lines and contractions both run as slices."""
    import synth.configs as sc
    from oracle.liouvillian import Liouvillian
    from synth import random_br_vector
    sc.CONFIGS["_expiry"] = dataclasses.replace(
        sc.CONFIGS["C1"], name="C1", nocc=24, natom=6, kgrid=(1, 24, 1), seed=67)
    try:
        gs = sc.make_ground_state("_expiry", solver="random")
    finally:
        del sc.CONFIGS["_expiry"]
    x = random_br_vector(gs, seed=9)
    return gs, x, Liouvillian(gs).apply(x)


def context(monkeypatch, n):
    from paper_2203_01120_gb300 import Context
    monkeypatch.setenv("TDLZ_TEST_INJECT_TC_TIMEOUT", str(n))
    return Context(0)


def product(torch, c, gs, x, mixed=False):
    from paper_2203_01120_gb300 import TDLZ_FP64, TDLZ_MIXED
    q = c.load_ground_state(gs)
    xt = torch.as_tensor(x, device="cuda").to(torch.complex64 if mixed else torch.complex128)
    yt = torch.empty_like(xt)
    torch.cuda.synchronize()
    c.apply_liouvillian(q, xt, yt, False, TDLZ_MIXED if mixed else TDLZ_FP64)
    return yt


# one wait; some of both kinds (for operands, for products), of several kernels
@pytest.mark.parametrize("n", [1, 2, 7, 100, 5000])
def test_apply_fp64(torch, system, monkeypatch, n):
    from paper_2203_01120_gb300 import TdlzError
    gs, x, ref = system
    c = context(monkeypatch, n)
    try:
        product(torch, c, gs, x)
        with pytest.raises(TdlzError) as e:
            c.synchronize()
        assert e.value.status == TDLZ_ERR_TIMEOUT
        c.synchronize()  # reported once
    finally:
        c.close()
    c = context(monkeypatch, 0)
    try:
        y = product(torch, c, gs, x)
        c.synchronize()
        assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    finally:
        c.close()


@pytest.mark.parametrize("n", [1, 3, 200, 2000])
@pytest.mark.parametrize("mixed", [False, True])
def test_chain_creation(torch, system, monkeypatch, n, mixed):
    from paper_2203_01120_gb300 import TDLZ_FP64, TDLZ_MIXED, TdlzError
    gs, prec = system[0], TDLZ_MIXED if mixed else TDLZ_FP64
    c = context(monkeypatch, n)
    try:
        q = c.load_ground_state(gs)
        with pytest.raises(TdlzError) as e:
            c.chain_create([q, q], [0, 2], 4, "nh", prec)
        assert e.value.status == TDLZ_ERR_TIMEOUT
    finally:
        c.close()
    c = context(monkeypatch, 0)
    try:
        q = c.load_ground_state(gs)
        got = c.lanczos_run([q, q], [0, 2], 4, "nh", prec)
        assert list(got["status"]) == [0, 0] and np.isfinite(got["alpha"]).all()
    finally:
        c.close()


def test_save_reports(torch, system, monkeypatch):
    from paper_2203_01120_gb300 import TDLZ_FP64, TdlzError
    c = context(monkeypatch, 0)
    try:
        q = c.load_ground_state(system[0])
        a = c.chain_create([q], [0], 4, "nh", TDLZ_FP64)
        a.advance(1)
        a.save()
        other = context(monkeypatch, 1)
        a.advance(1)
        other.synchronize()  # another context's work is sound
        with pytest.raises(TdlzError) as e:
            a.save()
        assert e.value.status == TDLZ_ERR_TIMEOUT
        other.close()
        a.close()
    finally:
        c.close()
        context(monkeypatch, 0).close()


def test_another_context_does_not_take_the_report(torch, system, monkeypatch):
    from paper_2203_01120_gb300 import TdlzError
    gs, x, _ = system
    a = context(monkeypatch, 1)
    try:
        y = product(torch, a, gs, x, mixed=True)
        torch.cuda.synchronize()
        monkeypatch.delenv("TDLZ_TEST_INJECT_TC_TIMEOUT")
        from paper_2203_01120_gb300 import Context
        b = Context(0)
        b.synchronize()
        b.close()
        with pytest.raises(TdlzError) as e:
            a.synchronize()
        assert e.value.status == TDLZ_ERR_TIMEOUT
        assert y.shape == x.shape
    finally:
        a.close()
