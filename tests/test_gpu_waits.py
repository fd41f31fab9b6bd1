"""The bounded waits of the plane pass: one that runs out (LL_WAIT_POLLS=0: every one does, though
each copy arrives) ends its call with LL_ETIMEOUT, in ll_create, ll_lanczos and ll_apply alike;
the context, other chains and, after an application, the chain itself go on as if nothing had been."""
import numpy as np
import pytest

from .test_gpu_work_grid import _system, lib  # noqa: F401  (lib: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nfft,ecut", [(12, 4.4), (24, 17.8), (32, 30.0), (48, 50.0)])
def test_a_wait_that_runs_out(lib, precision, nfft, ecut, monkeypatch):  # noqa: F811
    d, x = _system(ecut, nfft)
    d["eps_k"], d["dij"] = d["eps_k"] - 30.0, abs(d["dij"])      # D is positive
    kw = dict(approx="rpa", precision=precision, max_steps=8, **d)
    ref = lib.Chain(**kw)
    app, want = [ref.apply(x, up) for up in (True, False)], ref.lanczos(8)
    ch = lib.Chain(**kw)
    ch.lanczos(2)
    monkeypatch.setenv("LL_WAIT_POLLS", "0")
    for up in (True, False):
        with pytest.raises(lib.LLError) as e:
            ch.apply(x, up)
        assert e.value.code == lib.LL_ETIMEOUT and "gave up" in str(e.value)
    with pytest.raises(lib.LLError) as e:
        lib.Chain(**kw)
    assert e.value.code == lib.LL_ETIMEOUT
    with pytest.raises(lib.LLError) as e:
        ref_nh = lib.Chain(flavour="nh", **kw)
        ref_nh.lanczos(4)
    assert e.value.code == lib.LL_ETIMEOUT
    monkeypatch.delenv("LL_WAIT_POLLS")
    for up, a in zip((True, False), app):
        for p, q in zip(ch.apply(x, up), a):
            assert np.array_equal(p, q)
    for a, b in zip(ch.lanczos(6), want):
        assert np.array_equal(a, b)
