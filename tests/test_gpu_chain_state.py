"""What one call leaves behind for another: chains of one process with spheres of different sizes
take turns, in any order, and give what each gives alone."""
import numpy as np
import pytest

from .test_gpu_work_grid import _system, lib  # noqa: F401  (lib: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_chains_of_other_spheres_take_turns(lib, precision, monkeypatch):  # noqa: F811
    """The shared-memory limit of a kernel is the process's: a chain of smaller spheres must not
    lower it under a larger one's launches (same grid side and line bound, other tile sizes)."""
    monkeypatch.setenv("LL_PRUNE", "1")
    big, small = (_system(e, 48, nproj=8, nbnd=4) for e in (50.0, 38.0))
    kw = dict(approx="rpa", precision=precision, max_steps=4)
    alone = []
    for d, x in (big, small):
        ch = lib.Chain(**kw, **d)
        alone.append([ch.apply(x, up) for up in (True, False)])
        ch.close()
    chains = [lib.Chain(**kw, **d) for d, _ in (big, small)]
    for i in (0, 1, 0, 1, 0):
        x = (big, small)[i][1]
        for up, want in zip((True, False), alone[i]):
            for p, q in zip(chains[i].apply(x, up), want):
                assert np.array_equal(p, q)
    for ch in chains:
        ch.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("flavour", ["ph", "nh"])
@pytest.mark.parametrize("split", ["0", "1"])
def test_applications_between_steps(lib, precision, flavour, split, monkeypatch):  # noqa: F811
    """Chain.apply between Chain.lanczos calls: the coefficients are those of the recursion left
    alone, bit for bit (graphs on, on a stream of its own, and eager), and the applications those of
    a fresh chain."""
    torch = pytest.importorskip("torch")
    monkeypatch.setenv("LL_SPLIT_PERK", split)
    d, x = _system(10.0, 18)
    d["eps_k"] = d["eps_k"] - 30.0       # D is positive
    d["dij"] = abs(d["dij"])
    kw = dict(approx="rpa", precision=precision, flavour=flavour, max_steps=12)
    ref = lib.Chain(**kw, **d)
    want, app = ref.lanczos(12), [ref.apply(x, up) for up in (True, False)]
    ref.close()
    for stream in (None, torch.cuda.Stream()):
        ch = lib.Chain(stream=stream.cuda_stream if stream else None, **kw, **d)
        got = []
        for i in range(4):
            for up, a in zip((True, False), app):
                for p, q in zip(ch.apply(x, up), a):
                    assert np.array_equal(p, q)
            got = ch.lanczos(3)
        ch.close()
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
