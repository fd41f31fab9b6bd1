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
