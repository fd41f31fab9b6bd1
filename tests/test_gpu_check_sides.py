"""The bounds-checked build on every grid side, line bound and lane split of the plane pass, in both
precisions, on the per-k paths, and on spheres that only the general plane kernel takes: no index out
of its table's range, and the plain build's results."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from .test_gpu_check_build import check_lib  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import json, os, sys
import numpy as np
sys.path.insert(0, {root!r})
os.environ["LL_PRUNE"] = "1"
from tests.test_gpu_fixed_lines import GRIDS
from tests.test_gpu_far_q import FAR, WIDE, zones
from tests.test_gpu_work_grid import _system
from paper_2111_06623_gb300 import ll
systems = [_system(e, n) for n, e in GRIDS] + [_system(e, n, q=(q, 0.2, 0.1)) for n, e, q in FAR]
systems += [_system(e, n, q=q, nbnd=2) for n, e, q in WIDE[:3]]
for n, e in ((12, 4.4), (18, 10.0), (24, 17.8), (48, 50.0)):
    systems.append(_system(e, n))
    zones(systems[-1][0])
out = []
for split in ("0", "1"):
    os.environ["LL_SPLIT_PERK"] = split
    for d, x in systems:
        for prec in ("fp32", "fp64"):
            ch = ll.Chain(approx="rpa", precision=prec, flavour="nh", max_steps=2, **d)
            for up in (False, True):
                y = np.concatenate([v.ravel() for v in ch.apply(x, up)])
                out.append([float(np.linalg.norm(y)), float(y[0].real), float(y[-1].imag)])
            b, g, z = ch.lanczos(2)
            out.append([float(b[1]), float(z[0].real), float(z[1].real)])
            ch.close()
print(json.dumps(out))
"""


def _run(lib_path):
    env = dict(os.environ)
    env.pop("LL_LIBRARY", None)
    if lib_path:
        env["LL_LIBRARY"] = lib_path
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT)], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    return np.array(json.loads(r.stdout.strip().splitlines()[-1]))


def test_every_side_without_an_index_out_of_range(check_lib):  # noqa: F811
    got, want = _run(check_lib), _run(None)       # raises on LL_EINVAL (an index out of range)
    assert np.all(abs(got - want) <= 2e-5 * abs(want).max(axis=1, keepdims=True))
