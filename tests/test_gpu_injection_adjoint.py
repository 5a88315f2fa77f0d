"""An armed olb_inject_stalled_copy and a gradient run: the injection applies to one step,
the first one of the forward sweep, and is used up by it whichever way the sweep runs its
segments.  (The wait that runs out is bounded at 20 ms; see the test of the timeout path.)
In a child process, because the kernel selection is read from the environment once."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import json, sys
sys.path.insert(0, %(root)r); sys.path.insert(0, %(tests)r)
from paper_2307_11752_gb300 import olb
from _cases import porous_channel_case
lib = olb.load()
out = {}
for every in (8, 3):
    g = porous_channel_case(nx=64, ny=21, nz=13).gpu("f32", "pull")  # even nx: the TMA-fed kernel
    g.step(2)
    rc = [lib.olb_synchronize(g.handle), lib.olb_inject_stalled_copy(g.handle, 16, 20_000_000)]
    g.adjoint_run(8, every, (0, 63, 0))
    rc.append(lib.olb_synchronize(g.handle))
    g.step(1)
    rc.append(lib.olb_synchronize(g.handle))
    g.close()
    out[every] = rc
print(json.dumps(out))
'''


@pytest.fixture(scope="module")
def gpu():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_11752_gb300 import build
    build.build()


def test_an_injection_is_used_up_by_one_step_of_a_gradient(gpu):
    code = CHILD % {"root": ROOT, "tests": os.path.join(ROOT, "tests")}
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, OLB_TMA="1"))
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    for every, rc in out.items():
        assert rc == [0, 0, -6, 0], (every, rc)  # the timeout is reported once, the next step is not affected
