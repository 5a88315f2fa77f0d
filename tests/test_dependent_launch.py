"""Kernels that start before the previous launch has finished (programmatic dependent
launch) must not promise the compiler that nobody else touches their memory: an access
through a __restrict__ pointer may be moved above griddepcontrol.wait.  Read from the
source; the promise cannot be seen in a run that happens to be ordered well."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2307_11752_gb300", "csrc")

# members of Params that only host-to-device copies write (a copy is complete before the
# next kernel starts)
COPIED = {"cls", "wmask", "mat", "wall_u", "pmask", "word", "wall_f"}


def _code(path):
    with open(path) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def _kernels(text):
    """(name, parameter list, body up to the next kernel) of every __global__ function."""
    parts = re.split(r"__global__", text)[1:]
    for part in parts:
        m = re.search(r"\b(k_\w+)\s*\(", part)
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(part[i], 0)
            i += 1
        yield m.group(1), part[m.end():i - 1], part[i:]


def test_dependent_kernels_take_unqualified_pointers():
    waiting = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for name, params, body in _kernels(_code(path)):
            if "pdl_wait" in body:
                waiting.append(name)
                assert "__restrict__" not in params, (os.path.basename(path), name)
    assert {"k_step", "k_step_pair", "k_step2", "k_strip", "k_adjoint", "k_step_pair_tma"} <= set(waiting)


def test_only_copied_tables_are_qualified_in_the_step_parameters():
    text = _code(os.path.join(CSRC, "olb_kernels.cuh"))
    params = text[text.index("struct Params {"):]
    params = params[:params.index("\n};")]
    qualified = set(re.findall(r"__restrict__\s+(\w+)", params))
    assert qualified <= COPIED, qualified - COPIED
    for name in ("olb_pair.cuh", "olb_march.cuh", "olb_strip.cuh", "olb_tma.cuh"):
        assert "__restrict__" not in _code(os.path.join(CSRC, name)), name
