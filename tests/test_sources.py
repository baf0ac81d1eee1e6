"""Properties of the kernels' source that no test can provoke on a GPU that works: what a wait does that runs out."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_18191_b200", "csrc")
WAIT = re.compile(r"\bmbar_wait(_cluster)?\(")
FILES = [f for f in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) if "mbar_wait" in open(f).read()]


def _read(path):
    with open(path) as f:
        return [line.split("//")[0] if "----------------" not in line else line for line in f]


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_every_bounded_wait_reports_that_it_ran_out(path):
    """A wait that gives up writes its code to the status word, in its own statement or within the next lines (two waits
    may share a report); without that the call would return success with an output that was never written."""
    lines, seen = _read(path), 0
    for i, line in enumerate(lines):
        if WAIT.search(line) and "__device__" not in line:
            seen += 1
            # "if (wait) { ... } else report", or the report close behind
            positive = re.search(r"if \(mbar_wait\w*\([^!]*\{\s*$", line)
            near = "".join(lines[i:]).split("} else")[1][:80] if positive else "".join(lines[i:i + 7])
            assert re.search(r"atomicExch\(status, DEV_TIMEOUT_", near), f"{os.path.basename(path)}:{i + 1}: {line.strip()}"
    assert seen


def test_roles_that_wait_for_input_start_after_the_dependency_wait():
    """gemm_pair_kernel: the time limit of a wait on data of the preceding kernel must not run while that kernel does."""
    text = "".join(_read(os.path.join(CSRC, "gemm_pair.cuh")))
    body = text[text.index("gemm_pair_kernel(const __grid_constant__"):text.index("__syncwarp();\n  tc_fence_before();\n  cluster_sync_all();")]
    roles = body.split("// ----------------")[1:]
    assert len(roles) == 4
    for role in roles:
        wait = WAIT.search(role)
        assert wait and "pdl_sync();" in role[:wait.start()], role[:60]
