"""Index checks (FLAME_DEBUG_BOUNDS build) of the adjoint step and of the sizes
where lines change length.

The source says which accesses are checked: each adjoint kernel checks the
arrays it reads and writes, and a failed check is recorded in the handle's
status, the step's pass A within an adjoint step included.  The gradient and
line-length tests then run clean against the index-checking library.
"""
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0911_2889_gb300", "csrc")

# arrays of each adjoint kernel, by the site their checks name
CHECKS = {"k_adjL": {"Lam": 2, "Row": 2}, "k_adjB": {"Row": 1, "Uv": 1, "Aw": 1}, "k_adjC": {"Aw": 1, "Lam": 2, "State": 1}}


def _body(name, text):
    at = text.index("void __launch_bounds__", text.index(f" {name}(") - 120)
    end = text.find("__global__", at)
    return text[at:end if end > 0 else len(text)]


@pytest.mark.parametrize("kernel", list(CHECKS))
def test_adjoint_kernels_check_their_indices(kernel):
    body = _body(kernel, open(os.path.join(CSRC, "flame_adjoint.cuh")).read())
    for site, n in CHECKS[kernel].items():
        assert len(re.findall(r"FLAME_IN\(d\.status,[^;]*?kSiteAdj" + site + r"\b", body)) >= n, (kernel, site)


def test_failed_checks_of_an_adjoint_step_reach_the_handle():
    ops = open(os.path.join(CSRC, "flame_ops.cuh")).read()
    step = ops[ops.index("Ops<R>::adj_step("):]
    assert "f.status = d.status" in step[:step.index("passA(f")]
    api = open(os.path.join(CSRC, "flame_api.cu")).read()
    adj = api[api.index("flame_status flame_adjoint("):]
    assert "d.status = h->status" in adj[:adj.index("adj_step(d, q)")]


@pytest.mark.gpu
def test_gradients_and_line_lengths_run_clean_under_index_checks():
    from paper_0911_2889_gb300 import build
    build.build_library(debug=True)
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider", "-k", "not 200_steps and not _fd",
           "tests/test_gpu_adjoint.py", "tests/test_gpu_grids.py"]
    r = subprocess.run(cmd, cwd=ROOT, env=dict(os.environ, FLAME_DEBUG_BOUNDS="1"), capture_output=True, text=True,
                       timeout=3000)
    tail = r.stdout[-4000:] + r.stderr[-2000:]
    assert r.returncode == 0 and " passed" in tail and "failed" not in tail, tail
