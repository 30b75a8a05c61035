"""The bounded wait of the FP32 row pass for its bulk copies (flame_step.cuh).

The index-checking build can announce those copies without issuing them
(FLAME_FAULT_INJECT=wait), so that every wait runs out.  The row pass then
uses nothing of what it read: G is NaN, hence the state and the mean mode, which
a caller of flame_step_noalloc sees as well, and a handle's status is
FLAME_ETIMEOUT.  Both work on afterwards.
"""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STALLED_STEP = r"""
import os
import torch
from paper_0911_2889_gb300 import flame, inputs
assert flame.debug_bounds()
f = flame.Flame(256, 512, prec="fp32", t0=20.0, dt=1e-3)
st0 = torch.from_numpy(flame.box_to_abi(inputs.spectrum_ic(256, 512, 16, 3, amp=0.1, K1=f.K1, K2=f.K2))).cuda().to(f.cdtype)
def step():
    s = st0.clone()
    m = torch.zeros(1, dtype=torch.float64, device="cuda")
    t = torch.full((1,), 20.0, dtype=torch.float64, device="cuda")
    f.step(s, m, t, 1)
    return torch.view_as_real(s).cpu(), m.item(), t.item()
ref, mref, tref = step()
f.sync_status()
os.environ["FLAME_FAULT_INJECT"] = "wait"
got, m, t = step()
try:
    f.sync_status()
except flame.FlameError as e:
    assert e.status == flame.FLAME_ETIMEOUT, e
else:
    raise SystemExit("no FLAME_ETIMEOUT")
assert got.isnan().reshape(-1, 2).any(1).sum().item() >= got.numel() // 2 - 1 and m != m and t == tref
del os.environ["FLAME_FAULT_INJECT"]
got, m, t = step()
f.sync_status()
assert torch.equal(got, ref) and m == mref and t == tref
f.close()

# the step without allocations has no handle to ask
def noalloc():
    s = st0.clone()
    m = torch.zeros(1, dtype=torch.float64, device="cuda")
    t = torch.full((1,), 20.0, dtype=torch.float64, device="cuda")
    flame.flame_step_noalloc(f.params, s, m, t, 1)
    return torch.view_as_real(s).cpu(), m.item(), t.item()
ref, mref, tref = noalloc()
os.environ["FLAME_FAULT_INJECT"] = "wait"
got, m, t = noalloc()
assert got.isnan().reshape(-1, 2).any(1).sum().item() >= got.numel() // 2 - 1 and m != m and t == tref
del os.environ["FLAME_FAULT_INJECT"]
got, m, t = noalloc()
assert torch.equal(got, ref) and m == mref and t == tref
print("wait ok")
"""


@pytest.mark.gpu
@pytest.mark.parametrize("variants", ["1,0", "3,2"])
def test_row_pass_makes_its_output_nan_when_its_wait_runs_out(variants):
    from paper_0911_2889_gb300 import build
    build.build_library(debug=True)
    env = dict(os.environ, FLAME_DEBUG_BOUNDS="1", FLAME_FORCE_VARIANTS=variants)
    env.pop("FLAME_FAULT_INJECT", None)
    r = subprocess.run([sys.executable, "-c", STALLED_STEP], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "wait ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
