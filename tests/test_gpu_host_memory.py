"""Host memory that runs out inside a call: the C entries return TCM_ENOMEM with a message and the context
stays usable; nothing is thrown across the ABI.  In a process of its own whose address space is limited
to what it has plus 64 MiB, with calls whose descriptors take several hundred."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, resource, sys
import numpy as np, torch
from paper_0704_1672_gb300 import synth, tcm
rng = np.random.default_rng(1)
X = torch.tensor(synth.pack(synth.uniform_ball(rng, 20, 4.0), rng.normal(size=20)), device="cuda")
ctx = tcm.Context(lmax_cap=4)
n = 4_000_000
E = torch.empty(n, dtype=torch.float64, device="cuda")
R0 = np.zeros((n, 3))
R0[:, 2] = 30.0
sets, out = np.zeros(n * ctypes.sizeof(tcm.tcm_moments_t), np.uint8), np.zeros(n * ctypes.sizeof(tcm.tcm_moments_t), np.uint8)
rot = np.zeros((n, 9))
before = ctx.tcm_direct(X, X, R0[0], cA=np.zeros(3), cB=np.zeros(3))
s = [tcm.make_system(X, center=np.zeros(3), radius=4.0) for _ in range(2)]
torch.cuda.synchronize()
soft, hard = resource.getrlimit(resource.RLIMIT_AS)
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + (64 << 20), hard))
L = tcm.lib()
codes = [L.tcm_rotate_moments(ctx._h, n, sets.ctypes.data, rot.ctypes.data, out.ctypes.data),
         L.tcm_direct_batch(ctx._h, ctypes.addressof(s[0]), ctypes.addressof(s[1]), n, None, R0.ctypes.data, E.data_ptr())]
message = L.tcm_last_error().decode()
resource.setrlimit(resource.RLIMIT_AS, (soft, hard))
assert codes == [tcm.TCM_ENOMEM, tcm.TCM_ENOMEM], codes
assert "host allocation" in message, message
assert ctx.tcm_direct(X, X, R0[0], cA=np.zeros(3), cB=np.zeros(3)) == before
ctx.close()
print("child ok")
"""


def test_host_allocations_that_fail():
    from paper_0704_1672_gb300 import build
    build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, env={**os.environ, "PYTHONPATH": root}, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "child ok" in r.stdout, (r.returncode, r.stdout[-500:], r.stderr[-2000:])
