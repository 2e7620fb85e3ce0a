"""How a call waits: with the device's flags asking for blocking synchronisation,
the calling thread sleeps while a compression or decompression runs, instead of
watching for the result.  Each case runs in a process of its own, whose flags are
set before its context exists; the results equal the oracle's."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BODY = r"""
import ctypes, sys, time
flags = int(sys.argv[1])
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags_v2(0, flags) == 0
import torch
import numpy as np
import oracle, synth
import paper_2404_02826_gb300 as pc
small = synth.cosmology(30_001, seed=4)
ref, _ = oracle.compress(small, oracle.REL, 1e-3, want_perm=False)
c = pc.Compressor(small.shape[0], pc.PC_F32)
out = torch.empty(small.shape, device="cuda")
size = c.compress(torch.from_numpy(small).cuda(), pc.PC_EB_REL, 1e-3)
assert c.out[:size].cpu().numpy().tobytes() == ref
c.decompress(c.out, out, size)
assert out.cpu().numpy().tobytes() == oracle.decompress(ref).tobytes()
n = 1 << 26
pos = torch.rand((n, 3), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
c = pc.Compressor(n, pc.PC_F32)
for _ in range(3):
    size = c.compress(pos, pc.PC_EB_REL, 1e-4)
torch.cuda.synchronize()
wall, cpu = time.perf_counter(), time.thread_time()
for _ in range(20):
    c.compress(pos, pc.PC_EB_REL, 1e-4)
print("share", (time.thread_time() - cpu) / (time.perf_counter() - wall))
"""


# CU_CTX_SCHED_AUTO, SPIN, YIELD, BLOCKING_SYNC
@pytest.mark.parametrize("flags", [0, 1, 2, 4])
def test_a_blocking_device_lets_the_thread_sleep(flags, oracle_mod):
    r = subprocess.run([sys.executable, "-c", BODY, str(flags)], capture_output=True, text=True, timeout=300,
                       cwd=ROOT, env={**os.environ, "PYTHONPATH": ROOT + os.pathsep + os.environ.get("PYTHONPATH", "")})
    assert r.returncode == 0, r.stderr[-2000:]
    share = float(r.stdout.split("share")[1])
    print(f"flags {flags}: the thread ran {100 * share:.0f} % of the time")
    if flags == 4:  # a call of 3 ms: under 0.2 ms of launches
        assert share < 0.5
