"""What a process waits for before its first lattice runs."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CREATE = """
import time, torch, paper_1202_6130_gb300 as lbm
lbm.load()
torch.zeros(1, device="cuda")
torch.cuda.synchronize()
t = time.perf_counter()
sim = lbm.Simulation(64, 32, storage="fp16s")
torch.cuda.synchronize()
print((time.perf_counter() - t) * 1e3)
"""


def test_the_first_lattice_of_a_process_does_not_wait_for_its_code():
    """2.2 ms with the device code as it is, 16.5 ms where it has to be unpacked
    first; the shortest of three processes."""
    ms = [float(subprocess.run([sys.executable, "-c", CREATE], cwd=ROOT, check=True, text=True,
                               stdout=subprocess.PIPE).stdout) for _ in range(3)]
    assert min(ms) < 8.0, ms
