"""Surrogate contexts whose first calls come from several host threads at once: each gives what it
gives alone, in a process that has made no surrogate call before."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import threading
import numpy as np
from paper_1107_2619_gb300 import inputs as I, md

def run(seed, out):
    theta = I.sur_init_weights(seed).astype(np.float32)
    with md.SurrogateSystem(I.bcc_fe(12, seed=seed), theta, np.ones(32, np.float32), np.full(32, 0.5, np.float32)) as s:
        s.eam_forces()
        s.step(3)
        out[seed] = s.positions(), s.forces()

together, alone = {}, {}
threads = [threading.Thread(target=run, args=(q, together)) for q in range(6)]
for t in threads:
    t.start()
for t in threads:
    t.join()
for q in range(6):
    run(q, alone)
    assert all(np.array_equal(a, b) for a, b in zip(together[q], alone[q])), q
print("same")
"""


def test_first_calls_from_threads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_2619_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stderr[-2000:]
