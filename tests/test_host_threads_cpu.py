"""The host checks of a state where the process cannot have another thread: the caller does the work alone."""
import os
import resource
import subprocess
import sys

import pytest

from paper_2404_10223_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.skipif(not os.path.exists(build.LIB), reason="library not built")

SCRIPT = """
import resource
import numpy as np
from paper_2404_10223_gb300 import inputs, tnqe
w = inputs.workload("n14_mixed")
m = max(w.mps, key=lambda x: sum(t.size for t in x.tensors))
bad = [t.copy() for t in m.tensors]
bad[5][tuple(x[0] for x in np.nonzero(bad[5] == 0.0))] = 0.3
tnqe.load()
size = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (size + (256 << 20), resource.getrlimit(resource.RLIMIT_AS)[1]))
print(tnqe.tnqe_check_mps(m.tensors, m.U, w.n_alpha, w.n_beta), tnqe.tnqe_check_mps(bad, m.U, w.n_alpha, w.n_beta))
"""


def test_state_checks_without_threads():
    def stacks():                                    # a thread's stack does not fit the address space that is left
        hard = resource.getrlimit(resource.RLIMIT_STACK)[1]
        want = 1 << 30
        resource.setrlimit(resource.RLIMIT_STACK, (want if hard == resource.RLIM_INFINITY else min(want, hard), hard))

    env = dict(os.environ, PYTHONPATH=ROOT, OPENBLAS_NUM_THREADS="1", OMP_NUM_THREADS="1")
    p = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, preexec_fn=stacks, env=env, timeout=300)
    assert p.returncode == 0, p.stderr
    assert p.stdout.split()[0] == "(0," and "block structure" in p.stdout
