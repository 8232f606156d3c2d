"""The training samples where no thread can be started: the calling thread does all of
the work and the samples are the same."""
import os
import subprocess
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys, threading
sys.path.insert(0, %r)
import numpy as np
import paper_2605_08523_gb300 as ft
try:
    t = threading.Thread(target=lambda: None)
    t.start()
    t.join()
    print("threads start")
except RuntimeError:
    np.save(%r, ft.ftsp2_train_samples(100.0, 1 / 3, 40000, 7))
    print("done")
"""


def limits():
    # threads get stacks of the soft limit: larger than the address space allows
    import resource
    resource.setrlimit(resource.RLIMIT_STACK, (1 << 38, resource.getrlimit(resource.RLIMIT_STACK)[1]))
    resource.setrlimit(resource.RLIMIT_AS, (1 << 37, resource.getrlimit(resource.RLIMIT_AS)[1]))


def test_samples_without_threads(tmp_path):
    import pytest

    import __graft_entry__ as g
    g.build()
    import paper_2605_08523_gb300 as ft
    out = str(tmp_path / "x.npy")
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1")
    r = subprocess.run([sys.executable, "-c", CODE % (ROOT, out)], capture_output=True, text=True, env=env,
                       preexec_fn=limits)
    if "threads start" in r.stdout:
        pytest.skip("the limits do not keep threads from starting here")
    assert r.returncode == 0 and "done" in r.stdout, r.stderr
    assert np.array_equal(np.load(out), ft.ftsp2_train_samples(100.0, 1 / 3, 40000, 7))
