"""Calls from several host threads at once, on kernels that ask for different
amounts of shared memory by mechanism and batch: none may take away what
another has just asked for.
"""
import threading

import numpy as np
import pytest

from synth.configs import CONFIGS, load_mechanism, reactor_states

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _repeated(m, species, copies):
    """copies of m side by side, cut to the given number of species (no reactions)."""
    out = {k: np.concatenate([m[k]] * copies)[:species] for k in ("mw", "nasa", "tmid")}
    none = np.zeros((0, 3))
    out.update(reac=none.astype(np.int32), prod=none.astype(np.int32), arrh=none, arrh0=none,
               rtype=np.zeros(0, np.int32), rev=np.zeros(0, np.int32), eff_ptr=np.zeros(1, np.int32),
               eff_sp=np.zeros(0, np.int32), eff_val=np.zeros(0))
    return out


def test_shared_memory_of_one_kernel_from_two_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1608_05794_gb300.ck as ck
    large = load_mechanism(CONFIGS["large"]["mech"])
    # ROS4 teams of 256 threads with 86 and 113 KB, and with 118 KB in a small batch
    works = [(ck.load_mechanism(_repeated(large, 90, 1)), 400), (ck.load_mechanism(large), 400),
             (ck.load_mechanism(large), 40)]
    errors = []
    start = threading.Barrier(len(works))

    def run(gm, n):
        try:
            y = torch.ones((n, gm.n), dtype=torch.float64, device="cuda") / gm.S
            y[:, 0] = 1500.0
            p, dt = torch.full((n,), 1e5, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
            st = torch.empty(n, dtype=torch.int32, device="cuda")
            stream = torch.cuda.Stream()
            torch.cuda.synchronize()
            start.wait()
            for _ in range(400):
                ck.integrate_ros4(gm, p, y, dt, st, stream=stream)
            stream.synchronize()
            assert int(st.abs().sum()) == 0
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    threads = [threading.Thread(target=run, args=w) for w in works]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
