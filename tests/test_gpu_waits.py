"""Bounded device waits of every stage-1 walk: a compile whose waits may run
out at any step either finishes with the normal result or returns
GP_ERR_TIMEOUT, and the driver goes on working."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2604_16613_gb300 import circuits as C
from paper_2604_16613_gb300 import native
from paper_2604_16613_gb300.dem import Bounds, DeviceCircuit, Driver

from parity import compare_arrays, oracle_edges

pytestmark = pytest.mark.gpu

NM = C.NoiseModel.uniform(1e-3)
# (walk, max_qubits) as the driver's bounds choose it for circuits of at most 31 qubits
WALKS = [("role-split below 32 qubits", 31), ("one qubit a thread, 64", 64), ("one qubit a thread, 480", 480),
         ("role-split from 481 qubits", 481), ("listed", 4096), ("listed, widest", 8192)]


def make(circ, max_qubits):
    noise = np.asarray(C.log_uniform_noise(circ.n_locations, seed=8), dtype=np.float32)
    bd = Bounds.for_circuits([circ])
    bd.max_qubits = max_qubits
    drv = Driver(bd)
    dc, nz = DeviceCircuit(circ), torch.tensor(noise, device="cuda")
    return drv, noise, lambda: drv.compile(dc, nz).to_host()


@pytest.mark.parametrize("walk,max_qubits", WALKS, ids=[w[0].replace(" ", "-") for w in WALKS])
def test_short_wait_limit_with_windows_staged(walk, max_qubits):
    """Windows are staged and the limit is a few polls, so any wait of the
    walk (for a window, a ring slot, a checkpoint) may give up at any step,
    each role on its own."""
    # 161 layers: an observable walk of many checkpoints and stretches
    circ = C.repetition_code_memory(9, 40, NM)
    drv, noise, run = make(circ, max_qubits)
    before = run()
    for limit in (1, 2, 3, 5, 9, 17, 40, 100, 300, 1000):
        for _ in range(3):
            drv.set_debug(wait_limit=limit)
            t0 = time.perf_counter()
            try:
                got = run()
            except native.GpError as e:
                assert e.code == native.GP_ERR_TIMEOUT, str(e)
                got = None
            torch.cuda.synchronize()
            assert time.perf_counter() - t0 < 30.0
            drv.set_debug()
            after = run()
            for k in before:
                assert got is None or np.array_equal(got[k], before[k]), (limit, k)
                assert np.array_equal(after[k], before[k]), (limit, k)
    compare_arrays(before, 0, oracle_edges(circ, noise), walk)
