"""The stage-1 walks and the row records on a GPU: every walk that a driver's
bounds can choose gives the same compile bit for bit, equal to the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2604_16613_gb300 import circuits as C
from paper_2604_16613_gb300.dem import Bounds, DeviceCircuit, Driver

from parity import compare_arrays, oracle_arrays

pytestmark = pytest.mark.gpu


def f32(x):
    return np.asarray(x, dtype=np.float32)


NM = C.NoiseModel.uniform(1e-3)
# max_qubits either side of every rule: role-split (below 32 and from 481),
# one qubit a thread (256 and 480 threads), listed (two widths)
QUBITS = [31, 32, 64, 65, 480, 481, 3200, 4800, 4801, 8192]


@pytest.mark.parametrize("name,circ", [
    # 1 to 3 stretches of 16 layers: 32 layers or fewer are walked whole
    ("surface3", C.rotated_surface_code_memory(3, 3, NM)),
    ("surface3_long", C.rotated_surface_code_memory(3, 12, NM)),
    ("repetition", C.repetition_code_memory(9, 40, NM)),
    ("surface5", C.rotated_surface_code_memory(5, 4, NM)),
    ("random", C.random_circuit(11)),
])
def test_every_walk_gives_the_same_model(name, circ):
    noise = f32(circ.default_noise)
    dc, nz = DeviceCircuit(circ), torch.tensor(noise, device="cuda")
    base = None
    for nq in [circ.n_qubits] + [q for q in QUBITS if q >= circ.n_qubits]:
        bd = Bounds.for_circuits([circ])
        bd.max_qubits = nq
        drv = Driver(bd)
        for segments in (3, 1):
            drv.set_tuning(obs_segments=segments)
            got = drv.compile(dc, nz).to_host()
            if base is None:
                base = got
                compare_arrays(base, 0, oracle_arrays((circ.ops, circ.recs, circ.n_qubits, noise.astype(np.float64),
                                                       "L2")), name)
            for k in base:
                assert np.array_equal(base[k], got[k]), (nq, segments, k)


@pytest.mark.parametrize("level", ["L0", "L1", "L2"])
def test_rows_of_many_columns(level):
    """With an observable word each for up to eight of the [[144,12,12]] code's
    logicals, some noise rows are seen by more word columns than a row's eight
    slots: the rest go through the overflow list."""
    circ = C.bb_memory(3, NM, seed=3)
    noise = f32(circ.default_noise)
    drv = Driver.for_circuits([circ])
    drv.set_tuning(obs_words=8)
    got = drv.compile(DeviceCircuit(circ), torch.tensor(noise, device="cuda"), level).to_host()
    compare_arrays(got, 0, oracle_arrays((circ.ops, circ.recs, circ.n_qubits, noise.astype(np.float64), level)), level)
