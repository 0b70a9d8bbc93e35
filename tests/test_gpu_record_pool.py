"""Capacity of stage 1's record pool."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2604_16613_gb300 import circuits as C
from paper_2604_16613_gb300.dem import Bounds, DeviceCircuit, Driver

from parity import compare_arrays, oracle_edges

pytestmark = pytest.mark.gpu


def many_words(n_rows, n_qubits=64, more=16):
    """n_rows X errors, each flipping one detector in every one of four word
    columns, on the last `more` qubits in five: one component a row, as many
    mask words as the driver's pool has to hold."""
    c = C.Circuit(n_qubits)
    qubits = list(range(n_qubits))
    c.gate1(C.R, qubits)
    per_layer = 24000                     # rows of one TICK layer: at most 32,767
    for at in range(0, n_rows, per_layer):
        c.tick()
        now = min(n_rows - at, per_layer)
        c.noise(C.X_ERROR, [q for i in range(at, at + now, n_qubits) for q in qubits[:at + now - i]], 1e-6)
    c.tick()
    rec = c.measure(C.M, qubits)
    for k in range(5):
        for q in range(64):
            c.detector([rec[q]] if k < 4 or q >= n_qubits - more else [])
    return c


@pytest.mark.parametrize("n_rows", [1000, 5_000_000])
def test_pool_holds_four_and_a_quarter_words_a_mechanism(n_rows):
    """21.25 million records of 5 million mechanisms, 24,000 rows a layer."""
    circ = many_words(n_rows)
    noise = np.asarray(C.log_uniform_noise(circ.n_locations, seed=3) * 1e-4, dtype=np.float32)
    drv = Driver.for_circuits([circ])
    got = drv.compile(DeviceCircuit(circ), torch.tensor(noise, device="cuda")).to_host()
    compare_arrays(got, 0, oracle_edges(circ, noise), f"{n_rows}")


def mixed(n_qubits=24, layers=12, seed=7):
    """One- and two-qubit noise of every kind on qubits whose planes are zero
    in one basis, in the other, in both or in neither: records of every number
    of entries."""
    rng = np.random.default_rng(seed)
    c = C.Circuit(n_qubits)
    z, x = list(range(0, n_qubits, 2)), list(range(1, n_qubits, 2))
    c.gate1(C.R, z)
    c.gate1(C.RX, x)
    for _ in range(layers):
        c.tick()
        for kind in (C.X_ERROR, C.Z_ERROR, C.DEPOLARIZE1):
            c.noise(kind, [int(q) for q in rng.permutation(n_qubits)[:n_qubits - 3]], 1e-3)
        pairs = [int(q) for q in rng.permutation(n_qubits)[:n_qubits - 4]]
        c.noise(C.DEPOLARIZE2, pairs, 1e-3)
    c.tick()
    rz, rx = c.measure(C.M, z[:-1]), c.measure(C.MX, x[:-2])
    for i, r in enumerate(list(rz) + list(rx)):
        for _ in range(1 + (i % 3) * 40):       # detectors spread over several word columns
            c.detector([r])
    return c


@pytest.mark.parametrize("level", ["L0", "L1", "L2"])
@pytest.mark.parametrize("max_qubits", [24, 64, 481, 4096])
def test_records_of_every_number_of_entries(level, max_qubits):
    circ = mixed()
    noise = np.asarray(C.log_uniform_noise(circ.n_locations, seed=4), dtype=np.float32)
    bd = Bounds.for_circuits([circ])
    bd.max_qubits = max_qubits
    got = Driver(bd).compile(DeviceCircuit(circ), torch.tensor(noise, device="cuda"), level).to_host()
    compare_arrays(got, 0, oracle_edges(circ, noise, level), level)


def test_rows_indexed_by_mechanism_in_a_batch():
    """Bounds of fewer mechanisms than circuit rows: the rows of every circuit
    go by their first mechanism."""
    circs = [many_words(1000), many_words(77), mixed(n_qubits=64, layers=1), many_words(3)]
    circs[2]._ops = [np.concatenate([circs[2].ops[circs[2].ops[:, 0] < 34]])]     # X and Z errors only
    circs[2]._frozen = None
    noises = [np.asarray(C.log_uniform_noise(c.n_locations, seed=6 + i), dtype=np.float32) for i, c in enumerate(circs)]
    bd = Bounds.for_circuits(circs)
    assert bd.max_mechanisms < bd.max_ops
    host = Driver(bd).compile(circs, np.concatenate(noises)).to_host()
    for i, (c, nz) in enumerate(zip(circs, noises)):
        compare_arrays(host, i, oracle_edges(c, nz), f"circuit {i}")
