"""Launch shapes and sizes of the stage-1 walks that only some bounds reach:
the role-split walk at each of its block sizes, the listed walk on circuits
that fill more than one stride of its threads, and a server whose windows are
role-split."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2604_16613_gb300 import circuits as C
from paper_2604_16613_gb300 import native
from paper_2604_16613_gb300.dem import Bounds, DeviceCircuit, Driver
from paper_2604_16613_gb300.serve import Server

from parity import compare_arrays, compare_edges, oracle_edges

pytestmark = pytest.mark.gpu

NM = C.NoiseModel.uniform(1e-3)


def make(circ, max_qubits):
    noise = np.asarray(C.log_uniform_noise(circ.n_locations, seed=5), dtype=np.float32)
    bd = Bounds.for_circuits([circ])
    bd.max_qubits = max_qubits
    drv = Driver(bd)
    dc, nz = DeviceCircuit(circ), torch.tensor(noise, device="cuda")
    return drv, noise, lambda level="L2": drv.compile(dc, nz, level).to_host()


@pytest.mark.parametrize("max_qubits,circ", [
    (31, C.repetition_code_memory(9, 40, NM)),             # a long observable, few candidates a step
    (31, C.rotated_surface_code_memory(3, 12, NM)),
    (481, C.rotated_surface_code_memory(9, 9, NM)),
    (481, C.bb_memory(3, NM, seed=3)),                     # steps of more than 64 candidates: the helper walkers
    (577, C.rotated_surface_code_memory(17, 4, NM)),       # every qubit of the bounds in use
], ids=["repetition9", "surface3", "surface9", "bb", "surface17"])
def test_role_split_block_sizes(max_qubits, circ):
    drv, noise, run = make(circ, max_qubits)
    for level in ("L0", "L2"):
        ref = oracle_edges(circ, noise, level)
        base = None
        for threads in (128, 256, 512, 1024):
            for segments in (1, 2, 3):
                drv.set_tuning(stage1_threads=threads, obs_segments=segments)
                got = run(level)
                if base is None:
                    base = got
                    compare_arrays(base, 0, ref, f"{level} {threads}")
                for k in base:
                    assert np.array_equal(base[k], got[k]), (level, threads, segments, k)


@pytest.mark.parametrize("max_qubits,threads", [(31, 512), (481, 128), (481, 256), (481, 512), (481, 1024)])
def test_role_split_wait_that_runs_out(max_qubits, threads):
    """No window is staged and the limit is short, so the walker's first wait
    runs out: every role leaves (helpers, emitters, producer), the compile
    returns GP_ERR_TIMEOUT and the next one is right again."""
    circ = C.repetition_code_memory(9, 40, NM) if max_qubits < 32 else C.bb_memory(3, NM, seed=3)
    drv, noise, run = make(circ, max_qubits)
    drv.set_tuning(stage1_threads=threads)
    before = run()
    drv.set_debug(wait_limit=256, stall_windows=1)
    t0 = time.perf_counter()
    with pytest.raises(native.GpError) as e:
        run()
    assert e.value.code == native.GP_ERR_TIMEOUT, str(e.value)
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 30.0
    drv.set_debug()
    after = run()
    compare_arrays(after, 0, oracle_edges(circ, noise), "after the timeout")
    for k in before:
        assert np.array_equal(after[k], before[k]), k


@pytest.mark.parametrize("d,rounds,max_qubits", [
    (23, 5, 3200),      # 1,057 qubits, 41 layers: checkpoints over two strides of 960 threads
    (37, 2, 2737),      # 2,737 qubits, 17 layers: bounds too wide for the role-split tables
    (37, 5, 2880),      # the same with 41 layers
    (41, 5, 3840),      # 3,361 qubits, four strides
    (45, 5, 4049),      # 4,049 qubits, five strides
    (49, 5, 4801),      # 4,801 qubits: the widest instance, six strides, 41 layers
], ids=["d23", "d37", "d37_long", "d41", "d45", "d49"])
def test_listed_walk_over_several_strides(d, rounds, max_qubits):
    circ = C.rotated_surface_code_memory(d, rounds, NM)
    drv, noise, run = make(circ, max_qubits)
    base = run()
    compare_arrays(base, 0, oracle_edges(circ, noise), f"d={d}")
    drv.set_tuning(obs_segments=1)                          # the role-split walk's: the same walk here
    got = run()
    for k in base:
        assert np.array_equal(base[k], got[k]), k


def test_stream_of_a_role_split_patch():
    """A patch of 577 qubits streamed cycle by cycle, with and without a
    narrow patch beside it, equals its full compile and the oracle's model."""
    circ = C.rotated_surface_code_memory(17, 4, NM)
    small = C.rotated_surface_code_memory(3, 6, NM)
    noise = np.asarray(circ.default_noise, dtype=np.float32)
    ref = Driver.for_circuits([circ]).compile(circ, noise).edges()
    small_ref = Driver.for_circuits([small]).compile(small, np.asarray(small.default_noise, np.float32)).edges()
    assert Server.for_circuits([circ], max_cycles_per_step=1, max_horizon=1).stream([circ], [1])[0] == ref
    both = Server.for_circuits([circ, small], max_cycles_per_step=2, max_horizon=1).stream([circ, small], [1, 1])
    assert both[0] == ref and both[1] == small_ref
    compare_edges(ref, oracle_edges(circ, noise).edges(), "d=17")


@pytest.mark.parametrize("max_qubits", [2520, 2521, 2880, 2881, 3840, 3841])
def test_bounds_either_side_of_the_listed_widths(max_qubits):
    circ = C.rotated_surface_code_memory(5, 6, NM)
    noise = np.asarray(C.log_uniform_noise(circ.n_locations, seed=5), dtype=np.float32)
    base = Driver.for_circuits([circ]).compile(DeviceCircuit(circ), torch.tensor(noise, device="cuda")).to_host()
    got = make(circ, max_qubits)[2]()
    for k in base:
        assert np.array_equal(base[k], got[k]), k


@pytest.mark.parametrize("max_qubits,threads", [(31, 512), (481, 512), (577, 256), (1249, 512), (2500, 512)])
def test_more_blocks_per_sm_than_fit(max_qubits, threads):
    """Blocks per SM beyond what the shared memory holds: as many as fit."""
    circ = C.rotated_surface_code_memory(3, 12, NM)
    drv, noise, run = make(circ, max_qubits)
    base = run()
    compare_arrays(base, 0, oracle_edges(circ, noise), f"{max_qubits}")
    for blocks in (1, 2, 5, 64):
        drv.set_tuning(stage1_threads=threads, stage1_blocks_per_sm=blocks)
        got = run()
        for k in base:
            assert np.array_equal(base[k], got[k]), (blocks, k)
