"""The tensor-core step's tiles and stores (rows taken m_hi first, 32-byte
stores, items loaded 32 at a time) against the oracles, at the shapes where
they change: P below, at and above a tile's rows, runs of 1 to 16 entries,
batches, ragged lane counts around 32 items, bonds that are not powers of two,
and a workspace that is aligned to 16 bytes only.  Tolerance: 1e-5 normwise
(FP16X3), as for every other path of that form."""
import numpy as np
import pytest

from oracle import peps as op
from oracle import statevector as sv
from paper_1905_08394_gb300 import binding as B
from rqc_inputs import make_circuit, make_circuit_general, uniform_bitstrings

pytestmark = pytest.mark.gpu

TOL = 1e-5


def relerr(a, ref):
    return float(np.linalg.norm(a - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("R,C,d,n,kw", [
    (5, 6, 16, 33, dict()),                                  # dv = 4: runs of 16 bytes
    (6, 5, 20, 65, dict(max_lanes=64)),                      # more than 32 items per launch
    (5, 5, 22, 31, dict(max_lanes=31, fuse_rows=1)),         # odd lanes, one site per step
    (5, 5, 24, 7, dict(scheme="quadrants")),                 # odd side: open legs with P > 1
    (4, 6, 24, 70, dict(scheme="quadrants", max_lanes=60)),  # batches of open legs
    (4, 6, 24, 40, dict(scheme="quadrants", max_lanes=33, hold_ties=True)),
])
def test_steps_on_the_tensor_cores(cuda_device, R, C, d, n, kw):
    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit(R, C, d, 3)
    bits = uniform_bitstrings(R * C, n, 3)
    ref = op.amplitudes(op.build(R, C, circ.gates), bits)
    sim = Simulator(R, C, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    out = sim.amplitudes(bits, precision="fp16x3", flags=B.PEPS_FLAG_STEPWISE, **kw)
    assert sim.stats()["launches_contract_tc"] > 0
    assert relerr(out, ref) < TOL
    sim.close()


@pytest.mark.parametrize("prec,tol", [("fp16x3", TOL), ("bf16x3", 3e-5)])
@pytest.mark.parametrize("R,C,d,n,kw", [
    (6, 6, 24, 18, dict()),                                 # runs of 8 over h' and v'
    (6, 6, 24, 12, dict(scheme="quadrants")),               # merges, the fused dot, open legs
    (5, 5, 28, 5, dict(scheme="quadrants")),                # odd side, few tiles
])
def test_separate_corrections_with_one_accumulator_buffer(cuda_device, prec, tol, R, C, d, n, kw):
    # tc_ksplit = -1 gives every step a correction accumulator, so wide steps
    # take the epilogue that drains TMEM into registers
    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit(R, C, d, 5)
    bits = uniform_bitstrings(R * C, n, 5)
    ref = op.amplitudes(op.build(R, C, circ.gates), bits)
    sim = Simulator(R, C, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    out = sim.amplitudes(bits, precision=prec, tc_ksplit=-1, **kw)
    assert relerr(out, ref) < tol
    sim.close()


@pytest.mark.parametrize("R,C,layers,n,kw", [
    (4, 5, 5, 35, dict(max_lanes=35)),
    (4, 6, 4, 9, dict(scheme="quadrants")),   # a merge operand of 48 x 8
])
def test_bonds_that_are_not_powers_of_two(cuda_device, R, C, layers, n, kw):
    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit_general(R, C, layers, 7)
    bits = uniform_bitstrings(R * C, n, 7)
    ref = sv.amplitudes(R * C, circ.gates, bits)
    sim = Simulator(R, C, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    out = sim.amplitudes(bits, precision="fp16x3", **kw)
    assert sim.stats()["launches_contract_tc"] > 0
    assert relerr(out, ref) < TOL
    sim.close()


def test_workspace_aligned_to_16_bytes(cuda_device):
    import torch

    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit(6, 5, 20, 3)
    bits = uniform_bitstrings(30, 20, 3)
    sim = Simulator(6, 5, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    want = sim.amplitudes(bits, precision="fp16x3")
    o, keep = B.make_opts(precision="fp16x3")
    need = B.peps_workspace_bytes(sim.h, len(bits), o)
    ws = torch.empty(need + 16, dtype=torch.uint8, device=cuda_device)
    got = B.peps_amplitudes(sim.h, bits, o, ws.data_ptr() + 16, need,
                            torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(got, want)
    sim.close()
