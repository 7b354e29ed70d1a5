"""The CUDA-core step's tiles (contract_simt.cu) against the oracles, at shapes
that take every tile of its rule: many and few tiles, few columns, K and N
that are odd, three or not a multiple of four, rows that fill a tile and rows
that do not, storage in FP32 and in split 16-bit planes.  Tolerance: 1e-5
normwise, as for every FP32-equivalent form."""
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


@pytest.mark.parametrize("prec", ["fp32", "fp16x3"])
@pytest.mark.parametrize("R,C,d,n,kw", [
    (5, 5, 24, 37, dict(max_lanes=32)),                      # 128 x 64 and 64 x 64 tiles
    (5, 5, 24, 2, dict(fuse_rows=1)),                        # 32 x 64, 64 x 32
    (6, 5, 13, 130, dict(max_lanes=128)),                    # N from 2 to 16
    (4, 6, 16, 70, dict(scheme="quadrants", max_lanes=60)),  # open legs, batches
    (5, 5, 16, 3, dict(scheme="quadrants")),                 # odd side
])
def test_every_tile(cuda_device, prec, R, C, d, n, kw):
    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit(R, C, d, 9)
    bits = uniform_bitstrings(R * C, n, 9)
    ref = op.amplitudes(op.build(R, C, circ.gates), bits)
    sim = Simulator(R, C, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    out = sim.amplitudes(bits, precision=prec, flags=B.PEPS_FLAG_STEPWISE | B.PEPS_FLAG_NO_TC, **kw)
    assert sim.stats()["launches_contract_tc"] == 0
    assert relerr(out, ref) < TOL
    sim.close()


@pytest.mark.parametrize("prec", ["fp32", "fp16x3", "bf16x3"])
@pytest.mark.parametrize("R,C,layers,n", [(4, 5, 5, 19), (5, 4, 4, 64), (3, 3, 6, 5)])
def test_bonds_of_two_three_and_four(cuda_device, prec, R, C, layers, n):
    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit_general(R, C, layers, 4)
    bits = uniform_bitstrings(R * C, n, 4)
    ref = sv.amplitudes(R * C, circ.gates, bits)
    sim = Simulator(R, C, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    out = sim.amplitudes(bits, precision=prec, flags=B.PEPS_FLAG_STEPWISE | B.PEPS_FLAG_NO_TC)
    assert relerr(out, ref) < (3e-5 if prec == "bf16x3" else TOL)
    sim.close()
