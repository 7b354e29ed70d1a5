"""Tensor-core tiles of 96 and 192 columns (bonds of three) by pairs and by
single CTAs, in launches of few and of many tiles, against the state vector.
Tolerance: 1e-5 normwise (FP16X3), as for every other path of that form."""
import numpy as np
import pytest

from oracle import statevector as sv
from rqc_inputs import make_circuit_general, uniform_bitstrings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,C,layers,seed,n,kw", [
    (5, 4, 5, 4, 1, dict()),
    (5, 4, 5, 4, 64, dict(max_lanes=64)),
    (4, 6, 4, 7, 9, dict(scheme="quadrants")),
    (5, 4, 5, 4, 3, dict(tc_ksplit=-1)),
])
def test_columns_that_are_not_powers_of_two(cuda_device, R, C, layers, seed, n, kw):
    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit_general(R, C, layers, seed)
    bits = uniform_bitstrings(R * C, n, 3)
    ref = sv.amplitudes(R * C, circ.gates, bits)
    sim = Simulator(R, C, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    for pairs in (0, 1, 2):
        out = sim.amplitudes(bits, precision="fp16x3", tc_cluster=pairs, **kw)
        assert sim.stats()["launches_contract_tc"] > 0
        assert np.linalg.norm(out - ref) < 1e-5 * np.linalg.norm(ref), pairs
    sim.close()
