"""A fused dot product over a merge of N = 8 and many rows (16-column tiles,
whose idle epilogue warps have slots too) against the state vector, on a first
call and on calls of the plan that it leaves.  Tolerance: the unit roundoff of
TF32, 2^-11, times the square root of the number of steps, times 8, as for
every TF32 call of the square partition."""
import math

import numpy as np
import pytest

from oracle import statevector as sv
from rqc_inputs import make_circuit, uniform_bitstrings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,d", [(10, 22), (8, 26)])
def test_narrow_merge_with_many_rows(cuda_device, C, d):
    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit(2, C, d, 1)
    psi = sv.run(2 * C, circ.gates)
    sim = Simulator(2, C, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    for seed in (1, 2, 2):
        bits = uniform_bitstrings(2 * C, 20, seed)   # 16 lanes and 4
        ref = psi[bits.astype(np.int64)]
        out = sim.amplitudes(bits, precision="tf32", scheme="quadrants")
        tol = 8 * 2.0 ** -11 * math.sqrt(sim.stats()["n_steps"])
        assert np.linalg.norm(out - ref) < tol * np.linalg.norm(ref), seed
    sim.close()
