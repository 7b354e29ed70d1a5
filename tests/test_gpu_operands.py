"""Site operands made for the bitstrings of a call only: whichever variants a
call reads, its amplitudes are those of a call that reads (and makes) them all."""
import numpy as np
import pytest

from paper_1905_08394_gb300 import binding as B
from rqc_inputs import make_circuit, uniform_bitstrings

pytestmark = pytest.mark.gpu


# one launch per step, so that the operands of every step pass through the
# builders; more than 1024 bitstrings make all of them.  The lanes' arithmetic
# does not depend on their number: FP32 sums in one order, tensor-core tiles
# with the same K passes.  1e-6 of the largest amplitude allows for the tile
# variants that a launch's size picks.
@pytest.mark.parametrize("R,C,d,kw", [
    (4, 4, 12, dict(precision="fp32", flags=B.PEPS_FLAG_STEPWISE)),
    (4, 4, 12, dict(precision="fp16x3", flags=B.PEPS_FLAG_STEPWISE)),
    (4, 4, 16, dict(precision="fp16x3", scheme="quadrants", hold_ties=True)),
    (5, 4, 12, dict(precision="fp16x3", flags=B.PEPS_FLAG_STEPWISE, sliced_cz=[0, 7])),
])
def test_amplitudes_do_not_depend_on_the_other_bitstrings(cuda_device, R, C, d, kw):
    from paper_1905_08394_gb300 import Simulator

    bits = uniform_bitstrings(R * C, 1025, 5)
    sim = Simulator(R, C, device=cuda_device.index or 0)
    sim.apply_circuit(make_circuit(R, C, d, 3))
    every = sim.amplitudes(bits, **kw)
    tol = 1e-6 * np.abs(every).max()
    for n in (1, 2, 33, 1024):
        for first in (0, 1, 1025 - n):   # one plan, other bitstrings: marks of a call before are cleared
            got = sim.amplitudes(bits[first:first + n], **kw)
            assert np.abs(got - every[first:first + n]).max() <= tol, (n, first)
    sim.close()
