"""Every operand that a call's bitstrings select is made by that call: in a
workspace filled with NaN, a call of a fresh context (its first: nothing made
by another call) and further calls of its plan, with bitstrings that select
other operands than the calls before, agree with the state vector.  An operand
that is passed over leaves NaN in the amplitude.  Tolerance: 1e-5 of the
largest amplitude (or probability), as for every FP32-equivalent form."""
import numpy as np
import pytest

from oracle import statevector as sv
from paper_1905_08394_gb300 import binding as B
from rqc_inputs import make_circuit, prefix_group_bitstrings, uniform_bitstrings

pytestmark = pytest.mark.gpu

STEP = B.PEPS_FLAG_STEPWISE


@pytest.mark.parametrize("R,C,d,n,kw", [
    (4, 4, 12, 1, dict(precision="fp32", flags=STEP)),
    (4, 4, 12, 3, dict(precision="fp16x3", flags=STEP, fuse_rows=1)),
    (4, 4, 16, 1, dict(precision="fp16x3", scheme="quadrants", hold_ties=True)),
    (4, 4, 16, 2, dict(precision="bf16x3", scheme="quadrants")),
    (3, 3, 14, 2, dict(precision="fp32", scheme="quadrants", hold_ties=True)),
    (5, 4, 12, 2, dict(precision="fp16x3", flags=STEP, sliced_cz=[0, 7])),
    (4, 4, 16, 6, dict(precision="fp16x3", scheme="quadrants", prefix_cols=2, prefix_group=3)),
    (4, 4, 12, 8, dict(precision="fp16x3", flags=STEP, prefix_cols=1, prefix_group=4)),
    (4, 4, 8, 1, dict(precision="fp32", scheme="quadrants", measured_mask=(1 << 9) - 1)),
])
@pytest.mark.parametrize("replay", [False, True])
def test_calls_in_a_workspace_of_nan(cuda_device, R, C, d, n, kw, replay):
    import torch

    circ = make_circuit(R, C, d, 3)
    psi = sv.run(R * C, circ.gates)
    measured = kw.get("measured_mask", 0)
    if measured:
        want = (np.abs(psi) ** 2).reshape(-1, measured + 1).sum(0)
    else:
        measured, want = (1 << R * C) - 1, psi
    tol = (3e-5 if kw["precision"] == "bf16x3" else 1e-5) * np.abs(want).max()
    if "prefix_cols" in kw:
        first = prefix_group_bitstrings(R, C, kw["prefix_cols"], n // kw["prefix_group"],
                                        kw["prefix_group"], 5)
    else:
        first = uniform_bitstrings(R * C, n, 5)
    h = B.peps_create(R, C)
    for g in circ.gates:
        a, b = g.qubits[0], g.qubits[-1]
        if g.kind == "1q":
            B.peps_apply_1q(h, a // C, a % C, g.U)
        else:
            B.peps_apply_cz(h, a // C, a % C, b // C, b % C)
    o, keep = B.make_opts(**kw)
    if replay:
        o.flags |= B.PEPS_FLAG_GRAPH
    need = B.peps_workspace_bytes(h, n, o)
    ws = torch.full((need,), 0xFF, dtype=torch.uint8, device=cuda_device)
    stream = torch.cuda.current_stream().cuda_stream
    every = np.uint64((1 << R * C) - 1)
    # all bits turned (every site reads its other operands), half of them, the first again
    for flip in (np.uint64(0), every, np.uint64(0x5A5A5A5A) & every, np.uint64(0)):
        bits = first ^ flip
        out = B.peps_amplitudes(h, bits, o, ws.data_ptr(), need, stream)
        ref = want[(bits & np.uint64(measured)).astype(np.int64)]
        assert np.abs(out - ref).max() <= tol, flip
    B.peps_destroy(h)
