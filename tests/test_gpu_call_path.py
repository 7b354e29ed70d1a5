"""The host side of a call: the workspace size asked of a context that holds a
plan equals that of a fresh context, whatever changed since; and a call that
fails leaves the caller's array as it was."""
import numpy as np
import pytest

from paper_1905_08394_gb300 import binding as B
from rqc_inputs import make_circuit, uniform_bitstrings

pytestmark = pytest.mark.gpu


def fresh_bytes(circ, extra, n, kw):
    h = B.peps_create(circ.R, circ.C)
    C = circ.C
    for g in circ.gates:
        if g.kind == "1q":
            B.peps_apply_1q(h, g.qubits[0] // C, g.qubits[0] % C, g.U)
        else:
            a, b = g.qubits
            B.peps_apply_cz(h, a // C, a % C, b // C, b % C)
    for e in extra:
        B.peps_apply_cz(h, *e)
    o, keep = B.make_opts(**kw)
    need = B.peps_workspace_bytes(h, n, o)
    B.peps_destroy(h)
    return need


def test_workspace_size_of_a_planned_context(cuda_device):
    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit(4, 4, 12, 2)
    bits = uniform_bitstrings(16, 40, 2)
    sim = Simulator(4, 4, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    step = B.PEPS_FLAG_STEPWISE
    asked = [dict(), dict(precision="fp16x3", flags=step), dict(flags=step, max_lanes=7),
             dict(sliced_cz=[0, 5]), dict(sliced_cz=[0, 6]), dict(sliced_cz=[0, 6], slice_ids=[1, 2]),
             dict(sliced_cz=[0, 6], slice_ids=[1, 3]), dict(fixed_cz=[3], fixed_s=[1]),
             dict(fixed_cz=[3], fixed_s=[0]), dict(scheme="quadrants", tc_epi=4)]
    for run in asked:
        sim.amplitudes(bits, **run)
        for kw in asked:
            for n in (40, 41):
                o, keep = B.make_opts(**kw)
                assert B.peps_workspace_bytes(sim.h, n, o) == fresh_bytes(circ, [], n, kw), (run, kw)
    sim.apply_cz(1, 1, 1, 2)   # a gate more: the plan held is of another circuit
    o, keep = B.make_opts(**asked[-1])
    assert B.peps_workspace_bytes(sim.h, 40, o) == fresh_bytes(circ, [(1, 1, 1, 2)], 40, asked[-1])
    sim.close()


def test_a_failed_call_leaves_the_output(cuda_device):
    import torch

    from paper_1905_08394_gb300 import Simulator

    circ = make_circuit(4, 4, 12, 2)
    bits = uniform_bitstrings(16, 8, 3)   # no shared prefix bits
    sim = Simulator(4, 4, device=cuda_device.index or 0)
    sim.apply_circuit(circ)
    o, keep = B.make_opts(prefix_cols=2, prefix_group=4)
    need = B.peps_workspace_bytes(sim.h, 8, o)
    ws = torch.empty(need, dtype=torch.uint8, device=cuda_device)
    out = np.full(8, 3 + 4j)
    rc = B.load().peps_amplitudes(sim.h, bits.ctypes.data, 8, out.ctypes.data, o, ws.data_ptr(),
                                  need, torch.cuda.current_stream().cuda_stream)
    assert rc == B.PEPS_EINVAL and np.array_equal(out, np.full(8, 3 + 4j))
    sim.close()
