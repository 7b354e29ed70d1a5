"""The work that a user of this framework has it do: amplitudes (or marginal
probabilities) of batches of output bitstrings of one circuit, through
`Simulator.amplitudes` (host bitstrings in, host results out) and
`Simulator.amplitudes_device` (device tensors).  The circuits, depths, batch
sizes and options are those of the repository's workloads, tests and
benchmark; `draw` takes more of the same ranges.

A case holds
  family    "cz" (random CZ circuit), "general" (random two-qubit gates with
            Schmidt ranks 2, 3 and 4)
  R, C, depth, circuit   the lattice, the depth (layers) and the circuit's seed
  n         bitstrings of the call
  api       "host" or "device"
  precision, scheme, hold   the arithmetic, the contraction order, and whether
            bond bits that the output fixes are held
  prefix    columns that the bitstrings of a group share (0: none); group = its size
  lanes     bitstrings per launch (0: the library's choice)
  graph, rebuild   replay the call as a CUDA graph; evolve the circuit anew
  measured  qubits 0 .. measured-1 are measured, the rest summed (0: amplitudes)
  cuts      the sliced CZ gates of one amplitude, "1,80,..." ("": none)
"""
import math

import numpy as np
import torch

from paper_1905_08394_gb300 import Simulator, slicing
from paper_1905_08394_gb300 import binding as B
from rqc_inputs import (make_circuit, make_circuit_general, prefix_group_bitstrings,
                        uniform_bitstrings)

_DEFAULTS = dict(family="cz", R=4, C=4, depth=8, circuit=1, n=64, api="host", precision="fp32",
                 scheme="columns", hold=False, prefix=0, group=0, lanes=0, graph=False,
                 rebuild=False, measured=0, cuts="")


def _case(name=None, **kw):
    c = dict(_DEFAULTS, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small lattice checked against a state vector: one call is a few
        # microseconds of arithmetic, so launches and the host path are the cost
        _case("4x4-d8-small-batch", R=4, C=4, depth=8, circuit=1, n=64),
        # a medium lattice, a thousand amplitudes of one circuit in FP32
        _case("5x5-d16-batch", R=5, C=5, depth=16, circuit=2, n=1024),
        # gates that are not CZ: bonds of dimension 2, 3 and 4, nothing a power of two
        _case("5x5-general-gates", family="general", R=5, C=5, depth=4, circuit=5, n=331,
              precision="fp16x3"),
        # a rectangular lattice whose bitstrings share their first columns
        _case("6x5-d16-prefix-groups", R=6, C=5, depth=16, circuit=11, n=240, precision="fp16x3",
              prefix=2, group=24),
        # the precision study's circuit by the column sweep, default lanes
        _case("6x6-d24-columns", R=6, C=6, depth=24, circuit=3, n=256, precision="fp16x3"),
        # the same in a single-pass 16-bit form, device tensors
        _case("6x6-d24-columns-bf16", R=6, C=6, depth=24, circuit=3, n=250, precision="bf16",
              api="device"),
        # one amplitude of the deepest 6x6 circuit: latency of a chain of launches
        _case("6x6-d32-one-amplitude", R=6, C=6, depth=32, circuit=4, n=1, precision="fp16x3",
              scheme="quadrants", hold=True),
        # the benchmark's batch: 8 groups of 64, evolution and contraction as one graph
        _case("6x6-d32-groups", R=6, C=6, depth=32, circuit=4, n=512, precision="fp16x3",
              scheme="quadrants", hold=True, prefix=3, group=64, lanes=512, graph=True,
              api="device"),
        # one of those groups in the plain FP32 form
        _case("6x6-d32-group-fp32", R=6, C=6, depth=32, circuit=4, n=64, precision="fp32",
              scheme="quadrants", hold=True, prefix=3, group=64, api="device"),
        # uniform bitstrings of the paper's workstation experiment (no groups)
        _case("8x8-d25-uniform", R=8, C=8, depth=25, circuit=6, n=500, precision="fp16x3",
              scheme="quadrants", hold=True, lanes=32),
        # probabilities of half of the qubits: the double-layer network
        _case("6x6-d16-marginals", R=6, C=6, depth=16, circuit=24, n=64, precision="fp16x3",
              scheme="quadrants", measured=18),
        # one amplitude of a 7x7 circuit, evolved anew and sliced so that it
        # fits a few GiB (the cuts that the slice chooser gives for 4 GiB)
        _case("7x7-d32-sliced-amplitude", R=7, C=7, depth=32, circuit=5, n=1, precision="fp16x3",
              scheme="quadrants", rebuild=True,
              cuts="1,80,85,155,164,248,253,254,257,260,265,270,271,274,288,292,300,303,311"),
    ]


def _circuit(case):
    make = make_circuit_general if case["family"] == "general" else make_circuit
    return make(case["R"], case["C"], case["depth"], case["circuit"])


def _bits(case, seed):
    if case["prefix"]:
        return prefix_group_bitstrings(case["R"], case["C"], case["prefix"],
                                       case["n"] // case["group"], case["group"], seed)
    return uniform_bitstrings(case["R"] * case["C"], case["n"], seed)


def _options(case, circ, bits):
    kw = dict(precision=case["precision"], scheme=case["scheme"], hold_ties=case["hold"],
              max_lanes=case["lanes"])
    if case["prefix"]:
        kw.update(prefix_cols=case["prefix"], prefix_group=case["group"])
    if case["measured"]:
        kw.update(measured_mask=(1 << case["measured"]) - 1)
    if case["cuts"]:
        cuts = [int(k) for k in case["cuts"].split(",")]
        kw.update(sliced_cz=cuts, slice_ids=slicing.consistent_slice_ids(circ, cuts, int(bits[0])))
    kw["flags"] = ((B.PEPS_FLAG_GRAPH if case["graph"] else 0) |
                   (B.PEPS_FLAG_REBUILD if case["rebuild"] else 0))
    return kw


def prepare(case, seed):
    """A simulator that holds the circuit, and the bitstrings wanted of it."""
    circ = _circuit(case)
    bits = _bits(case, seed)
    sim = Simulator(case["R"], case["C"])
    sim.apply_circuit(circ)
    state = {"sim": sim, "bits": bits, "kw": _options(case, circ, bits)}
    if case["api"] == "device":
        state["d_bits"] = torch.from_numpy(bits.view(np.int64)).cuda()
        state["d_out"] = torch.empty(len(bits), dtype=torch.complex128, device="cuda")
    return state


def run(state):
    if "d_bits" in state:
        return state["sim"].amplitudes_device(state["d_bits"], state["d_out"], **state["kw"])
    return state["sim"].amplitudes(state["bits"], **state["kw"])


# ---------------------------------------------------------------------------
# Work, and the draws
# ---------------------------------------------------------------------------

def _plan(case):
    """(flops, launches, workspace bytes) of the contraction the case asks for."""
    circ = _circuit(case)
    C = case["C"]
    h = B.peps_create(case["R"], C)
    try:
        for g in circ.gates:
            a, b = g.qubits[0], g.qubits[-1]
            if g.kind == "1q":
                B.peps_apply_1q(h, a // C, a % C, g.U)
            elif g.kind == "2q":
                B.peps_apply_2q(h, a // C, a % C, b // C, b % C, g.U)
            else:
                B.peps_apply_cz(h, a // C, a % C, b // C, b % C)
        opts, keep = B.make_opts(**_options(case, circ, _bits(case, 0)))
        info = B.peps_plan_info_get(h, case["n"], opts)
        space = B.peps_workspace_bytes(h, case["n"], opts)
        del keep
    finally:
        B.peps_destroy(h)
    return info["flops_call"], info["n_launches"], space


def work(case):
    """Real flops of the contraction in the order that the case asks for (8 per
    complex multiply-add); bytes: bitstrings and gates in, results out."""
    gates = len(_circuit(case).gates)
    return {"bytes": 24.0 * case["n"] + 64.0 * gates, "flops": _plan(case)[0]}


# useful flops a second of each form, for the cost of a drawn case
_RATE = {"fp32": 2e13, "tf32": 8e13, "bf16": 1e14, "fp16": 1e14, "bf16x3": 8e13, "fp16x3": 8e13}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _drawn(rng):
    kind = rng.choice(["small", "small", "general", "columns", "columns", "quadrants",
                       "quadrants", "groups", "marginals", "sliced"])
    circuit = rng.randrange(1, 10000)
    if kind == "small":
        R, C = rng.choice([(1, 7), (6, 1), (2, 7), (3, 3), (3, 5), (4, 4), (4, 5), (5, 4), (5, 5)])
        return _case(R=R, C=C, depth=rng.randint(4, 20), circuit=circuit, n=_log(rng, 1, 3000),
                     precision=rng.choice(["fp32", "fp32", "fp16x3", "bf16"]),
                     hold=rng.random() < 0.3, api=rng.choice(["host", "device"]))
    if kind == "general":
        R, C = rng.choice([(3, 4), (4, 4), (5, 4), (5, 5)])
        return _case(family="general", R=R, C=C, depth=rng.randint(1, 4), circuit=circuit,
                     n=_log(rng, 1, 600), precision=rng.choice(["fp32", "fp16x3"]))
    if kind == "columns":
        R, C = rng.choice([(5, 6), (6, 5), (6, 6), (6, 7), (7, 6)])
        case = _case(R=R, C=C, depth=rng.randint(10, 25), circuit=circuit, n=_log(rng, 1, 300),
                     precision=rng.choice(["fp16x3", "fp16x3", "fp32", "tf32", "bf16", "fp16",
                                           "bf16x3"]),
                     hold=rng.random() < 0.5, lanes=rng.choice([0, 0, 7, 16, 32, 64]),
                     rebuild=rng.random() < 0.3, api=rng.choice(["host", "device"]))
        if rng.random() < 0.3:
            group = rng.randint(2, 40)
            case.update(prefix=rng.randint(1, C - 2), group=group,
                        n=group * max(1, case["n"] // group))
        return case
    if kind == "quadrants":
        R, C = rng.choice([(4, 6), (6, 4), (6, 6), (6, 6), (5, 5), (7, 7), (6, 8), (8, 8)])
        return _case(R=R, C=C, depth=rng.randint(12, 32), circuit=circuit, n=_log(rng, 1, 400),
                     precision=rng.choice(["fp16x3", "fp16x3", "fp16x3", "fp32", "tf32"]),
                     scheme="quadrants", hold=rng.random() < 0.8,
                     lanes=rng.choice([0, 16, 32, 64]), api=rng.choice(["host", "device"]))
    if kind == "groups":
        R, C = rng.choice([(4, 6), (6, 6), (6, 6), (6, 8)])
        group = rng.randint(3, 80)
        return _case(R=R, C=C, depth=rng.randint(16, 32), circuit=circuit,
                     n=group * rng.randint(1, 8), prefix=C // 2, group=group,
                     precision=rng.choice(["fp16x3", "fp16x3", "fp32"]), scheme="quadrants",
                     hold=rng.random() < 0.9, lanes=rng.choice([0, 64, 128, 256]),
                     graph=rng.random() < 0.5, api="device")
    if kind == "marginals":
        R, C = rng.choice([(4, 4), (5, 5), (4, 6), (6, 6)])
        return _case(R=R, C=C, depth=rng.randint(4, 16), circuit=circuit, n=_log(rng, 1, 100),
                     precision=rng.choice(["fp16x3", "fp32"]),
                     scheme=rng.choice(["columns", "quadrants"]), measured=rng.randint(1, R * C - 1))
    side = rng.choice([5, 7])
    depth = rng.randint(12, 27)
    circ = make_circuit(side, side, depth, circuit)
    cuts = sorted(rng.sample(range(sum(g.kind == "cz" for g in circ.gates)), rng.randint(1, 6)))
    return _case(R=side, C=side, depth=depth, circuit=circuit, n=1,
                 precision=rng.choice(["fp16x3", "fp32"]), scheme="quadrants",
                 rebuild=rng.random() < 0.5, cuts=",".join(map(str, cuts)))


def draw(rng):
    """One more case; drawn again until it costs no more than the listed ones."""
    while True:
        case = _drawn(rng)
        try:
            flops, launches, space = _plan(case)
        except B.PepsError:   # larger than the library takes
            continue
        if flops / _RATE[case["precision"]] + launches * 8e-6 < 0.12 and space < 20 << 30:
            return case


# ---------------------------------------------------------------------------
# The same results in 64 bits, by plain torch
# ---------------------------------------------------------------------------

def _state_vector(n, gates, dev):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device=dev)
    psi[0] = 1
    for g in gates:
        if g.kind == "1q":
            q = g.qubits[0]
            U = torch.tensor(np.asarray(g.U), device=dev)
            v = psi.view(1 << (n - 1 - q), 2, 1 << q)
            a, b = v[:, 0].clone(), v[:, 1].clone()
            v[:, 0] = U[0, 0] * a + U[0, 1] * b
            v[:, 1] = U[1, 0] * a + U[1, 1] * b
            continue
        hi, lo = max(g.qubits), min(g.qubits)
        v = psi.view(1 << (n - 1 - hi), 2, 1 << (hi - lo - 1), 2, 1 << lo)
        if g.kind == "cz":
            v[:, 1, :, 1] *= -1
            continue
        U = torch.tensor(np.asarray(g.U), device=dev).reshape(2, 2, 2, 2)   # t0 t1 s0 s1
        if g.qubits[0] == lo:
            U = U.permute(1, 0, 3, 2)                                       # high qubit first
        old = {(s, t): v[:, s, :, t].clone() for s in (0, 1) for t in (0, 1)}
        for s in (0, 1):
            for t in (0, 1):
                v[:, s, :, t] = sum(U[s, t, i, j] * old[i, j] for i in (0, 1) for j in (0, 1))
    return psi


def _peps(R, C, gates, dev):
    """Site tensors [2][l][r][u][d] of a circuit of single-qubit and CZ gates."""
    A = [torch.tensor([1, 0], dtype=torch.complex128, device=dev).reshape(2, 1, 1, 1, 1)
         for _ in range(R * C)]
    keep = torch.eye(2, dtype=torch.complex128, device=dev)
    sign = torch.tensor([[1, 1], [1, -1]], dtype=torch.complex128, device=dev)
    for g in gates:
        if g.kind == "1q":
            q = g.qubits[0]
            A[q] = torch.einsum("ts,slrud->tlrud", torch.tensor(np.asarray(g.U), device=dev), A[q])
            continue
        a, b = g.qubits
        for q, leg, f in ((a, 2 if b == a + 1 else 4, keep), (b, 1 if b == a + 1 else 3, sign)):
            s = list(A[q].shape)
            one = [1] * (leg + 1) + [2] + [1] * (4 - leg)
            one[0] = 2
            t = A[q].unsqueeze(leg + 1) * f.reshape(one)
            s[leg] *= 2
            A[q] = t.reshape(s)
    return A


def _columns_flops(R, C, A):
    total = 0.0
    for c in range(C):
        for r in range(R):
            m = math.prod(A[k * C + c].shape[1] for k in range(r + 1, R)) * \
                math.prod(A[k * C + c].shape[2] for k in range(r))
            total += 8.0 * m * math.prod(A[r * C + c].shape[1:])
    return total


def _columns(R, C, A, bits):
    """Amplitudes of `bits`, one site at a time down the columns."""
    dev = A[0].device
    largest = max(math.prod(A[k * C + c].shape[2] for k in range(R)) *
                  max(A[k * C + c].shape[4] for k in range(R)) *
                  max(A[k * C + c].shape[1] for k in range(R)) for c in range(C))
    out = []
    step = max(1, int((4 << 30) / (16.0 * largest)))
    for i in range(0, len(bits), step):
        x = [[int(v) >> q & 1 for v in bits[i:i + step]] for q in range(R * C)]
        n = len(x[0])
        T = torch.ones((n, 1), dtype=torch.complex128, device=dev)
        for c in range(C):
            u = 1
            for r in range(R):
                q = r * C + c
                E = A[q][torch.tensor(x[q], device=dev)]
                _, l, rr, u, d = E.shape
                T = T.reshape(n, l, -1, u).transpose(1, 2).reshape(n, -1, l * u)
                T = torch.bmm(T, E.permute(0, 1, 3, 2, 4).reshape(n, l * u, rr * d))
                T = T.reshape(n, -1)
        out.append(T.reshape(n))
    return torch.cat(out)


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    circ, bits = _circuit(case), _bits(case, seed)
    R, C = case["R"], case["C"]
    idx = torch.from_numpy(bits.view(np.int64)).to(dev)
    # (cuts: the slices that are left out vanish, so the sum is the amplitude)
    if R * C <= 28:
        psi = _state_vector(R * C, circ.gates, dev)
        if not case["measured"]:
            out = psi[idx]
        else:
            k = case["measured"]
            p = (psi.real ** 2 + psi.imag ** 2).reshape(-1, 1 << k).sum(0)
            out = p[idx & ((1 << k) - 1)].to(torch.complex128)
    else:
        if case["measured"] or case["family"] == "general":
            return None
        A = _peps(R, C, circ.gates, dev)
        if _columns_flops(R, C, A) * case["n"] > 1.2e13:
            return None
        out = _columns(R, C, A, bits)
    return out if case["api"] == "device" else out.cpu().numpy()
