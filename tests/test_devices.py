"""A kernel's shared-memory limit belongs to a device: a process that has run on
one device runs the same calls on another, and a set-up that failed once is
tried again.  Host code against a fake runtime, which refuses a launch above
the limit set on its device; no device."""
import pytest

from fake_cuda import fake_lib, run  # noqa: F401  (fixture)

SCRIPT = """
h = context(make_circuit(5, 5, {d}, 3))
bits = uniform_bitstrings(25, {n}, 3)
kw = dict({kw})
lib.fake_refuse_attributes({refuse})
rcs, smem = [], []
for device in (0, 1, 1, 3, 0):
    rc, log, ws, out = call(h, bits, device=device, **kw)
    rcs.append(rc)
    smem.append(max([int(l[7]) for l in log if l[0] == "launch" and {kernel!r} in l[1]], default=0))
print(json.dumps([rcs, smem]))
"""

CALLS = [
    # the CUDA-core step's tiles with K passes of 32
    (24, 2, dict(fuse_rows=1, flags=132), "k_contract_simt"),
    # whole sweeps of a small lattice
    (16, 64, dict(), "k_sweep_small"),
    # the tensor-core step
    (24, 20, dict(precision="fp16x3", flags=128), "k_contract_tc"),
]


@pytest.mark.parametrize("d,n,kw,kernel", CALLS)
def test_second_device(fake_lib, d, n, kw, kernel):
    rcs, smem = run(fake_lib, SCRIPT.format(d=d, n=n, kw=kw, kernel=kernel, refuse=0))
    assert rcs == [0] * 5 and len(set(smem)) == 1 and smem[0] > 48 * 1024, (rcs, smem)


@pytest.mark.parametrize("d,n,kw,kernel", CALLS)
def test_a_failed_set_up_is_tried_again(fake_lib, d, n, kw, kernel):
    rcs, smem = run(fake_lib, SCRIPT.format(d=d, n=n, kw=kw, kernel=kernel, refuse=1))
    assert rcs == [-4] + [0] * 4, rcs
