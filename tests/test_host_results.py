"""Where a host call's results go: a small call's come back with the status
words in one copy, a large call's straight into the caller's array (a pinned
one is then the copy's target), and either way the array is written only after
the status was seen to be good.  Host code against a fake runtime whose kernels
do nothing: a call returns the zeros of its workspace; no device."""
import pytest

from fake_cuda import fake_lib, run  # noqa: F401  (fixture)

SCRIPT = """
h = context(make_circuit(3, 3, 4, 1))
n = {n}
bits = np.arange(n, dtype=np.uint64) % np.uint64(512)
o, keep = B.make_opts()
need = B.peps_workspace_bytes(h, n, o)
ws = np.zeros(need + 1024, dtype=np.uint8)
base = (ws.ctypes.data + 511) // 512 * 512
status = np.ctypeslib.as_array((ctypes.c_int32 * 4).from_address(base))
got = []
for error in (0, 1, 0):
    status[:] = 0
    status[0] = error
    out = np.full(n, 3 + 4j)
    lib.fake_clear()
    rc = lib.peps_amplitudes(h, bits.ctypes.data, n, out.ctypes.data, o, base, need, None)
    log = [l.split() for l in lib.fake_log().decode().splitlines()]
    back = [("out" if int(l[2]) == out.ctypes.data else "other", int(l[4])) for l in log
            if l[0] == "copy" and l[1] == "2"]
    got.append([rc, back, bool((out == 3 + 4j).all()), bool((out == 0).all()),
                sum(l[0] == "sync" for l in log)])
print(json.dumps(got))
"""


@pytest.mark.parametrize("n", [1, 2, 4096, 4097, 50000])
def test_results_of_a_host_call(fake_lib, n):
    first, failed, again = run(fake_lib, SCRIPT.format(n=n))
    for rc, back, kept, written, syncs in (first, again):
        assert rc == 0 and written
        if n > 4096:
            assert back == [["other", 16], ["out", 16 * n]]
        else:
            assert back == [["other", 16 * (n + 1)]] and syncs == 1
    rc, back, kept, written, syncs = failed
    assert rc == -1 and kept and all(to == "other" for to, size in back)
