"""The partial sums of a fused dot product stay inside their part of the
workspace, whatever the merge's tile width: the slots that the tiles of a launch
write (one of every epilogue warp of every tile, as the final pass reads them)
end before the next part.  Host code against a fake runtime; no device."""
import pytest

from fake_cuda import fake_lib, run  # noqa: F401  (fixture)

SCRIPT = """
h = context({circ})
kw = dict(scheme="quadrants", **{kw})
bits = uniform_bitstrings({circ}.R * {circ}.C, 20, 3)
o, keep = B.make_opts(**kw)
merge = B.peps_plan_steps(h, len(bits), o)[-1]
rc, log, ws, out = call(h, bits, **kw)
args = lambda l: [int(v) for v in l[9:]]
begin = args(next(l for l in log if l[0] == "launch" and "k_begin" in l[1]))
dots = []
for l in log:
    if l[0] == "launch" and "k_dot_final" in l[1]:
        entries, recs, partials, acc = args(l)
        n = int(l[3])
        # DotEntry: 40 bytes, the last word is the number of slots
        words = np.ctypeslib.as_array((ctypes.c_int32 * (10 * n)).from_address(entries))
        slots = int(words[9])
        assert (words[9::10] == slots).all()
        dots.append((slots, n, partials + 16 * n * slots))
print(json.dumps(dict(rc=rc, M=int(merge["M"]), N=int(merge["N"]), K=int(merge["K"]),
                      fused=int(merge["fused_dot"]), dots=dots, next=min(begin[5], begin[1]))))
"""


@pytest.mark.parametrize("circ,kw,M,N,tile,warps", [
    # N = 8: tiles of 16 columns, eight warps to each (or the four asked for)
    ("make_circuit(2, 10, 22, 1)", dict(precision="tf32"), 32768, 8, 16, 8),
    ("make_circuit(2, 10, 22, 1)", dict(precision="tf32", max_lanes=20), 32768, 8, 16, 8),
    ("make_circuit(2, 10, 22, 1)", dict(precision="tf32", tc_epi=4), 32768, 8, 16, 4),
    ("make_circuit(2, 8, 26, 1)", dict(precision="tf32"), 16384, 8, 16, 8),
    # wider merges: tiles of 256 columns, of 128 where the corrections stand apart
    ("make_circuit(4, 6, 24, 1)", dict(precision="tf32"), 512, 64, 128, 8),
    ("make_circuit(6, 6, 24, 1)", dict(precision="fp16x3"), 512, 512, 256, 8),
    ("make_circuit(6, 6, 24, 1)", dict(precision="fp16x3", tc_ksplit=-1), 512, 512, 128, 8),
])
def test_slots_end_before_the_next_part(fake_lib, circ, kw, M, N, tile, warps):
    r = run(fake_lib, SCRIPT.format(circ=circ, kw=kw))
    assert r["rc"] == 0 and r["fused"] == 1, r
    assert (r["M"], r["N"]) == (M, N), r
    assert r["dots"]
    for slots, n, end in r["dots"]:
        assert slots == M // 128 * (2 * N // tile) * warps, r
        assert end <= r["next"], r
