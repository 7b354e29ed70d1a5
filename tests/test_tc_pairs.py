"""The tiles of the tensor-core launches are shapes that the MMA is specified
for: one CTA takes 128 rows by a multiple of 16 columns, a pair 256 rows by a
multiple of 32, neither more than 256, and a tile's columns divide the
operand's.  Host code against a fake runtime: the boxes of the operands' tensor
maps and the kernels that are launched; no device."""
import pytest

from fake_cuda import fake_lib, run  # noqa: F401  (fixture)

SCRIPT = """
import re
circ = {circ}
h = context(circ)
bits = uniform_bitstrings(circ.R * circ.C, {n}, 3)
rc, log, ws, out = call(h, bits, **{kw})
# per launch, in the same order: map of A (rank 4 or 5), maps of the planes of B (rank 3)
maps, tiles = [], []
for l in log:
    if l[0] == "encode":
        dims = [tuple(map(int, d.split(":"))) for d in l[2:]]
        if len(dims) > 3:
            maps.append([dims])
        else:
            maps[-1].append(dims)
launches = [l for l in log if l[0] == "launch" and "k_contract_tcI" in l[1]]
for m, l in zip(maps, launches):
    pair = int(re.search(r"k_contract_tcILi[0-9]ELi[0-9]+ELi([12])E", l[1]).group(1))
    rows = int(np.prod([box for _, box in m[0][1:]]))
    tiles.append((pair, int(l[8]), rows, m[1][1][1] * pair, m[1][1][0]))
print(json.dumps(dict(rc=rc, n=[len(maps), len(launches)], tiles=sorted(set(tiles)))))
"""


@pytest.mark.parametrize("circ,n,kw,cols,paired", [
    # N = 8: 16-column tiles
    ("make_circuit(2, 10, 22, 1)", 4, dict(precision="tf32", scheme="quadrants"), 16, False),
    ("make_circuit(6, 6, 24, 3)", 20, dict(precision="bf16"), 16, False),
    # bonds of three: tiles of 96 and 192 columns, in launches of few tiles and of many
    ("make_circuit_general(5, 4, 5, 4)", 1, dict(precision="fp16x3"), 96, True),
    ("make_circuit_general(5, 4, 5, 4)", 64, dict(precision="fp16x3", max_lanes=64), 192, True),
    ("make_circuit_general(4, 6, 4, 7)", 9, dict(precision="fp16x3", scheme="quadrants"), 96, True),
    ("make_circuit_general(5, 5, 4, 5)", 2, dict(precision="fp16x3", tc_ksplit=-1), 96, False),
    # powers of two, narrowed for launches of few tiles
    ("make_circuit(6, 6, 32, 4)", 1, dict(precision="fp16x3", scheme="quadrants", hold_ties=True),
     64, True),
])
@pytest.mark.parametrize("pairs", [0, 2])
def test_tiles_are_specified_shapes(fake_lib, circ, n, kw, cols, paired, pairs):
    r = run(fake_lib, SCRIPT.format(circ=circ, n=n, kw=dict(kw, tc_cluster=pairs)))
    assert r["rc"] == 0 and r["tiles"] and r["n"][0] == r["n"][1], r
    for pair, cluster, rows, bn, nr in r["tiles"]:
        assert cluster == pair and rows == 128 and bn <= 256 and nr % bn == 0, r
        assert bn % (32 if pair == 2 else 16) == 0, r
    # the width in question is among them, in pairs where its row tiles are even
    assert any(t[3] == cols and (t[0] == 2) == paired for t in r["tiles"]), r
