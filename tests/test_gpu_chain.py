"""The 15-puzzle search step (one child per lane and round) at the edges of
its dispatch and of its stacks, and the two splitter block sizes, against the
stored oracle results and the oracle. Every output is a whole number: exact."""
import numpy as np
import pytest

import oracle
from paper_1705_02843_gb300 import bpida
from paper_1705_02843_gb300 import inputs as I
from tests.test_gpu_parity import _golden, gpu_solve

pytestmark = pytest.mark.gpu


# 16 / 17 warps: the two register builds; 32: 13 stack entries per lane, where
# the deep trees of random permutations overflow into the warps' global stacks
@pytest.mark.parametrize("cfg", [
    dict(warps_per_block=1), dict(warps_per_block=16), dict(warps_per_block=17),
    dict(warps_per_block=32, stack_entries=256), dict(warps_per_block=32, stack_entries=256, split_target=1),
    dict(exit_fraction_pct=1, min_rounds=1, min_pass_us=-1),
])
@pytest.mark.parametrize("form", ["one", "batch"])
def test_block_sizes_and_stacks(cfg, form):
    gold = sorted(_golden("perms15_100")["instances"], key=lambda r: sum(r["nodes"]))
    picked = [gold[60]] if form == "one" else gold[40:60]
    perms = I.perms15_100()
    rc, got = gpu_solve(4, [perms[r["index"]].tiles for r in picked], **cfg)
    assert rc == bpida.OK
    for r, g in zip(picked, got):
        assert (g["status"], g["length"], g["nodes"]) == (0, r["length"], r["nodes"])
        assert "".join(map(str, g["moves"])) == r["moves"] and g["solutions"] == r["solutions"]


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049])
def test_splitter_block_sizes(n):
    """Calls on both sides of the splitter's change of block size."""
    insts = [I.make_walk(4, 7000 + i, 1 + i % 26) for i in range(n)]
    tiles = [x.tiles for x in insts]
    rc, got = gpu_solve(4, tiles)
    assert rc == bpida.OK
    step = max(1, n // 64)
    ref = oracle.solve_batch(4, np.array(tiles[::step], dtype=np.uint8), count_all=True)
    for g, r in zip(got[::step], ref):
        assert (g["status"], g["length"], g["nodes"], g["moves"]) == (0, r.length, r.nodes, r.moves)
