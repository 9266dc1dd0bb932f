"""The splitter's two block sizes against the oracle. Every output is a whole
number: exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_1705_02843_gb300 import bpida
from paper_1705_02843_gb300 import inputs as I
from tests.test_gpu_parity import gpu_solve
from tests.test_gpu_parity import _golden

pytestmark = pytest.mark.gpu


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


@pytest.fixture(scope="module")
def hard24():
    """24-puzzle walks whose frontiers are longer than a block has threads."""
    tiles = [I.make_walk(5, 8000 + i, 46 + i % 9).tiles for i in range(24)]
    return tiles, oracle.solve_batch(5, np.array(tiles, dtype=np.uint8), count_all=True)


@pytest.mark.parametrize("n", [2047, 2048, 2049])
def test_splitter_block_sizes_24puzzle(n, hard24):
    """128-bit boards, most of them short walks."""
    tiles = hard24[0] + [I.make_walk(5, 9000 + i, i % 22).tiles for i in range(n - 24)]
    rc, got = gpu_solve(5, tiles)
    assert rc == bpida.OK
    ref = hard24[1] + oracle.solve_batch(5, np.array(tiles[24::32], dtype=np.uint8), count_all=True)
    for g, r in zip(got[:24] + got[24::32], ref):
        assert (g["status"], g["length"], g["nodes"], g["moves"], g["solutions"]) == \
            (0, r.length, r.nodes, r.moves, r.solutions)


@pytest.mark.parametrize("n", [2047, 2048, 2049])
def test_splitter_block_sizes_pattern_databases(n):
    """Pattern databases (5-5-5): 20 permutations with stored results of that
    heuristic, the rest short walks, whose solutions are the Manhattan
    distance's."""
    gold = sorted(_golden("perms15_100_pdb555")["instances"], key=lambda r: sum(r["nodes"]))[60:80]
    perms = I.perms15_100()
    tiles = [perms[r["index"]].tiles for r in gold] + [I.make_walk(4, 9000 + i, i % 30).tiles for i in range(n - 20)]
    t = torch.from_numpy(np.array([I.pack(4, x) for x in tiles], dtype=np.uint64).reshape(-1).view(np.int64)).cuda()
    with bpida.PatternDb(4, I.PDB_PARTITIONS["555"]) as pdb:
        sol = bpida.solve(t, 4, bpida.make_config(4), pdb=pdb)
        got = sol.to_host()
    assert sol.status == bpida.OK
    for r, g in zip(gold, got):
        assert (g["status"], g["length"], g["nodes"], g["solutions"]) == (0, r["length"], r["nodes"], r["solutions"])
        assert "".join(map(str, g["moves"])) == r["moves"]
    ref = oracle.solve_batch(4, np.array(tiles[20::32], dtype=np.uint8), count_all=True)
    for g, r in zip(got[20::32], ref):
        assert (g["status"], g["length"], g["moves"], g["solutions"]) == (0, r.length, r.moves, r.solutions)
