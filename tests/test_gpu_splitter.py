"""The splitter's two block sizes against the oracle. Every output is a whole
number: exact."""
import numpy as np
import pytest

import oracle
from paper_1705_02843_gb300 import bpida
from paper_1705_02843_gb300 import inputs as I
from tests.test_gpu_parity import gpu_solve

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
