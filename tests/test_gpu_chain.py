"""The 15-puzzle search of larger calls (one child per lane and round) at the
edges of its dispatch and of its stacks, against the stored oracle results.
Every output is a whole number: exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_1705_02843_gb300 import bpida
from paper_1705_02843_gb300 import inputs as I
from tests.test_gpu_parity import _golden, gpu_solve

pytestmark = pytest.mark.gpu


# 16 / 17 warps: the two register builds; 32: 13 stack entries per lane, where
# deep trees overflow into the warps' global stacks; the last two: hand-backs
# of half-taken nodes as often as possible, and single roots
@pytest.mark.parametrize("cfg", [
    dict(), dict(warps_per_block=1), dict(warps_per_block=16), dict(warps_per_block=17),
    dict(warps_per_block=32, stack_entries=256), dict(exit_fraction_pct=1, min_rounds=1, min_pass_us=-1),
    dict(warps_per_block=32, stack_entries=256, split_target=1, driver=1),
])
@pytest.mark.parametrize("n", [63, 64, 65])
def test_block_sizes_and_stacks(cfg, n):
    gold = sorted(_golden("perms15_100")["instances"], key=lambda r: sum(r["nodes"]))[:n]
    perms = I.perms15_100()
    rc, got = gpu_solve(4, [perms[r["index"]].tiles for r in gold], **cfg)
    assert rc == bpida.OK
    for r, g in zip(gold, got):
        assert (g["status"], g["length"], g["nodes"]) == (0, r["length"], r["nodes"])
        assert "".join(map(str, g["moves"])) == r["moves"] and g["solutions"] == r["solutions"]


def test_first_solution_and_budget():
    gold = sorted(_golden("perms15_100")["instances"], key=lambda r: sum(r["nodes"]))[:64]
    perms = I.perms15_100()
    tiles = [perms[r["index"]].tiles for r in gold]
    rc, got = gpu_solve(4, tiles, count_all=False)
    assert rc == bpida.OK
    for r, g in zip(gold, got):
        assert (g["status"], g["length"], g["nodes"][:-1]) == (0, r["length"], r["nodes"][:-1])
        assert 1 <= g["nodes"][-1] <= r["nodes"][-1]
    budget = sum(gold[40]["nodes"])
    rc, got = gpu_solve(4, tiles, node_budget=budget)
    assert rc == bpida.OK
    for r, g in zip(gold, got):
        if sum(r["nodes"]) <= budget:
            assert (g["status"], g["nodes"], g["solutions"]) == (0, r["nodes"], r["solutions"])
        else:
            assert g["status"] == bpida.EBUDGET and g["nodes"] == r["nodes"][:len(g["nodes"])]


def test_very_hard_batch_stays_within_the_queues():
    """A batch whose hardest board expands more than 1e11 nodes: every board
    ends with its result, the same as in calls of k_search's size."""
    rng = I.Xoshiro256ss(0x5EED0000 + 31)
    tiles = []
    for _ in range(100):
        s = rng.next_u64()
        rng.below(100)
        tiles.append(I.make_perm(4, s).tiles)
    rc, got = gpu_solve(4, tiles)
    assert rc == bpida.OK
    halves = gpu_solve(4, tiles[:50])[1] + gpu_solve(4, tiles[50:])[1]
    for g, h in zip(got, halves):
        assert g["status"] == h["status"] == bpida.OK
        assert (g["length"], g["nodes"], g["moves"], g["solutions"]) == (h["length"], h["nodes"], h["moves"], h["solutions"])


@pytest.mark.parametrize("driver", [0, 1])
@pytest.mark.parametrize("n", [64, 256, 700])
def test_easy_batches_keep_the_short_steps_kernel(n, driver):
    """Calls of many easy boards: no step is large enough for the kernel of
    large steps, which would be the slower one."""
    insts = [I.make_walk(4, 9000 + i, 40) for i in range(n)]
    tiles = [x.tiles for x in insts]
    rc, got = gpu_solve(4, tiles, driver=driver)
    assert rc == bpida.OK and bpida.chain_passes() == 0
    ref = oracle.solve_batch(4, np.array(tiles[::n // 16], dtype=np.uint8), count_all=True)
    for g, r in zip(got[::n // 16], ref):
        assert (g["status"], g["length"], g["nodes"], g["moves"]) == (0, r.length, r.nodes, r.moves)


@pytest.mark.parametrize("driver", [0, 1])
def test_hard_batches_use_both_kernels(driver):
    """Small first steps on one kernel, large ones on the other; no call of
    fewer than 64 boards uses the latter."""
    gold = sorted(_golden("perms15_100")["instances"], key=lambda r: sum(r["nodes"]))[:64]
    perms = I.perms15_100()
    for n in (63, 64):
        rc, got = gpu_solve(4, [perms[r["index"]].tiles for r in gold[:n]], driver=driver)
        assert rc == bpida.OK
        if n < 64:
            assert bpida.chain_passes() == 0
        else:
            assert 0 < bpida.chain_passes() < bpida.last_stats()["passes"]
        for r, g in zip(gold, got):
            assert (g["status"], g["length"], g["nodes"], g["solutions"]) == (0, r["length"], r["nodes"], r["solutions"])


def _used(make):
    """Device bytes that make() leaves allocated."""
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    kept = make()
    torch.cuda.synchronize()
    after = torch.cuda.mem_get_info()[0]
    return before - after, kept


QUEUES = 2 * 24 * ((1 << 24) + 1024)  # the two hand-back queues' bytes (24-byte records)


@pytest.mark.parametrize("cfg", [dict(), dict(warps_per_block=32, stack_entries=256)])
def test_workspace_is_no_larger_than_a_smaller_calls(cfg):
    """The large steps' overflow stacks take room of the hand-back queues. In
    a call's bytes: the queues, the frontiers (2 * 16388 records a board) and
    less than 16 MiB of the rest (per-board state, the graph)."""
    boards = torch.from_numpy(I.packed_array([I.make_walk(4, 100 + i, 30) for i in range(64)]).view(np.int64)).cuda()
    c = bpida.make_config(4, **cfg)
    for n in (63, 64):  # loads the kernels
        bpida.solve(boards[:n], 4, c).synchronize()
    for n in (63, 64):
        bpida.release_workspace()
        used, _ = _used(lambda: bpida.solve(boards[:n], 4, c).synchronize())
        assert used < QUEUES + n * 2 * 16388 * 24 + (16 << 20), n
    bpida.release_workspace()


def test_server_memory():
    """A server's bytes: its frontier memory, the queues, less than 16 MiB of
    the rest (16 slots)."""
    bpida.Server(frontier_bytes=64 << 20, max_slots=16).close()  # loads the kernels
    used, sv = _used(lambda: bpida.Server(frontier_bytes=64 << 20, max_slots=16))
    sv.close()
    assert used < QUEUES + (64 << 20) + (16 << 20)


@pytest.fixture
def limits():
    yield bpida.set_search_limits
    bpida.set_search_limits()


def _easiest_perms(n):
    gold = sorted(_golden("perms15_100")["instances"], key=lambda r: sum(r["nodes"]))[:n]
    perms = I.perms15_100()
    return gold, [perms[r["index"]].tiles for r in gold]


def _exact(r, g):
    assert (g["status"], g["length"], g["nodes"], g["solutions"]) == (0, r["length"], r["nodes"], r["solutions"])
    assert "".join(map(str, g["moves"])) == r["moves"]


# the edges of test_block_sizes_and_stacks, with every step after the first on
# the large steps' kernel
@pytest.mark.parametrize("cfg", [
    dict(), dict(warps_per_block=1), dict(warps_per_block=16), dict(warps_per_block=17),
    dict(warps_per_block=32, stack_entries=256), dict(exit_fraction_pct=1, min_rounds=1, min_pass_us=-1),
    dict(warps_per_block=32, stack_entries=256, split_target=1, driver=1),
])
def test_small_steps_on_the_large_steps_kernel(cfg, limits):
    gold, tiles = _easiest_perms(64)
    gpu_solve(4, tiles, **cfg)
    large = bpida.chain_passes()
    limits(large_step_nodes=1)
    rc, got = gpu_solve(4, tiles, **cfg)
    assert rc == bpida.OK and bpida.chain_passes() > large
    for r, g in zip(gold, got):
        _exact(r, g)


@pytest.mark.parametrize("driver", [0, 1])
def test_easy_boards_on_the_large_steps_kernel(driver, limits):
    """Goals at the root and above the split depth, first solutions, budgets."""
    tiles = [I.make_walk(4, 7000 + i, i % 44).tiles for i in range(200)]
    ref = oracle.solve_batch(4, np.array(tiles, dtype=np.uint8), count_all=True)
    limits(large_step_nodes=1)
    rc, got = gpu_solve(4, tiles, driver=driver)
    assert rc == bpida.OK and bpida.chain_passes() > 0
    for g, r in zip(got, ref):
        assert (g["status"], g["length"], g["nodes"], g["moves"]) == (0, r.length, r.nodes, r.moves)
    rc, got = gpu_solve(4, tiles, driver=driver, count_all=False)
    for g, r in zip(got, ref):
        assert (g["status"], g["length"], g["nodes"][:-1]) == (0, r.length, r.nodes[:-1])
        assert 1 <= g["nodes"][-1] <= r.nodes[-1]
    budget = sorted(sum(r.nodes) for r in ref)[120]
    rc, got = gpu_solve(4, tiles, driver=driver, node_budget=budget)
    for g, r in zip(got, ref):
        if sum(r.nodes) <= budget:
            assert (g["status"], g["nodes"], g["moves"]) == (0, r.nodes, r.moves)
        else:
            assert g["status"] == bpida.EBUDGET and g["nodes"] == r.nodes[:len(g["nodes"])]


@pytest.mark.parametrize("cfg", [dict(stack_entries=1024), dict(warps_per_block=32, stack_entries=384)])
def test_full_overflow_stacks_hand_entries_to_the_next_pass(cfg, limits):
    """Without room in the overflow stacks, full lanes hand entries back in
    the middle of a run, and every result is the same. (With the hand-back
    threshold at all warps, which a busy warp never sees, nothing else is
    handed back.)"""
    gold, tiles = _easiest_perms(64)
    limits(large_step_nodes=1)
    gpu_solve(4, tiles, exit_fraction_pct=100, **cfg)
    assert bpida.last_stats()["handed_back"] == 0
    limits(overflow_entries=1, large_step_nodes=1)
    rc, got = gpu_solve(4, tiles, exit_fraction_pct=100, **cfg)
    assert rc == bpida.OK and bpida.last_stats()["handed_back"] > 0
    for r, g in zip(gold, got):
        _exact(r, g)


@pytest.mark.parametrize("driver", [0, 1])
@pytest.mark.parametrize("n", [60, 64])
def test_a_full_queue_ends_the_unfinished_boards(n, driver, limits):
    """Both kernels on a queue of 20000 records: the boards that were not
    finished when it overflowed end with BPIDA_ENOMEM, the others (here
    boards of at most three moves) have their results, and the next
    call is unharmed."""
    gold, tiles = _easiest_perms(n - 4)
    easy = [I.make_walk(4, 40 + i, i).tiles for i in range(4)]
    ref = oracle.solve_batch(4, np.array(easy, dtype=np.uint8), count_all=True)
    limits(queue_records=20000, overflow_entries=1, large_step_nodes=1)
    rc, got = gpu_solve(4, easy + tiles, stack_entries=256, driver=driver)
    assert rc == (bpida.ENOMEM if driver else bpida.OK)
    assert {g["status"] for g in got} == {bpida.OK, bpida.ENOMEM}
    for g, r in zip(got[:4], ref):
        assert (g["status"], g["length"], g["nodes"], g["moves"]) == (0, r.length, r.nodes, r.moves)
    for g, r in zip(got[4:], gold):
        if g["status"] == bpida.OK:
            _exact(r, g)
        else:
            assert g["length"] == -1 and g["nodes"] == r["nodes"][:len(g["nodes"])]
    limits()
    rc, got = gpu_solve(4, easy + tiles, driver=driver)
    assert rc == bpida.OK
    for g, r in zip(got[4:], gold):
        _exact(r, g)
