"""The solver's performance cases: what a program that uses it has it do.

Every case goes through a public entry point (`bpida.solve`, with the
Manhattan distance or with pattern databases, or `bpida.Server`) and returns
everything that the call computes. Boards are seeded random walks from the
goal (easy to ordinary) and uniformly random solvable permutations (ordinary
to very hard: the node counts of single boards spread over seven orders of
magnitude), as in `paper_1705_02843_gb300/inputs.py` and the benchmark.

A case is a dict of
  entry    "solve", "pdb" or "serve"
  width    board width (3, 4, 5)
  boards   boards of one pass
  per_call boards of one solve call (the pass makes boards / per_call calls)
  lo, hi   walk lengths drawn from [lo, hi]
  perm_pct percentage of the boards that are random permutations
  budget   node budget per board (0: none)
  count_all  True: all optimal solutions; False: stop at the first one
  groups   tile groups of the pattern databases ("555", "663", "" for none)
"""
import time

import numpy as np
import torch

from paper_1705_02843_gb300 import bpida
from paper_1705_02843_gb300 import inputs as I


def _case(entry="solve", width=4, boards=1, per_call=0, lo=40, hi=40, perm_pct=0, budget=0, count_all=True, groups=""):
    return {"entry": entry, "width": width, "boards": boards, "per_call": per_call or boards, "lo": lo, "hi": hi,
            "perm_pct": perm_pct, "budget": budget, "count_all": count_all, "groups": groups}


def listed():
    return [
        # one easy 15-puzzle per call: an interactive user's request, all latency
        dict(_case(boards=1), name="walk40_one"),
        # a small batch of easy boards (walks15_16x40)
        dict(_case(boards=16), name="walks40_16"),
        # hard boards as they come, one per call: the paper's own form of use
        dict(_case(boards=8, per_call=1, perm_pct=100), name="perms_plain_8"),
        # the same in first-solution mode, the paper's main timing experiment
        dict(_case(boards=5, per_call=1, perm_pct=100, count_all=False), name="perms_first_5"),
        # the paper's benchmark size in one call: 100 random permutations
        dict(_case(boards=100, perm_pct=100), name="perms_batch_100"),
        # a production batch: mostly easy boards, 5 % hard ones (mixed15_4096's mix)
        dict(_case(boards=1024, lo=20, hi=90, perm_pct=5), name="mix_1024"),
        # the smallest board size in bulk: random 8-puzzles
        dict(_case(width=3, boards=5000, perm_pct=100), name="eight_5000"),
        # one 24-puzzle per call
        dict(_case(width=5, boards=1, lo=46, hi=46), name="walk24_one"),
        # 24-puzzles under a node budget (walks24_1024's mix)
        dict(_case(width=5, boards=256, lo=40, hi=100, budget=50_000_000), name="walks24_256"),
        # pattern databases in L2 (5-5-5), the benchmark's 100 boards in one call
        dict(_case("pdb", boards=100, perm_pct=100, groups="555"), name="pdb555_batch_100"),
        # pattern databases in HBM (6-6-3), one board per call
        dict(_case("pdb", boards=4, per_call=1, perm_pct=100, groups="663"), name="pdb663_plain_4"),
        # a burst of requests to the solve service (serving_stream's mix)
        dict(_case("serve", boards=300, lo=30, hi=90, perm_pct=2), name="serve_burst_300"),
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["walks", "plain", "first", "perms", "mix", "eight", "walk24", "walks24", "pdb", "pdb_plain", "serve"])
    if kind == "walks":
        a, b = rng.randint(20, 60), rng.randint(20, 60)
        return _case(boards=_log(rng, 1, 700), lo=min(a, b), hi=max(a, b))
    if kind in ("plain", "first"):
        n = rng.randint(1, 6)
        return _case(boards=n, per_call=1, lo=40, hi=rng.randint(60, 90), perm_pct=rng.choice([50, 100]), count_all=kind == "plain")
    if kind == "perms":
        return _case(boards=_log(rng, 2, 80), perm_pct=100)
    if kind == "mix":
        return _case(boards=_log(rng, 9, 900), lo=20, hi=90, perm_pct=rng.randint(1, 5))
    if kind == "eight":
        return _case(width=3, boards=_log(rng, 1, 5000), perm_pct=100)
    if kind == "walk24":
        n = rng.randint(1, 3)
        return _case(width=5, boards=n, per_call=1, lo=30, hi=rng.randint(38, 46))
    if kind == "walks24":
        return _case(width=5, boards=_log(rng, 9, 250), lo=40, hi=rng.randint(50, 100), budget=rng.choice([3_000_000, 50_000_000]))
    if kind == "pdb":
        return _case("pdb", boards=_log(rng, 2, 100), perm_pct=100, groups=rng.choice(["555", "663"]))
    if kind == "pdb_plain":
        n = rng.randint(1, 6)
        return _case("pdb", boards=n, per_call=1, lo=40, hi=90, perm_pct=rng.choice([50, 100]), groups=rng.choice(["555", "663"]))
    return _case("serve", boards=_log(rng, 8, 300), lo=30, hi=90, perm_pct=rng.randint(0, 2))


def _boards(case, seed):
    """The pass's packed boards on the host."""
    rng = I.Xoshiro256ss(0x5EED0000 + int(seed))
    out = []
    for _ in range(case["boards"]):
        s = rng.next_u64()
        if rng.below(100) < case["perm_pct"]:
            out.append(I.make_perm(case["width"], s))
        else:
            out.append(I.make_walk(case["width"], s, rng.uniform_int(case["lo"], case["hi"])))
    return I.packed_array(out)


class _State:
    """What the program keeps: its boards and, where it uses them, the pattern
    databases or the running service."""

    def __init__(self, case, seed):
        self.case, self.pdb, self.server = case, None, None
        packed = _boards(case, seed)
        if case["entry"] == "serve":
            self.packed = [int(w) for w in packed]
            self.server = bpida.Server(frontier_bytes=256 << 20, max_slots=4096)
            return
        dev = torch.from_numpy(packed.view(np.int64)).cuda()
        self.calls = list(torch.split(dev, case["per_call"]))
        self.config = bpida.make_config(case["width"], node_budget=case["budget"], count_all=case["count_all"])
        if case["groups"]:
            self.pdb = bpida.PatternDb(case["width"], I.PDB_PARTITIONS[case["groups"]])

    def __del__(self):
        for held in (self.pdb, self.server):
            if held is not None:
                held.close()


def prepare(case, seed):
    return _State(case, seed)


def _serve(server, packed):
    for i, w in enumerate(packed):
        server.submit(w, i)
    got = {}
    while len(got) < len(packed):
        results = server.poll()
        for r in results:
            got[r["req_id"]] = r
        if not results:
            time.sleep(0.0001)
    n = len(packed)
    moves = np.zeros((n, bpida.max_len(4)), np.uint8)
    nodes = np.zeros((n, bpida.max_iters(4)), np.int64)
    for i in range(n):
        moves[i, :len(got[i]["moves"])] = got[i]["moves"]
        nodes[i, :len(got[i]["nodes"])] = got[i]["nodes"]
    out = {k: np.array([got[i][k] for i in range(n)], np.int64) for k in ("length", "iters", "status", "solutions")}
    return dict(out, moves=moves, nodes=nodes)


def run(state):
    case = state.case
    if case["entry"] == "serve":
        return _serve(state.server, state.packed)
    out = []
    for boards in state.calls:
        sol = bpida.solve(boards, case["width"], state.config, pdb=state.pdb)
        if sol.status != bpida.OK:
            raise RuntimeError(bpida.status_str(sol.status))
        got = {"length": sol.length, "iters": sol.iters, "status": sol.inst_status}
        if case["count_all"]:
            got.update(moves=sol.moves, nodes=sol.nodes, solutions=sol.solutions)
        # first-solution mode: which optimal solution is found first, and how
        # much of the last iteration was searched by then, depend on timing
        out.append(got)
    return out


# Mean nodes per board that IDA* expands (stored oracle results of the
# benchmark's workloads): walks by length, random permutations by heuristic.
_WALK15 = {20: 2.6e3, 30: 4.4e4, 40: 5.3e5, 50: 2.8e6, 60: 7.5e6, 70: 2.8e7, 80: 3.3e7, 90: 4.5e7}
_WALK24 = {30: 1e5, 40: 8.3e5, 50: 8.9e6, 60: 1.7e7, 70: 3.1e7, 80: 3.9e7, 90: 4.3e7, 100: 4.6e7}
_PERM = {"": 4.2e8, "555": 5.3e6, "663": 2.5e6}


def _nodes(case):
    perm = case["perm_pct"] / 100.0
    if case["width"] == 3:
        mean = 2e3
    else:
        table = _WALK15 if case["width"] == 4 else _WALK24
        lengths = range(case["lo"], case["hi"] + 1)
        mean = sum(table[max(min(table), min(max(table), n // 10 * 10))] for n in lengths) / len(lengths)
        if case["groups"]:
            mean /= 80
        if perm:
            mean = (1 - perm) * mean + perm * _PERM[case["groups"]]
    return mean * case["boards"]


def work(case):
    """Bytes: the boards read, the result rows written. Operations: about 20
    integer operations per expanded node (the pop, the goal test, the moves'
    heuristic changes, the child boards) for the mean node count of such
    boards; with pattern databases one table byte per node comes on top."""
    w = case["width"]
    row = 4 + 4 + 4 + 8 + bpida.max_len(w) + 8 * bpida.max_iters(w)
    nodes = _nodes(case)
    return {"bytes": case["boards"] * (8 * I.words_per_board(w) + row) + (nodes if case["groups"] else 0),
            "flops": 20 * nodes}


def exact(case, seed):
    """Every output is a whole number: there is none to compute in 64 bits."""
    return None
