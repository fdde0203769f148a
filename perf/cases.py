"""The calls whose time matters: what users of the library have it do, at the
sizes they do it.

Two families, as in the C ABI: midgame solves (every filling of a board's
empty cells) and retrograde steps over sections and slices.  Boards and the
choice of sections come from the seed; child values are the true values of
the slice above, computed by the library while a case is prepared.

Every output is a table of bits (int64 words of 256-bit win and not-lose
tables), so results are compared bit for bit.
"""
import functools

import numpy as np
import torch

import paper_1404_0743_gb300 as pp
from paper_1404_0743_gb300 import inputs

DEV = "cuda"
VALUE_BYTES = 64


def listed():
    return [
        # the plain midgame workload of the benchmark definition: a small
        # one-shot call on device boards, where latency and launches count
        {"name": "solve_64x6", "kind": "solve", "boards": 64, "kmin": 6, "kmax": 6},
        # one deep query as the paper's backend gets it: 16 empty cells, 10.2
        # million fills of a single board
        {"name": "solve_1x16", "kind": "solve", "boards": 1, "kmin": 16, "kmax": 16},
        # the headline workload: a plan over 1024 boards with 12 empty cells
        {"name": "plan_1024x12", "kind": "plan", "boards": 1024, "kmin": 12, "kmax": 12},
        # an odd-sized batch of unequal queries, end to end from host arrays
        {"name": "host_101_mixed", "kind": "host", "boards": 101, "kmin": 8, "kmax": 13},
        # half storage: one parity class of the rotations, one-shot
        {"name": "parity_203x12", "kind": "parity", "boards": 203, "kmin": 12, "kmax": 12, "parity": 0},
        # the request server, a burst of queries submitted at once
        {"name": "server_400", "kind": "server", "boards": 400, "kmin": 8, "kmax": 14},
        # the terminal slice: three quarters of the boards of slice 36
        {"name": "slice36", "kind": "slice", "n": 36, "d4": False, "boards": 36_000_000},
        # the step of the benchmark definition, half of slice 35 from slice 36
        {"name": "slice35", "kind": "slice", "n": 35, "d4": False, "boards": 400_000_000},
        # a batch of the D4-reduced slice-34 stream, its input made ready first
        {"name": "slice34_d4", "kind": "slice", "n": 34, "d4": True, "boards": 300_000_000},
        # part of D4 slice 33 through its dependency cone, one-shot from raw values
        {"name": "sparse33_d4", "kind": "sparse", "n": 33, "d4": True, "boards": 60_000_000},
        # one section by pointers to its children: a tiny one, latency alone
        {"name": "section35_2k", "kind": "section", "n": 35, "boards": 2_000},
        # and an ordinary one below slice 35, from raw child values
        {"name": "section34_200k", "kind": "section", "n": 34, "boards": 200_000},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["solve", "plan", "host", "parity", "server", "slice", "slice", "sparse", "section", "section"])
    if kind in ("solve", "plan", "host", "parity"):
        kmax = rng.randint(5, 13)
        kmin = max(4, kmax - rng.randint(0, 5)) if kind == "host" else kmax
        # at most the fills of the largest listed batch
        most = max(2, min(1500, 1024 * _fills(12) // _fills(kmax)))
        c = {"kind": kind, "boards": _log(rng, 1, most), "kmin": kmin, "kmax": kmax}
        if kind == "parity":
            c["parity"] = rng.randint(0, 1)
        return c
    if kind == "server":
        return {"kind": kind, "boards": _log(rng, 20, 500), "kmin": 8, "kmax": rng.randint(11, 14)}
    if kind == "slice":
        n, d4 = rng.choice([36, 35, 34]), rng.random() < 0.5
        most = {36: (45_000_000, 9_000_000), 35: (400_000_000, 110_000_000), 34: (250_000_000, 300_000_000)}[n][d4]
        return {"kind": kind, "n": n, "d4": d4, "boards": _log(rng, 200_000, most)}
    if kind == "sparse":
        return {"kind": kind, "n": rng.choice([34, 33]), "d4": rng.random() < 0.5,
                "boards": _log(rng, 500_000, 60_000_000)}
    return {"kind": "section", "n": rng.choice([35, 34, 34, 33]), "boards": _log(rng, 1_000, 2_000_000)}


# ---- sizes -------------------------------------------------------------------

def _comb(n, r):
    c = 1
    for i in range(r):
        c = c * (n - i) // (i + 1)
    return c


def _level_fills(k, m):
    return _comb(k, m) * _comb(m, (m + 1) // 2)


def _fills(k):
    return sum(_level_fills(k, m) for m in range(k + 1))


@functools.lru_cache(maxsize=None)
def _sections(n, d4):
    secs, total = pp.slice_sections(n, d4)
    return secs, np.prod(secs["dim"].astype(np.int64), axis=1), total


def work(case):
    if case["kind"] in ("solve", "plan", "host", "parity", "server"):
        ks = range(case["kmin"], case["kmax"] + 1)
        # 32-bit word operations: per fill, both tables take one OR per move
        # and word, and one rmax (eight neighbours through three-input
        # operations: four per word); a parity class is half of a table
        words = 8 if case["kind"] == "parity" else 16
        ops = sum(words * _level_fills(k, m) * (k - m + 4) for k in ks for m in range(k + 1)) / len(ks)
        return {"bytes": case["boards"] * (8 + VALUE_BYTES), "flops": case["boards"] * ops}
    n, boards = case["n"], case["boards"]
    read = 0
    if n < 36:  # this part's share of the slice above, read once
        read = boards * _sections(n + 1, case.get("d4", False))[2] / _sections(n, case.get("d4", False))[2]
    return {"bytes": VALUE_BYTES * (boards + read), "flops": 0}


# ---- preparation ---------------------------------------------------------------

def _boards(case, seed):
    """Boards with kmin..kmax empty cells, as many of each as divides evenly,
    in a drawn order."""
    rng = np.random.default_rng(seed)
    ks = rng.permutation(np.resize(np.arange(case["kmin"], case["kmax"] + 1), case["boards"]))
    out = np.zeros(case["boards"], dtype=np.uint64)
    for i, k in enumerate(ks):
        stream = inputs.SplitMix64(inputs.SEED_SERVING + seed * 1_000_003 + i)
        stones = 36 - int(k)
        out[i] = inputs.random_board(stream, (stones + 1) // 2, stones // 2)
    return out


def _pick_sections(n, d4, boards, seed):
    """A filter over the sections of slice n, drawn until about that many
    boards are kept (never more)."""
    _, sizes, _ = _sections(n, d4)
    keep = np.zeros(len(sizes), dtype=np.uint8)
    left = boards
    for i in np.random.default_rng(seed).permutation(len(sizes)):
        if sizes[i] <= left:
            keep[i] = 1
            left -= sizes[i]
    return keep


def _zeros(count):
    return torch.zeros((count, 8), dtype=torch.int64, device=DEV)


def _slice_above(n, d4, keep):
    """The sections of slice n+1 that the kept sections of slice n read:
    (values, row of each section), from slice 36 down."""
    if n == 35:
        secs, _, total = _sections(36, d4)
        values = _zeros(total)
        pp.slice_step(36, None, values, d4=d4)
        return values, secs["offset"].copy()
    need = pp.slice_children(n, keep, d4=d4)
    above, rows = _slice_above(n + 1, d4, need)
    offs, count = pp.compact_offsets(n + 1, need, d4)
    values = _zeros(count)
    if n + 1 == 35:
        pp.slice_step(35, above, values, filter=need, d4=d4)
    else:
        pp.slice_step_sparse(n + 1, above, rows, values, filter=need, d4=d4)
    return values, offs


def prepare(case, seed):
    pp.init()
    kind = case["kind"]
    if kind in ("solve", "plan", "host", "parity", "server"):
        return _prepare_midgame(case, seed)
    n, d4, boards = case["n"], case.get("d4", False), case["boards"]
    if kind == "section":
        return _prepare_section(n, boards, seed)
    keep = _pick_sections(n, d4, boards, seed)
    state = {"case": case, "out": _zeros(boards), "keep": keep}
    if n < 36:
        state["above"], state["rows"] = _slice_above(n, d4, keep)
    if kind == "slice":
        if n < 35:
            state["ready"] = torch.empty_like(state["above"])
            state["plan"] = pp.SlicePlan(n, state["ready"], state["out"], filter=keep, d4=d4, in_offsets=state["rows"])
            state["plan"].set_prepared(2)
        else:
            state["plan"] = pp.SlicePlan(n, state.get("above"), state["out"], filter=keep, d4=d4)
    return state


def _prepare_midgame(case, seed):
    boards, kind, kmax = _boards(case, seed), case["kind"], case["kmax"]
    count = len(boards)
    state = {"case": case, "boards": boards}
    if kind == "server":
        state["server"] = pp.Server(torch.empty(8 << 30, dtype=torch.uint8, device=DEV), max_slots=256,
                                    max_empty=case["kmax"])
        state["queries"] = [int(b) for b in boards]
        return state
    size = pp.midgame_parity_workspace_bytes if kind == "parity" else pp.midgame_workspace_bytes
    state["workspace"] = torch.empty(size(count, kmax), dtype=torch.uint8, device=DEV)
    if kind == "host":
        state["h_boards"] = torch.from_numpy(boards.view(np.int64)).pin_memory()
        state["h_out"] = torch.zeros((count, 8), dtype=torch.int64).pin_memory()
        return state
    state["out"] = _zeros(count)
    if kind == "plan":
        state["plan"] = pp.MidgamePlan(boards, kmax)
    else:
        state["d_boards"] = torch.from_numpy(boards.view(np.int64)).to(DEV)
    return state


def _prepare_section(n, boards, seed):
    """One section of slice n, drawn from the sixteen whose sizes are nearest
    to (and at most) the number of boards, and its child sections."""
    secs, sizes, _ = _sections(n, False)
    near = [i for i in np.argsort(-sizes, kind="stable") if sizes[i] <= boards][:16]
    i = near[int(np.random.default_rng(seed).integers(len(near)))]
    keep = np.zeros(len(secs), dtype=np.uint8)
    keep[i] = 1
    above, rows = _slice_above(n, False, keep)
    next_secs, next_sizes, _ = _sections(n + 1, False)
    index = {c["bw"].tobytes(): j for j, c in enumerate(next_secs)}
    children = []
    for q in range(4):
        bw = secs[i]["bw"].copy()
        if int(bw[q].sum()) == 9:
            children.append(None)
            continue
        bw[q][n % 2] += 1  # black moves on an even number of stones
        j = index[bw.tobytes()]
        children.append(above[int(rows[j]):int(rows[j]) + int(next_sizes[j])].clone())
    return {"case": {"kind": "section", "n": n}, "section": secs[i], "children": children, "out": _zeros(boards)}


# ---- one pass ------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        pp.midgame_solve(state["d_boards"], state["out"], case["kmax"], state["workspace"])
    elif kind == "plan":
        state["plan"].run(state["workspace"], state["out"])
    elif kind == "host":
        pp.midgame_solve_host(state["h_boards"], state["h_out"], case["kmax"], state["workspace"])
        return state["h_out"]
    elif kind == "parity":
        pp.midgame_solve_parity(state["d_boards"], state["out"], case["kmax"], case["parity"], state["workspace"])
    elif kind == "server":
        return _serve(state["server"], state["queries"])
    elif kind == "section":
        pp.section_compute(case["n"], state["section"], state["children"], state["out"])
    elif kind == "sparse":
        pp.slice_step_sparse(case["n"], state["above"], state["rows"], state["out"], filter=state["keep"],
                             d4=case["d4"])
    else:
        if case["n"] < 35:
            pp.prepare_children_ready(case["n"], state["above"], state["ready"], d4=case["d4"],
                                      in_offsets=state["rows"])
        state["plan"].run()
    return state["out"]


def _serve(server, queries):
    for i, board in enumerate(queries):
        server.submit(board, i)
    values = np.zeros((len(queries), 8), dtype=np.uint64)
    got = 0
    while got < len(queries):
        server.wait(min(64, len(queries) - got))
        for r in server.poll(1024):
            if r["status"]:
                raise RuntimeError(f"query {r['req_id']}: status {r['status']}")
            values[r["req_id"]] = r["value"]
            got += 1
    return values.view(np.int64)


def exact(case, seed):
    """Every output is a bit table, equal or not: there is no rounding."""
    return None
