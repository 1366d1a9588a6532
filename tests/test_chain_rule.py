"""Which dependency levels of direct steps a plan runs as one launch (host
only): levels of a task a warp and few terms a task, where the chain saves more
than its start."""
import json

import pytest

import paper_1907_11217_gb300 as tz
from tests.gpu_util import grid_spec


def make(rows, cols, t, batch_log2, prec="c64", restarts=16):
    net = tz.tz_network_from_circuit(tz.tz_circuit_from_spec(grid_spec(rows, cols, t, 4)), batch_log2)
    tree = tz.tz_path_greedy(net, restarts=restarts, seed=7, log2_max_intermediate=26, precision=prec,
                             algorithm="elimination")
    plan = tz.tz_plan_create(net, tree, tz.tz_slice_select(net, tree, 26, 40), precision=prec,
                             max_bitstrings=1 << batch_log2)
    return plan, json.loads(plan.describe())


def level(desc, item):
    """Warp tasks of a level, and the most terms a task adds in series."""
    tasks = terms = 0
    for a, _, c in (d[:3] for d in desc["dsteps"][item[3]:item[3] + item[4]]):
        lay = {t["id"]: t["lay"] for t in desc["tensors"] if t["id"] in (a, c)}
        nc, nk = len(lay[c]), len(set(lay[a]) - set(lay[c]))
        split = min(nk, max(0, 12 - nc), 8)
        tasks += max(1, 2 ** (nc + split) // 32)
        terms = max(terms, 2 ** (nk - min(split, 5)))
    return tasks, terms


@pytest.mark.parametrize("rows,cols,t,batch_log2,prec", [
    (6, 6, 24, 2, "c64"), (6, 6, 20, 6, "c64"), (5, 6, 16, 6, "c64"), (5, 5, 24, 2, "c64"), (5, 5, 20, 3, "c64"),
    (4, 5, 16, 2, "c128"), (4, 5, 18, 4, "fp16x3"), (4, 4, 10, 2, "c64")])
def test_no_long_level_is_chained(rows, cols, t, batch_log2, prec):
    plan, desc = make(rows, cols, t, batch_log2, prec)
    for items in (desc["var_items"], desc["const_items"]):
        for i, it in enumerate(items):
            n = it[7]
            assert n == 0 or n >= 3
            for lv in items[i:i + n]:
                assert lv[0] == 1 and lv[6] == 0
                tasks, terms = level(desc, lv)
                assert tasks <= 128 and terms <= (1 if prec == "c128" else 16)
            if n and prec == "c128":
                assert n >= 4
    chained = sum(it[7] - 1 for it in desc["var_items"] if it[7])
    if prec in ("c64", "c128"):  # (no tensor-core steps: a launch an item)
        assert plan.stats()["n_launches_per_group"] == len(desc["var_items"]) - chained


def test_small_circuit_chains_its_narrow_levels():
    """4 x 4, depth 10: levels of 22, then 8 to 1 tasks; the first alone, the
    others on one CTA."""
    _, desc = make(4, 4, 10, 2)
    levels = [it for it in desc["var_items"] if it[0] == 1]
    chains = [it[7] for it in levels if it[7]]
    tasks = [level(desc, it)[0] for it in levels]
    narrow = max(len(r) for r in "".join("n" if t <= 16 else "w" for t in tasks).split("w"))
    assert narrow >= 8 and chains == [narrow]
