"""Execution order of the persistent grids: every (unit, head) once, whatever the head range, longest sequences first."""
import numpy as np
import pytest

from paper_2602_21788_b200 import build, fcp


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _items(groups, heads, per):
    """(place in the unit list, head) of work items 0, 1, ... as the kernels' producer thread computes them."""
    out = []
    for first, n, gh, _ in groups.tolist():
        gh = min(gh, heads)
        block = n * gh * per
        for r in range(n * heads * per):
            hb, rest = divmod(r, block)
            inner = min(gh, heads - hb * gh) * per
            out.append((first + rest // inner, hb * gh * per + rest % inner))
    return out


CASES = [
    ([5], 1, 1, 64),
    ([300, 4000, 129, 2000, 2000, 64], 8, 2, 128),
    ([70000, 70000, 900, 1500, 300], 32, 8, 128),      # one sequence's dQ rows of a KV head exceed a group: blocks of one head
    ([9000, 20000, 9000, 128], 24, 8, 128),            # blocks of several heads, the last one smaller
]


@pytest.mark.parametrize("lens,hq,hkv,D", CASES)
@pytest.mark.parametrize("heads", [None, 1, 3])
def test_work_order_visits_every_item_once(lens, hq, hkv, D, heads):
    plan = fcp.Plan(lens, [1] * len(lens), hq, hkv, D)
    n_kv = min(heads or hkv, hkv)
    for table, n_units, per in (("fwd_groups", plan.info("n_fwd_units"), hq // hkv), ("fused_groups", plan.info("n_fused_units"), hq // hkv),
                                ("bwd_groups", plan.info("n_bwd_units"), 1), ("fwd_groups", plan.info("n_fwd_units"), 1)):
        items = _items(plan.table(table), n_kv, per)
        assert len(items) == len(set(items)) == n_units * n_kv * per
        assert {u for u, _ in items} == set(range(n_units)) and {h for _, h in items} == set(range(n_kv * per))


@pytest.mark.parametrize("lens,hq,hkv,D", CASES)
def test_groups_go_longest_sequence_first_and_by_cost_within(lens, hq, hkv, D):
    plan = fcp.Plan(lens, [1] * len(lens), hq, hkv, D)
    units = plan.table("bwd_units")[plan.table("bwd_work")]
    shortest_so_far = max(lens)
    groups = plan.table("bwd_groups").tolist()
    late = groups.pop() if len(groups) > 1 and groups[-1][2] == 1 << 16 else None   # the cheapest units of all sequences
    for first, n, _, _ in groups:
        g = units[first:first + n]
        group_lens = [lens[b] for b in g[:, 6]]
        assert max(group_lens) <= shortest_so_far
        shortest_so_far = min(group_lens)
        assert np.all(np.diff(g[:, 5]) <= 0)
    if late:
        g = units[late[0]:]
        assert np.all(np.diff(g[:, 5]) <= 0) and g[:, 5].sum() <= 0.15 * units[:, 5].sum()
        assert g[:, 5].max() <= min(units[f:f + n, 5].min() for f, n, _, _ in groups)


@pytest.mark.parametrize("lens,hq,hkv,D", [
    ([64486, 1], 1, 1, 128),              # exactly the built-in arena
    ([63487] + [1] * 12, 2, 1, 64),       # the same, thirteen sequences
    ([1500, 300, 77], 4, 2, 128),
    ([32243] + [1] * 7, 2, 1, 128),
])
def test_noalloc_arena_holds_tables_and_scratch_and_nothing_for_the_order(lens, hq, hkv, D):
    al = lambda x: (x + 255) // 256 * 256
    T, tpad = sum(lens), al(sum(lens)) + 256
    units = sum(-(-n // 128) for n in lens)
    need = 256 + al(32 * units) + al(16 * len(lens)) + al(4 * units) + al(4 * T * hq * D + 8 * tpad * hq)
    plan = fcp.Plan(lens, [1] * len(lens), hq, hkv, D)
    assert fcp.fcp_noalloc_bytes_needed(plan) == need <= fcp.FCP_NOALLOC_MAX_BYTES
    assert len(plan.table("bwd_groups")) <= 2


@pytest.mark.parametrize("lens,hq,split", [
    ([256] * 74, 1, 1), ([256] * 80, 1, 0), ([256] * 36, 4, 0),      # second items on some SMs cost more than the tiles apart save
    ([512] * 40, 1, 1), ([512] * 72, 1, 0),
    ([1024] * 28, 1, 1), ([1024] * 36, 1, 0), ([1024] * 9, 4, 0),
    ([2048] * 18, 1, 1), ([2048] * 6, 3, 1),
    ([128] * 20, 2, 0), ([100, 128, 7], 3, 0),                       # one Q tile per unit
    ([700, 520, 300, 1000, 450, 640, 130, 613], 4, 1),               # 88 items or so of a small model's batch
    ([2560] * 15, 1, 0), ([256] * 37, 4, 0),                         # as many items as SMs, or more
])
def test_q_tiles_are_items_of_their_own_where_that_is_the_shorter_launch(lens, hq, split):
    assert fcp.Plan(lens, [1] * len(lens), hq, 1, 64).info("fused_split") == split


@pytest.mark.parametrize("lens,degs,hq,hkv,D", [
    ([300, 4000, 129, 2000, 2000, 64], [1, 5, 1, 3, 3, 2], 8, 2, 128),
    ([8192, 700, 700, 1], [31, 1, 2, 1], 32, 8, 128),
    ([512] * 30, [2] * 30, 4, 4, 64),                  # equal costs throughout
])
def test_units_of_equal_cost_keep_the_order_of_the_list(lens, degs, hq, hkv, D):
    plan = fcp.Plan(lens, degs, hq, hkv, D)
    order, cost = plan.table("bwd_work"), plan.table("bwd_units")[:, 5]
    for first, n, _, _ in plan.table("bwd_groups").tolist():
        g = order[first:first + n].tolist()
        assert g == sorted(g, key=lambda u: (-cost[u], u))
    f = plan.table("fwd_units")                        # item numbers are the places in the unsorted list
    for first, n, _, _ in plan.table("fwd_groups").tolist():
        rows = f[first:first + n]
        keys = [(-(r[10] + r[11]), r[13], r[0]) for r in rows.tolist()]
        assert keys == sorted(keys)
