"""The bench's count of T-table lookups where each distinct tree node is visited once."""
import numpy as np

import bench
import workload as W


def test_column_nodes_counts_distinct_prefixes():
    assert bench.column_nodes(np.uint32([0, 1, 2, 3]), 2) == 2 + 4
    assert bench.column_nodes(np.uint32([5, 5, 5]), 3) == 3          # one value: a path
    assert bench.column_nodes(np.uint32([0, 7]), 3) == 2 + 2 + 2
    v = np.random.default_rng(1).integers(0, 1 << 9, 300, dtype=np.uint64).astype(np.uint32)
    assert bench.column_nodes(v, 9) == sum(len({int(x) >> (9 - lv) for x in v}) for lv in range(1, 10))


def test_node_lookups_over_tables_and_groups():
    tables = {0: np.uint32([[0, 1, 2, 3]]), 1: np.uint32([[5, 5, 5], [0, 7, 7]])}
    preds = [W.eq_pred(0, 0, 0, 1), W.range_pred(0, 0, 0, 1, 2), W.eq_pred(1, 1, 1, 7)]
    nodes = {}
    got = bench.node_lookups(preds[:2], tables, 3, nodes) + bench.node_lookups(preds[2:], tables, 3, nodes)
    col0, col1 = bench.column_nodes(tables[0][0], 3), bench.column_nodes(tables[1][1], 3)
    prf = 148 * 3 * (4 * 3 + 3 * 1)                                  # (2 P - 1) re-shares of each element
    assert got == col0 * (960 + 12 * 308) + col1 * 960 + prf
    assert bench.node_lookups(preds, tables, 3) == got and nodes == {(0, 0): col0, (1, 1): col1}
