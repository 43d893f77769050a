"""CPU tests of the benchmark's roofline models: work is charged to what does it."""
import bench


def _hard(table):
    st = {"clears": 10 ** 9, "steps": 10 ** 7, "hard_leaves": 2 * 10 ** 9, "table_leaves": table}
    return bench.hard_roofline(st, 45.0, 42.0, 152, 2070.0, None)["terms"]


def test_table_leaves_touch_no_shared_memory():
    none, half = _hard(0), _hard(10 ** 9)
    assert none["smem"]["work"] - half["smem"]["work"] == bench.HARD_SMEM["leaf"] * 10 ** 9
    assert none["int32"]["work"] - half["int32"]["work"] == \
        (bench.HARD_INT["leaf"] - bench.HARD_INT["table_leaf"]) * 10 ** 9
    assert half["smem"]["work"] == 10 ** 9 + 5 * 10 ** 9
