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


def _phases(total):
    return {"ms_s1": 0.5, "ms_easy": 3.8, "ms_hard": 4.3, "ms_p2": 0.5, "ms_total": total, "ms_easy_kernel": 3.8,
            "ms_p2_kernel": 0.5, "easy_leaves": 10 ** 8, "easy_runs": 10 ** 8, "easy_run_leaves": 10 ** 9,
            "p2_clears": 10 ** 8}


def test_no_rate_from_overlapped_kernels():
    shared = bench.other_rooflines(_phases(4.4), 152, 2070.0)
    assert shared == {"overlapped": True, "easy_kernel_ms": 3.8, "p2_sieve_kernel_ms": 0.5}
    alone = bench.other_rooflines(_phases(9.2), 152, 2070.0)
    assert alone["easy_kernel"]["frac"] > 0 and alone["p2_sieve_kernel"]["frac"] > 0
