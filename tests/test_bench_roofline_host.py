"""The bench's roofline of the dense runs: bytes of the layout that the kernels
have, and the form that the timed steps ran."""
import importlib.util
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
spec = importlib.util.spec_from_file_location("bench_roofline", os.path.join(ROOT, "bench.py"))
B = importlib.util.module_from_spec(spec)
spec.loader.exec_module(B)


def test_bytes_of_the_sparse_layout():
    # one species: count 4 + four inbox words 16
    assert B.sparse_bytes_per_tet_period(1, 0, False) == 20
    # three species: counts 12 + masks 4, unit factors 8
    assert B.sparse_bytes_per_tet_period(3, 3, False) == 24
    # the bar: eight counts 32 + masks 4 + unit factors 8 + reaction mask 4
    assert B.sparse_bytes_per_tet_period(8, 14, True) == 48
    # 16-bit masks from nine species on
    assert B.sparse_bytes_per_tet_period(9, 0, False) == 36 + 8


def test_the_line_names_the_form_that_was_timed():
    args = dict(T=2_400_000, S=8, R=14, masked=True, periods=724, steps=3, ms_per_step=724 * 0.125, launch_us=124.6,
                sampled=91, kernel="k_period (block 64)")
    one = B.dense_roofline(launches=724 * 3 + 6, **args)
    assert one["kernel"] == "k_period (block 64)" and one["period_us"] == 125.0
    assert abs(one["achieved"] - 48 * 2.4e6 / 125e-6 / 1e9) < 0.1 and one["frac"] < 1.0 and "hbm" not in one["bound"]
    many = B.dense_roofline(launches=9, **args)
    assert "k_run" in many["kernel"] and many["one_period_launch"] == "k_period (block 64)"
