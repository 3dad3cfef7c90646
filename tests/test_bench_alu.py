"""The benchmark's share of the FP64 rate: never the formulas' flops of a kernel
that does part of them off the FP64 pipe, and the two forms of the column solve
apart."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_share_of_the_fp64_rate():
    import bench
    assert bench.alu_rate("k_nh_solve", 0.52, 0.76, 1.04) == (0.52, 0.5, "algorithmic")
    for k in bench.INTEGER_FORMS:
        assert k in bench.FP64_ALG
        achieved, frac, _ = bench.alu_rate(k, 1.2, None, 1.0)
        assert achieved == 1.2 and frac is None
        assert bench.alu_rate(k, 1.2, 0.8, 1.0)[:2] == (0.8, 0.8)


def test_the_solve_forms_are_counted_apart():
    import bench
    src = open(os.path.join(ROOT, "paper_2404_08849_gb300", "csrc", "dycore.cu")).read()
    assert 'PN("k_nh_solve_block")' in src and 'PN("k_nh_solve")' in src
    args = (40962, 122880, 81920, 30, 4, "mix")
    assert bench.algorithmic_bytes("k_nh_solve/mix", *args) == bench.algorithmic_bytes("k_nh_solve_block/mix", *args)
    assert "k_nh_solve_block" not in bench.FP64_WORK_MIX      # the table's counts are the one-warp form's
