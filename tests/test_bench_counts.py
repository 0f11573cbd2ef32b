"""CPU: the bench counts the sweeps and words that the kernels it timed execute."""
import bench


def test_counts_follow_the_kernels_that_ran():
    four = {"rows_H": 1, "rows_pass2": 1, "rows_pass4": 1, "cols_final_pass1": 1}
    nested = {"cols_nested": 1, "rows_nested": 1, "cols_nested_rhs": 1, "rows_nested_rhs": 1}
    assert bench.path_counts(four) == (4, 7, 8, 18)
    assert bench.path_counts(nested) == (4, 6, 4, 10)      # 40 B a point and iteration in FP32
    # every nested kernel has its fields, so that a dominant one is found among them
    assert all(k in bench.KERNEL_FIELDS for k in nested)


def test_counts_of_the_side_legs_are_those_of_their_passes():
    # vector: per component s, b, t, a along y and two inverses along x; right side two copies per axis and component
    assert (bench.VCH_SWEEPS_ITER, bench.VCH_SWEEPS_RHS) == (2 * (4 + 2), 2 * 4)
    # 3D: two inverses of two fields (z), three (y) and one (x)
    assert (bench.SPLIT3D_SWEEPS_ITER, bench.SPLIT3D_SWEEPS_RHS) == (2 * (2 + 3 + 1), 6)
    # sixth order: three inverses on lines; y pass 3 x 2, x pass 2, H_y W and two for v and X W on grids
    assert (bench.FCH1D_SWEEPS_ITER, bench.FCH2D_SWEEPS_ITER) == (3, 6 + 2 + 1 + 2)
