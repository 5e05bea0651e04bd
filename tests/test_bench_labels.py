"""The kernels that the bench line names for the triangular solves.  CPU only."""
import pytest

import bench

OPT = {"solve_mode": 2, "solve_mode_bwd": -1, "wide_slices": -1, "solve_blocks_per_sm": 1}


@pytest.mark.parametrize("opt,nrhs,mixed,fwd,bwd", [
    ({}, 4, False, "k_blocks/k_rows_vec", "k_blocks/k_rows_vec"),
    ({}, 16, False, "k_blocks/k_rows", "k_blocks/k_rows"),
    ({}, 8, True, "k_blocks/k_rows_vec", "k_blocks/k_rows_vec"),
    ({}, 1, False, "k_blocks/k_rows_vec/k_rows_pack", "k_blocks/k_rows_vec/k_rows_pack"),
    ({"solve_blocks_per_sm": 0}, 1, True, "k_blocks/k_rows_vec/k_rows_pack", "k_blocks/k_rows/k_rows_pack"),
    ({"wide_slices": 32}, 1, True, "k_blocks/k_rows", "k_blocks/k_rows"),
    ({"solve_mode": 1}, 1, False, "k_rows_vec", "k_rows_vec"),
    ({"solve_mode": 1, "solve_mode_bwd": 2}, 3, False, "k_rows_vec", "k_blocks/k_rows_vec"),
    ({"solve_mode": 0}, 3, False, "k_blocks/k_wide", "k_blocks/k_wide"),
])
def test_solve_kernels(opt, nrhs, mixed, fwd, bwd):
    assert bench._solve_kernels({**OPT, **opt}, nrhs, mixed) == f"{fwd} (forward) + {bwd} (backward)"
