"""Sizes of the device workspaces, by the size queries (no GPU)."""
import ctypes

import pytest
import torch


@pytest.fixture(scope="module")
def B():
    from paper_2608_09713_b200 import build
    build.build_cuda()
    from paper_2608_09713_b200 import binding
    return binding


@pytest.mark.parametrize("mode", [0, 1])
def test_plan_of_few_rows_and_many_columns(B, mode):
    """What is kept per output row goes by the rows: 1000 rows over 1e8 columns need the column pointers, counts and bit
    numbers (13 bytes a column) and little else."""
    n = 100_000_000
    assert B.spsyrk_plan_workspace_bytes(1000, n, 10_000, torch.float64, mode) < 14 * n


@pytest.mark.parametrize("mode", [0, 1])
def test_plan_of_a_small_matrix_reserves_no_row_parts(B, mode):
    """3001 rows over 2^17 columns: no row can outgrow the slots of the rank kernel."""
    nnz = 300_100
    per_nonzero = 2 * (12 + 4) + 8 * (1 + mode) + 8  # two buffer sets of the sort, descriptors, status words
    assert B.spsyrk_plan_workspace_bytes(3001, 1 << 17, nnz, torch.int32, mode) < per_nonzero * nnz + 14 * (1 << 17) + 1_500_000


def test_plan_of_the_large_random_matrix(B):
    """2^22 rows of 16 nonzeros in double precision: at most 4.55 times A."""
    m, nnz = 1 << 22, 16 << 22
    assert B.spsyrk_plan_workspace_bytes(m, m, nnz) < 4.55 * (8 * (m + 1) + 12 * nnz)
