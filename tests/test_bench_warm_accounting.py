"""The flop counts of bench.py for warm-started cells, pinned by hand counts of the water and by their growth."""
import numpy as np
import pytest

import bench


def test_water_products_by_hand():
    # n = 6, o = 4, v = 2: S C 216, lower C^T S C 126, C E 216; an evaluation: S C_o 144, populations 24, H 36,
    # H C_o 144, A_vo 48; a rotation 96; A_oo 60, t of two rows 32, nine entries of P and of W 72
    once, evaluation, rotation, end = 558, 396, 96, 60 + 32 + 72
    for k in (1, 2, 3):
        fma = once + k * evaluation + (k - 1) * rotation + end
        assert bench._warm_flops_per_cell(k) == pytest.approx(2 * fma + 3000.0)
    np.testing.assert_allclose(bench._warm_flops_per_cell(np.array([2, 3])), [2 * 1610 + 3000, 2 * 2102 + 3000])


def test_interatomic_entries_of_two_waters():
    # (H2O)_2: 12 x 12 symmetric, less the blocks of one atom: (144 - 2 (16 + 1 + 1)) / 2 = 54
    a = bench._warm_products(2, 12, 8, 54)
    assert bench._warm_flops_per_cell(2, 12, 8, 15) == pytest.approx(2 * a + 15000.0)


def test_periodic_products_near_their_leading_term():
    # n = 198, o = 132: 2.5 n^3 + 2 (2 n^2 o + n o v) + 2 n o v + n o^2 / 2 + n o^2 + n^2 o = 7.39 n^3
    n = 198.0
    assert bench._periodic_warm_flops_per_cell(2, n, 132) == pytest.approx(2 * 7.39 * n ** 3, rel=0.01)


def test_cells_are_counted_by_their_path():
    cells = [(2, 198, 132), (12, 198, 132)]
    got = bench._flops_by_path(cells, bench._periodic_warm_flops_per_cell, bench._periodic_flops_per_cell)
    assert got == pytest.approx(bench._periodic_warm_flops_per_cell(2, 198, 132)
                                + bench._periodic_flops_per_cell(12, 198, 132))
