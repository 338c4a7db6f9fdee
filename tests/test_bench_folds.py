"""bench.py's count of the float64 stages' folded columns and multiply-adds.

The columns are the classes of a row's cells under phi -> -phi, pi - phi and pi / 2 - phi
about the mirror axis, as far as the images are cells of the row: counted here
by joining cells whose distances from the axis are such images of each other."""

import math
from fractions import Fraction as F

import numpy as np
import pytest

import bench
from paper_1806_04593_gb300 import inputs

R = np.array([0.5, 1.0])


def yy(n_phi, buffer, lmax=8):
    # n cells span 3 pi / 2 and `buffer` cells on either side
    return inputs.GridSpec("fold", R, 8, n_phi, 0.0, buffer * 1.5 * math.pi / (n_phi - 2 * buffer), lmax)


def classes(n_phi, cell):
    """cell: the width of a cell in units of pi, exactly (None: pi is no whole number of cells)."""
    # distances of the cells from the axis, in cells; mirror images are one already
    x = {abs(F(2 * k + 1 - n_phi, 2)) for k in range(n_phi)}
    pi = None if cell is None else 1 / cell
    if pi is None or pi.denominator != 1:
        return len(x), False
    quarter = pi % 2 == 0
    seen, count = set(), 0
    for a in sorted(x):
        if a in seen:
            continue
        count += 1
        todo = [a]
        while todo:
            b = todo.pop()
            if b in seen:
                continue
            seen.add(b)
            images = [pi - b] + ([abs(pi / 2 - b), pi / 2 + b] if quarter else [])
            todo += [c for c in images if c in x]
    return count, quarter


@pytest.mark.parametrize("n_phi, buffer", [(270, 0), (135, 0), (48, 2), (185, 1), (34, 2), (25, 0), (3, 0), (27, 0), (30, 0), (36, 0), (120, 0), (77, 1)])
def test_yinyang_columns(n_phi, buffer):
    assert bench.fold_columns(yy(n_phi, buffer)) == classes(n_phi, F(3, 2) / (n_phi - 2 * buffer))


@pytest.mark.parametrize("n_phi", [2, 4, 16, 17, 18, 60, 360, 362])
def test_polar_columns(n_phi):
    # the axis is phi = pi (or 0: the same distances); an odd number of cells has none at pi / 2 from it
    spec = inputs.polar_grid(R, 8, n_phi, 8)
    assert bench.fold_columns(spec) == classes(n_phi, F(2, n_phi) if n_phi % 2 == 0 else None)


def test_one_degree_grid():
    spec = yy(270, 0, lmax=25)
    assert bench.fold_columns(spec) == (45, True)
    assert bench.fold_products(spec, 1) == 45 * (25 + 2 * 26)   # 25 slots of even order, 26 of odd order twice
    rows, half, n_lm = 2 * 8, 4, 26 * 26
    assert bench.kernel_work("k_sep_phi64", spec, n_lm, True, "fp64")["flop"] == 2 * rows * 3465
    assert bench.kernel_work("k_synth_f64", spec, n_lm, True, "fp64")["flop"] == 2 * (4 * rows * 3420 + 3 * 2 * half * n_lm)
