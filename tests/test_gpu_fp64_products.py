"""The FP64 assignment's integer products, node by node against exact rational arithmetic."""

import math
import random
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_1512_07295_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _spline(p, s):
    """W^(p)(s), the top hat convolved with itself p - 1 times, exactly: sum_k (-1)^k C(p, k) (s + p/2 - k)_+^(p-1) / (p-1)!."""
    x, out = s + Fraction(p, 2), Fraction(0)
    for k in range(p + 1):
        if x - k > 0:
            out += (-1) ** k * math.comb(p, k) * (x - k) ** (p - 1)
    return out / math.factorial(p - 1)


# Offsets: on a node and half way (a weight is zero: FP64 products), next to both, tiny enough that an end weight falls
# below the products' range (2^-44 with the higher orders), generic. Weights: signs, subnormal and large floats, zero.
OFFSETS = [Fraction(0), Fraction(1, 2), Fraction(1, 2**20), 1 - Fraction(1, 2**20), Fraction(1, 2**44),
           Fraction(358235907, 2**30), Fraction(914322651, 2**30)]
WEIGHTS = [1.0, -1.0, 0.3, -2.5e-40, 3e38, 1.4e-45, 0.0, 7.25]


@pytest.mark.parametrize("order", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("weighted", [False, True])
def test_every_node_product(order, weighted):
    ng, rng = 64, random.Random(order)
    cells = [(8 * a + 3, 8 * b + 3, 8 * c + 3) for a in range(8) for b in range(8) for c in range(8)]  # stencils apart
    offs = [tuple(rng.choice(OFFSETS) for _ in range(3)) for _ in cells]
    w = np.array([rng.choice(WEIGHTS) if weighted else 1.0 for _ in cells], dtype=np.float32)
    u = [[c + f for c, f in zip(cell, off)] for cell, off in zip(cells, offs)]
    pos = torch.tensor([[float(x) for x in p] for p in u], dtype=torch.float64, device=DEV)  # exact: box = N
    cfg = api.Config(ng=ng, box=float(ng), order=order, interlace=True, prec="fp64")
    grids = api.assign(pos, cfg, torch.from_numpy(w).to(DEV) if weighted else None)
    memo = {}
    for grid, shift in zip(grids, (Fraction(0), Fraction(1, 2))):
        ref = np.zeros((ng, ng, ng))
        for p, wi in zip(u, w):
            axes = []
            for x in p:
                lo = math.floor(x + shift) - 3
                for j in range(lo, lo + 8):
                    memo.setdefault((x, shift, j), _spline(order, j - x - shift))
                axes.append([(j, memo[(x, shift, j)]) for j in range(lo, lo + 8) if memo[(x, shift, j)] > 0])
            for jx, wx in axes[0]:
                for jy, wy in axes[1]:
                    for jz, wz in axes[2]:
                        ref[jx, jy, jz] = float(Fraction(float(wi)) * wx * wy * wz)
        got = grid.cpu().numpy()
        # three weights of at most ten roundings each, and their products: below 40 ulp of the node's value; what falls
        # below 2^-1022 is off by its spacing there
        assert np.all(np.abs(got - ref) <= 40 * 2.0**-52 * np.abs(ref) + 1e-320)
        assert np.array_equal(got == 0, ref == 0) or order > 4  # the higher orders' recurrence may round an end weight to 0


@pytest.mark.parametrize("order", [5, 6])
def test_no_product_outside_a_stencil(order):
    ng, rng = 64, random.Random(order)
    cells = [(8 * a + 3, 8 * b + 3, 8 * c + 3) for a in range(8) for b in range(8) for c in range(8)]  # stencils apart
    u = [[c + rng.choice(OFFSETS) for c in cell] for cell in cells]
    w = torch.tensor([rng.choice(WEIGHTS) for _ in cells], dtype=torch.float32, device=DEV)
    pos = torch.tensor([[float(x) for x in p] for p in u], dtype=torch.float64, device=DEV)  # exact: box = N
    cfg = api.Config(ng=ng, box=float(ng), order=order, interlace=True, prec="fp64")
    for grid, shift in zip(api.assign(pos, cfg, w), (Fraction(0), Fraction(1, 2))):
        inside = np.zeros((ng, ng, ng), dtype=bool)
        for p in u:
            ax = [[j for j in range(math.floor(x + shift) - 3, math.floor(x + shift) + 5) if _spline(order, j - x - shift) > 0]
                  for x in p]
            inside[np.ix_(*ax)] = True
        assert not grid.cpu().numpy()[~inside].any()
