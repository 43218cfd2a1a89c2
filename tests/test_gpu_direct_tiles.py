"""GPU parity of the FP32 direct sum at the edges of its tiles: every column width of a block (N/2 + 1 values
of n_y in blocks of 8, 16, 24, 32, 40, and two blocks), pair tiles filled in part, and particle counts at
the ends of chunks (16), runs (64) and of the record ring (4 runs). Tolerance: the bound of the sums over
64 particles, (2 x 2^-21.4 + 3 x 2^-21 + 68 eps_32) sum|w| / sum w = 6.3e-6, taken as 7e-6."""

import numpy as np
import pytest
import torch

import _ref
import oracle
from paper_1512_07295_gb300 import api, catalogs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng,n", [(8, 1), (14, 63), (16, 65), (30, 16), (46, 17), (62, 321), (64, 64), (78, 255),
                                  (80, 257), (82, 1025)])
def test_direct_modes_tc_tile_edges(ng, n):
    box = 120.0
    pos = catalogs.poisson(n, box, seed=1000 + ng)
    w = catalogs.random_weights(n, seed=2000 + ng).astype(np.float32)
    ref = _ref.half_complex(oracle.direct.direct_modes(pos, box, ng, w.astype(np.float64)))
    got = api.direct_modes(torch.from_numpy(pos).cuda(), api.Config(ng=ng, box=box, prec="fp32"),
                           weights=torch.from_numpy(w).cuda()).cpu().numpy()
    assert api.device_error() == 0
    assert np.max(np.abs(got - ref)) <= 7e-6


@pytest.mark.parametrize("ng,n", [(46, 70_001), (64, 50_000)])
def test_direct_modes_tc_stages_reused_many_times(ng, n):
    # hundreds of chunks per particle slice: every operand stage and both accumulators in turn are overwritten behind
    # the MMAs that read them
    box = 120.0
    pos = catalogs.poisson(n, box, seed=3000 + ng)
    w = catalogs.random_weights(n, seed=4000 + ng).astype(np.float32)
    rng = np.random.default_rng(ng)
    idx = rng.integers(0, [ng, ng, ng // 2 + 1], (200, 3))
    nvec = np.where(idx < ng // 2, idx, idx - ng)  # slot N/2 is n = -N/2 on every axis
    ref = oracle.direct.direct_modes_at(pos, box, nvec, w.astype(np.float64))
    got = api.direct_modes(torch.from_numpy(pos).cuda(), api.Config(ng=ng, box=box, prec="fp32"),
                           weights=torch.from_numpy(w).cuda())
    assert api.device_error() == 0
    got = got.cpu().numpy()[idx[:, 0], idx[:, 1], idx[:, 2]]
    assert np.max(np.abs(got - ref)) <= 7e-6


def test_direct_modes_tc_both_operands_are_split_alike():
    # one particle with x = y = z = t: the modes (m, 0, 0), (0, 0, m) and (0, m, 0) have the same phase, which the first
    # two take through operand A and the last through operand B, times 1 or 0 exactly; with the same split the
    # results are equal bit for bit
    ng, box = 80, 1.0
    cfg = api.Config(ng=ng, box=box, prec="fp32")
    m = np.arange(1, ng // 2)
    for t in np.random.default_rng(11).uniform(0.0, 1.0, 12):
        d = api.direct_modes(torch.full((1, 3), t, dtype=torch.float64, device="cuda"), cfg).cpu().numpy()
        assert np.array_equal(d[m, 0, 0], d[0, m, 0])
        assert np.array_equal(d[0, 0, m], d[0, m, 0])


def test_direct_modes_tc_sums_keep_a_small_total_beside_large_ones():
    # particles at the origin (every factor is exactly 1 or 0): runs of 64 with weights 1, 2^30 and -2^30 in turn, 64
    # slices of three runs each. Sum w is the number of unit weights, so delta = 1 on every stored mode, and
    # every sum is exact if the totals of a slice's runs are
    run, ng = 64, 8
    w = np.tile(np.repeat(np.float32([1.0, 2.0**30, -(2.0**30)]), run), 64)
    d = api.direct_modes(torch.zeros((len(w), 3), dtype=torch.float64, device="cuda"), api.Config(ng=ng, box=1.0, prec="fp32"),
                         weights=torch.from_numpy(w).cuda()).cpu().numpy()
    assert d[0, 0, 0] == 0
    assert np.all(d.ravel()[1:] == 1.0)
