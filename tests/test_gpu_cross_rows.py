"""GPU parity of the binned cross power by rows: row lengths that fill a warp's lanes in part (several rows per
warp, ragged last lanes), bins that are wide, narrow, start at k = 0 or end below the Nyquist corner, and
bins too many for the private copies (the one-atomic-per-mode kernel). FP64 sums of at most N^3 exact
products in any order: 1e-12 relative to the largest bin (fields of random sign), counts exact."""

import numpy as np
import pytest
import torch

import oracle
from paper_1512_07295_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("ng,lo2,w2,nbins", [(8, 1, 2, 4), (10, 0, 1, 24), (14, 3, 5, 2), (64, 0, 2, 60), (66, 1, 2, 33),
                                             (100, 7, 3, 40), (18, 0, 1, 2048), (12, 40000, 3, 8)])
def test_cross_rows(prec, ng, lo2, w2, nbins):
    rng = np.random.default_rng(ng * 7 + nbins)
    shape = (ng, ng, ng // 2 + 1)
    dt = np.complex64 if prec == "fp32" else np.complex128
    a = (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(dt)
    b = (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(dt)
    edges2 = lo2 + w2 * np.arange(nbins + 1)
    ref, ref_k, cnt = oracle.power.cross_power_half(a.astype(np.complex128), b.astype(np.complex128), 150.0, edges2)
    cfg = api.Config(ng=ng, box=150.0, prec=prec, bin_lo2=lo2, bin_w2=w2, nbins=nbins)
    pk, km, nm = (t.cpu().numpy() for t in api.cross_power(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), cfg))
    assert np.array_equal(nm, cnt)
    full = cnt > 0
    assert np.isnan(pk[~full]).all() and np.isnan(km[~full]).all()
    if full.any():
        assert np.max(np.abs(pk - ref)[full]) <= 1e-12 * np.max(np.abs(ref[full]))
        assert np.max(np.abs(km / ref_k - 1)[full]) <= 1e-12


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("ng,lo2,w2,nbins", [(64, 40, 6, 5), (96, 0, 3, 7), (130, 100, 1, 12), (48, 83, 1, 3), (20, 1, 20000, 4),
                                             (22, 5, 10**9, 1), (66, 57, 60000, 2), (16, 1, 2, 8)])
def test_cross_rows_bins_that_hold_few_or_all_modes(prec, ng, lo2, w2, nbins):
    # only the slots within the bins are read: shells away from k = 0, a ball, the last corner, bins beyond every mode
    test_cross_rows(prec, ng, lo2, w2, nbins)


@pytest.mark.parametrize("ng", [16, 66])
def test_cross_rows_subnormal_and_nonfinite_fields(ng):
    # floats that the integer widening leaves to the conversion instructions: subnormals (beside normal values and alone),
    # zeros; an infinity and a NaN reach the bins that hold them and no other
    rng = np.random.default_rng(ng)
    shape = (ng, ng, ng // 2 + 1)
    field = lambda: (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(np.complex64)
    a, b = field(), field()
    cfg = api.Config(ng=ng, box=150.0, prec="fp32")
    run = lambda x, y: [t.cpu().numpy() for t in api.cross_power(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), cfg)]
    for scale in (np.where(rng.random(shape) < 0.3, 1e-41, 1.0), np.full(shape, 1e-42), np.where(rng.random(shape) < 0.5, 0.0, 1e-39)):
        x = (a * scale.astype(np.complex64)).astype(np.complex64)
        ref, _, _ = oracle.power.cross_power_half(x.astype(np.complex128), b.astype(np.complex128), 150.0)
        pk, _, _ = run(x, b)
        assert np.max(np.abs(pk - ref)) <= 1e-12 * np.max(np.abs(ref))
    clean, _, _ = run(a, b)
    bad = a.copy()
    bad[2, 1, 0], bad[0, 3, 4] = np.inf, np.nan  # |n|^2 = 5 and 25: bins 1 and 4
    bad[ng // 2, ng // 2, ng // 2] = np.nan      # in no bin
    pk, _, _ = run(bad, b)
    assert not np.isfinite(pk[[1, 4]]).any()
    rest = np.delete(np.arange(ng // 2), [1, 4])
    assert np.max(np.abs(pk - clean)[rest]) <= 1e-12 * np.max(np.abs(clean))
