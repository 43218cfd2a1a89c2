"""GPU parity of the adjoint's mode kernel by rows and of its gather: grids whose rows fill a warp in part or need
several passes, every order, one and two grids, positions at the seam, in other periodic images and as
packed records, and non-finite positions (zero gradient). FP32: the forward grids, two transforms and the
gather each err by a few FP32 ulps of the largest gradient; 1e-4 of it, as in the single-size test."""

import numpy as np
import pytest
import torch

import _ref
import oracle
from paper_1512_07295_gb300 import api, catalogs, ffi

pytestmark = pytest.mark.gpu


def _grad(pos, cfg, dl, w=None):
    t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return api.power_backward(t(pos), cfg, t(dl), weights=t(w)).cpu().numpy()


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-4), ("fixed64", 1e-4), ("fp64", 1e-9)])
@pytest.mark.parametrize("ng,order,interlace", [(8, 4, True), (18, 3, True), (34, 4, False), (66, 4, True), (10, 2, True)])
def test_backward_rows_and_seam(prec, tol, ng, order, interlace):
    box = 90.0
    rng = np.random.default_rng(ng)
    pos = rng.uniform(0.0, box, (700, 3))
    pos[:40] = rng.uniform(-0.6, 0.6, (40, 3)) * box / ng  # both sides of the seam, as other periodic images too
    pos[40:60] += box * rng.integers(-3, 4, (20, 3))
    dl = rng.standard_normal(ng // 2)
    ref = oracle.adjoint.position_gradient(np.mod(pos, box), box, ng, order, dl, interlace=interlace)
    got = _grad(pos, api.Config(ng=ng, box=box, order=order, interlace=interlace, prec=prec), dl)
    assert api.device_error() == 0
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))


def test_backward_packed_records_and_nonfinite_positions():
    box, ng = 64.0, 16
    rng = np.random.default_rng(3)
    cells = _ref.pack_cellpos(rng.uniform(0.0, ng, (500, 3)), ng)
    dl = rng.standard_normal(ng // 2)
    ref = oracle.adjoint.position_gradient(_ref.cellpos_to_units(cells, ng) * (box / ng), box, ng, 4, dl)
    cfg = api.Config(ng=ng, box=box, prec="fp32")
    assert np.max(np.abs(_grad(cells, cfg, dl) - ref)) <= 1e-4 * np.max(np.abs(ref))
    pos = catalogs.poisson(300, box, seed=4)
    pos[7, 1], pos[9, 2] = np.nan, np.inf
    got = _grad(pos, cfg, dl)
    assert api.device_error() & ffi.PK_DERR_NONFINITE
    assert np.all(got[[7, 9]] == 0.0) and np.all(np.isfinite(got))
