"""The binning's placing pass from ranks and its 16-byte record accesses: the binned layout holds exactly the input's
records (and each one's weight), tile by tile and slab by slab, at the ends of the blocks' rounds, for
spatially ordered, random and one-cell catalogues, and from packed records at addresses that are not
multiples of 16 bytes; shifted records (multi-grid interlacing) equal the shift of the records. Offsets are
the exact fraction rounded to FP32, also next to cell faces. All exact."""

import ctypes

import numpy as np
import pytest
import torch

import _ref
from paper_1512_07295_gb300 import api, catalogs, ffi

pytestmark = pytest.mark.gpu


def _misaligned(cells):
    buf = torch.empty(cells.numel() + 1, dtype=torch.int32, device="cuda")
    out = buf[1:].view(cells.shape)
    out.copy_(cells)
    assert out.data_ptr() % 16 == 4
    return out


def _check(cells, w, cfg):
    s, ws, off = (t.cpu().numpy() for t in api.bin_particles(cells, cfg, w))
    c, wc = cells.cpu().numpy(), w.cpu().numpy()
    pairs = lambda r, v: np.sort(np.rec.fromarrays([*r.T, v.view(np.int32)]), axis=0)
    assert np.array_equal(pairs(s, ws), pairs(c, wc))
    nt = -(-cfg.ng // 8)
    k = s[:, 0].view(np.uint32).astype(np.int64)
    cx, cy, cz = k >> 20, (k >> 10) & 1023, k & 1023
    tile = ((cx // 8) * nt + cy // 8) * nt + cz // 8
    slab = 2 * (cx % 8) + (s[:, 1].view(np.float32) >= 0.5)
    assert np.all(np.diff(tile * 16 + slab) >= 0)
    assert np.array_equal(off, np.searchsorted(tile, np.arange(nt**3 + 1)))


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1025, 70_001])
@pytest.mark.parametrize("kind", ["random", "ordered", "one-cell"])
def test_binned_layout_holds_every_record(n, kind):
    ng = 36  # ragged tiles
    rng = np.random.default_rng(n)
    u = rng.uniform(0, ng, (n, 3)) if kind != "one-cell" else 17.0 + rng.uniform(0, 1, (n, 3))
    if kind == "ordered":
        u = u[np.lexsort((u[:, 2], u[:, 1], np.floor(u[:, 0])))]
    cells = torch.from_numpy(_ref.pack_cellpos(u, ng)).cuda()
    w = torch.from_numpy(rng.uniform(0.5, 1.5, n).astype(np.float32)).cuda()
    cfg = api.Config(ng=ng, box=100.0)
    _check(cells, w, cfg)
    _check(_misaligned(cells), w, cfg)
    pk, _, _ = api.power(cells, cfg, w)
    pk2, _, _ = api.power(_misaligned(cells), cfg, w)
    assert api.device_error() == 0
    assert torch.allclose(pk, pk2, rtol=1e-5, atol=0)


def test_offsets_are_the_exact_fraction_rounded():
    ng, box = 64, 64.0  # u = x exactly
    rng = np.random.default_rng(5)
    c = rng.integers(0, ng, (4000, 3)).astype(np.float64)
    d = np.concatenate([2.0 ** -rng.uniform(1, 52, 6000), np.zeros(1000), 0.5 - 2.0**-25 + 2.0 ** -rng.integers(26, 46, 1000),
                        1.0 - 2.0 ** -rng.uniform(20, 45, 4000)]).reshape(-1, 3)
    x = np.concatenate([c + d, rng.uniform(0, 2.0**-70, (50, 3)), np.nextafter(c[:500], 0.0).clip(0)])
    cells = api.prepare(torch.from_numpy(x).cuda(), api.Config(ng=ng, box=box)).cpu().numpy()
    assert np.array_equal(cells, _ref.pack_cellpos(x, ng))


@pytest.mark.parametrize("ngrids", [4, 8])
def test_shift_in_the_binning_equals_shifted_positions(ngrids):
    ng, box = 40, 200.0
    pos = catalogs.zeldovich(24, box, rms=6.0, seed=9)
    cfg = api.Config(ng=ng, box=box, prec="fp32")
    tpos = torch.from_numpy(pos).cuda()
    cells = api.prepare(tpos, cfg)
    a = api.power_multigrid(tpos, cfg, ngrids)
    b = api.power_multigrid(_misaligned(cells), cfg, ngrids)
    f = api.power_multigrid(tpos, api.Config(ng=ng, box=box, prec="fp64"), ngrids)
    for q in (a, b):
        assert torch.allclose(q[0], f[0], rtol=1e-5, atol=0) and torch.equal(q[2], f[2])


@pytest.mark.parametrize("prec", ["fp32", "fixed64"])
@pytest.mark.parametrize("ng,n", [(8, 5), (16, 2047), (64, 2049), (200, 300_001), (296, 100_000), (304, 100_000), (16, 40_000)])
def test_assignment_from_the_tile_binning_equals_that_from_the_slab_layout(prec, ng, n):
    # the internal binning by tile (one to many chunks, up to its largest grid, above its population limit and
    # above its largest grid) against pk_bin's layout: P(k) of the two agree to FP32 rounding, exactly where
    # the sums are integers (fixed64)
    rng = np.random.default_rng(ng + n)
    cells = torch.from_numpy(_ref.pack_cellpos(rng.uniform(0, ng, (n, 3)), ng)).cuda()
    w = torch.from_numpy(rng.uniform(0.5, 1.5, n).astype(np.float32)).cuda()
    cfg = api.Config(ng=ng, box=100.0, prec=prec)
    a = api.power(cells, cfg, w)
    b = api.power_binned(api.bin_particles(cells, cfg, w), cfg)
    assert api.device_error() == 0
    assert torch.equal(a[2], b[2])
    ok = a[2] > 0
    assert torch.allclose(a[0][ok], b[0][ok], rtol=1e-12 if prec == "fixed64" else 1e-5, atol=0)


@pytest.mark.parametrize("prec", ["fp32", "fixed64"])
def test_assignment_on_the_first_grid_beyond_the_tile_binning(prec):
    # 38^3 counters (N = 304, above) still fit a block's shared memory, 39^3 (N = 306) do not: the slab layout
    test_assignment_from_the_tile_binning_equals_that_from_the_slab_layout(prec, 306, 100_000)


@pytest.mark.parametrize("shift", [0, 5])
@pytest.mark.parametrize("n", [1, 33, 5000, 70_001])
def test_placing_through_cursors(n, shift):
    # the placing pass without ranks (2^32 records or more take it), called with small counts: every record and its weight,
    # tile by tile and slab by slab. launch_bin by its C++ name
    ng, nt = 36, 5
    rng = np.random.default_rng(n + shift)
    u = rng.uniform(0, ng, (n, 3))
    u[: n // 2] = 17.0 + 0.25 * u[: n // 2] / ng  # half of them in one slab
    cells = torch.from_numpy(_ref.pack_cellpos(u, ng)).cuda()
    w = torch.from_numpy(rng.uniform(0.5, 1.5, n).astype(np.float32)).cuda()
    nkeys = 16 * nt**3
    new = lambda k, t: torch.zeros(k, dtype=t, device="cuda")
    out, wout, offsets = torch.empty_like(cells), torch.empty_like(w), new(nt**3 + 1, torch.int64)
    counts, sub, scan = new(nkeys, torch.int64), new(nkeys + 1, torch.int64), new(nkeys, torch.int64)
    fn = getattr(ffi.lib(), "_ZN2pk10launch_binEPK10pk_cellposPKfliiiPS0_PfPlPyPjS7_PxP11CUstream_st")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    torch.cuda.synchronize()
    assert fn(p(cells), p(w), ctypes.c_int64(n), ng, nt, shift, p(out), p(wout), p(offsets), p(counts), ctypes.c_void_p(0),
              p(sub), p(scan), ctypes.c_void_p(0)) == 0
    torch.cuda.synchronize()
    assert api.device_error() == 0
    half = np.array([0.5 * ((shift >> a) & 1) for a in range(3)])
    x = np.mod(_ref.cellpos_to_units(cells.cpu().numpy(), ng) + half, ng)
    want = _ref.pack_cellpos(x, ng)  # the shifted offsets are those of the FP32 sum: one rounding of the exact one
    s, ws, off = out.cpu().numpy(), wout.cpu().numpy(), offsets.cpu().numpy()
    pairs = lambda r, v: np.sort(np.rec.fromarrays([*r.T, v.view(np.int32)]), axis=0)
    assert np.array_equal(pairs(s, ws), pairs(want, w.cpu().numpy()))
    k = s[:, 0].view(np.uint32).astype(np.int64)
    cx, cy, cz = k >> 20, (k >> 10) & 1023, k & 1023
    tile = ((cx // 8) * nt + cy // 8) * nt + cz // 8
    assert np.all(np.diff(tile * 16 + 2 * (cx % 8) + (s[:, 1].view(np.float32) >= 0.5)) >= 0)
    assert np.array_equal(off, np.searchsorted(tile, np.arange(nt**3 + 1)))
