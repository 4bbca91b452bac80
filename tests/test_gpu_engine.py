"""GPU parity of the tile engine where its strips are densest: masks whose
strips have more extra contacts than the engine's list holds (several passes,
every site resolved), contacts of every row at once, and joins across every
strip boundary, on whole and ragged tiles of every tile width."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


def _mask(kind, H, W, seed):
    """Bond arrays: `rungs` -- every second row fully joined east, all north
    bonds open but one in eight (31 contacts in a joined row's strip word, 496
    in a strip); `dense` -- every bond open with probability 0.9; `stairs` --
    two-site runs shifted by one from row to row, so that every run touches two
    runs below."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H, 0:W]
    if kind == "rungs":
        east, north = (y % 2 == 0), rng.random((H, W)) < 0.875
    elif kind == "dense":
        east, north = rng.random((H, W)) < 0.9, rng.random((H, W)) < 0.9
    else:
        east, north = (x + y) % 2 == 0, rng.random((H, W)) < 0.95
    return oracle.pack_mask(east.astype(np.uint8).reshape(-1), north.astype(np.uint8).reshape(-1))


@pytest.mark.parametrize("tile_w", sw.TILE_WIDTHS)
@pytest.mark.parametrize("H,W", [(32, 32), (33, 64), (64, 256), (97, 290), (160, 513)])
@pytest.mark.parametrize("kind", ["rungs", "dense", "stairs"])
def test_labels_of_dense_strips(tile_w, H, W, kind):
    L = sw.lib(tile_w)
    mask = _mask(kind, H, W, H * 1000 + W)
    dev = torch.from_numpy(mask).cuda()
    for periodic in (0, 1):
        ref, _ = oracle.label(mask, H, W, bool(periodic))
        lab = torch.full((H * W,), -7, dtype=torch.int32, device="cuda")
        rc = L.ccl_label(ctypes.c_void_p(dev.data_ptr()), ctypes.c_void_p(lab.data_ptr()), H, W, periodic, None)
        assert rc == 0, L.sw_last_error()
        torch.cuda.synchronize()
        sw.ccl_status()
        assert np.array_equal(lab.cpu().numpy(), ref), periodic


@pytest.mark.parametrize("off", [1, 2, 4])
def test_labels_of_an_unaligned_mask(off):
    """A mask that starts 1, 2 or 4 bytes past an aligned address (byte loads,
    and 32-bit loads that are not 64-bit aligned), rows of odd and even width."""
    for H, W in [(40, 96), (37, 131), (5, 257)]:
        mask = oracle.perc_mask(H, W, 3)
        buf = torch.zeros(mask.size + 8, dtype=torch.uint8, device="cuda")
        buf[off:off + mask.size] = torch.from_numpy(mask).cuda()
        lab = torch.full((H * W,), -7, dtype=torch.int32, device="cuda")
        sw.ccl_label(buf[off:off + mask.size], lab, H, W, True)
        sw.ccl_status()
        ref, _ = oracle.label(mask, H, W, True)
        assert np.array_equal(lab.cpu().numpy(), ref), (H, W)


@pytest.mark.parametrize("tile_w,W", [(256, 7001), (128, 6500), (64, 6410)])
@pytest.mark.parametrize("rows", [41, 40])
def test_merge_with_several_tiles_per_block(tile_w, W, rows):
    """Grids just above the size where a merge block takes two tiles, with an
    odd and an even number of tiles, ragged in both directions."""
    H = rows * 32 - 5
    n_tiles = rows * ((W + tile_w - 1) // tile_w)
    assert n_tiles * (32 + tile_w) > 152 * 2048
    L = sw.lib(tile_w)
    mask = oracle.perc_mask(H, W, rows)
    dev = torch.from_numpy(mask).cuda()
    lab = torch.full((H * W,), -7, dtype=torch.int32, device="cuda")
    for periodic in (0, 1):
        rc = L.ccl_label(ctypes.c_void_p(dev.data_ptr()), ctypes.c_void_p(lab.data_ptr()), H, W, periodic, None)
        assert rc == 0, L.sw_last_error()
        torch.cuda.synchronize()
        sw.ccl_status()
        ref, _ = oracle.label(mask, H, W, bool(periodic))
        assert np.array_equal(lab.cpu().numpy(), ref), periodic


@pytest.mark.parametrize("H,W", [(1, 1), (1, 16), (3, 16), (16, 1), (40, 1), (2, 3), (9, 7), (5, 17), (7, 15), (40, 33),
                                 (64, 128), (33, 1000), (129, 515), (2, 300), (300, 2), (61, 36)])
@pytest.mark.parametrize("px_off,mask_off", [(0, 0), (1, 0), (16, 1), (32, 4)])
def test_pixel_bonds(H, W, px_off, mask_off):
    """Masks of images of any width (row ends anywhere in a thread's sites, the
    last row and the last sites), aligned or not, and nothing written past the
    mask's end."""
    rng = np.random.default_rng(H * 1000 + W)
    px = rng.integers(0, 2, (H, W)).astype(np.uint8)
    buf = torch.zeros(H * W + px_off, dtype=torch.uint8, device="cuda")
    buf[px_off:] = torch.from_numpy(px.reshape(-1)).cuda()
    nb = sw.mask_bytes(H * W)
    for periodic in (False, True):
        out = torch.full((nb + mask_off + 16,), 0xA5, dtype=torch.uint8, device="cuda")
        sw.ccl_bonds_from_pixels(buf[px_off:], out[mask_off:], H, W, periodic)
        got = out.cpu().numpy()
        assert np.array_equal(got[mask_off:mask_off + nb], oracle.bonds_from_pixels(px, periodic))
        assert (got[:mask_off] == 0xA5).all() and (got[mask_off + nb:] == 0xA5).all()
