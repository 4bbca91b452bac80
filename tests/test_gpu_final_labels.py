"""GPU parity of the final labels where rows start at every offset from a
16-byte word: widths around the tile widths and the words, label arrays that
start off a word, ragged last tiles, every tile width and height."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_w", sw.TILE_WIDTHS)
@pytest.mark.parametrize("W", [1, 2, 3, 4, 5, 61, 62, 63, 64, 65, 66, 67, 125, 127, 128, 129, 131, 254, 255, 256, 257, 258, 259, 515])
@pytest.mark.parametrize("H", [1, 33])
@pytest.mark.parametrize("off", [0, 1, 2, 3])
def test_offsets(tile_w, W, H, off):
    m = torch.empty(sw.mask_bytes(H * W), dtype=torch.uint8, device="cuda")
    sw.ccl_perc_mask(W + off, m, H, W)
    lab = torch.full((H * W + 8,), -7, dtype=torch.int32, device="cuda")
    L = sw.lib(tile_w)
    rc = L.ccl_label(ctypes.c_void_p(m.data_ptr()), ctypes.c_void_p(lab.data_ptr() + 4 * off), H, W, 1, None)
    assert rc == 0, L.sw_last_error()
    torch.cuda.synchronize()
    out = lab.cpu().numpy()
    assert np.array_equal(out[off:off + H * W], oracle.label(m.cpu().numpy(), H, W, True)[0])
    assert (out[:off] == -7).all() and (out[off + H * W:] == -7).all()


@pytest.mark.parametrize("H,W", [(1200, 1203), (1501, 1502), (2000, 1537), (15000, 131)])
def test_tall_tiles(H, W):
    m = torch.empty(sw.mask_bytes(H * W), dtype=torch.uint8, device="cuda")
    sw.ccl_perc_mask(5, m, H, W)
    lab = torch.full((H * W,), -7, dtype=torch.int32, device="cuda")
    sw.ccl_label(m, lab, H, W, False)
    sw.ccl_status()
    assert np.array_equal(lab.cpu().numpy(), oracle.label(m.cpu().numpy(), H, W, False)[0])
