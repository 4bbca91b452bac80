"""GPU parity of stand-alone labeling on tiles of 8 and 16 rows (grids and
groups with few tiles) against the oracle: both sides of the sizes where the
height changes, ragged last tiles, one row, wraps, every tile width, the calls
that bring their own scratch (which stay inside it), and a group whose grids
alone would take lower tiles."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu

# 128-wide tiles: 8 rows up to 608 of them, then 16 rows up to 912
SHAPES = [(1, 300), (7, 200), (8, 128), (9, 129), (15, 640), (17, 301), (4864, 128), (4865, 128), (779, 775),
          (785, 770), (14592, 128), (14593, 128), (1104, 1111)]


def _mask(H, W, seed):
    m = torch.empty(sw.mask_bytes(H * W), dtype=torch.uint8, device="cuda")
    sw.ccl_perc_mask(seed, m, H, W)
    return m, m.cpu().numpy()


@pytest.mark.parametrize("H,W", SHAPES)
@pytest.mark.parametrize("periodic", [True, False])
def test_labels(H, W, periodic):
    m, m_np = _mask(H, W, H + W)
    ref, _ = oracle.label(m_np, H, W, periodic)
    need = sw.ccl_workspace_bytes(H, W)
    ws = torch.full((need + 256,), 0x5A, dtype=torch.uint8, device="cuda")
    lab = torch.full((H * W,), -7, dtype=torch.int32, device="cuda")
    sw.ccl_label_ws(m, lab, H, W, periodic, ws[:need])
    sw.ccl_status()
    assert np.array_equal(lab.cpu().numpy(), ref)
    assert bool((ws[need:] == 0x5A).all())
    lab.fill_(-7)
    sw.ccl_label(m, lab, H, W, periodic)
    sw.ccl_status()
    assert np.array_equal(lab.cpu().numpy(), ref)


@pytest.mark.parametrize("tile_w", sw.TILE_WIDTHS)
@pytest.mark.parametrize("H,W", [(40, 70), (333, 517), (900, 1000)])
def test_tile_widths(tile_w, H, W):
    m, m_np = _mask(H, W, 3)
    lab = torch.full((H * W,), -7, dtype=torch.int32, device="cuda")
    L = sw.lib(tile_w)
    assert L.ccl_label_noalloc(ctypes.c_void_p(m.data_ptr()), ctypes.c_void_p(lab.data_ptr()), H, W, 1, None) == 0
    torch.cuda.synchronize()
    assert np.array_equal(lab.cpu().numpy(), oracle.label(m_np, H, W, True)[0])


@pytest.mark.parametrize("sides", [[(5, 9)], [(200, 300), (64, 64), (1, 700)], [(400, 500)] * 5, [(700, 800)] * 4])
def test_groups(sides):
    H, W = [x[0] for x in sides], [x[1] for x in sides]
    per = [j % 2 == 0 for j in range(len(sides))]
    masks = [_mask(h, w, 10 + j) for j, (h, w) in enumerate(sides)]
    labs = [torch.full((h * w,), -7, dtype=torch.int32, device="cuda") for h, w in sides]
    need = sw.ccl_batch_workspace_bytes(H, W)
    ws = torch.full((need + 256,), 0x5A, dtype=torch.uint8, device="cuda")
    sw.ccl_label_batch([m[0] for m in masks], labs, H, W, per, ws[:need])
    sw.ccl_status()
    for j, (h, w) in enumerate(sides):
        assert np.array_equal(labs[j].cpu().numpy(), oracle.label(masks[j][1], h, w, per[j])[0]), j
    assert bool((ws[need:] == 0x5A).all())
