"""The column-walk kernels at the edges of their tiles, segments and warps:
the forward iteration (k_walk.cuh) and the samples adjoint (k_bw_walk.cuh)
against the FP64 oracle, and the claims their dispatch rests on.

Tolerances: forward 1e-3 px and gradients 1e-4 relative L2, as derived in
test_gpu_parity.py and test_gpu_backward.py for the same quantities.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2509_25924_gb300 as ofv  # noqa: E402
import synth  # noqa: E402
from test_gpu_backward import _rel, _smooth, gpu_grad, oracle_grad  # noqa: E402
from test_gpu_parity import DEV, compare, gpu_flow, mask_max, oracle_flow  # noqa: E402

pytestmark = pytest.mark.gpu


def _pair(H, W, shift=(1.3, -0.7), seed=3):
    I1, I2 = synth.smooth_pair(H, W, shift, seed=seed)
    return I1.astype(np.float32), I2.astype(np.float32)


@pytest.mark.parametrize("kr", range(1, 11))
def test_tiles_of_any_size_give_the_same_field(kr):
    # the default and the smaller tiles, bitwise: sizes one over, at and one
    # under whole tiles, and a stream (default tiles) against single pairs.  Up
    # to radius 4 these pairs run the smaller tiles for both edges (radii 1 and 2
    # have one tile), so that only the stream's tiles differ there
    edge = 48 if kr <= 5 else 64
    for H, W in ((2 * edge + 1, 113), (81, 2 * edge - 1), (120, 168)):
        I1, I2 = _pair(H, W)
        kw = dict(levels_psl=1, kernel_radius=kr, iterations=2)
        a = gpu_flow(I1, I2, tile_edge=0, **kw)
        b = gpu_flow(I1, I2, tile_edge=32, **kw)
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
        h = ofv.ofv_create(H, W, ofv.ofv_default_params(input=ofv.OFV_IN_F32, **kw))
        fr = torch.from_numpy(np.stack([I1, I2, I1])).to(DEV)
        uv = torch.empty((2, 2, H, W), device=DEV)
        ofv.ofv_compute_sequence(h, 3, fr, H * W * 4, uv[0], uv[1], H * W)
        torch.cuda.synchronize()
        ofv.ofv_destroy(h)
        assert np.array_equal(uv[0, 0].cpu().numpy(), a[0]) and np.array_equal(uv[1, 0].cpu().numpy(), a[1])


@pytest.mark.parametrize("storage", [ofv.OFV_STORE_F32, ofv.OFV_STORE_F16, ofv.OFV_STORE_BF16])
@pytest.mark.parametrize("kr,H,W", [(3, 1304, 1409), (4, 1304, 1409), (5, 145, 113), (6, 129, 201), (8, 190, 131),
                                    (10, 129, 201)])
def test_each_tile_shape_of_a_single_pair_gives_the_same_field(kr, H, W, storage):
    # pairs of radii 3 and 4 need 760 of the default tiles to take them (small
    # pairs run the smaller tiles whatever tile_edge says)
    I1, I2 = _pair(H, W)
    kw = dict(levels_psl=0 if kr <= 4 else 1, kernel_radius=kr, iterations=2, storage=storage)
    a = gpu_flow(I1, I2, tile_edge=0, **kw)
    b = gpu_flow(I1, I2, tile_edge=32, **kw)
    assert np.isfinite(a[0]).all()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("H,W,kr", [(39, 55, 4), (40, 56, 4), (41, 57, 4), (24, 224, 2), (25, 113, 1), (48, 97, 5),
                                    (64, 64, 6), (65, 129, 8), (63, 65, 10)])
def test_walk_at_tile_remainders_matches_oracle(H, W, kr):
    # seed 4: the oracle leaves no pixel of these fields out but at KR 1 (0.35 %)
    I1, I2 = _pair(H, W, seed=4)
    u, v = gpu_flow(I1, I2, levels_psl=0, kernel_radius=kr, iterations=3)
    ou, ov, nd, _ = oracle_flow(I1, I2, psl=0, kr=kr, it=3)
    compare(u, v, ou, ov, nd, max_masked=mask_max(kr), label=f"{H}x{W} KR {kr}")


def test_fields_at_unaligned_addresses():
    # outputs that start at an odd element, rows of 16-byte and of odd length
    for H, W in ((56, 64), (57, 63)):
        I1, I2 = _pair(H, W)
        a = gpu_flow(I1, I2)
        h = ofv.ofv_create(H, W, ofv.ofv_default_params(input=ofv.OFV_IN_F32))
        buf = torch.empty(2 * H * W + 3, device=DEV)
        u, v = buf[1:1 + H * W], buf[2 + H * W:2 + 2 * H * W]
        ofv.ofv_compute(h, torch.from_numpy(I1).to(DEV), torch.from_numpy(I2).to(DEV), u, v)
        torch.cuda.synchronize()
        ofv.ofv_destroy(h)
        assert np.array_equal(u.cpu().numpy().reshape(H, W), a[0])
        assert np.array_equal(v.cpu().numpy().reshape(H, W), a[1])


@pytest.mark.parametrize("H,W,kr,shift", [(31, 33, 4, (0.8, -0.5)), (32, 64, 3, (0.8, -0.5)), (65, 31, 8, (-1.2, 0.4)),
                                          (40, 56, 10, (0.3, 0.2)), (96, 80, 4, (9.3, -8.7))])
def test_samples_adjoint_at_remainders_matches_oracle(H, W, kr, shift):
    psl = 2 if abs(shift[0]) > 4 else 0
    I1, I2, gu, gv = _smooth(H, W, seed=H, shift=shift)
    g1, g2, _ = gpu_grad(I1, I2, gu, gv, levels_psl=psl, kernel_radius=kr, iterations=3)
    o1, o2, _ = oracle_grad(I1, I2, gu, gv, psl=psl, kr=kr, it=3)
    assert _rel(g1, o1) <= 1e-4, _rel(g1, o1)
    assert _rel(g2, o2) <= 1e-4, _rel(g2, o2)


@pytest.mark.parametrize("H,W,psl,kr,it,edge", [
    (801, 833, 1, 4, 2, 0),     # 8-row walks (above 152 x 16 of them), with and without a gradient of V0
    (1304, 1409, 0, 4, 1, 0),   # 40-row tiles of the recompute that keeps the window sums
    (1304, 1409, 0, 3, 2, 0),
    (1304, 1409, 0, 4, 1, 32),  # the smaller ones at the same size
    (801, 833, 0, 10, 2, 0),    # 8-row walks behind 64-px tiles
])
def test_gradients_of_large_frames_match_oracle(H, W, psl, kr, it, edge):
    I1, I2, gu, gv = _smooth(H, W, seed=H, shift=(0.8, -0.5))
    g1, g2, _ = gpu_grad(I1, I2, gu, gv, levels_psl=psl, kernel_radius=kr, iterations=it, tile_edge=edge)
    o1, o2, _ = oracle_grad(I1, I2, gu, gv, psl=psl, kr=kr, it=it)
    assert _rel(g1, o1) <= 1e-4, _rel(g1, o1)
    assert _rel(g2, o2) <= 1e-4, _rel(g2, o2)


def test_samples_adjoint_of_zero_motion_matches_oracle():
    # every sample lies on a cell corner, where each frame's slope is that of
    # its own cell: the walk leaves such pixels to the general form
    I1, _, gu, gv = _smooth(70, 66, seed=5)
    g1, g2, _ = gpu_grad(I1, I1, gu, gv, levels_psl=1, kernel_radius=4, iterations=2)
    o1, o2, _ = oracle_grad(I1, I1, gu, gv, psl=1, kr=4, it=2)
    assert _rel(g1, o1) <= 1e-4, _rel(g1, o1)
    assert _rel(g2, o2) <= 1e-4, _rel(g2, o2)
