"""Launches that overlap the one ahead of them, against plain launches.

One pair's launches and the reverse mode's form chains in which a kernel may
start while the one before it still writes.  A read ahead of the wait, or of a
stale line, shows only when the buffers hold something else than this call's
values: so the calls here follow one another on one handle without a
synchronisation, each on other frames.

Forward fields are compared bitwise with those of a handle whose kernel timing
is on, which launches everything plainly and in order.  Gradients are sums of
float atomics, whose order varies from run to run: two runs of one computation
differ by rounding alone, a few 2^-24 of a sum of at most a few dozen terms, so
1e-6 relative (measured over twelve runs of each case: 6e-8 at most).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2509_25924_gb300 as ofv  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
SHIFTS = [(1.3, -0.7), (-2.1, 0.4), (0.2, 2.6), (-0.9, -1.8)]


def _pairs(H, W, n=4):
    out = []
    for k in range(n):
        I1, I2 = synth.smooth_pair(H, W, SHIFTS[k % 4], seed=50 + k)
        out.append(tuple(torch.from_numpy(I.astype(np.float32)).to(DEV) for I in (I1, I2)))
    return out


def _plain(pairs, H, W, w25=None, **kw):
    """Each pair on its own, launched plainly."""
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(input=ofv.OFV_IN_F32, **kw))
    try:
        if w25 is not None:
            ofv.ofv_set_prefilter(h, w25)
        ofv.ofv_profile_enable(h, True)
        out = []
        for a, b in pairs:
            u, v = torch.empty((2, H, W), device=DEV)
            ofv.ofv_compute(h, a, b, u, v)
            torch.cuda.synchronize()
            out.append((u, v))
        return out
    finally:
        ofv.ofv_destroy(h)


@pytest.mark.parametrize("H,W,kw", [
    (64, 80, dict(levels_psl=2)),                                        # a few tiles
    (300, 260, dict(levels_psl=2, iterations=4)),
    (1024, 1024, dict(levels_psl=2)),                                    # 1.6 waves at level 0
    (1304, 1408, dict(levels_psl=1)),                                    # the larger tiles of KR 4
    (257, 511, dict(levels_psl=3, kernel_radius=2)),
    (719, 403, dict(levels_psl=2, kernel_radius=10, norm_radius=2)),
    (300, 260, dict(levels_psl=1, kernel_radius=5, storage=ofv.OFV_STORE_F16)),
    (300, 260, dict(levels_psl=2, storage=ofv.OFV_STORE_BF16)),
    (280, 310, dict(levels_psl=2, norm_radius=1, prefilter=1)),          # ingest, pre-filter and reductions chained
    (96, 96, dict(levels_psl=0, iterations=1)),                          # the first iteration is the last
])
def test_calls_in_a_row_give_the_fields_of_plain_launches(H, W, kw):
    pairs = _pairs(H, W)
    w25 = None
    if kw.get("prefilter"):
        w25 = torch.zeros(25, device=DEV)
        w25[12], w25[7], w25[11] = 0.7, 0.2, 0.1
    want = _plain(pairs, H, W, w25=w25, **kw)
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(input=ofv.OFV_IN_F32, **kw))
    try:
        if w25 is not None:
            ofv.ofv_set_prefilter(h, w25)
        got = torch.empty((12, 2, H, W), device=DEV)
        torch.cuda.synchronize()
        for k in range(12):
            ofv.ofv_compute(h, *pairs[k % 4], got[k, 0], got[k, 1])
        torch.cuda.synchronize()
    finally:
        ofv.ofv_destroy(h)
    for k in range(12):
        assert torch.equal(got[k, 0], want[k % 4][0]) and torch.equal(got[k, 1], want[k % 4][1]), k


@pytest.mark.parametrize("H,W,kw", [(96, 120, dict(levels_psl=2)), (256, 300, dict(levels_psl=1, kernel_radius=3)),
                                    (801, 833, dict(levels_psl=2)), (130, 150, dict(levels_psl=1, kernel_radius=10)),
                                    (140, 170, dict(levels_psl=1, norm_radius=2, prefilter=1))])
def test_gradients_after_forward_calls_are_those_of_calls_on_their_own(H, W, kw):
    pairs = _pairs(H, W)
    gu, gv = torch.randn((2, H, W), device=DEV, generator=torch.Generator(DEV).manual_seed(1))
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(input=ofv.OFV_IN_F32, **kw))
    try:
        w25 = torch.zeros(25, device=DEV)
        w25[12], w25[7], w25[11] = 0.7, 0.2, 0.1
        if kw.get("prefilter"):
            ofv.ofv_set_prefilter(h, w25)

        def grad(k, out):
            ofv.ofv_backward(h, *pairs[k], gu, gv, out[0], out[1], gw)

        gw = torch.empty(25, device=DEV)
        want = torch.empty((4, 2, H, W), device=DEV)
        for k in range(4):
            torch.cuda.synchronize()
            grad(k, want[k])
        torch.cuda.synchronize()
        got = torch.empty((8, 2, H, W), device=DEV)
        u, v = torch.empty((2, H, W), device=DEV)
        for k in range(8):
            ofv.ofv_compute(h, *pairs[(k + 1) % 4], u, v)
            grad(k % 4, got[k])
        torch.cuda.synchronize()
    finally:
        ofv.ofv_destroy(h)
    for k in range(8):
        for f in range(2):
            w = want[k % 4, f].double()
            rel = float((got[k, f].double() - w).norm() / w.norm())
            assert rel <= 1e-6, (k, f, rel)
