"""GPU parity of the estimator variants against the FP64 oracle, through the
C ABI: the Gaussian-weighted window, the increment form of the Gauss-Newton
step, the warm start of a time-resolved sequence from an earlier field and
the region mask (no vector, NaN, at masked pixels, exactly where the oracle
has none).

Tolerances as for the default estimator: FP32 max |dV| <= 1e-3 px over
pixels whose oracle det/(Sxx+Syy)^2 >= 1e-3.  For a warm-started sequence
the GPU chain starts from its own earlier fields and the oracle chain from
its own, so the comparison also checks that the differences do not grow
along the chain.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2509_25924_gb300 as ofv  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
FP32_TOL = 1e-3
NDET_MIN = 1e-3
PATHS = [ofv.OFV_PATH_FUSED, ofv.OFV_PATH_PLAIN, ofv.OFV_PATH_TILE]


def _variant_params(gauss_sigma=0.0, inc=False, **kw):
    p = dict(kw)
    if gauss_sigma > 0:
        p.update(window=ofv.OFV_WINDOW_GAUSS, window_sigma=gauss_sigma)
    if inc:
        p["increment_form"] = 1
    return p


def _gpu(I1, I2, **kw):
    H, W = I1.shape
    kw.setdefault("input", ofv.OFV_IN_F32 if I1.dtype == np.float32 else ofv.OFV_IN_U16)
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(**kw))
    try:
        t1 = torch.from_numpy(np.ascontiguousarray(I1)).to(DEV)
        t2 = torch.from_numpy(np.ascontiguousarray(I2)).to(DEV)
        u = torch.empty((H, W), device=DEV); v = torch.empty_like(u)
        ofv.ofv_compute(h, t1, t2, u, v)
        torch.cuda.synchronize()
        return u.cpu().numpy(), v.cpu().numpy()
    finally:
        ofv.ofv_destroy(h)


def _oracle(I1, I2, psl, kr, it, sigma=0.0, inc=False, init=None):
    bits = 0 if I1.dtype == np.float32 else 12
    return oracle.flow(I1.astype(np.float64), I2.astype(np.float64),
                       oracle.Params(psl=psl, kr=kr, it=it, bits=bits, win_sigma=sigma, increment_form=inc,
                                     init=init), diagnostics=True)


def _compare(u, v, ou, ov, nd, label, tol=FP32_TOL, max_masked=0.01):
    m = nd >= NDET_MIN
    masked = 1.0 - m.mean()
    assert np.isfinite(u).all() and np.isfinite(v).all(), f"{label}: non-finite output"
    assert masked <= max_masked, f"{label}: {masked:.3%} ill-conditioned pixels"
    dmax = max(np.abs(u - ou)[m].max(), np.abs(v - ov)[m].max())
    print(f"{label}: max|dV|={dmax:.3e} masked={masked:.4%}")
    assert dmax <= tol, f"{label}: max |dV| {dmax:.3e} > {tol}"
    return dmax


@pytest.fixture(scope="module")
def rankine():
    I1, I2, _, _ = synth.rankine_pair()
    return I1, I2


VARIANTS = [
    ("gauss_s1.5_kr4", dict(gauss_sigma=1.5), 4),
    ("gauss_s3_kr7", dict(gauss_sigma=3.0), 7),
    ("increment_kr4", dict(inc=True), 4),
    ("gauss_increment_kr3", dict(gauss_sigma=2.0, inc=True), 3),
]


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("name,var,kr", VARIANTS, ids=[v[0] for v in VARIANTS])
def test_variant_matches_oracle(rankine, path, name, var, kr):
    I1, I2 = rankine
    u, v = _gpu(I1, I2, path=path, levels_psl=2, kernel_radius=kr, iterations=3, **_variant_params(**var))
    ou, ov, nd, _ = _oracle(I1, I2, 2, kr, 3, var.get("gauss_sigma", 0.0), var.get("inc", False))
    _compare(u, v, ou, ov, nd, f"{name} path {path}")


def test_gaussian_window_beyond_the_block_kernel_radius(rankine):
    """KR 12 runs the one-tile-per-CTA kernel on the fused path."""
    I1, I2 = rankine
    u, v = _gpu(I1, I2, levels_psl=1, kernel_radius=12, iterations=2, **_variant_params(gauss_sigma=5.0))
    ou, ov, nd, _ = _oracle(I1, I2, 1, 12, 2, 5.0)
    _compare(u, v, ou, ov, nd, "gauss kr12")


@pytest.mark.parametrize("storage", [ofv.OFV_STORE_F16, ofv.OFV_STORE_BF16])
def test_variants_with_reduced_storage(rankine, storage):
    I1, I2 = rankine
    var = _variant_params(gauss_sigma=2.0, inc=True)
    u, v = _gpu(I1, I2, storage=storage, **var)
    ou, ov, nd, _ = _oracle(I1, I2, 2, 4, 3, 2.0, True)
    m = nd >= NDET_MIN
    rms = float(np.sqrt(np.mean((np.hypot(u - ou, v - ov)[m]) ** 2)))
    assert rms <= 1e-2, rms


def test_gaussian_with_wide_sigma_approaches_the_box(rankine):
    I1, I2 = rankine
    ub, vb = _gpu(I1, I2)
    uw, vw = _gpu(I1, I2, **_variant_params(gauss_sigma=1e4))
    ou, ov, nd, _ = _oracle(I1, I2, 2, 4, 3)
    m = nd >= NDET_MIN
    assert max(np.abs(uw - ub)[m].max(), np.abs(vw - vb)[m].max()) < 2e-3


def test_batched_and_noalloc_run_the_variants_bitwise_like_compute():
    var = _variant_params(gauss_sigma=1.8, inc=True, levels_psl=1, kernel_radius=3, iterations=2,
                          input=ofv.OFV_IN_F32)
    shapes = [(96, 128), (80, 72), (128, 128)]
    H, W = 128, 128
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(**var))
    try:
        pairs, ref = [], []
        for k, (hh, ww) in enumerate(shapes):
            I1, I2, _, _ = synth.rankine_pair(hh, ww, seed=30 + k, R=16.0, dmax=1.5)
            t1 = torch.from_numpy(I1).to(DEV); t2 = torch.from_numpy(I2).to(DEV)
            u = torch.empty((hh, ww), device=DEV); v = torch.empty_like(u)
            pairs.append((t1, t2, u, v))
            hk = ofv.ofv_create(hh, ww, ofv.ofv_default_params(**var))
            try:
                ru = torch.empty_like(u); rv = torch.empty_like(u)
                ofv.ofv_compute(hk, t1, t2, ru, rv)
                nu = torch.empty_like(u); nv = torch.empty_like(u)
                ofv.ofv_compute_noalloc(hh, ww, ofv.ofv_default_params(**var), None, t1, t2, nu, nv)
                torch.cuda.synchronize()
                assert torch.equal(nu, ru) and torch.equal(nv, rv)
                ref.append((ru, rv))
            finally:
                ofv.ofv_destroy(hk)
        ofv.ofv_compute_batched(h, pairs)
        torch.cuda.synchronize()
        for (_, _, u, v), (ru, rv) in zip(pairs, ref):
            assert torch.equal(u, ru) and torch.equal(v, rv)
    finally:
        ofv.ofv_destroy(h)


# --------------------------------------------------------------------------
# warm start of a time-resolved sequence
# --------------------------------------------------------------------------
def _oracle_chain(F, d, psl, kr, it):
    out = []
    for k in range(F.shape[0] - 1):
        init = (out[k - d][0], out[k - d][1]) if d > 0 and k >= d else None
        out.append(_oracle(F[k], F[k + 1], psl, kr, it, init=init))
    return out


@pytest.mark.parametrize("d,batch,psl,it,path", [
    (1, 8, 0, 2, ofv.OFV_PATH_FUSED), (2, 2, 2, 3, ofv.OFV_PATH_FUSED), (3, 4, 1, 2, ofv.OFV_PATH_FUSED),
    (1, 1, 1, 2, ofv.OFV_PATH_PLAIN), (4, 2, 0, 2, ofv.OFV_PATH_FUSED), (6, 2, 1, 2, ofv.OFV_PATH_FUSED),
])
def test_warm_started_sequence_matches_the_oracle_chain(d, batch, psl, it, path):
    """d <= batch: groups of d pairs; d = m batch: groups of batch pairs,
    each started from the group m back (device sequence only; the host-memory
    form refuses it)."""
    n, H, W, kr = 11, 96, 128, 4
    F = synth.stream_frames(H, W, n, seed=5)
    p = ofv.ofv_default_params(levels_psl=psl, kernel_radius=kr, iterations=it, max_batch=batch, warm_start=d,
                               path=path)
    h = ofv.ofv_create(H, W, p)
    try:
        fr = torch.from_numpy(F).to(DEV)
        us = torch.empty((n - 1, H, W), device=DEV); vs = torch.empty_like(us)
        ofv.ofv_compute_sequence(h, n, fr, H * W * 2, us, vs, H * W)
        torch.cuda.synchronize()
        hu = torch.empty((n - 1, H, W)).pin_memory(); hv = torch.empty_like(hu).pin_memory()
        if d <= batch:  # the same sequence from host memory gives the same fields bitwise
            ofv.ofv_compute_sequence_host(h, n, torch.from_numpy(F).pin_memory(), H * W * 2, hu, hv, H * W)
            torch.cuda.synchronize()
            assert torch.equal(hu, us.cpu()) and torch.equal(hv, vs.cpu())
        else:
            with pytest.raises(ofv.OfvError) as ei:
                ofv.ofv_compute_sequence_host(h, n, torch.from_numpy(F).pin_memory(), H * W * 2, hu, hv, H * W)
            assert ei.value.status == ofv.OFV_ERR_INVALID_ARG
        ref = _oracle_chain(F, d, psl, kr, it)
        for k in range(n - 1):
            ou, ov, nd, _ = ref[k]
            _compare(us[k].cpu().numpy(), vs[k].cpu().numpy(), ou, ov, nd, f"warm d={d} pair {k}")
    finally:
        ofv.ofv_destroy(h)


def test_warm_start_pairs_before_d_equal_the_cold_start():
    n, H, W = 6, 96, 128
    F = synth.stream_frames(H, W, n, seed=6)
    fr = torch.from_numpy(F).to(DEV)
    res = []
    for d in (0, 3):
        h = ofv.ofv_create(H, W, ofv.ofv_default_params(max_batch=4, warm_start=d))
        try:
            us = torch.empty((n - 1, H, W), device=DEV); vs = torch.empty_like(us)
            ofv.ofv_compute_sequence(h, n, fr, H * W * 2, us, vs, H * W)
            torch.cuda.synchronize()
            res.append((us.clone(), vs.clone()))
        finally:
            ofv.ofv_destroy(h)
    assert torch.equal(res[0][0][:3], res[1][0][:3]) and torch.equal(res[0][1][:3], res[1][1][:3])
    assert not torch.equal(res[0][0][3:], res[1][0][3:])


def test_warm_start_beyond_the_batch_is_rejected():
    """d above the pairs per launch and not a multiple of it."""
    H, W = 96, 128
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(max_batch=2, warm_start=3))
    try:
        F = torch.zeros((4, H, W), dtype=torch.uint16, device=DEV)
        u = torch.empty((3, H, W), device=DEV)
        with pytest.raises(ofv.OfvError) as ei:
            ofv.ofv_compute_sequence(h, 4, F, H * W * 2, u, torch.empty_like(u), H * W)
        assert ei.value.status == ofv.OFV_ERR_INVALID_ARG
    finally:
        ofv.ofv_destroy(h)


@pytest.mark.parametrize("var", [dict(gauss_sigma=2.0), dict(inc=True)])
def test_reverse_mode_rejects_the_variants(var):
    H, W = 64, 64
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(input=ofv.OFV_IN_F32, levels_psl=1, **_variant_params(**var)))
    try:
        z = torch.zeros((H, W), device=DEV)
        with pytest.raises(ofv.OfvError) as ei:
            ofv.ofv_backward(h, z, z, z, z, torch.empty_like(z), torch.empty_like(z))
        assert ei.value.status == ofv.OFV_ERR_UNSUPPORTED
    finally:
        ofv.ofv_destroy(h)


# --------------------------------------------------------------------------
# region mask
# --------------------------------------------------------------------------
def _disk_and_band_mask(H, W):
    yy, xx = np.mgrid[0:H, 0:W]
    m = np.ones((H, W), np.uint8)
    m[(xx - 0.6 * W) ** 2 + (yy - 0.4 * H) ** 2 < (0.08 * W) ** 2] = 0
    m[int(0.75 * H):int(0.75 * H) + 7, :int(0.5 * W)] = 0
    return m


def _gpu_masked(I1, I2, m, **kw):
    H, W = I1.shape
    kw.setdefault("input", ofv.OFV_IN_F32 if I1.dtype == np.float32 else ofv.OFV_IN_U16)
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(**kw))
    try:
        ofv.ofv_set_mask(h, torch.from_numpy(m).to(DEV))
        t1 = torch.from_numpy(np.ascontiguousarray(I1)).to(DEV)
        t2 = torch.from_numpy(np.ascontiguousarray(I2)).to(DEV)
        u = torch.empty((H, W), device=DEV); v = torch.empty_like(u)
        ofv.ofv_compute(h, t1, t2, u, v)
        torch.cuda.synchronize()
        return u.cpu().numpy(), v.cpu().numpy()
    finally:
        ofv.ofv_destroy(h)


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("kr,psl", [(4, 2), (2, 1), (12, 1)])
def test_masked_field_matches_oracle(rankine, path, kr, psl):
    I1, I2 = rankine
    m = _disk_and_band_mask(*I1.shape)
    u, v = _gpu_masked(I1, I2, m, path=path, levels_psl=psl, kernel_radius=kr, iterations=2)
    ou, ov, nd, _ = oracle.flow(I1.astype(np.float64), I2.astype(np.float64),
                                oracle.Params(psl=psl, kr=kr, it=2, mask=m), diagnostics=True)
    assert np.array_equal(np.isnan(u), m == 0) and np.array_equal(np.isnan(v), m == 0)
    sel = m != 0
    _compare(u[sel], v[sel], ou[sel], ov[sel], nd[sel], f"mask kr{kr} psl{psl} path {path}")


def test_masked_sequence_and_clearing_the_mask():
    n, H, W = 6, 96, 128
    F = synth.stream_frames(H, W, n, seed=9)
    m = _disk_and_band_mask(H, W)
    fr = torch.from_numpy(F).to(DEV)
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(max_batch=2))
    try:
        u0 = torch.empty((H, W), device=DEV); v0 = torch.empty_like(u0)
        ofv.ofv_compute(h, fr[1], fr[2], u0, v0)
        ofv.ofv_set_mask(h, torch.from_numpy(m).to(DEV))
        us = torch.empty((n - 1, H, W), device=DEV); vs = torch.empty_like(us)
        ofv.ofv_compute_sequence(h, n, fr, H * W * 2, us, vs, H * W)
        u1 = torch.empty_like(u0); v1 = torch.empty_like(u0)
        ofv.ofv_compute(h, fr[1], fr[2], u1, v1)
        torch.cuda.synchronize()
        assert torch.equal(u1.isnan(), torch.from_numpy(m == 0).to(DEV))
        assert torch.equal(us[1].nan_to_num(7.0), u1.nan_to_num(7.0)) and torch.equal(vs[1].nan_to_num(7.0),
                                                                                      v1.nan_to_num(7.0))
        ou, ov, nd, _ = oracle.flow(F[1].astype(np.float64), F[2].astype(np.float64),
                                    oracle.Params(bits=12, mask=m), diagnostics=True)
        sel = m != 0
        _compare(u1.cpu().numpy()[sel], v1.cpu().numpy()[sel], ou[sel], ov[sel], nd[sel], "masked u16 pair")
        for fn in (lambda: ofv.ofv_compute_batched(h, [(fr[0], fr[1], u1, v1)]),
                   lambda: ofv.ofv_backward(h, fr[0], fr[1], u1, v1, torch.empty_like(u1), torch.empty_like(u1))):
            with pytest.raises(ofv.OfvError) as ei:
                fn()
            assert ei.value.status == ofv.OFV_ERR_UNSUPPORTED
        ofv.ofv_set_mask(h, None)
        ofv.ofv_compute(h, fr[1], fr[2], u1, v1)
        torch.cuda.synchronize()
        assert torch.equal(u1, u0) and torch.equal(v1, v0)
    finally:
        ofv.ofv_destroy(h)


@pytest.mark.parametrize("kr,storage,edge", [(1, ofv.OFV_STORE_F32, 0), (3, ofv.OFV_STORE_F32, 0),
                                             (4, ofv.OFV_STORE_F32, 32), (4, ofv.OFV_STORE_F16, 0),
                                             (5, ofv.OFV_STORE_BF16, 0), (6, ofv.OFV_STORE_F32, 32),
                                             (10, ofv.OFV_STORE_F32, 0)])
def test_masked_launches_stage_by_tensor_copies_as_unmasked_ones_do(kr, storage, edge):
    """The kernels a mask runs have a staged box of their own: with tensor maps
    of the box window's kernels they would copy their tiles row by row."""
    H, W = 230, 300
    I1, I2 = (I.astype(np.float32) for I in synth.smooth_pair(H, W, (1.3, -0.7), seed=12))
    m = _disk_and_band_mask(H, W)
    kw = dict(levels_psl=1, kernel_radius=kr, iterations=2)
    h = ofv.ofv_create(H, W, ofv.ofv_default_params(input=ofv.OFV_IN_F32, storage=storage, tile_edge=edge, **kw))
    try:
        assert ofv.ofv_debug_tma_levels(h) == 2
        t1, t2 = torch.from_numpy(I1).to(DEV), torch.from_numpy(I2).to(DEV)
        u0 = torch.empty((H, W), device=DEV); v0 = torch.empty_like(u0)
        ofv.ofv_compute(h, t1, t2, u0, v0)
        ofv.ofv_set_mask(h, torch.from_numpy(m).to(DEV))
        assert ofv.ofv_debug_tma_levels(h) == 2
        u = torch.empty_like(u0); v = torch.empty_like(u0)
        ofv.ofv_compute(h, t1, t2, u, v)
        ofv.ofv_set_mask(h, None)
        assert ofv.ofv_debug_tma_levels(h) == 2
        u1 = torch.empty_like(u0); v1 = torch.empty_like(u0)
        ofv.ofv_compute(h, t1, t2, u1, v1)
        torch.cuda.synchronize()
        assert torch.equal(u1, u0) and torch.equal(v1, v0)
    finally:
        ofv.ofv_destroy(h)
    ou, ov, nd, _ = oracle.flow(I1.astype(np.float64), I2.astype(np.float64),
                                oracle.Params(psl=1, kr=kr, it=2, mask=m), diagnostics=True)
    u, v = u.cpu().numpy(), v.cpu().numpy()
    assert np.array_equal(np.isnan(u), m == 0)
    sel = m != 0
    # a 3x3 window leaves more pixels nearly singular; 16-bit levels by the RMS rule
    if storage == ofv.OFV_STORE_F32:
        _compare(u[sel], v[sel], ou[sel], ov[sel], nd[sel], f"mask kr{kr}", max_masked=0.05 if kr == 1 else 0.01)
    else:
        d = np.hypot(u[sel] - ou[sel], v[sel] - ov[sel])[nd[sel] >= 1e-3]
        assert np.sqrt(np.mean(d ** 2)) <= 1e-2


def test_graph_replay_runs_the_variants_and_the_mask_like_compute(rankine):
    """A CUDA graph recorded with the Gaussian window, the increment form and
    a region mask replays bitwise the field of ofv_compute."""
    I1, I2 = rankine
    H, W = I1.shape
    m = _disk_and_band_mask(H, W)
    p = ofv.ofv_default_params(input=ofv.OFV_IN_F32, **_variant_params(gauss_sigma=2.5, inc=True))
    h = ofv.ofv_create(H, W, p)
    try:
        ofv.ofv_set_mask(h, torch.from_numpy(m).to(DEV))
        t1 = torch.from_numpy(I1).to(DEV); t2 = torch.from_numpy(I2).to(DEV)
        u = torch.empty((H, W), device=DEV); v = torch.empty_like(u)
        ofv.ofv_compute(h, t1, t2, u, v)
        gu = torch.empty_like(u); gv = torch.empty_like(u)
        g = ofv.ofv_graph_create(h, t1, t2, gu, gv)
        try:
            ofv.ofv_graph_launch(g)
            torch.cuda.synchronize()
        finally:
            ofv.ofv_graph_destroy(g)
        assert torch.equal(gu.nan_to_num(9.0), u.nan_to_num(9.0)) and torch.equal(gv.nan_to_num(9.0), v.nan_to_num(9.0))
        assert torch.equal(gu.isnan().cpu(), torch.from_numpy(m == 0))
    finally:
        ofv.ofv_destroy(h)


def _random_variant_configs(n=14, seed=20251203):
    r = np.random.default_rng(seed)
    out = []
    while len(out) < n:
        psl, it = int(r.integers(0, 4)), int(r.integers(1, 4))
        path = int(r.integers(0, 3))
        kr = int(r.integers(1, 11)) if path != ofv.OFV_PATH_TILE or r.random() < 0.7 else 12
        minsz = max(8, 2 * kr + 1) * (1 << psl)
        H, W = int(r.integers(minsz, minsz + 120)), int(r.integers(minsz, minsz + 120))
        dm = 0.9 if psl == 0 else 2.5
        d = (float(r.uniform(-dm, dm)), float(r.uniform(-dm, dm)))
        sigma = float(r.uniform(0.8, 4.0)) if r.random() < 0.5 else 0.0
        inc = bool(r.random() < 0.5)
        mask = bool(r.random() < 0.4)
        store = int(r.integers(0, 3))
        if store != ofv.OFV_STORE_F32 and kr == 1:
            # a 3 x 3 window is too sensitive for 16-bit level storage: FP16-sized
            # input noise moves half the FP64 field by more than 1e-3 px
            kr = 2
        out.append((H, W, psl, kr, it, path, d, sigma, inc, mask, store, int(r.integers(0, 2**31))))
    return out


@pytest.mark.parametrize("H,W,psl,kr,it,path,d,sigma,inc,mask,store,seed", _random_variant_configs())
def test_random_variant_configurations_match_oracle(H, W, psl, kr, it, path, d, sigma, inc, mask, store, seed):
    """Seeded random shapes, pyramid depths, radii, iterations, paths,
    displacements, storage types and combinations of the Gaussian window,
    the increment form and a region mask: FP32 by the max rule on the pixels
    FP32 data determines (an oracle-only perturbation mask, as in the
    default-path test), FP16 / BF16 by the RMS rule on the pixels the stored
    precision determines (the same perturbation at the storage's rounding);
    no vector exactly at the masked pixels."""
    I1, I2 = synth.translation_pair(H, W, d, seed=seed % 100000, kind=synth.OUT_F32)
    m = _disk_and_band_mask(H, W) if mask else None
    kw = dict(path=path, levels_psl=psl, kernel_radius=kr, iterations=it, storage=store,
              **_variant_params(gauss_sigma=sigma, inc=inc))
    if m is not None:
        u, v = _gpu_masked(I1, I2, m, **kw)
    else:
        u, v = _gpu(I1, I2, **kw)
    prm = dict(psl=psl, kr=kr, it=it, win_sigma=sigma, increment_form=inc, mask=m)
    ou, ov, nd, _ = oracle.flow(I1.astype(np.float64), I2.astype(np.float64), oracle.Params(**prm),
                                diagnostics=True)
    valid = np.ones((H, W), bool) if m is None else (m != 0)
    assert np.array_equal(np.isnan(u), ~valid) and np.array_equal(np.isnan(v), ~valid)
    label = f"{H}x{W} psl={psl} kr={kr} it={it} path={path} sigma={sigma:.2f} inc={inc} mask={mask} store={store}"
    sel = valid & (nd >= NDET_MIN)
    if store == ofv.OFV_STORE_F32:
        rng = np.random.default_rng(1234)
        worst = np.zeros((H, W))
        for _ in range(2):
            a1 = I1.astype(np.float64) * (1 + 1e-7 * rng.standard_normal(I1.shape))
            a2 = I2.astype(np.float64) * (1 + 1e-7 * rng.standard_normal(I2.shape))
            pu, pv = oracle.flow(a1, a2, oracle.Params(**prm))
            worst = np.maximum(worst, np.nan_to_num(np.hypot(pu - ou, pv - ov)))
        sel &= worst <= 0.1 * FP32_TOL
        masked = 1.0 - sel[valid].mean()
        assert masked <= 0.05, f"{label}: {masked:.3%} excluded"
        dmax = max(np.abs(u - ou)[sel].max(), np.abs(v - ov)[sel].max())
        print(f"{label}: max|dV|={dmax:.3e} excluded={masked:.4%}")
        assert dmax <= FP32_TOL, f"{label}: max |dV| {dmax:.3e}"
    else:
        # the storage rounds the level images to 2^-11 (FP16) or 2^-8 (BF16)
        # relative: leave out the pixels where input noise of that size moves
        # the FP64 field by more than the tolerance itself (small windows,
        # e.g. KR 1, are that sensitive)
        rel = 2.0 ** -11 if store == ofv.OFV_STORE_F16 else 2.0 ** -8
        rng = np.random.default_rng(4321)
        worst = np.zeros((H, W))
        for _ in range(2):
            a1 = I1.astype(np.float64) * (1 + rel * rng.standard_normal(I1.shape))
            a2 = I2.astype(np.float64) * (1 + rel * rng.standard_normal(I2.shape))
            pu, pv = oracle.flow(a1, a2, oracle.Params(**prm))
            worst = np.maximum(worst, np.nan_to_num(np.hypot(pu - ou, pv - ov)))
        sel &= worst <= 1e-2
        masked = 1.0 - sel[valid].mean()
        assert masked <= 0.25, f"{label}: {masked:.3%} excluded"
        rms = float(np.sqrt(np.mean(np.hypot(u - ou, v - ov)[sel] ** 2)))
        print(f"{label}: rms={rms:.3e} excluded={masked:.4%}")
        assert rms <= 1e-2, f"{label}: rms {rms:.3e}"
