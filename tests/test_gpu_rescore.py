"""mf_rescore_topk: candidate selection is exact integer work (bit-exact against
the oracle's ordering rule on the same snr_max/argmax maps, generated on the
host), and the FP64 re-score matches the FP64 oracle, evaluated at the
oracle's own selection, to 1e-9 relative (two FP64 sums in different
order)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mf():
    import paper_2209_09848_gb300 as m
    assert torch.cuda.is_available()
    m.load()
    return m


@pytest.mark.parametrize("k_top,T,H,W,mask_frac", [(64, 20, 70, 90, 0.02), (500, 12, 48, 64, 0.0),
                                                   (4096, 8, 64, 80, 0.01), (1, 5, 16, 16, 0.0)])
def test_rescore_matches_oracle(mf, oracle, k_top, T, H, W, mask_frac):
    from paper_2209_09848_gb300 import synth
    c = synth.small_case(T, H, W, 17 + k_top, mask_frac=mask_frac, movers=4)
    vx, vy = synth.velocity_grid(4, 3, -0.3, 0.3)
    K = len(vx)
    table = mf.prf_table_create(vx, vy, T)
    # a best-score map and its trajectories from the host generator: the
    # selection and the re-score read them, not a search's output
    s_max, a_max = synth.score_map(H, W, seed=k_top + H, K=K, mask_frac=mask_frac)
    dev = "cuda"
    r = torch.from_numpy(c["res"]).to(dev)
    s = torch.from_numpy(c["sigma"]).to(dev)
    m = None if c["mask"] is None else torch.from_numpy(c["mask"]).to(dev)
    k_eff = min(k_top, H * W)
    raw, n = mf.rescore_topk(r, s, table, torch.from_numpy(s_max).to(dev), torch.from_numpy(a_max).to(dev),
                             k_eff, mask=m)
    torch.cuda.synchronize()
    assert mf.device_status() == 0
    n = int(n.item())
    cands = mf.decode_candidates(raw, n)
    want = oracle.topk_order(s_max, a_max, k_eff)
    assert n == len(want)
    got_idx = cands["y"].astype(np.int64) * W + cands["x"]
    assert np.array_equal(got_idx, want)
    wy, wx = want // W, want % W
    wk = a_max.ravel()[want]
    assert np.array_equal(cands["k"], wk)
    assert np.array_equal(cands["snr_search"], s_max.ravel()[want])
    sh, tp = oracle.trajectory_table(vx, vy, T)
    lam = oracle.inverse_variance(c["sigma"], c["mask"])
    N, D = oracle.search_points(c["res"], lam, sh, tp, wy.astype(np.int32), wx.astype(np.int32), wk)
    ok = D > 0
    np.testing.assert_allclose(cands["snr"][ok], N[ok] / np.sqrt(D[ok]), rtol=1e-9, atol=1e-12)
    np.testing.assert_allclose(cands["flux"][ok], N[ok] / D[ok], rtol=1e-9, atol=1e-12)
    assert np.all(cands["snr"][~ok] == 0) and np.all(cands["flux"][~ok] == 0)


def test_rescore_reads_bf16_master_as_stored(mf, oracle):
    from paper_2209_09848_gb300 import synth
    T, H, W = 10, 40, 56
    c = synth.small_case(T, H, W, 5, mask_frac=0.01, movers=3)
    vx, vy = synth.velocity_grid(3, 3, -0.2, 0.2)
    table = mf.prf_table_create(vx, vy, T)
    q = torch.from_numpy(c["res"]).to(torch.bfloat16)
    r = q.cuda()
    s = torch.from_numpy(c["sigma"]).cuda()
    m = torch.from_numpy(c["mask"]).cuda()
    s_max, a_max = synth.score_map(H, W, seed=6, K=len(vx), mask_frac=0.0)
    raw, n = mf.rescore_topk(r, s, table, torch.from_numpy(s_max).cuda(), torch.from_numpy(a_max).cuda(), 50,
                             mask=m)
    torch.cuda.synchronize()
    cands = mf.decode_candidates(raw, int(n.item()))
    want = oracle.topk_order(s_max, a_max, 50)
    assert np.array_equal(cands["y"].astype(np.int64) * W + cands["x"], want)
    sh, tp = oracle.trajectory_table(vx, vy, T)
    lam = oracle.inverse_variance(c["sigma"], c["mask"])
    N, D = oracle.search_points(q.float().numpy(), lam, sh, tp, (want // W).astype(np.int32),
                                (want % W).astype(np.int32), a_max.ravel()[want])
    ok = D > 0
    np.testing.assert_allclose(cands["snr"][ok], N[ok] / np.sqrt(D[ok]), rtol=1e-9, atol=1e-12)


def test_rescore_argument_errors(mf):
    T, H, W = 4, 8, 8
    table = mf.prf_table_create([0.1], [0.0], T)
    r = torch.zeros((T, H, W), device="cuda")
    s = torch.ones((H, W), device="cuda")
    smax = torch.zeros((H, W), device="cuda")
    amax = torch.zeros((H, W), dtype=torch.int32, device="cuda")
    with pytest.raises(mf.MFError):
        mf.rescore_topk(r, s, table, smax, amax, 0)
    with pytest.raises(mf.MFError):
        mf.rescore_topk(r, s, table, smax, amax, H * W + 1)


@pytest.mark.parametrize("kind", ["noise", "constant", "rounded", "negative", "wide", "infinite"])
@pytest.mark.parametrize("valid", [1.0, 0.001])
def test_selection_of_hard_maps(mf, oracle, kind, valid):
    # ties by the hundred thousand (the list past the ranking's limit is cut
    # by the radix select), every sign and exponent, few valid pixels; the
    # selection is exact integer work
    H, W = 371, 523
    g = np.random.default_rng(len(kind))
    m = {"noise": lambda: g.normal(2.5, 0.45, (H, W)), "constant": lambda: np.full((H, W), 2.5),
         "rounded": lambda: np.round(g.normal(2.5, 0.45, (H, W)), 1), "negative": lambda: -np.abs(g.normal(size=(H, W))),
         "wide": lambda: g.normal(size=(H, W)) * 10.0 ** g.uniform(-40, 30, (H, W)),
         "infinite": lambda: np.where(g.random((H, W)) < 0.1, np.inf, g.normal(size=(H, W)))}[kind]().astype(np.float32)
    a = np.where(g.random((H, W)) < valid, 0, -1).astype(np.int32)
    table = mf.prf_table_create([0.0], [0.0], 1)
    r, sg = torch.zeros((1, H, W), device="cuda"), torch.ones((H, W), device="cuda")
    for k in (1, 33, 4096, 16384):
        raw, n = mf.rescore_topk(r, sg, table, torch.from_numpy(m).cuda(), torch.from_numpy(a).cuda(), k)
        c = mf.decode_candidates(raw, int(n.item()))
        assert np.array_equal(c["y"].astype(np.int64) * W + c["x"], oracle.topk_order(m, a, k))


@pytest.mark.parametrize("k_top,T", [(3, 37), (700, 9), (2500, 5)])
def test_rescore_custom_footprints_and_scales(mf, oracle, k_top, T):
    # candidates shared by 8, 8 and 2 warps; a base pixel that changes every
    # frame, footprints that do not factor, frame scales, and a masked pixel
    # holding NaN (its value does not matter); 1e-9: FP64 sums in other orders
    from paper_2209_09848_gb300 import synth
    H, W, K = 61, 70, 5
    c = synth.small_case(T, H, W, 40 + T, mask_frac=0.03, movers=1)
    g = np.random.default_rng(T)
    sh = g.integers(-9, 10, size=(K, T, 2)).astype(np.int32)
    tp = g.uniform(-0.2, 1.0, size=(K, T, 5, 5))
    table = mf.prf_table_create_custom(sh, tp)
    scale = g.uniform(0.5, 2.0, T).astype(np.float32)
    res = np.where(c["mask"][None] > 0, np.nan, c["res"]).astype(np.float32)
    s_max, a_max = synth.score_map(H, W, seed=T, K=K, mask_frac=0.0)
    dev = "cuda"
    raw, n = mf.rescore_topk(torch.from_numpy(res).to(dev), torch.from_numpy(c["sigma"]).to(dev), table,
                             torch.from_numpy(s_max).to(dev), torch.from_numpy(a_max).to(dev), k_top,
                             mask=torch.from_numpy(c["mask"]).to(dev), frame_scale=torch.from_numpy(scale).to(dev))
    got = mf.decode_candidates(raw, int(n.item()))
    want = oracle.topk_order(s_max, a_max, k_top)
    lam = oracle.inverse_variance(c["sigma"], c["mask"])
    N, D = oracle.search_points(c["res"], lam, sh, tp, (want // W).astype(np.int32), (want % W).astype(np.int32),
                                a_max.ravel()[want], frame_scale=scale.astype(np.float64))
    ok = D > 0
    np.testing.assert_allclose(got["snr"][ok], N[ok] / np.sqrt(D[ok]), rtol=1e-9, atol=1e-9)
    np.testing.assert_allclose(got["flux"][ok], N[ok] / D[ok], rtol=1e-9, atol=1e-9)


@pytest.mark.parametrize("scattered", [False, True])
@pytest.mark.parametrize("k_top,T", [(3, 301), (1500, 130), (2000, 33)])
def test_rescore_trajectories_off_the_image(mf, oracle, k_top, T, scattered):
    # trajectories that leave the image, return to it or never reach it (only
    # the frames and rows between count), and with one that jumps by hundreds
    # of pixels D from the taps instead of the collapsed kernel's rows;
    # candidates shared by 8 to 2 warps; 1e-9: FP64 sums in other orders
    from paper_2209_09848_gb300 import synth
    H, W = 43, 50
    g = np.random.default_rng(T)
    t = np.arange(T)
    paths = [(3.0 * t, 2.0 * t), (-0.7 * t, 0.0 * t), (90 * np.sin(t / 11.0), 5 * np.sin(t / 3.0)),
             (0.0 * t, -70 + 0.5 * t), (0.1 * t, -0.05 * t), (0.0 * t + 200, 0.0 * t - 200)]
    if scattered:
        paths.append((g.integers(-400, 401, T), g.integers(-400, 401, T)))
    sh = np.round(np.array(paths)).transpose(0, 2, 1).astype(np.int32)
    K = len(paths)
    tp = g.uniform(0.0, 1.0, size=(K, T, 5, 5))
    c = synth.small_case(T, H, W, 60 + T, mask_frac=0.03, movers=1)
    table = mf.prf_table_create_custom(sh, tp)
    s_max, a_max = synth.score_map(H, W, seed=T, K=K, mask_frac=0.0)
    raw, n = mf.rescore_topk(torch.from_numpy(c["res"]).cuda(), torch.from_numpy(c["sigma"]).cuda(), table,
                             torch.from_numpy(s_max).cuda(), torch.from_numpy(a_max).cuda(), k_top,
                             mask=torch.from_numpy(c["mask"]).cuda())
    got = mf.decode_candidates(raw, int(n.item()))
    want = oracle.topk_order(s_max, a_max, k_top)
    assert np.array_equal(got["y"].astype(np.int64) * W + got["x"], want)
    lam = oracle.inverse_variance(c["sigma"], c["mask"])
    N, D = oracle.search_points(c["res"], lam, sh, tp, (want // W).astype(np.int32), (want % W).astype(np.int32),
                                a_max.ravel()[want])
    ok = D > 0
    np.testing.assert_allclose(got["snr"][ok], N[ok] / np.sqrt(D[ok]), rtol=1e-9, atol=1e-9)
    np.testing.assert_allclose(got["flux"][ok], N[ok] / D[ok], rtol=1e-9, atol=1e-9)
    assert np.all(got["snr"][~ok] == 0) and np.all(got["flux"][~ok] == 0)


def test_rescore_ignores_scales_of_frames_without_a_pixel(mf, oracle):
    # a frame whose footprint lies off the image or on masked pixels adds
    # nothing, whatever its scale
    from paper_2209_09848_gb300 import synth
    T, H, W = 21, 40, 60
    c = synth.small_case(T, H, W, 77, movers=1)
    mask = np.zeros((H, W), np.uint8)
    mask[20:34, 30:44] = 1
    sh = np.zeros((2, T, 2), np.int32)
    sh[:, 3] = (500, 0)
    sh[:, 9] = (0, -300)
    sh[:, 14] = (30, 20)  # from rows 4 .. 9, columns 4 .. 9 onto the mask
    g = np.random.default_rng(3)
    tp = g.uniform(0.1, 1.0, size=(2, T, 5, 5))
    scale = g.uniform(0.5, 2.0, T).astype(np.float32)
    bad = scale.copy()
    bad[[3, 9, 14]] = np.inf, np.nan, -np.inf
    a_max = np.full((H, W), -1, np.int32)
    a_max[4:10, 4:10] = g.integers(0, 2, (6, 6))
    s_max = g.normal(size=(H, W)).astype(np.float32)
    table = mf.prf_table_create_custom(sh, tp)
    raw, n = mf.rescore_topk(torch.from_numpy(c["res"]).cuda(), torch.from_numpy(c["sigma"]).cuda(), table,
                             torch.from_numpy(s_max).cuda(), torch.from_numpy(a_max).cuda(), 30,
                             mask=torch.from_numpy(mask).cuda(), frame_scale=torch.from_numpy(bad).cuda())
    got = mf.decode_candidates(raw, int(n.item()))
    want = oracle.topk_order(s_max, a_max, 30)
    N, D = oracle.search_points(c["res"], oracle.inverse_variance(c["sigma"], mask), sh, tp,
                                (want // W).astype(np.int32), (want % W).astype(np.int32), a_max.ravel()[want],
                                frame_scale=scale.astype(np.float64))
    assert np.all(D > 0)
    np.testing.assert_allclose(got["snr"], N / np.sqrt(D), rtol=1e-9, atol=1e-9)
    np.testing.assert_allclose(got["flux"], N / D, rtol=1e-9, atol=1e-9)
