"""mf_background_refit (Section 3.1: per-pixel Huber fit of the background
and its jitter Taylor terms, with the low-resolution scattered light
subtracted) against the FP64 oracle.  The kernel sums in FP32 over an
orthonormal basis; residuals agree to |delta r| <= 2e-6 max|D| (the
rounding of FP32 frames of that size), and the fitted background phi . beta
(the coefficients themselves are ill-conditioned in the Taylor basis) to
the same bound."""
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


def _check(mf, c, delta, M, scatter=True, in_place=False):
    from oracle import background as ob
    D = torch.from_numpy(c["D"]).cuda()
    S = torch.from_numpy(c["S"]).cuda() if scatter else None
    out = D if in_place else None
    R, coef = mf.background_refit(D.clone() if not in_place else D, c["jitter"], delta, M, scatter=S,
                                  resid=out if in_place else None)
    torch.cuda.synchronize()
    assert mf.device_status() == 0
    co, Ro = ob.refit(c["D"], c["jitter"], delta, M, S=c["S"] if scatter else None)
    tol = 2e-6 * max(1.0, float(np.abs(c["D"]).max()))
    err = np.abs(R.cpu().numpy().astype(np.float64) - Ro)
    assert err.max() <= tol, "residual max err %.3g > %.3g" % (err.max(), tol)
    phi = ob.basis(c["jitter"])
    fit_g = np.einsum("tk,hwk->thw", phi, coef.cpu().numpy().astype(np.float64))
    fit_o = np.einsum("tk,hwk->thw", phi, co)
    assert np.abs(fit_g - fit_o).max() <= 4 * tol
    return R, coef


@pytest.mark.parametrize("T,H,W,n,M,delta", [
    (100, 64, 48, 8, 10, 1.345),
    (300, 37, 53, 4, 5, 1.0),        # pixel count not a multiple of the CTA, > 1 basis chunk
    (6, 20, 30, 2, 3, 1.345),         # the smallest frame count
    (64, 33, 17, 16, 0, 1.345),       # least-squares start only
    (80, 40, 40, 8, 4, float("inf")),  # least squares throughout
    (600, 16, 16, 8, 20, 0.5),       # many clipped residuals, three basis chunks
])
def test_refit_matches_oracle(mf, T, H, W, n, M, delta):
    from paper_2209_09848_gb300 import synth
    c = synth.background_case(T, H, W, seed=T + H, n=n, n_movers=2)
    _check(mf, c, delta, M)


def test_refit_without_scatter_and_in_place(mf):
    from paper_2209_09848_gb300 import synth
    c = synth.background_case(50, 30, 40, seed=3, n=4)
    _check(mf, c, 1.345, 6, scatter=False)
    _check(mf, c, 1.345, 6, in_place=True)


def test_refit_removes_background_and_keeps_movers(mf):
    # a bright mover survives in the residual; the background does not
    from paper_2209_09848_gb300 import synth
    c = synth.background_case(200, 64, 64, seed=8, n=8, n_movers=4, outlier_frac=0.0)
    R, coef = mf.background_refit(torch.from_numpy(c["D"]).cuda(), c["jitter"], 1.345, 10,
                                  scatter=torch.from_numpy(c["S"]).cuda())
    r = R.cpu().numpy()
    inner = r[:, 8:-8, 8:-8]
    assert abs(np.median(inner)) < 0.1 and np.percentile(np.abs(inner), 50) < 1.0
    assert r.max() > 1.0  # the movers


def test_refit_deterministic(mf):
    from paper_2209_09848_gb300 import synth
    c = synth.background_case(90, 50, 50, seed=9, n=8)
    D = torch.from_numpy(c["D"]).cuda()
    a = mf.background_refit(D, c["jitter"], 1.345, 5, scatter=torch.from_numpy(c["S"]).cuda())
    b = mf.background_refit(D, c["jitter"], 1.345, 5, scatter=torch.from_numpy(c["S"]).cuda())
    torch.cuda.synchronize()
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_refit_rejects_bad_arguments(mf):
    D = torch.zeros((10, 4, 4), device="cuda")
    jit = np.random.default_rng(0).uniform(-0.2, 0.2, size=(10, 2))
    for kw in (dict(delta=0.0), dict(delta=float("nan")), dict(iterations=-1), dict(iterations=1001)):
        args = dict(delta=1.0, iterations=2)
        args.update(kw)
        with pytest.raises(mf.MFError):
            mf.background_refit(D, jit, args["delta"], args["iterations"])
    with pytest.raises(mf.MFError):  # constant jitter: x and x^2 collinear with 1
        mf.background_refit(D, np.zeros((10, 2)), 1.0, 2)
    with pytest.raises(mf.MFError):  # fewer frames than coefficients
        mf.background_refit(torch.zeros((5, 4, 4), device="cuda"), jit[:5], 1.0, 2)
    bad = jit.copy()
    bad[3, 1] = np.inf
    with pytest.raises(mf.MFError):
        mf.background_refit(D, bad, 1.0, 2)


@pytest.mark.parametrize("T", [6, 7, 176, 177, 352, 353, 528, 529, 768, 769, 1152, 1153, 1920, 1921])
@pytest.mark.parametrize("H,W", [(8, 12), (5, 7)])
def test_refit_series_lengths(mf, T, H, W):
    # the edges of the layouts that keep a series on the chip, and the first
    # length that is re-read from memory; pixel counts that allow 128-bit rows
    # and one that does not (nor fills a CTA's pixels)
    from paper_2209_09848_gb300 import synth
    c = synth.background_case(T, H, W, seed=T, n=3)
    _check(mf, c, 1.345, 4)


@pytest.mark.parametrize("T,H,W,M", [
    (40, 171, 171, 2),     # one warp to a CTA
    (177, 128, 128, 2),    # two, pixel count a multiple of 4
    (353, 101, 99, 3),     # three, an odd number of steps
    (600, 101, 99, 4),     # four
    (1000, 80, 80, 10),    # six
    (1200, 53, 47, 0),     # six on 8 pixels, least squares only
])
def test_refit_more_pixel_blocks_than_ctas(mf, T, H, W, M):
    # every CTA goes on to a second block of pixels, with the shared memory of
    # the first: the buffers in which its warps exchange their sums change hands
    # after even and odd numbers of steps; in place, the residuals of one block
    # are written beside the reads of the next
    from paper_2209_09848_gb300 import synth
    c = synth.background_case(T, H, W, seed=T + M, n=4)
    a = _check(mf, c, 1.345, M)
    b = _check(mf, c, 1.345, M, in_place=True)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("frame", [0, -1])
@pytest.mark.parametrize("T,outlier", [(300, 150.0), (600, 300.0), (1500, 300.0)])
def test_refit_outlier_in_an_end_frame(mf, T, outlier, frame):
    # frames whose background is already gone, one of them hundreds of sigma
    # off: the other frames' residuals are as good as without it (the bound of
    # the other tests, for those frames' values) at every pixel whose FP64 fit
    # has let go of it in these steps; elsewhere the fit is of the outlier's size,
    # and the bound the other tests' own
    from oracle import background as ob
    H, W = 12, 20
    g = np.random.default_rng(T)
    jit = np.clip(np.cumsum(g.normal(0, 0.04, (T, 2)), 0), -0.15, 0.15)
    D = g.normal(size=(T, H, W)).astype(np.float32)
    D[frame] += np.float32(outlier)
    R, _ = mf.background_refit(torch.from_numpy(D).cuda(), jit, 1.345, 10)
    torch.cuda.synchronize()
    _, Ro = ob.refit(D, jit, 1.345, 10)
    rest = np.arange(T) != frame % T
    gone = np.abs(D[rest] - Ro[rest]).max(axis=0) <= 1.0
    err = np.abs(R.cpu().numpy().astype(np.float64) - Ro)[rest].max(axis=0)
    tol = np.where(gone, 2e-6 * max(1.0, float(np.abs(D[rest]).max())), 2e-6 * float(np.abs(D).max()))
    assert (err <= tol).all(), "residual max err / bound %.3g" % (err / tol).max()


@pytest.mark.parametrize("T,H,W", [
    (6, 344, 340), (15, 350, 337), (32, 344, 340), (33, 350, 337),  # 64 pixels to a warp, and past them
    (49, 245, 239), (96, 244, 240), (97, 245, 239),                 # 32 pixels, and past them
    (48, 7, 9), (49, 7, 9),
])
def test_refit_short_series(mf, T, H, W):
    # few frames: a warp takes more pixels where the image has enough of them;
    # pixel counts that allow 128-bit rows and ones that do not, blocks past the
    # grid's
    from paper_2209_09848_gb300 import synth
    _check(mf, synth.background_case(T, H, W, seed=T, n=5), 1.345, 3)
