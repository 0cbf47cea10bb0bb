"""The tile kernels that keep their frame in registers, at the sizes and data where their tiling, their
border handling or their shortcuts change: against the one-iteration kernels (a pinned block or strip
height), whose arithmetic they repeat, so the comparison is for equality."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_10979_gb300 import flow, synth  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = flow.Context(0)
    yield c
    c.close()


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def images(H, W, kind="plain"):
    if min(H, W) > 8:
        p = synth.random_affine_rect_pair(H, W, H + W)
        I0, I1 = p.I0.copy(), p.I1.copy()
    else:
        I0, I1 = np.random.default_rng(H + W).random((2, H, W)).astype(np.float32)
    if kind == "flat":  # zero residuals and gradients beside textured pixels
        I0[:, W // 2:] = I1[:, W // 2:] = 0.25
    elif kind == "faint":  # squared gradients and residuals near and below the smallest normal number
        I0, I1 = I0 * np.float32(1e-19), I1 * np.float32(1e-19)
    return cu(I0), cu(I1)


def both(ctx, im, pinned, ref_engine=None, **kw):
    ref = dict(kw, engine=kw["engine"] if ref_engine is None else ref_engine)
    a = flow.of_solve(ctx, *im, flow.default_params(rows_per_warp=pinned, **ref), want_w=True)
    b = flow.of_solve(ctx, *im, flow.default_params(rows_per_warp=0, **kw), want_w=True)
    for x, y in zip(a[:2], b[:2]):
        assert torch.equal(x, y)
    if kw.get("beta", 1.0) != 0.0:
        assert torch.equal(a[2], b[2])
    assert a[3]["iters_run"] == b[3]["iters_run"]


@pytest.mark.parametrize("method", [flow.OF_PADMM_I, flow.OF_CP, flow.OF_PDR])
@pytest.mark.parametrize("engine", [flow.OF_ENGINE_FUSED, flow.OF_ENGINE_STREAM, flow.OF_ENGINE_RESIDENT])
@pytest.mark.parametrize("prec", [0, 2])
def test_without_beta_w_is_zero_whatever_the_launch_count(ctx, method, engine, prec):
    """The iterations leave w alone without beta: it is zero in whichever buffer the last launch ends, also
    where the workspace held another solve's w."""
    im = images(150, 200)
    for iters in (11, 12, 13, 14):
        kw = dict(method=method, engine=engine, precision=prec, lam=3.0, levels=2, warps=2, iters=iters)
        w = flow.of_solve(ctx, *im, flow.default_params(beta=0.05, **kw), want_w=True)[2]
        assert w.abs().max() > 0
        w = flow.of_solve(ctx, *im, flow.default_params(beta=0.0, **kw), want_w=True)[2]
        assert torch.equal(w, torch.zeros_like(w))


# One frame and its neighbours: 64 columns less the halo (8 to 16), 24, 36 or 48 rows less theirs.
@pytest.mark.parametrize("H,W", [(1, 1), (2, 300), (300, 2), (35, 49), (36, 50), (47, 65), (130, 171), (391, 590)])
@pytest.mark.parametrize("iters", [20, 47])
def test_alg1_tiles_at_their_edges(ctx, H, W, iters):
    eng = flow.OF_ENGINE_STREAM if H * W < 7000 else flow.OF_ENGINE_FUSED  # (the fused engine's small levels are resident)
    both(ctx, images(H, W), 8, method=flow.OF_CP, lam=3.0, levels=1, warps=2, iters=iters, engine=eng)


@pytest.mark.parametrize("kind", ["flat", "faint"])
@pytest.mark.parametrize("beta", [0.05, 0.0, 1e-16])
def test_alg1_quotients_outside_the_usual_range(ctx, kind, beta):
    both(ctx, images(150, 202, kind), 8, method=flow.OF_CP, lam=3.0, beta=beta, levels=1, warps=2, iters=40,
         engine=flow.OF_ENGINE_FUSED)


# Tiles of the cluster engine: one column of up to 64 pixels or several of up to 60, two to twelve rows; the last
# size does not fit it.  Launches of an odd and an even number of iterations, and fewer than one exchange takes.
@pytest.mark.parametrize("H,W", [(1, 1), (2, 3), (1, 64), (3, 65), (48, 64), (49, 63), (33, 120), (192, 2), (60, 80),
                                 (12, 700), (96, 122), (97, 119)])
@pytest.mark.parametrize("iters", [1, 2, 37])
@pytest.mark.parametrize("kw", [dict(), dict(method=flow.OF_PADMM_II, rho=1.7), dict(beta=0.0, a_tilde_mode=1),
                                dict(precision=2, fp32_flow=0)], ids=["I", "II", "per-pixel", "bf16"])
def test_admm_cluster_engine_at_its_edges(ctx, H, W, iters, kw):
    P = dict(dict(method=flow.OF_PADMM_I, lam=3.0, levels=1, warps=2, iters=iters, engine=flow.OF_ENGINE_RESIDENT), **kw)
    both(ctx, images(H, W), 1, flow.OF_ENGINE_STREAM, **P)


@pytest.mark.parametrize("H,W", [(30, 40), (60, 80)])
@pytest.mark.parametrize("iters", [40, 25])
def test_admm_cluster_engine_stops_where_the_streamed_solve_does(ctx, H, W, iters):
    im = images(H, W)
    kw = dict(method=flow.OF_PADMM_I, lam=3.0, levels=1, iters=iters, engine=flow.OF_ENGINE_RESIDENT)
    tol = flow.of_solve(ctx, *im, flow.default_params(warps=1, **dict(kw, iters=20)))[3]["residual"] * 1.001
    for t in (tol, 1e-30):
        both(ctx, im, 1, flow.OF_ENGINE_STREAM, warps=2, tol=t, **kw)


# pDR's register tiles (levels from 40,000 pixels) against the tile kernel that batches run: frames of 64 x 48 less a
# halo of 7 to 31 pixels, odd sizes, strips narrower and lower than a frame, one launch of every length.
@pytest.mark.parametrize("H,W", [(200, 201), (201, 200), (127, 641), (41, 1000), (1000, 41), (7, 5801), (5801, 7), (480, 640)])
@pytest.mark.parametrize("kw", [dict(), dict(beta=0.0), dict(precision=2, fp32_flow=1), dict(precision=1, fp32_flow=0),
                                dict(tol=1e-30)], ids=["f32", "beta0", "bf16", "f16", "tested"])
def test_pdr_register_tiles_equal_the_batched_tile_kernel(ctx, H, W, kw):
    im = images(H, W)
    for iters in (1, 13, 20):
        P = flow.default_params(method=flow.OF_PDR, lam=3.0, levels=1, warps=2, iters=iters, engine=flow.OF_ENGINE_STREAM, **kw)
        u, v, _, st = flow.of_solve(ctx, *im, P)
        ub, vb, sb = flow.of_solve_batch(ctx, [im[0]] * 2, [im[1]] * 2, P)
        assert torch.equal(u, ub[0]) and torch.equal(v, vb[0])
        assert st["iters_run"] == sb[0]["iters_run"]
        assert st["residual"] == pytest.approx(sb[0]["residual"], rel=1e-5, abs=1e-12)


@pytest.mark.parametrize("kind", ["flat", "faint"])
@pytest.mark.parametrize("beta", [0.05, 0.0, 1e-16])
def test_pdr_quotients_outside_the_usual_range(ctx, kind, beta):
    im = images(202, 206, kind)
    P = flow.default_params(method=flow.OF_PDR, lam=3.0, beta=beta, levels=1, warps=2, iters=30, engine=flow.OF_ENGINE_STREAM)
    u, v, _, _ = flow.of_solve(ctx, *im, P)
    ub, vb, _ = flow.of_solve_batch(ctx, [im[0]] * 2, [im[1]] * 2, P)
    assert torch.equal(u, ub[0]) and torch.equal(v, vb[0])


def np64(t):
    return t.cpu().double().numpy()


# The one-launch pyramid step at tile edges (32 x 16 coarse pixels) and, for the smallest ratio, the three kernels it
# falls back to where its tile does not fit: the bar of the operator's parity test.
@pytest.mark.parametrize("H,W", [(2, 2), (63, 33), (65, 131), (128, 64)])
@pytest.mark.parametrize("eta", [0.5, 0.8, 0.2])
def test_pyramid_step_on_either_route(orc, H, W, eta):
    img = np.random.default_rng(H + W).random((H, W)).astype(np.float32)
    Hc, Wc = orc.level_size(H, eta), orc.level_size(W, eta)
    got = np64(flow.of_pyr_down(cu(img), Hc, Wc, eta))
    assert np.max(np.abs(got - orc.downsample(img.astype(np.float64), Hc, Wc, eta))) < 2e-5


# Twofold FP32 with the rounding test: FP64's results rounded once.  The oracle forms the same terms in FP64 in its own
# order, each below 16, so a value may differ where 2^-48 of that crosses a rounding boundary: one FP32 unit at most.
@pytest.mark.parametrize("flow_kind", ["fractions", "integers", "zero", "far outside"])
@pytest.mark.parametrize("H,W", [(1, 1), (1, 33), (9, 32), (45, 61)])
def test_warp_gives_the_fp64_results(orc, H, W, flow_kind):
    rng = np.random.default_rng(H * W)
    I0, I1 = rng.random((2, H, W)).astype(np.float32)
    u0, v0 = {"fractions": rng.uniform(-5, 5, (2, H, W)), "integers": rng.integers(-4, 5, (2, H, W)),
              "zero": np.zeros((2, H, W)), "far outside": rng.uniform(-5, 5, (2, H, W)) + 3 * max(H, W)}[flow_kind].astype(np.float32)
    gx, gy = flow.of_derivatives(cu(I1))
    Ix, Iy, It, _ = flow.of_warp_linearise(cu(I0), cu(I1), gx, gy, cu(u0), cu(v0), 0.05)
    ref = orc.warp_linearise(I0, I1, np64(gx), np64(gy), u0, v0, 0.05)
    scale = max(1.0, float(np.abs(u0).max() + np.abs(v0).max()))
    for a, b in zip((Ix, Iy, It), ref):
        assert np.all(np.abs(np64(a) - b) <= np.spacing(np.abs(b).astype(np.float32)) + scale * 2.0 ** -48)
