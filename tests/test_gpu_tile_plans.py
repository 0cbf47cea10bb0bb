"""The ADMM tile kernel in every tiling that the cost rule picks by itself (frame height, iterations per launch, one
tile per block or looping), single pairs and batches, against the row-streaming kernel whose arithmetic it repeats:
for equality."""
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


def images(H, W):
    p = synth.random_affine_rect_pair(H, W, H + W)
    return cu(p.I0), cu(p.I1)


KINDS = {"f32": dict(), "II": dict(method=flow.OF_PADMM_II, rho=1.8), "beta0": dict(beta=0.0), "per-pixel": dict(a_tilde_mode=1),
         "f16": dict(precision=1, fp32_last_warp=0), "bf16all": dict(precision=2, fp32_flow=0, fp32_last_warp=0)}


# One tile per block with two, three and four rows per warp, and the looping form; odd and even widths; launches of
# three to eight iterations with a remainder.
@pytest.mark.parametrize("H,W", [(150, 202), (201, 301), (240, 320), (391, 590), (480, 640), (600, 801), (375, 1242), (436, 1024)])
@pytest.mark.parametrize("kind", list(KINDS))
def test_single_pairs(ctx, H, W, kind):
    im = images(H, W)
    kw = dict(lam=3.0, levels=1, warps=2, iters=23, **KINDS[kind])
    a = flow.of_solve(ctx, *im, flow.default_params(engine=flow.OF_ENGINE_STREAM, rows_per_warp=8, **kw), want_w=True)
    b = flow.of_solve(ctx, *im, flow.default_params(**kw), want_w=True)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    assert a[3]["iters_run"] == b[3]["iters_run"]
    assert a[3]["residual"] == pytest.approx(b[3]["residual"], rel=1e-5)


BATCH = [(391, 590), (150, 202), (480, 641), (201, 301), (375, 1242), (97, 131), (436, 1024)]


# More tiles than blocks: the tiles of a block lie in several pairs, and a pair that has met the stopping test is
# passed over while its neighbours go on.
@pytest.mark.parametrize("kind", [k for k in KINDS if k != "per-pixel"])
def test_batches_of_more_tiles_than_blocks(ctx, kind):
    ims = [images(H, W) for H, W in BATCH]
    for tol in (0.0, None):
        kw = dict(lam=3.0, levels=1, warps=2, iters=40, **KINDS[kind])
        ref = dict(kw, engine=flow.OF_ENGINE_STREAM, rows_per_warp=8)
        if tol is None:  # between the pairs' residuals: some stop early
            res = [flow.of_solve(ctx, *im, flow.default_params(**dict(ref, warps=1, iters=20)))[3]["residual"] for im in ims]
            tol = float(np.median(res)) * 1.001
        kw["tol"] = ref["tol"] = tol
        us, vs, st = flow.of_solve_batch(ctx, [i[0] for i in ims], [i[1] for i in ims],
                                         flow.default_params(engine=flow.OF_ENGINE_STREAM, **kw))
        counts = set()
        for k, im in enumerate(ims):
            u, v, _, s = flow.of_solve(ctx, *im, flow.default_params(**ref))
            assert s["iters_run"] == st[k]["iters_run"], BATCH[k]
            assert torch.equal(u, us[k]) and torch.equal(v, vs[k]), BATCH[k]
            counts.add(s["iters_run"])
        assert len(counts) == (1 if tol == 0.0 else len(counts)) and (tol == 0.0 or len(counts) > 1)


# The stopping test's launches, 5 and 5 or 3, 3, 3 and 1 per ten iterations, with remainders of one to nine iterations.
@pytest.mark.parametrize("H,W", [(120, 160), (80, 107), (150, 201), (3, 4000), (4000, 2), (240, 320), (375, 1242)])
@pytest.mark.parametrize("method,pinned", [(flow.OF_PADMM_I, 8), (flow.OF_PADMM_II, 8), (flow.OF_CP, 8)])
@pytest.mark.parametrize("prec", [0, 2])
def test_single_pairs_with_the_stopping_test(ctx, H, W, method, pinned, prec):
    im = images(H, W) if min(H, W) > 8 else [cu(a) for a in np.random.default_rng(H).random((2, H, W))]
    kw = dict(method=method, lam=3.0, levels=1, precision=prec, fp32_last_warp=0)
    ref = dict(kw, engine=flow.OF_ENGINE_STREAM, rows_per_warp=pinned)
    met = flow.of_solve(ctx, *im, flow.default_params(warps=1, iters=20, **ref))[3]["residual"] * 1.001
    for iters in (20, 21, 25, 39):
        for tol in (met, 1e-30):
            a = flow.of_solve(ctx, *im, flow.default_params(warps=2, iters=iters, tol=tol, **ref), want_w=True)
            b = flow.of_solve(ctx, *im, flow.default_params(warps=2, iters=iters, tol=tol, **kw), want_w=True)
            assert all(torch.equal(x, y) for x, y in zip(a[:3], b[:3])), (iters, tol)
            assert a[3]["iters_run"] == b[3]["iters_run"]
            assert a[3]["residual"] == pytest.approx(b[3]["residual"], rel=1e-5)


# pDR's register tiles and one-iteration tiles on either side of the rule that chooses: strips, odd widths near its
# smallest level, with and without the stopping test.
@pytest.mark.parametrize("H,W", [(2, 20000), (3, 32768), (8, 5000), (5000, 8), (4000, 11), (200, 201), (240, 320)])
@pytest.mark.parametrize("tol", [0.0, 1e-30])
def test_pdr_on_either_tile_kernel(ctx, H, W, tol):
    im = images(H, W) if min(H, W) > 8 else [cu(a) for a in np.random.default_rng(H).random((2, H, W))]
    P = flow.default_params(method=flow.OF_PDR, lam=3.0, levels=1, warps=2, iters=23, tol=tol, engine=flow.OF_ENGINE_STREAM)
    u, v, _, st = flow.of_solve(ctx, *im, P)
    ub, vb, sb = flow.of_solve_batch(ctx, [im[0]] * 2, [im[1]] * 2, P)  # one iteration per launch
    assert torch.equal(u, ub[0]) and torch.equal(v, vb[0])
    assert st["iters_run"] == sb[0]["iters_run"]


# Pyramid steps that keep nearly all of the pixels: three kernels take the larger image and one the smaller, its upper
# rows, with the same sampling positions in both.
@pytest.mark.parametrize("eta", [0.95, 0.9])
def test_pyramid_steps_that_keep_most_pixels(eta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    big = torch.rand(1400, 1900, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    a = flow.of_pyr_down(big, round(1400 * eta), round(1900 * eta), eta)
    b = flow.of_pyr_down(big[:1300], round(1300 * eta), round(1900 * eta), eta)
    assert torch.equal(a[:1100], b[:1100])
