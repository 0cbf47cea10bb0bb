"""The quotients of the ALG1 and pDR register kernels on images with regions without data: beside textured pixels the
flow and the illumination decay through every magnitude to zero, pixels without any gradient have no divisor, and
clipped images mix both in every warp.  Against the kernels that divide, for equality."""
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


def images(H, W, kind):
    p = synth.random_affine_rect_pair(H, W, 5)
    I = np.stack([p.I0, p.I1]).astype(np.float32)
    y, x = np.mgrid[:H, :W]
    if kind == "box":  # texture on an empty background
        I *= (abs(x - W / 2) < W / 12) & (abs(y - H / 2) < H / 12)
    elif kind == "half":
        I[:, :, W // 2:] = 1.0
    elif kind == "clipped":
        I = np.clip(4.0 * (I - I.mean()) + 0.5, 0.0, 1.0)
    elif kind == "faint":  # quotients that are subnormal from the first iteration
        I *= np.float32(1e-36)
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in I]


@pytest.mark.parametrize("kind", ["box", "half", "clipped", "faint"])
@pytest.mark.parametrize("beta", [0.05, 0.0])
@pytest.mark.parametrize("H,W", [(260, 350), (203, 301)])
def test_alg1(ctx, kind, beta, H, W):
    im = images(H, W, kind)
    kw = dict(method=flow.OF_CP, lam=3.0, beta=beta, levels=1, warps=2, iters=70, engine=flow.OF_ENGINE_STREAM)
    a = flow.of_solve(ctx, *im, flow.default_params(rows_per_warp=8, **kw), want_w=True)
    b = flow.of_solve(ctx, *im, flow.default_params(**kw), want_w=True)
    assert all(torch.equal(x, y) for x, y in zip(a[:3], b[:3]))


@pytest.mark.parametrize("kind", ["box", "half", "clipped", "faint"])
@pytest.mark.parametrize("beta", [0.05, 0.0])
@pytest.mark.parametrize("H,W", [(260, 350), (203, 301)])
@pytest.mark.parametrize("prec", [0, 2])
def test_pdr(ctx, kind, beta, H, W, prec):
    im = images(H, W, kind)
    P = flow.default_params(method=flow.OF_PDR, lam=3.0, beta=beta, levels=1, warps=2, iters=70, precision=prec,
                            engine=flow.OF_ENGINE_STREAM)
    u, v, _, _ = flow.of_solve(ctx, *im, P)
    ub, vb, _ = flow.of_solve_batch(ctx, [im[0]] * 2, [im[1]] * 2, P)  # k_pdr_tile
    assert torch.equal(u, ub[0]) and torch.equal(v, vb[0])
