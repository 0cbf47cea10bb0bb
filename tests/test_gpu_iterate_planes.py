"""The step-level iterations leave the planes alone that their method does not use, also where the caller passes
them: w, p1, p2 and wb without beta, the barred planes of the ADMM methods, s of pDR and ALG1."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_10979_gb300 import flow  # noqa: E402

PLANES = ("w", "u", "v", "p1", "p2", "q11", "q12", "q21", "q22", "s", "wb", "ub", "vb")


@pytest.mark.parametrize("method,entry", [(flow.OF_PADMM_I, "of_admm_iterate"), (flow.OF_PADMM_II, "of_admm_iterate"),
                                          (flow.OF_CP, "of_cp_iterate"), (flow.OF_PDR, "of_pdr_iterate")])
@pytest.mark.parametrize("beta", [0.0, 0.05])
@pytest.mark.parametrize("iters", [1, 2, 3, 7, 8])
def test_unused_planes_are_left_alone(method, entry, beta, iters):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    H, W = 70, 131
    g = torch.Generator(device="cuda").manual_seed(iters)
    planes = {n: 0.1 * torch.randn(H, W, device="cuda", generator=g) for n in PLANES}
    Ix, Iy, It = (0.2 * torch.randn(H, W, device="cuda", generator=g) for _ in range(3))
    old = {n: t.clone() for n, t in planes.items()}
    nbytes = flow.lib().of_fields_bytes(H, W)
    scratch = torch.full((nbytes // 4 + 1,), float("nan"), device="cuda")
    P = flow.default_params(method=method, beta=beta, lam=2.0)
    at = (ctypes.c_float(0.5),) if entry == "of_admm_iterate" else ()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    flow.check(getattr(flow.lib(), entry)(flow._fields(planes), ptr(Ix), ptr(Iy), ptr(It), H, W, W, *at, ctypes.byref(P),
                                          iters, ptr(scratch), None, flow._stream(None)))
    torch.cuda.synchronize()
    admm = entry == "of_admm_iterate"
    unused = (() if beta else ("w", "p1", "p2", "wb")) + (("wb", "ub", "vb") if admm else ("s",))
    for n in PLANES:
        assert torch.isfinite(planes[n]).all(), n
        if n in unused:
            assert torch.equal(planes[n], old[n]), n
        elif n in ("u", "v", "q11", "q22"):
            assert not torch.equal(planes[n], old[n]), n


# Sizes and counts on either side of the rule that chooses between the tile kernel and the row-streaming one.
@pytest.mark.parametrize("H,W", [(1, 1), (48, 64), (2, 9000), (3, 30000), (241, 323), (700, 900)])
@pytest.mark.parametrize("kw", [dict(), dict(method=flow.OF_PADMM_II, rho=1.8), dict(beta=0.0), dict(a_tilde_mode=1)],
                         ids=["I", "II", "beta0", "per-pixel"])
def test_admm_iterations_in_one_call_equal_single_ones(H, W, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = torch.Generator(device="cuda").manual_seed(H + W)
    Ix, Iy, It = (0.2 * torch.randn(H, W, device="cuda", generator=g) for _ in range(3))
    start = {n: torch.zeros(H, W, device="cuda") for n in PLANES[:10]}
    P = flow.default_params(lam=2.0, **kw)
    single = {n: t.clone() for n, t in start.items()}
    done = 0
    for iters in (2, 3, 5, 14):
        while done < iters:
            r1 = flow.of_admm_iterate(single, Ix, Iy, It, 0.5, P, 1)
            done += 1
        many = {n: t.clone() for n, t in start.items()}
        r = flow.of_admm_iterate(many, Ix, Iy, It, 0.5, P, iters)
        assert all(torch.equal(many[n], single[n]) for n in start), iters
        assert r == pytest.approx(r1, rel=1e-5)
        tested = {n: t.clone() for n, t in start.items()}
        flow.of_admm_iterate(tested, Ix, Iy, It, 0.5, flow.default_params(lam=2.0, tol=1e-30, **kw), iters)
        assert all(torch.equal(tested[n], single[n]) for n in start), iters
