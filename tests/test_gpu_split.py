"""GPU: applies whose terms are split over several CTAs (few right-hand sides).

1D, N <= 8192: cluster sizes 1 to 8 by batch and m, with remainders (terms that do not
divide into rounds, odd m, one term), batches on both sides of each size's last one,
both directions and both storage precisions, against the FP64 oracle.

Bar: an FFT of n points in FP32 has a relative l2 error of at most about
eps log2 n (eps = 6e-8); a forward and an inverse one with the products between them,
n <= 8192, stay below 30 eps = 2e-6.  Reduced storage: the project's bar of 3e-3.
"""
import numpy as np
import pytest

import synth
from oracle import direct as O

pytestmark = pytest.mark.gpu

TOL = 2e-6
TOL_LOWP = 3e-3


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    from paper_1604_04374_gb300 import build
    build.build()
    O.build()
    torch.cuda.init()
    return torch


def dev(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel(got, ref):
    got = got.detach().cpu().numpy().astype(np.float64).reshape(ref.shape[0], -1)
    ref = ref.reshape(ref.shape[0], -1)
    return float(np.max(np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)))


def problem_1d(n, m, batch):
    rng = np.random.default_rng(1000 * n + 10 * m + batch)
    w = synth.hat_windows_1d(n, m) if m >= 2 else np.ones((1, n), np.float32)
    h = np.zeros((m, n), np.float32)
    offs = np.unique(np.arange(-6, 7) % n)
    h[:, offs] = rng.standard_normal((m, offs.size)).astype(np.float32)
    return w, h, rng.standard_normal((batch, n)).astype(np.float32)


@pytest.mark.parametrize("n", [16, 64, 256, 512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("m,batch", [(1, 1), (2, 3), (5, 1), (9, 38), (17, 19), (33, 1), (32, 20), (6, 77)])
def test_1d_clusters(torch_cuda, n, m, batch):
    torch = torch_cuda
    from paper_1604_04374_gb300 import Plan, pce
    w, h, u = problem_1d(n, m, batch)
    yr, xr = O.apply(u, w, h), O.apply_adjoint(u, w, h)
    for flags, tol in ((0, TOL), (pce.PCE_FLAG_LOWP_STORAGE, TOL_LOWP)):
        plan = Plan(dev(torch, w), h=dev(torch, h), flags=flags)
        assert rel(plan.apply(dev(torch, u)), yr) <= tol
        assert rel(plan.apply_adjoint(dev(torch, u)), xr) <= tol
        plan.close()


def problem_2d(ny, nx, gy, gx, batch, zero=()):
    rng = np.random.default_rng(ny + 7 * nx + 100 * gy + 1000 * gx + batch)
    wy, wx = synth.hat_factors_2d(ny, nx, gy, gx)
    for k in zero:
        wy[k] = 0.0
    h = np.zeros((gy * gx, ny, nx), np.float32)
    offs = np.arange(-2, 3)
    h[:, (offs % ny)[:, None], (offs % nx)[None, :]] = rng.standard_normal((gy * gx, 5, 5)).astype(np.float32)
    return wy, wx, h, rng.standard_normal((batch, ny, nx)).astype(np.float32)


@pytest.mark.parametrize("ny,nx", [(16, 32), (64, 64), (256, 128), (512, 64), (1024, 32), (2048, 32)])
@pytest.mark.parametrize("gy,gx,batch,zero", [(1, 1, 1, ()), (3, 3, 1, ()), (4, 4, 3, (0, 1, 2, 15)),
                                              (5, 1, 2, ()), (3, 5, 1, (14, 13))])
def test_2d_column_splits(torch_cuda, ny, nx, gy, gx, batch, zero):
    """The terms (or slots) of a column tile over CTAs: dense and separable plans, the column variants that split, empty windows in a CTA's share, the
    product form and reduced storage."""
    torch = torch_cuda
    from paper_1604_04374_gb300 import Plan, pce
    wy, wx, h, u = problem_2d(ny, nx, gy, gx, batch, zero)
    w = (wy[:, :, None] * wx[:, None, :]).astype(np.float32)
    yr, xr = O.apply(u, w, h), O.apply_adjoint(u, w, h)
    ud, hd = dev(torch, u), dev(torch, h)

    def check(plan, tol):
        assert rel(plan.apply(ud), yr) <= tol
        assert rel(plan.apply_adjoint(ud), xr) <= tol

    plan = Plan(dev(torch, w), h=hd)
    check(plan, TOL)
    if ny >= 512:
        plan.set_tuning(0, 1, 0)   # block Stockham columns
        check(plan, TOL)
    check(Plan(dev(torch, w), h=hd, flags=pce.PCE_FLAG_LOWP_STORAGE), TOL_LOWP)
    p = Plan(dev(torch, w), h=hd, flags=pce.PCE_FLAG_PRODUCT_CONVOLUTION)
    # P_m = sum_k w_k . (h_k * u): the adjoint operator's structure with h reversed
    hr = np.ascontiguousarray(np.roll(h[:, ::-1, ::-1], (1, 1), (1, 2)))
    assert rel(p.apply(ud), O.apply_adjoint(u, w, hr)) <= TOL
    sep = Plan(wy=dev(torch, wy), wx=dev(torch, wx), h=hd)
    check(sep, TOL)
    for cv in {512: (0, 2), 1024: (0, 2)}.get(ny, ()):
        sep.set_tuning(0, cv, 2)
        check(sep, TOL)


@pytest.mark.parametrize("ny,nx,gy,gx,zero", [(16, 32, 3, 3, ()), (64, 128, 1, 2, ()), (128, 64, 5, 1, (0, 3)),
                                              (256, 256, 4, 4, (0, 1, 15)), (512, 128, 3, 3, ()), (1024, 64, 1, 3, ()),
                                              (1024, 128, 5, 1, (2,))])
def test_2d_forward_splits_keep_the_bits(torch_cuda, ny, nx, gy, gx, zero):
    """A right-hand side alone (terms over a cluster) equals the same one in a batch
    (fewer or no CTAs a tile) bit for bit: dense plans, both storages, and separable ones."""
    torch = torch_cuda
    from paper_1604_04374_gb300 import Plan, pce
    wy, wx, h, u = problem_2d(ny, nx, gy, gx, 40, zero)
    w = (wy[:, :, None] * wx[:, None, :]).astype(np.float32)
    ud, hd = dev(torch, u), dev(torch, h)
    plans = [Plan(dev(torch, w), h=hd), Plan(dev(torch, w), h=hd, flags=pce.PCE_FLAG_LOWP_STORAGE),
             Plan(wy=dev(torch, wy), wx=dev(torch, wx), h=hd)]
    for plan in plans:
        y = plan.apply(ud)
        for b in (0, 17, 39):
            assert torch.equal(plan.apply(ud[b:b + 1].contiguous())[0], y[b])


def forward_split(ny, nx, nb, units, sep):
    """CTAs that share a column tile's terms in a forward launch of nb right-hand sides."""
    cols = 4 if sep or ny >= 256 else 128 // (ny // 8)
    ctas = nb * -(-(nx // 2) // cols)
    if sep:
        return 4 if units >= 4 and ctas * 4 <= 152 * (6 if ny == 512 else 4) else 1
    if units >= 8 and (ny < 256 or units >= 5 * -(-units // 8)) and ctas * 8 <= 152 * 4:
        return 8
    if units >= {256: 28, 64: 40}.get(ny, 8) and units >= 3 * -(-units // 4) and ctas * 4 <= 152 * 4:
        return 4
    return 1


@pytest.mark.parametrize("ny,nx,gy,gx,zero", [(16, 512, 2, 4, ()), (32, 256, 3, 4, (9,)), (64, 128, 8, 5, (0, 1)),
                                              (128, 64, 5, 4, (4,)), (256, 32, 4, 8, ()), (512, 64, 3, 3, (0,)),
                                              (1024, 64, 2, 3, ())])
def test_2d_forward_split_and_unsplit_launches_agree(torch_cuda, ny, nx, gy, gx, zero):
    """Launches of 64, 30 and 1 right-hand sides, which take one, four and eight CTAs a tile
    (separable columns one and four), give the same bits."""
    torch = torch_cuda
    from paper_1604_04374_gb300 import Plan, pce
    wy, wx, h, u = problem_2d(ny, nx, gy, gx, 64, zero)
    w = (wy[:, :, None] * wx[:, None, :]).astype(np.float32)
    ud, hd = dev(torch, u), dev(torch, h)
    sep = ny >= 512
    few = (1,) if sep else (30, 1)
    terms = gy * gx - (len(zero) if sep else 0)
    assert [forward_split(ny, nx, nb, terms, sep) for nb in (64, *few)] == ([1, 4] if sep else [1, 4, 8])
    plans = ([Plan(wy=dev(torch, wy), wx=dev(torch, wx), h=hd)] if sep else
             [Plan(dev(torch, w), h=hd), Plan(dev(torch, w), h=hd, flags=pce.PCE_FLAG_LOWP_STORAGE)])
    for plan in plans:
        assert plan.info()[2] >= 64 * ny * nx * 4   # scratch for all 64 at once
        y = plan.apply(ud)
        for nb in few:
            for b in (0, 64 - nb):
                assert torch.equal(plan.apply(ud[b:b + nb].contiguous()), y[b:b + nb])
        plan.close()


TOL_LONG = 2.2e-6


@pytest.mark.parametrize("n,batch", [(16384, 38), (65536, 10), (262144, 3)])
@pytest.mark.parametrize("m", [1, 5, 16])
def test_long_1d_splits_keep_the_bits(torch_cuda, n, m, batch):
    """N > 8192: a right-hand side alone (one row pair a CTA, the adjoint's term pairs over
    CTAs) equals the same one in the smallest batch of packed CTAs bit for bit, and the
    FFT convolution in FP64 (bar: 18 stages each way of eps = 6e-8, 2.2e-6)."""
    torch = torch_cuda
    from paper_1604_04374_gb300 import Plan
    w, h, u = problem_1d(n, m, batch)
    wd, hd, ud = dev(torch, w), dev(torch, h), dev(torch, u)
    plan = Plan(wd, h=hd)
    y, x = plan.apply(ud), plan.apply_adjoint(ud)
    hh = torch.fft.rfft(hd.double())
    yr = torch.fft.irfft((torch.fft.rfft(wd.double() * ud[-1].double()) * hh).sum(0), n=n)
    xr = (wd.double() * torch.fft.irfft(torch.fft.rfft(ud[-1].double()) * hh.conj(), n=n)).sum(0)
    assert rel(y[-1:], host(yr)) <= TOL_LONG and rel(x[-1:], host(xr)) <= TOL_LONG
    for b in (0, batch - 1):
        assert torch.equal(plan.apply(ud[b:b + 1].contiguous())[0], y[b])
        assert torch.equal(plan.apply_adjoint(ud[b:b + 1].contiguous())[0], x[b])


def host(t):
    return t.detach().cpu().numpy()[None]


@pytest.mark.parametrize("n,ms", [(16, (257, 600)), (32, (129, 300)), (64, (65, 300)), (128, (33, 70)),
                                  (256, (17, 40, 131)), (512, (17, 40, 131)), (1024, (9, 20, 67)), (2048, (9, 17, 67)),
                                  (4096, (5, 11, 40)), (8192, (3, 7, 32))])
def test_1d_results_do_not_depend_on_the_batch(torch_cuda, n, ms):
    """N <= 8192: a right-hand side alone, in clusters of eight, four and two and in CTAs of
    its own gives the same bits, both directions, both storages; for the lengths whose
    CTAs do not change with the batch also beyond 304 right-hand sides."""
    torch = torch_cuda
    from paper_1604_04374_gb300 import Plan, pce
    full = 310 if n <= 256 or n == 8192 else 80
    for m in ms:
        w, h, u = problem_1d(n, m, full)
        ud = dev(torch, u)
        for flags in (0, pce.PCE_FLAG_LOWP_STORAGE):
            plan = Plan(dev(torch, w), h=dev(torch, h), flags=flags)
            for apply in (plan.apply, plan.apply_adjoint):
                ref = apply(ud)
                for nb in (1, 3, 20, 39, 80):
                    assert torch.equal(apply(ud[:nb].contiguous()), ref[:nb]), (m, flags, apply.__name__, nb)
                assert torch.equal(apply(ud[79:80].contiguous())[0], ref[79])
            plan.close()
