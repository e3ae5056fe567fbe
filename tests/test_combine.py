"""The per-pixel FP64 steps against the same formulas in torch float64 on the CPU: the gradient combine at
every remainder of its four-order groups and with zeros, subnormals, infinities and NaN among the
coefficients (which leave its fast widening), the adjoint source's quotient, and eps over few and many
partial sums."""
import math

import pytest
import torch

from paper_1608_05238_gb300 import _build, mcr
from parity_util import f32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    mcr.load()


def _med(nz, nx, seed):
    g = torch.Generator().manual_seed(seed)
    mua = 0.01 + 0.1 * torch.rand(nz, nx, generator=g)
    return mcr.Medium(mua.cuda(), torch.full((nz, nx), 10.0).cuda(), f32(0.03), f32(0.9))


@pytest.mark.parametrize("K", [0, 1, 3, 4, 5, 7, 8, 9, 64])
@pytest.mark.parametrize("special", [False, True])
def test_gradient_orders_and_special_values(K, special):
    nz, nx, C = 9, 37, 2 * K + 1
    g = torch.Generator().manual_seed(K)
    med = _med(nz, nx, K)
    c, a = (torch.randn(C, nz, nx, generator=g) for _ in range(2))
    v = 1e-3 * torch.randn(nz, nx, generator=g)
    if special:
        for t in (c, a):
            flat = t.view(-1)
            at = torch.randperm(flat.numel(), generator=g)[:flat.numel() // 3]
            flat[at] = torch.tensor([0.0, -0.0, 1e-42, -3e-45, 1e38, 2e-38])[torch.arange(len(at)) % 6]
        c[-1, 0, 0], a[-1, 0, 1], c[0, 0, 2] = math.inf, math.nan, -math.inf
    d_mua, d_mus = mcr.gradient(med, c.cuda(), a.cuda(), v.cuda())
    C64, A64, area, gg = c.double(), a.double(), med.dx * med.dx, med.g
    pr = C64[1:] * A64[1:]
    w = (1.0 - gg ** torch.arange(1, K + 1, dtype=torch.float64)).repeat_interleave(2).reshape(-1, 1, 1)
    ref_a = v.double() * C64[0] + area * (C64[0] * A64[0] / (2 * math.pi) + pr.sum(0) / math.pi)
    ref_s = area * (w * pr).sum(0) / math.pi
    # FP64: each of the 2K+2 terms and additions rounds to 2^-53 of the sum of magnitudes
    size = area * ((C64 * A64).abs().sum(0) + 1e-300) + (v.double() * C64[0]).abs()
    for got, ref in ((d_mua.cpu(), ref_a), (d_mus.cpu(), ref_s)):
        fine = torch.isfinite(ref)
        assert torch.equal(fine, torch.isfinite(got)) and torch.equal(torch.isnan(ref), torch.isnan(got))
        fine &= torch.isfinite(size)  # (at K = 0 d_mus is 0 where a_0 is not finite)
        assert ((got - ref).abs()[fine] <= (2 * K + 8) * 2.0 ** -52 * size[fine]).all()


@pytest.mark.parametrize("nz,nx", [(1, 1), (7, 33), (300, 1000)])
def test_adjoint_source_and_eps(nz, nx):
    g = torch.Generator().manual_seed(nx)
    med = _med(nz, nx, nx)
    v = torch.randn(nz, nx, generator=g)
    v.view(-1)[::5] = 0.0
    area = med.dx * med.dx
    ref = (-(med.mua.cpu().double()) * v.double() / area).float()
    assert torch.equal(mcr.adjoint_source(med, v.cuda()).cpu(), ref)
    a0 = torch.rand(1, nz, nx, generator=g)
    hm = torch.rand(nz, nx, generator=g)
    H, dv, eps = mcr.h_eps(med, a0.cuda(), hm.cuda())
    r2 = ((hm.double() - H.cpu().double()) ** 2).sum()
    assert abs(eps.item() - 0.5 * area * r2.item()) <= 1e-13 * 0.5 * area * r2.item() + 1e-300
