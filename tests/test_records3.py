"""The 3D record deposit at the edges of its tiles, orders and launches: disjoint packet ranges add up to
the whole run at every order L (the sums are integers; the FP32 outputs round them once), on grids of less
than a tile, ragged tiles and two sorting passes, and for packets so long-lived that the record launches
end before they do and the closing direct launch takes them over."""
import numpy as np
import pytest
import torch

from paper_1608_05238_gb300 import _build, mcr, mcr3
from parity_util import f32

pytestmark = pytest.mark.gpu

COUNTERS = ("launched", "flights", "collisions", "segments", "escapes", "rr_kill", "rr_survive")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    mcr.load()


def _ranges_add_up(med, src, K, cuts, **kw):
    """Runs [0, cuts[-1]) whole and in the given ranges; 2^-22 relative: two FP32 roundings a range."""
    n = cuts[-1]
    whole, st = mcr3.forward(med, src, mcr.Run(K=K, n_packets=n, seed=3, **kw), stats=True)
    acc = torch.zeros_like(whole, dtype=torch.float64)
    total = dict.fromkeys(COUNTERS, 0)
    for a, b in zip([0] + cuts[:-1], cuts):
        part, sp = mcr3.forward(med, src, mcr.Run(K=K, n_packets=b - a, first_packet=a, seed=3, **kw), stats=True)
        acc += part.double() * (b - a)
        for k in COUNTERS:
            total[k] += sp[k]
    ref = whole.double() * n
    assert total == {k: st[k] for k in COUNTERS}
    per_voxel = ref[0].abs() * 4.0 * np.sqrt(2 * K + 1)  # every |Y_lm| <= sqrt((2l+1)/4 pi)
    assert ((acc - ref).abs() <= 2.0 ** -22 * len(cuts) * (per_voxel + 1e-30)).all()
    return st


@pytest.mark.parametrize("L", range(9))
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 4, 8), (5, 7, 11), (41, 40, 43)])
def test_ranges_add_up_at_every_order(L, shape):
    r = np.random.default_rng(L)
    med = mcr3.Medium3(torch.from_numpy((0.01 + 0.1 * r.random(shape)).astype(np.float32)).cuda(),
                       torch.from_numpy((5 + 10 * r.random(shape)).astype(np.float32)).cuda(), f32(0.1), f32(0.9))
    src = mcr3.Source3(mcr.ISO_POINT, x0=f32(0.05 * shape[2]), y0=f32(0.05 * shape[1]), z0=f32(0.05 * shape[0]))
    _ranges_add_up(med, src, L, [1_000, 1_001, 6_000], w_threshold=0.01, roulette_p=0.2)


def test_packets_that_outlast_the_record_launches():
    """Isotropic scattering with a mean free path of 1/150 mm in a 16 mm cube: some 7e5 segments a packet,
    beyond the 4,096 a packet that record launches are enqueued for."""
    shape = (16, 16, 16)
    med = mcr3.Medium3(torch.zeros(shape, device="cuda"), torch.full(shape, 150.0, device="cuda"), 1.0, 0.0)
    st = _ranges_add_up(med, mcr3.Source3(mcr.ISO_POINT, x0=8.3, y0=8.2, z0=8.1), 4, [25, 50, 75, 100])
    assert st["segments"] > 40_000_000 and st["escapes"] == 100
