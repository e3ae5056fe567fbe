"""The record deposit (packets' segments as records, sorted by tally row, summed in registers) against the
direct deposit: bit-identical coefficients and equal run counters at the edges of its tiles, passes and
launches -- orders per register pass, rows per tile, one and two sorting passes, buffers that pause a
launch and buffers so small that the closing direct launch finishes the packets, batches and graphs."""
import numpy as np
import pytest
import torch

from paper_1608_05238_gb300 import _build, batch, mcr
from parity_util import f32

pytestmark = pytest.mark.gpu

DIRECT, RECORDS = (0, 0, 1, 0, 1, 1, 0), (0, 0, 0, 0, 0, 2, 0)
COUNTERS = ("launched", "flights", "collisions", "segments", "escapes", "rr_kill", "rr_survive", "scatter_limit",
            "event_limit")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    mcr.load()


def _medium(nz, nx, dx, seed):
    r = np.random.default_rng(seed)
    mua = torch.from_numpy((0.01 + 0.1 * r.random((nz, nx))).astype(np.float32)).cuda()
    mus = torch.from_numpy((5.0 + 10.0 * r.random((nz, nx))).astype(np.float32)).cuda()
    return mcr.Medium(mua, mus, f32(dx), f32(0.9))


def _line(nx, dx):
    return mcr.Source(mcr.LINE, x0=0.0, z0=0.0, x1=f32(nx * dx), z1=0.0, dir_x=0.2, dir_z=1.0)


def _compare(problems, common, records=RECORDS):
    ref, st_ref = mcr.run_batch(problems, common, launch=DIRECT, stats=True)
    ref = [x.clone() for x in ref]
    got, st = mcr.run_batch(problems, common, launch=records, stats=True)
    assert all(torch.equal(a, b) for a, b in zip(ref, got))
    assert [st[k] for k in COUNTERS] == [st_ref[k] for k in COUNTERS]
    for k in ("launched_w", "escaped_w", "rr_net_w", "killed_w"):
        assert abs(st[k] - st_ref[k]) <= 1e-9 * max(1.0, st_ref["launched"])
    mcr.check()


@pytest.mark.parametrize("K", [0, 1, 4, 5, 8, 9, 12, 13, 16, 17, 24, 25, 32, 33, 47, 49, 64])
def test_every_order_split(K):
    med = _medium(40, 56, 0.08, K)
    _compare([mcr.Problem(med, 20_000, seed=K, source=_line(56, 0.08))], mcr.Run(K=K, n_packets=0))


@pytest.mark.parametrize("nz,nx", [(1, 31), (1, 32), (3, 11), (1, 300), (256, 257), (700, 601)])
def test_tile_edges_and_sorting_passes(nz, nx):
    """Fewer rows than a tile, exactly one, a ragged last tile; 2056 tiles (a second sorting pass, 65,792
    rows) and 420,700 rows (tiles of more than 32 rows)."""
    med = _medium(nz, nx, 0.1, nx)
    _compare([mcr.Problem(med, 3_000, seed=2, source=_line(nx, 0.1))], mcr.Run(K=7, n_packets=0))


@pytest.mark.parametrize("capacity", [1, 4_000, 3_000_000])
def test_launches_that_pause(capacity):
    """One block of slots (the closing direct launch does nearly everything), a few blocks, and several
    full launches; an adjoint source with roulette."""
    q = torch.from_numpy(np.random.default_rng(1).normal(size=(40, 56)).astype(np.float32)).cuda()
    med = _medium(40, 56, 0.08, 3)
    n = 300 if capacity < 100 else 40_000
    _compare([mcr.Problem(med, n, seed=5, stream_id=1, qstar=q)],
             mcr.Run(K=16, n_packets=0, w_threshold=0.05, roulette_p=0.3), (0, 0, 0, 0, 0, 2, capacity))


@pytest.mark.parametrize("limits", [dict(max_scatter=3), dict(max_events=5)])
def test_caps_end_the_same_packets(limits):
    med = _medium(24, 24, 0.2, 6)
    run = mcr.Run(K=6, n_packets=0, **limits)
    problems = [mcr.Problem(med, 5_000, seed=7, source=_line(24, 0.2))]
    out = []
    for launch in (DIRECT, RECORDS):
        out.append(mcr.run_batch(problems, run, launch=launch)[0].clone())
        try:
            mcr.check()
        except mcr.McrError:  # the event cap is reported, by either
            assert "max_events" in limits
    assert torch.equal(*out)


def test_ragged_batch_and_graph_replay():
    problems = [mcr.Problem(_medium(30 + 7 * i, 50 - 3 * i, 0.1, i), 4_000 + 137 * i, seed=i, stream_id=i,
                            source=mcr.Source(mcr.ISO_POINT, x0=1.0, z0=1.0)) for i in range(7)]
    common = mcr.Run(K=12, n_packets=0)
    _compare(problems, common)
    ref = [x.clone() for x in mcr.run_batch(problems, common, launch=DIRECT)]
    runner = batch.BatchRunner(problems, common)
    runner.capture()
    for p in problems:
        p.out.zero_()
    assert all(torch.equal(a, b) for a, b in zip(ref, runner.replay()))
