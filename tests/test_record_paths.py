"""Paths of the record deposit that short runs do not reach: many work units of one tally row, two sorting
passes, small launch shapes, full buffers -- each against the direct deposit, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1608_05238_gb300 import _build, batch, mcr, mcr3
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


def _same(problems, common, records=RECORDS):
    ref, st_ref = mcr.run_batch(problems, common, launch=DIRECT, stats=True)
    ref = [x.clone() for x in ref]
    got, st = mcr.run_batch(problems, common, launch=records, stats=True)
    assert all(torch.equal(a, b) for a, b in zip(ref, got))
    assert [st[k] for k in COUNTERS] == [st_ref[k] for k in COUNTERS]
    mcr.check()


@pytest.mark.parametrize("nz,nx", [(1, 1), (1, 2), (2, 33)])
@pytest.mark.parametrize("K", [4, 64])
def test_many_units_of_few_rows(nz, nx, K):
    """Every unit of the deposit holds records of one or a few rows: runs of the greatest length only, as
    many units as the run has batches, each of which lists its runs anew."""
    med = _medium(nz, nx, 2.0, K)
    _same([mcr.Problem(med, 100_000, seed=K, source=mcr.Source(mcr.ISO_POINT, x0=1.0, z0=1.0))],
          mcr.Run(K=K, n_packets=0))


@pytest.mark.parametrize("nz,nx", [(256, 512), (1, 131_073), (363, 362), (700, 601)])
def test_both_sides_of_the_second_sorting_pass(nz, nx):
    """131,072 rows are 2,048 tiles of 64, one pass; one row more takes the second pass (and its count)."""
    med = _medium(nz, nx, 0.05, nx)
    src = mcr.Source(mcr.LINE, x0=0.0, z0=0.0, x1=f32(nx * 0.05), z1=0.0, dir_x=0.2, dir_z=1.0)
    _same([mcr.Problem(med, 40_000, seed=2, source=src)], mcr.Run(K=7, n_packets=0))
    assert mcr.record_passes() == (1 if nz * nx <= 131_072 else 2)


@pytest.mark.parametrize("launch", [None, DIRECT])
def test_a_graph_outlives_larger_calls(launch):
    """Later calls with more packets, and then with a larger grid and order, grow every buffer of the workspace;
    the graph goes on with its own."""
    mcr.release_workspace()
    problems = [mcr.Problem(_medium(64, 64, 0.1, i), 10_000, seed=i, stream_id=i,
                            source=mcr.Source(mcr.ISO_POINT, x0=3.0, z0=3.0)) for i in range(3)]
    q = torch.from_numpy(np.random.default_rng(4).normal(size=(64, 64)).astype(np.float32)).cuda()
    problems.append(mcr.Problem(_medium(64, 64, 0.1, 9), 10_000, seed=9, stream_id=1, qstar=q))
    common = mcr.Run(K=16, n_packets=0)
    ref = [x.clone() for x in mcr.run_batch(problems, common, launch=DIRECT)]
    runner = batch.BatchRunner(problems, common, launch=launch)
    runner.capture()
    for n, K, packets in ((64, 16, 1_000_000), (300, 33, 2_000_000), (64, 16, 1_000)):
        med = _medium(n, n, 0.05, n)
        big = torch.ones(n, n, device="cuda")
        a = mcr.adjoint(med, big, mcr.Run(K=K, n_packets=packets, seed=2))
        for p in problems:
            p.out.zero_()
        assert all(torch.equal(x, y) for x, y in zip(ref, runner.replay()))
        assert torch.equal(a, mcr.adjoint(med, big, mcr.Run(K=K, n_packets=packets, seed=2)))
    mcr.check()
    torch.cuda.synchronize()
    mcr.release_workspace()


@pytest.mark.parametrize("threads,blocks", [(32, 1), (64, 1), (32, 2), (96, 1), (256, 1)])
def test_small_launch_shapes_run_by_records(threads, blocks):
    """Shapes with fewer lanes than the tail takes packets: the record launches go through the packets all the
    same, a few at a time, and leave none to the closing launch."""
    med = _medium(64, 80, 0.1, threads)
    src = mcr.Source(mcr.LINE, x0=0.0, z0=0.0, x1=8.0, z1=0.0, dir_x=0.1, dir_z=1.0)
    _same([mcr.Problem(med, 60_000, seed=3, source=src)], mcr.Run(K=8, n_packets=0), (threads, blocks, 0, 0, 0, 2, 0))
    kernels, closing = mcr.record_info()
    assert kernels > 0 and closing == 0
    mcr.run_batch([mcr.Problem(med, 100, seed=3, source=src)], mcr.Run(K=8, n_packets=0), DIRECT)
    assert mcr.record_info() == (0, -1)


@pytest.mark.parametrize("mua", [0.2, 0.22, 0.41])
def test_weight_counters_are_summed_in_64_bits(mua):
    """2^26 packets of equal weight through one absorbing pixel, few lanes: some 13,800 additions to a lane's sum.
    FP64 sums of them err by at most 2^-53 of the whole per addition of the longest chain: a lane's additions (at
    most four times the mean), the warps' sums and their 152 atomic additions in each of two launches."""
    n, lanes = 1 << 26, 152 * 32
    med = mcr.Medium(torch.full((1, 1), mua, device="cuda"), torch.zeros(1, 1, device="cuda"), 1.5, 0.0)
    src = mcr.Source(mcr.PENCIL, x0=0.7, z0=0.0, dir_x=0.0, dir_z=1.0)
    run = mcr.Run(K=0, n_packets=0)
    _, one = mcr.run_batch([mcr.Problem(med, 1, seed=1, source=src)], run, launch=RECORDS, stats=True)
    w = one["escaped_w"]  # FP32: a product of 2^26 and it is exact
    assert w == float(np.float32(w)) and 0.5 < w < 1.0
    _, st = mcr.run_batch([mcr.Problem(med, n, seed=1, source=src)], run, launch=(32, 1, 0, 0, 0, 2, 0), stats=True)
    assert mcr.record_info()[1] == 0 and st["escapes"] == n
    assert abs(st["escaped_w"] - n * w) <= (4 * n / lanes + 5 + 2 * 152) * 2.0 ** -53 * n * w


def test_runs_by_records_hold_no_launch_order():
    """The launch order is the direct deposit's: a line source (whose packets it would order once the tally is
    over 96 MB) takes no more memory by records than a pencil beam (whose packets it never orders)."""
    n = 1 << 24  # 64 MB of order; the packets leave the grid at once
    mua = torch.full((512, 512), 0.1, device="cuda")
    med = mcr.Medium(mua, mua, 0.1, 0.0)
    up = dict(x0=10.0, z0=0.0, dir_x=0.0, dir_z=-1.0)
    line, pencil = mcr.Source(mcr.LINE, x1=40.0, z1=0.0, **up), mcr.Source(mcr.PENCIL, **up)
    held = []
    mcr.forward(med, line, mcr.Run(K=32, n_packets=n))
    for src in (pencil, line):
        torch.cuda.synchronize()
        mcr.release_workspace()
        free = torch.cuda.mem_get_info()[0]
        mcr.forward(med, src, mcr.Run(K=32, n_packets=n))
        torch.cuda.synchronize()
        assert mcr.record_info()[0] > 0
        held.append(free - torch.cuda.mem_get_info()[0])
    assert held[1] - held[0] < n


@pytest.fixture
def little_memory():
    """Leaves `room` bytes of the GPU's memory free (asked for by calling it)."""
    held = []

    def leave(room):
        mcr.release_workspace()
        torch.cuda.empty_cache()
        torch.cuda.synchronize()
        while (take := min(torch.cuda.mem_get_info()[0] - room, 16 << 30)) > 1 << 26:
            held.append(torch.empty(take, dtype=torch.uint8, device="cuda"))

    leave.drop = held.clear
    yield leave
    held.clear()
    torch.cuda.empty_cache()
    mcr.release_workspace()


@pytest.mark.parametrize("room", [600 << 20, 6 << 30])
def test_little_memory_means_smaller_record_buffers(little_memory, room):
    """Where two buffers of 4 GB (3D: 5.4 GB) do not fit, smaller ones take more launches: the same sums, by
    records, in at most a quarter of what was free (or the least size); buffers of a smaller run are kept."""
    med = _medium(64, 64, 0.1, 5)
    src = mcr.Source(mcr.ISO_POINT, x0=3.0, z0=3.0)
    med3 = mcr3.Medium3(torch.full((24, 24, 24), 0.02, device="cuda"), torch.full((24, 24, 24), 8.0, device="cuda"),
                        f32(0.2), f32(0.9))
    src3 = mcr3.Source3(mcr.ISO_POINT, x0=2.1, y0=2.2, z0=2.3)
    run = mcr.Run(K=12, n_packets=400_000, seed=3)
    run3 = mcr.Run(K=3, n_packets=400_000, seed=3)
    ref, ref3 = mcr.forward(med, src, run), mcr3.forward(med3, src3, run3)
    small = mcr.forward(med, src, mcr.Run(K=12, n_packets=2_000, seed=3))
    torch.cuda.synchronize()
    little_memory(room)
    assert torch.equal(small, mcr.forward(med, src, mcr.Run(K=12, n_packets=2_000, seed=3)))
    free = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        assert torch.equal(ref, mcr.forward(med, src, run))
        kernels, closing = mcr.record_info(2)
        assert kernels > 0 and closing == 0
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= max(room // 4, 0) + (40 << 20)
    assert torch.equal(ref3, mcr3.forward(med3, src3, run3))
    assert mcr.record_info(3)[0] > 0 and mcr.record_info(3)[1] == 0
    mcr.check()


@pytest.fixture
def direct3(little_memory):
    """3D runs deposit directly: there was no room for record buffers when they were first asked for, and what
    was not to be had is not asked for again."""
    one = torch.ones(1, 1, 1, device="cuda")
    little_memory(100 << 20)
    mcr3.forward(mcr3.Medium3(one, one, 1.0, 0.0), mcr3.Source3(mcr.ISO_POINT, x0=0.5, y0=0.5, z0=0.5),
                 mcr.Run(K=0, n_packets=10))
    assert mcr.record_info(3) == (0, -1)
    little_memory.drop()
    torch.cuda.empty_cache()


COUNTERS3 = ("launched", "flights", "collisions", "segments", "escapes", "rr_kill", "rr_survive")
# a few tiles; and 132,192 voxels: 64-row tiles over two sorting passes
GRIDS3 = [((9, 14, 11), 0.25, 40_000), ((51, 54, 48), 0.08, 30_000)]


def _runs3(shape, dx, n, L, seed=5):
    r = np.random.default_rng(L)
    med = mcr3.Medium3(torch.from_numpy((0.01 + 0.1 * r.random(shape)).astype(np.float32)).cuda(),
                       torch.from_numpy((5 + 10 * r.random(shape)).astype(np.float32)).cuda(), f32(dx), f32(0.9))
    run = mcr.Run(K=L, n_packets=n, seed=seed, w_threshold=0.02, roulette_p=0.25)
    src = mcr3.Source3(mcr.PENCIL, x0=f32(0.4 * shape[2] * dx), y0=f32(0.6 * shape[1] * dx), z0=0.0, dir_x=0.2,
                       dir_y=-0.1, dir_z=1.0)
    q = torch.from_numpy(r.normal(size=shape).astype(np.float32)).cuda()
    out, st = mcr3.forward(med, src, run, stats=True)
    info = mcr.record_info(3)
    return out.cpu(), mcr3.adjoint(med, q, run).cpu(), [st[k] for k in COUNTERS3], info


@pytest.fixture(scope="module")
def by_records3():
    return {(g, L): _runs3(*GRIDS3[g], L) for g in range(2) for L in range(9)}


def test_records_equal_the_direct_deposit_in_3d(by_records3, direct3):
    """Every order L, forward (more packets than the tail takes: the main loop runs too) and adjoint: the same
    coefficients, bit for bit, and the same paths."""
    for (g, L), (fwd, adj, counts, info) in by_records3.items():
        assert info[0] > 0 and info[1] == 0, (g, L)
        d_fwd, d_adj, d_counts, d_info = _runs3(*GRIDS3[g], L)
        assert d_info == (0, -1)
        assert torch.equal(fwd, d_fwd) and torch.equal(adj, d_adj) and counts == d_counts, (g, L)


def test_3d_runs_refuse_a_capture_and_leave_it_whole():
    """A 3D run synchronises, so it is refused under capture, before it has enqueued anything: the capture goes on."""
    med = mcr3.Medium3(torch.full((8, 8, 8), 0.02, device="cuda"), torch.full((8, 8, 8), 8.0, device="cuda"), 0.2, 0.5)
    src, run = mcr3.Source3(mcr.ISO_POINT, x0=0.8, y0=0.8, z0=0.8), mcr.Run(K=2, n_packets=1_000)
    ref = mcr3.forward(med, src, run)
    x = torch.zeros(4, device="cuda")
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream), torch.cuda.graph(graph, stream=stream):
        x += 1.0
        with pytest.raises(mcr.McrError):
            mcr3.forward(med, src, run, stream=stream, out=ref)
    graph.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [1.0] * 4
    assert torch.equal(mcr3.forward(med, src, run), ref)
