"""The tiled launches (one per phase, in CUDA graphs, two of them side by side)
on boards that the resident launches would take: every tile, z segment and
graph chunk, both orders of the z-UPML and the interior launch, and batches.
All paths use the same arithmetic per node and round a halo value as its owner
stores it, so everything is equal bit for bit."""
import numpy as np
import pytest

from paper_1008_2602_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TUNES = [dict(tile_x=62, tile_y=8, zseg=64, graph_chunk=7), dict(tile_x=62, tile_y=4, zseg=5, graph_chunk=1),
         dict(tile_x=124, tile_y=4, zseg=9, graph_chunk=16), dict(tile_x=124, tile_y=8, zseg=3, graph_chunk=4), {}]


@pytest.fixture(scope="module")
def fdtd():
    import torch
    assert torch.cuda.is_available()
    from paper_1008_2602_gb300 import solver
    return solver


def _r(seed, *n, upml=4, **kw):
    return W.random_problem(seed, *n, upml=upml, n_steps=50, **kw)


BOARDS = {
    "two_tiles": _r(6, 75, 38, 29),
    "odd_first_column": _r(2, 20, 33, 18, upml=5).replace(upml_kappa_max=5.0),   # fused region from x = 5
    "three_wide": _r(5, 260, 21, 31, upml=6),
    "uneven": _r(9, 150, 36, 28).replace(upml_depth=(4, 0, 3, 5, 0, 6), walls=(0, 1, 0, 0, 1, 0)),
    "no_upml": _r(8, 70, 31, 22, upml=0).replace(walls=(1, 1, 0, 0, 1, 1)),
}


def _same(a, b):
    for c in range(6):
        assert np.array_equal(a.field(c), b.field(c)), c
    assert np.array_equal(a.traces(), b.traces()) and np.any(b.field(2))


@pytest.mark.parametrize("name", list(BOARDS))
def test_every_tile_equals_the_resident_steps(fdtd, name):
    p = BOARDS[name]
    ref = fdtd.Solver(p)
    assert ref.resident()
    ref.run()
    for tune in TUNES:
        s = fdtd.Solver(p, tuning=tune)
        s.set_tiled()
        assert not s.resident()
        s.run()
        _same(s, ref)
        s.close()
    ref.close()


@pytest.mark.parametrize("name", ["two_tiles", "odd_first_column", "three_wide"])
def test_every_tile_gives_the_same_fp16_board(fdtd, name):
    p = BOARDS[name]
    ref = fdtd.Solver(p, precision="fp16")
    ref.step_profiled(p.n_steps)
    for tune in TUNES:
        s = fdtd.Solver(p, precision="fp16", tuning=tune)
        s.run()
        _same(s, ref)
        s.close()
    ref.close()


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("zseg", [1, 40])
def test_both_launch_orders_equal_the_serial_launches(fdtd, precision, zseg):
    """62x4 tiles over 24 z-UPML planes: 2 x 98 x 24 items with one plane an
    item, more than the line between the two orders, and 2 x 98 x 2 with 40."""
    p = _r(12, 130, 400, 40, upml=12).replace(upml_depth=(4, 4, 4, 4, 12, 12), n_steps=40)
    tune = dict(tile_x=62, tile_y=4, zseg=zseg)
    a, b = (fdtd.Solver(p, precision=precision, tuning=tune) for _ in range(2))
    a.set_tiled()
    a.step(37).step(3)
    b.step_profiled(40)
    _same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
def test_a_tiled_batch_equals_each_board_alone(fdtd, precision):
    """Uneven boards and lengths; members that end within a call; one that
    joins later; in FP32 one member stays with the resident launches."""
    probs = [W.random_problem(20 + s, 30 + 17 * s, 24 + 9 * s, 14 + 2 * s, upml=3, n_steps=60) for s in range(6)]
    steps = [10 + 9 * (i % 4) for i in range(len(probs))]
    sols = [fdtd.Solver(p, precision=precision) for p in probs]
    for s in sols[1:]:
        s.set_tiled()
    b = fdtd.Batch()
    for s, n in zip(sols[:-1], steps):
        b.add(s, n)
    b.step(17)
    b.add(sols[-1], steps[-1])
    assert [s.resident() for s in sols] == [precision == "fp32"] + [False] * 5
    while any(b.remaining(s) for s in sols):
        b.step(5)
    b.sync()
    for s, p, n in zip(sols, probs, steps):
        ref = fdtd.Solver(p, precision=precision)
        ref.step_profiled(n)
        _same(s, ref)
        ref.close()
    b.close()
    for s in sols:
        s.close()


@pytest.mark.parametrize("axis,plane,rim,resident", [(0, 0, 0, True), (1, 0, 0, True), (2, 0, 0, True), (1, 17, 0, True),
                                                     (1, 17, 1, False), (0, 40, 0, False), (1, 33, 0, False), (2, 26, 0, False)])
def test_restored_planes_go_on_alike(fdtd, axis, plane, rim, resident):
    """A checkpoint of a board with a plane of E_x, E_z written from outside:
    only values behind a high PEC wall, which no step writes, keep it from the
    resident launches (rim: the plane's own edges there have some too); both
    ways give the same fields."""
    import torch
    from paper_1008_2602_gb300 import capi
    p = W.random_problem(16, 40, 33, 26, upml=3, n_steps=60)
    a, b, c = (fdtd.Solver(p) for _ in range(3))
    a.step(9)
    nodes = [n + 1 for n in (p.nz, p.ny, p.nx)]
    del nodes[2 - axis]
    vals = torch.rand([2] + nodes, generator=torch.Generator().manual_seed(1))
    if not rim:
        vals[:, -1, :] = vals[:, :, -1] = 0
    vals = vals.cuda()
    torch.cuda.synchronize()
    capi.fdtd_halo_unpack(a.ctx, axis, plane, 0b101, vals.data_ptr())
    state = a.save()
    for s in (b, c):
        s.load(state)
    assert b.resident() == resident
    c.set_tiled()
    for n in (1, 6, 5):
        b.step(n)
        c.step(n)
        _same(b, c)
    for s in (a, b, c):
        s.close()
