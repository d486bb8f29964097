"""Resident launches (many steps in one cooperative launch) against the
launch-per-phase path, which ``step_profiled`` always takes: both use the same
arithmetic per node, so fields, auxiliaries (through checkpoints), traces and
the energy must be equal bit for bit; the FP64 spectra fold their samples in
other chunks and agree to rounding (2^-52 times the few thousand terms summed
is below 1e-12)."""
import numpy as np
import pytest

from paper_1008_2602_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fdtd():
    import torch
    assert torch.cuda.is_available()
    from paper_1008_2602_gb300 import solver
    return solver


def _r(seed, *n, upml=3, **kw):
    return W.random_problem(seed, *n, upml=upml, n_steps=kw.pop("n_steps", 60), **kw)


def _ports(p, seed, n_src, n_prb):
    """Many sources (some on one edge) and probes, several to a warp unit."""
    rng = np.random.default_rng(seed)
    base = np.asarray(p.sources)
    src = np.concatenate([base, base[rng.integers(len(base), size=n_src)]])
    prm = np.concatenate([p.source_params, np.tile(p.source_params[:1], (n_src, 1)) * rng.uniform(0.5, 2, (n_src, 1))])
    prm[:, 1:] = p.source_params[0, 1:]
    prb = np.stack([rng.integers(0, p.nx, n_prb), rng.integers(0, p.ny, n_prb), rng.integers(0, 3, n_prb),
                    rng.integers(0, 3, n_prb)], axis=1).astype(np.int32)
    return p.replace(sources=src.astype(np.int32), source_params=prm, probes=np.concatenate([p.probes, prb]))


CASES = {
    "odd": _r(1, 37, 29, 23),
    "kappa": _r(2, 20, 33, 18, upml=5).replace(upml_kappa_max=5.0),
    "quads_cut": _r(3, 75, 40, 21, upml=4),                       # nx % 4 == 3
    "tiny": _r(4, 9, 8, 7, upml=2),
    "long_rows": _r(5, 150, 21, 31, upml=6),
    "no_upml": _r(6, 40, 31, 22, upml=0),
    "pmc_sides": _r(7, 41, 31, 22, upml=0).replace(walls=(1, 1, 1, 1, 0, 0)),
    "pmc_all": _r(8, 40, 31, 22, upml=0).replace(walls=(1,) * 6),
    "mixed_low": _r(9, 44, 36, 28, upml=4).replace(upml_depth=(4, 0, 3, 5, 0, 6), walls=(0, 1, 0, 0, 1, 0)),
    "mixed_high": _r(10, 44, 36, 28, upml=4).replace(upml_depth=(0, 4, 0, 5, 4, 0), walls=(1, 0, 1, 0, 0, 1)),
    "no_fused_region": _r(12, 4, 40, 12, upml=0, n_src=1),
    "more_units_than_warps": _r(13, 130, 120, 60, upml=5, n_steps=30),
    "voltage": W.add_voltage_sources(_r(11, 37, 29, 23), [(10, 10, 10, 2), (10, 10, 10, 2)]),
    "many_ports": _ports(_r(14, 37, 29, 23), 3, 12, 150),
    "table1": W.table1_board(n_steps=80),
    # past one unit a warp (the boards above but two have at most that)
    "large_odd": _r(31, 97, 61, 43, upml=5, n_steps=40).replace(upml_kappa_max=5.0),
    "large_pmc": _r(32, 121, 75, 31, upml=0, n_steps=40).replace(walls=(1,) * 6),
    "large_mixed": _r(33, 118, 66, 44, upml=4, n_steps=40).replace(upml_depth=(4, 0, 3, 5, 0, 6), walls=(0, 1, 0, 0, 1, 0)),
    "large_ports": _ports(_r(34, 97, 61, 43, upml=5, n_steps=40), 4, 12, 150),
    "large_8bit": W.realistic_board(n_steps=40),
}


@pytest.mark.parametrize("name", list(CASES))
def test_resident_steps_equal_the_tiled_ones(fdtd, name):
    p = CASES[name]
    n = p.n_steps
    a, b = fdtd.Solver(p), fdtd.Solver(p)
    a.step(n - 8)          # an even and an odd number of steps, a single one
    a.step(7)
    a.step(1)
    b.step_profiled(n)
    for c in range(6):
        assert np.array_equal(a.field(c), b.field(c)), c
    ta = a.traces()
    assert np.array_equal(ta, b.traces()) and np.any(a.field(2))
    sa, sb = a.spectra(), b.spectra()
    assert np.linalg.norm(sa - sb) <= 1e-12 * np.linalg.norm(sb)
    assert a.diagnostics() == b.diagnostics()
    # the two paths take turns: both field sets, every auxiliary and parity agree
    a.step_profiled(3)
    a.step(4)
    b.step(2)
    b.step_profiled(5)
    for c in range(6):
        assert np.array_equal(a.field(c), b.field(c)), c
    assert a.diagnostics() == b.diagnostics()
    # a checkpoint of one continues in the other
    state = a.save()
    b.load(state)
    a.step(5)
    b.step_profiled(5)
    for c in range(6):
        assert np.array_equal(a.field(c), b.field(c)), c
    a.close()
    b.close()


def test_probes_past_the_spectrum_and_unstable_runs(fdtd):
    """Samples after the spectrum's length are not recorded; a non-finite
    sample is reported as by the tiled launches."""
    p = CASES["odd"].replace(n_steps=20)
    a = fdtd.Solver(p)
    a.step(50)
    assert a.traces(max_len=50).shape[1] == 20
    a.close()
    from paper_1008_2602_gb300 import capi
    q = CASES["odd"].replace(courant=1.5, n_steps=4000)
    s = fdtd.Solver(q)
    with pytest.raises(capi.FdtdError) as e:
        for _ in range(40):
            s.step(100)
            s.sync()
    assert e.value.code == capi.FDTD_EUNSTABLE
    s.close()


def test_depth_switch_between_resident_runs(fdtd):
    """A board that leaves depth 2 keeps the set numbering of its steps."""
    p = _r(15, 64, 40, 30, upml=4, n_steps=90)
    a, b = fdtd.Solver(p), fdtd.Solver(p)
    a.step(11)
    a.set_tuning(depth=2)
    a.step(20)
    a.set_tuning(depth=1)
    a.step(9)
    b.step_profiled(40)
    for c in range(6):
        assert np.array_equal(a.field(c), b.field(c)), c
    a.close()
    b.close()


def test_batch_of_uneven_boards_and_lengths(fdtd):
    """Several groups of teams, members that finish within a call, one member
    too wide for nothing but the general rule, and a member joining later."""
    probs = [W.random_problem(20 + s, 20 + 7 * s, 24 + 5 * s, 14 + s, upml=3, n_steps=60) for s in range(9)]
    probs += [W.random_problem(40, 230, 190, 40, upml=6, n_steps=60), W.random_problem(41, 210, 220, 38, upml=6, n_steps=60)]
    sols = [fdtd.Solver(p) for p in probs]
    b = fdtd.Batch()
    steps = [10 + 3 * (i % 7) for i in range(len(probs))]
    for s, n in zip(sols[:-1], steps):
        b.add(s, n)
    b.step(13)
    b.add(sols[-1], steps[-1])
    while any(b.remaining(s) for s in sols):
        b.step(4)
    b.sync()
    for s, p, n in zip(sols, probs, steps):
        ref = fdtd.Solver(p)
        ref.step_profiled(n)
        assert np.array_equal(s.traces(), ref.traces()), p.name
        for c in range(6):
            assert np.array_equal(s.field(c), ref.field(c)), (p.name, c)
        ref.close()
    b.close()
    for s in sols:
        s.close()


def test_a_plane_written_from_outside_keeps_the_general_path(fdtd):
    """Values put on an outer wall plane differ between the two field sets, so
    several steps after such a write go the general way; all agree."""
    import torch
    p = _r(16, 40, 33, 26)
    out = []
    for general in (False, True):
        s = fdtd.Solver(p)
        s.step_profiled(9)
        from paper_1008_2602_gb300 import capi
        plane = torch.ones(2 * (p.nz + 1) * (p.nx + 1), device="cuda") * 0.25
        torch.cuda.synchronize()
        capi.fdtd_halo_unpack(s.ctx, 1, p.ny, 0b101, plane.data_ptr())
        s.sync()
        if general:
            s.step_profiled(1)
            s.step_profiled(5)
        else:
            s.step(1)
            s.step(5)
        out.append([s.field(c) for c in range(6)])
        s.close()
    for c in range(6):
        assert np.array_equal(out[0][c], out[1][c]), c


def test_steps_on_two_streams_at_once(fdtd):
    """Two boards stepped from two host threads: cooperative launches of
    different streams take turns on the device."""
    import threading
    probs = [_r(50 + s, 60, 50, 40, upml=5, n_steps=300) for s in range(2)]
    got = [None, None]

    def work(t):
        s = fdtd.Solver(probs[t])
        for _ in range(30):
            s.step(10)
        got[t] = s.traces()
        s.close()

    th = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in th:
        t.start()
    for t in th:
        t.join(timeout=120)
    for t in range(2):
        ref = fdtd.Solver(probs[t])
        ref.step_profiled(300)
        assert np.array_equal(got[t], ref.traces())
        ref.close()


def test_single_steps_in_a_caller_s_graph(fdtd):
    """A few steps captured into a caller's graph replay as further steps."""
    import torch
    p = _r(17, 37, 29, 23)
    st = torch.cuda.Stream()
    a, b = fdtd.Solver(p, stream=st), fdtd.Solver(p)
    a.step(2)
    a.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        g.capture_begin(capture_error_mode="thread_local")
        a.step(3)
        g.capture_end()
    for _ in range(4):
        g.replay()
    torch.cuda.synchronize()
    assert a.info()["step"] == 14
    a.step(1)                       # an odd distance from the counted steps: the device counter decides
    b.step_profiled(15)
    assert np.array_equal(a.traces(max_len=5), b.traces(max_len=5))
    a.close()
    b.close()
