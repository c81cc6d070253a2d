"""The kernels that the library chooses by the grid's size, where the choice
or its bookkeeping can go wrong: very wide rows, grids near the on-chip limit,
a constant drive, captured calls, several handles at once."""
import threading
import time

import numpy as np
import pytest

from paper_1401_6047_gb300 import bte
from paper_1401_6047_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _params(n_max, m_points, prec=W.FP32_MIXED, omega=2.2, periods=1.5, **kw):
    L = max(9.0, 0.01 * m_points)
    if omega == 0.0:
        kw.update(t_max=2.0)
    return W.Params(E_dc=1.4, E_omega=0.7, omega=omega, B=2.6, mu=1.7, n_max=n_max, m_points=m_points,
                    phiy_min=-L, phiy_max=L, dt=2e-3, periods=periods * omega / 2.2, avg_window=0.05, precision=prec,
                    B_omega=0.3, B_phase=0.4, **kw)


def _state(s):
    return (*s.get_state(0), *s.get_state(1))


def _run(p, steps, **kw):
    st = W.random_state(p, seed=p.n_max)
    with bte.Solver(p, **kw) as s:
        s.set_state(0, st[0], st[1])
        s.set_state(1, st[2], st[3])
        for k in steps:
            s.step(k)
        return (*_state(s), *s.trace())


def _equal(got, want):
    return all(np.array_equal(x, y) for x, y in zip(got, want))


# rows of more columns than one CTA of the row sums takes (16384 FP32, 8192
# FP64), one past a whole number of its pieces, and more than 393216 columns,
# whose sums once asked for more shared memory than a launch may
@pytest.mark.parametrize("shape,prec", [((19, 400001), W.FP32_MIXED), ((20, 98305), W.FP32_MIXED),
                                        ((2, 16385), W.FP32_MIXED), ((1, 60001), W.FP32_MIXED),
                                        ((9, 8193), W.FP64), ((3, 50001), W.FP64)])
def test_wide_rows_equal_one_launch_per_step(shape, prec):
    p = _params(*shape, prec)
    assert _equal(_run(p, (4, 5, 18)), _run(p, (4, 5, 18), graph_steps=16))


# FP32 grids that fit on chip in one form of the arithmetic only: with one
# column per thread (its bits are those of mode 3, so these take two steps per
# launch), and with two or four
@pytest.mark.parametrize("shape", [(400, 5000), (700, 2880), (137, 14600), (30, 60700)])
def test_grids_at_the_on_chip_limit_equal_one_launch_per_step(shape):
    p = _params(*shape)
    steps = (5, 2, 1, 33)
    assert _equal(_run(p, steps), _run(p, steps, graph_steps=16))


# drives whose table starts over with the entry it ended on (a constant one,
# from 0 and not) and without, inside a pair and between two
@pytest.mark.parametrize("omega,B_phase", [(0.0, 0.4), (30.0, 0.0), (31.0, 0.4), (1500.0, 0.4), (3141.0, 0.4)])
def test_two_steps_per_launch_under_every_drive(omega, B_phase):
    p = _params(699, 3000, omega=omega).replace(B_phase=B_phase)
    steps = (5, 2, 41, 70)
    assert _equal(_run(p, steps), _run(p, steps, graph_steps=16))


# two steps per launch: an odd number of pairs, of steps, and more steps than
# the handle keeps rows for (16 at 120001 columns); on chip: in place; one
# launch per step, shorter and longer than the handle's own graphs
@pytest.mark.parametrize("shape,n,kw", [((999, 2520), 2, {}), ((999, 2520), 3, {}), ((999, 2520), 5, {}),
                                        ((999, 2520), 6, {}), ((999, 2520), 8, {}), ((19, 120001), 16, {}),
                                        ((19, 120001), 42, {}), ((30, 201), 7, {}),
                                        ((30, 201), 40, dict(graph_steps=16))])
def test_captured_calls_replay(shape, n, kw):
    torch = pytest.importorskip("torch")
    p = _params(*shape)
    with bte.Solver(p, **kw) as ref:
        ref.step(4 + 3 * n)
        want = _state(ref)
    stream = torch.cuda.Stream()
    with bte.Solver(p, stream=stream.cuda_stream, **kw) as s:
        s.step(4)
        s.observables(check=False)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            s.step(n)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        assert _equal(_state(s), want)


# pairs of launch shapes whose shared memory differs: the first handle's calls
# after the second handle is made
@pytest.mark.parametrize("first,second", [(((400, 2001), dict(tile_m=768, chunk_n=64)), ((30, 201), dict(tile_m=32, chunk_n=8))),
                                          (((400, 4001), {}), ((8, 37), {})),
                                          (((60, 501), dict(resident=1)), ((30, 201), dict(resident=1))),
                                          (((60, 201), dict(resident=3, wide_cols=100)), ((30, 201), dict(resident=3, wide_cols=20)))])
def test_a_later_handle_leaves_an_earlier_one_running(first, second):
    with bte.Solver(_params(*first[0]), **first[1]) as a:
        with bte.Solver(_params(*second[0]), **second[1]) as b:
            for s in (b, a, b, a):
                s.step(3)
                s.step(8)
                assert s.observables(check=False).status == bte.OK


def test_handles_on_several_threads():
    """Each thread makes and steps its own handles; the launches of one are
    not refused for what another thread's handle needs."""
    errors = []

    def work(shape):
        try:
            for _ in range(6):
                with bte.Solver(_params(*shape, periods=20.0)) as s:
                    for _ in range(40):
                        s.step(8)
                        s.step(2)
                    s.observables()
        except bte.BteError as e:
            errors.append(f"{shape}: {e}")

    threads = [threading.Thread(target=work, args=(sh,)) for sh in ((119, 4000), (8, 37), (60, 1000), (30, 201))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors


# mode 3 on several clusters and on one, its shape given and not; mode 0
@pytest.mark.parametrize("shape,kw", [((30, 201), dict(resident=3)), ((47, 256), dict(resident=3)),
                                      ((16, 96), dict(resident=3)), ((30, 201), dict(resident=3, wide_cols=101)),
                                      ((30, 201), {}), ((999, 2520), {})])
@pytest.mark.parametrize("prec", [W.FP64, W.FP32_MIXED])
def test_cutting_a_run_into_calls_keeps_its_bits(shape, kw, prec):
    p = _params(*shape, prec)
    assert _equal(_run(p, (3, 1, 40, 2, 11), **kw), _run(p, (57,), **kw))


@pytest.mark.parametrize("prec", [W.FP64, W.FP32_MIXED])
def test_state_into_one_array_for_both(prec):
    """The second grid array is copied last, so it is what one array given for
    both ends with."""
    with bte.Solver(_params(30, 201, prec)) as s:
        s.step(10)
        for grid in (0, 1):
            x = np.zeros(s.shape)
            bte._check(bte.lib().bte_get_state(s._h, grid, bte._dp(x), bte._dp(x)))
            assert np.array_equal(x, s.get_state(grid)[1])


def _seconds(pts, **kw):
    best = 1e9
    for _ in range(3):
        t = time.perf_counter()
        bte.batch_run(pts, **kw)
        best = min(best, time.perf_counter() - t)
    return best


# points that fit no cluster: many that leave most of the GPU idle alone (3.7
# and 1.7 times the lock-step time one after another), few and large ones that
# do not, and both
@pytest.mark.parametrize("points,prec", [([(9, 4001, 64)], W.FP32_MIXED), ([(9, 2001, 64)], W.FP64),
                                         ([(200, 2001, 6)], W.FP32_MIXED), ([(400, 4001, 3), (9, 4001, 48)], W.FP32_MIXED)])
def test_batches_that_fit_no_cluster_are_no_slower_than_lock_step(points, prec):
    pts = [_params(n, m, prec).replace(periods=0.5, avg_window=0.1) for n, m, count in points for _ in range(count)]
    assert not bte.batch_plan(pts).any()
    assert _seconds(pts) < 1.3 * _seconds(pts, resident=1)
    for o, r in zip(bte.batch_run(pts), bte.batch_run(pts, resident=1)):
        assert o.status == r.status == bte.OK
        for x, y in zip((o.v_dr, o.norm, o.v_dc_avg, o.absorption), (r.v_dr, r.norm, r.v_dc_avg, r.absorption)):
            assert abs(x - y) <= 1e-10 * abs(y)  # the same cells, added in another order


def test_tuned_options_are_no_slower_than_none():
    """Points that run fastest one after another, which only options that leave
    the shape to the library do."""
    pts = [_params(88, 1001, W.FP64).replace(periods=0.3, avg_window=0.1) for _ in range(6)]
    best, secs = bte.batch_tune(pts, sample=6, steps=400)
    assert secs.argmin() == 0 and best["resident"] == 0
    assert _seconds(pts, **best) < 1.3 * _seconds(pts)


# few cells and many, an odd number of them, the two arrays of an FP32 grid
# widened one after the other and side by side, in one stretch and in several
@pytest.mark.parametrize("shape", [(1, 3), (2, 21), (30, 201), (398, 501), (399, 501), (1000, 2101)])
@pytest.mark.parametrize("prec", [W.FP64, W.FP32_MIXED])
def test_state_comes_back_as_it_was_set(shape, prec):
    p = _params(*shape, prec)
    st = W.random_state(p, seed=5)
    if prec == W.FP32_MIXED:
        st = [x.astype(np.float32).astype(np.float64) for x in st]
    with bte.Solver(p) as s:
        s.set_state(0, st[0], st[1])
        s.set_state(1, st[2], st[3])
        assert _equal(_state(s), st)
        for which in (0, 1):  # one array of a grid alone
            x = np.zeros(s.shape)
            args = [None, None]
            args[which] = bte._dp(x)
            bte._check(bte.lib().bte_get_state(s._h, 1, *args))
            assert np.array_equal(x, st[2 + which])


# points on chip whose column groups (2 columns in FP64, 4 in FP32) need the
# last warp's threads for another row block or to be walked once: on, just
# below and just above each edge, with few rows per CTA and many
@pytest.mark.parametrize("groups", [96, 97, 160, 161, 170, 171, 240, 241, 256, 257, 480, 481, 512, 513])
@pytest.mark.parametrize("n_max", [4, 24])
@pytest.mark.parametrize("prec", [W.FP64, W.FP32_MIXED])
def test_on_chip_points_at_the_edges_of_the_thread_split(groups, n_max, prec):
    """Against lock-step launches; FP32 states are equal, their sums added in
    FP32 pairs (1e-7 of the norm, 2e-6 of the drift)."""
    V = 2 if prec == W.FP64 else 4
    pts = [_params(n_max, groups * V - k, prec).replace(periods=0.06, avg_window=0.05) for k in (0, 1)]
    fits = bte.batch_plan(pts).all()
    if not fits:
        pytest.skip("does not fit a cluster")
    for o, r in zip(bte.batch_run(pts, resident_smem=232448), bte.batch_run(pts, resident=1)):
        assert o.status == r.status == bte.OK
        for k in ("v_dr", "norm", "v_dc_avg", "absorption"):
            x, y = getattr(o, k), getattr(r, k)
            assert abs(x - y) <= (1e-12 * max(abs(y), 1e-3) if prec == W.FP64 else 1e-7 if k == "norm" else 2e-6)
