"""Single-instance kernels that the library chooses by the grid's size (the
launch shape left to it): the whole grid on chip, one block per SM
(csrc/bte_grid.cu), and two steps per launch for FP32 grids that do not fit
(csrc/bte_pair.cu).  Both perform the one launch per step kernel's operations
per cell and add the rows 0 and 1 in its order, so state and trace agree with
it bit for bit (it runs when the launch shape is given, here graph_steps)."""
import numpy as np
import pytest

from paper_1401_6047_gb300 import bte
from paper_1401_6047_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _params(n_max, m_points, prec, omega=2.2, **kw):
    L = max(9.0, 0.01 * m_points)
    return W.Params(E_dc=1.4, E_omega=0.7, omega=omega, B=2.6, mu=1.7, n_max=n_max, m_points=m_points,
                    phiy_min=-L, phiy_max=L, dt=2e-3, periods=1.5 * omega / 2.2, avg_window=0.5, precision=prec,
                    B_omega=0.3, B_phase=0.4, **kw)


def _run(p, steps, **kw):
    st = W.random_state(p, seed=p.n_max)
    with bte.Solver(p, **kw) as s:
        s.set_state(0, st[0], st[1])
        s.set_state(1, st[2], st[3])
        for k in steps:
            s.step(k)
        return (*s.get_state(0), *s.get_state(1), *s.trace())


# one block, blocks of one row, of one column group, several of both, ragged
# last blocks, more columns than threads, the largest that fit
@pytest.mark.parametrize("shape", [(1, 3), (9, 37), (30, 201), (22, 129), (64, 1000), (3, 5000), (500, 64),
                                   (119, 4000), (400, 4001)])
@pytest.mark.parametrize("prec", [W.FP64, W.FP32_MIXED])
def test_blocks_on_chip_equal_one_launch_per_step(shape, prec):
    if prec == W.FP64 and shape[0] * shape[1] > 600000:
        pytest.skip("does not fit on chip in FP64")
    p = _params(*shape, prec)
    steps = (5, 1, 3, 60, 4)  # calls of fewer than four steps take single launches
    for x, y in zip(_run(p, steps), _run(p, steps, graph_steps=16)):
        assert np.array_equal(x, y)


# chunks of 8 rows and more, ragged last tile (1, 41 and 120 of its 120
# columns), states below and above the size from which the walk alternates,
# the drive table starting over inside a pair (period of an odd number of steps)
@pytest.mark.parametrize("shape,omega", [((700, 5041), 20.0), ((2100, 1081), 7.0), ((999, 2520), 2.2), ((19, 120001), 13.0)])
def test_two_steps_per_launch_equal_one(shape, omega):
    p = _params(*shape, W.FP32_MIXED, omega=omega)
    steps = (5, 1, 2, 37, 80)  # odd calls end with a single step
    for x, y in zip(_run(p, steps), _run(p, steps, graph_steps=16)):
        assert np.array_equal(x, y)


def test_routes_replay_in_a_captured_graph():
    """Calls captured on the caller's stream and replayed: the kernels take
    the step index from the device, so each replay advances further."""
    torch = pytest.importorskip("torch")
    p = _params(30, 201, W.FP32_MIXED)
    with bte.Solver(p) as ref:
        ref.step(4 + 3 * 8)
        want = (*ref.get_state(0), *ref.get_state(1))
    stream = torch.cuda.Stream()
    with bte.Solver(p, stream=stream.cuda_stream) as s:
        s.step(4)
        s.observables(check=False)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            s.step(8)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        got = (*s.get_state(0), *s.get_state(1))
    for x, y in zip(got, want):
        assert np.array_equal(x, y)


def _obs(o):
    return np.array([o.v_dr, o.norm, o.v_dc_avg, o.absorption, o.norm_max_abs_err])


def test_batched_points_that_fit_no_cluster_run_alone():
    """Two FP64 points too large for a cluster of 16 CTAs (tier 0 of the plan)
    among one that fits: run as single instances by default, streamed with
    resident = 1.  FP64 sums in another order: 1e-12 relative (the norm's
    error to 1e-13 absolute)."""
    pts = [_params(n, m, W.FP64).replace(periods=0.05 + 0.01 * n / 90, avg_window=0.02)
           for n, m in ((88, 1001), (30, 201), (90, 1345))]
    assert list(bte.batch_plan(pts)) [::2] == [0, 0]
    for o, r in zip(bte.batch_run(pts), bte.batch_run(pts, resident=1)):
        assert o.status == r.status == bte.OK and o.step == r.step == o.steps_total
        assert np.all(np.abs(_obs(o) - _obs(r))[:4] <= 1e-12 * np.abs(_obs(r))[:4])
        assert abs(o.norm_max_abs_err - r.norm_max_abs_err) <= 1e-13


@pytest.mark.parametrize("prec", [W.FP64, W.FP32_MIXED])
def test_larger_clusters_for_few_points_give_the_same_bits(prec):
    """Few points get larger clusters than they need; with resident_smem given
    (here its default) they keep the smallest."""
    pts = [_params(n, m, prec).replace(periods=0.1, avg_window=0.05) for n, m in ((60, 501), (33, 402), (9, 37))]
    for o, r in zip(bte.batch_run(pts), bte.batch_run(pts, resident_smem=232448)):
        assert np.array_equal(_obs(o), _obs(r))
