"""Mixed-precision, batched CG solves on the GPU through the C ABI; every solution is checked by the FP64
oracle's true residual |b - A x| / |b|."""
import numpy as np
import pytest

import hisq_inputs as hi
from gpu_util import gpu

pytestmark = pytest.mark.gpu

TOL = 1e-10
SLACK = 1.0   # the library stops at 0.95 tol, so the oracle's own FP64 residual is within tol


def _solve(g, rhs, mass, **params):
    p = g.hisq.hisq_default_solver_params()
    for k, v in params.items():
        setattr(p, k, v)
    g.hisq.hisq_set_solver_params(p)
    xs = [np.zeros_like(b) for b in rhs]
    g.hisq.hisq_cg_solve(g.fat, g.naik, list(rhs), xs, mass, TOL)
    iters = np.zeros(len(rhs), dtype=np.int32)
    res = np.zeros(len(rhs))
    stats = g.hisq.hisq_last_stats(iters, res)
    return np.stack(xs), stats, iters, res


def test_plain_fp64_cg_8c4():
    """8^3 x 4, one RHS, FP64 everywhere, m = 0.1, to true residual 1e-10; iteration count of
    the textbook oracle CG within a few."""
    dims = (8, 8, 8, 4)
    with gpu(dims, 0) as g:
        b = hi.gaussian_rhs(g.lat, 0)
        for graph in (0, 1, 2):
            x, stats, iters, res = _solve(g, [b], 0.1, inner_prec=0, use_graph=graph)
            true = g.oracle.true_residual(b, x[0], 0.1)[0]
            assert true <= TOL * SLACK and res[0] <= TOL
            _, it_oracle, _ = g.oracle.cg(b, 0.1, TOL)
            assert abs(int(iters[0]) - it_oracle) <= 2


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("graph", [0, 1, 2])
def test_mixed_precision_reaches_fp64_residual(prec, graph):
    dims = (8, 10, 8, 6)
    with gpu(dims, prec) as g:
        rhs = [hi.gaussian_rhs(g.lat, k) for k in range(3)]
        x, stats, iters, res = _solve(g, rhs, 0.05, inner_prec=prec, use_graph=graph)
        true = g.oracle.true_residual(np.stack(rhs), x, 0.05)
        assert np.all(true <= TOL * SLACK), true
        assert stats.converged == 3 and stats.reliable_updates >= 3


@pytest.mark.parametrize("graph", [0, 1, 2])
def test_bundle_uneven_convergence_masked(graph):
    """A bundle whose right-hand sides converge at different iterations (scaled norms 1e-3..1e3
    and spectral shaping b = A^q g): converged ones are masked while the rest iterate."""
    dims = (8, 10, 8, 6)
    mass = 0.05
    with gpu(dims, 1) as g:
        rhs = []
        for k in range(6):
            v = hi.gaussian_rhs(g.lat, 10 + k)
            for _ in range(k % 3):
                v = g.oracle.aop(v, mass)
            rhs.append(v / np.linalg.norm(v) * 10.0 ** (-3 + 6 * k / 5))
        x, stats, iters, res = _solve(g, rhs, mass, inner_prec=1, use_graph=graph, bundle=6)
        true = g.oracle.true_residual(np.stack(rhs), x, mass)
        assert np.all(true <= TOL * SLACK), true
        assert len(set(iters.tolist())) > 1
        assert stats.bundle_iterations == max(iters)


def test_many_rhs_in_several_bundles_and_zero_rhs():
    dims = (8, 8, 8, 4)
    with gpu(dims, 1) as g:
        rhs = [hi.gaussian_rhs(g.lat, 30 + k) for k in range(19)]
        rhs[5] = np.zeros_like(rhs[5])
        x, stats, iters, res = _solve(g, rhs, 0.1, inner_prec=1, bundle=8)
        assert stats.bundles == 3
        assert np.all(x[5] == 0) and iters[5] == 0
        ok = [k for k in range(19) if k != 5]
        true = g.oracle.true_residual(np.stack(rhs)[ok], x[ok], 0.1)
        assert np.all(true <= TOL * SLACK)


def test_not_converged_is_reported():
    dims = (8, 8, 8, 4)
    with gpu(dims, 1) as g:
        b = hi.gaussian_rhs(g.lat, 0)
        p = g.hisq.hisq_default_solver_params()
        p.max_iter = 5
        g.hisq.hisq_set_solver_params(p)
        x = np.zeros_like(b)
        rc = g.hisq.hisq_cg_solve(g.fat, g.naik, [b], [x], 0.1, TOL, raise_on_error=False)
        assert rc == -4
        stats = g.hisq.hisq_last_stats()
        assert stats.converged == 0 and stats.max_iterations == 5


def test_nan_rhs_is_breakdown():
    dims = (8, 8, 8, 4)
    with gpu(dims, 1) as g:
        b = hi.gaussian_rhs(g.lat, 0)
        b[3, 1] = np.nan
        x = np.zeros_like(b)
        rc = g.hisq.hisq_cg_solve(g.fat, g.naik, [b], [x], 0.1, TOL, raise_on_error=False)
        assert rc == -5


def test_device_pointers_and_timing():
    """rhs/x as device tensors; per-Dslash CUDA-event timing in host-driven mode."""
    import torch
    dims = (8, 10, 8, 6)
    with gpu(dims, 1) as g:
        b = hi.gaussian_rhs(g.lat, 3)
        bd = torch.from_numpy(b.view(np.float64).copy()).cuda()
        xd = torch.zeros_like(bd)
        p = g.hisq.hisq_default_solver_params()
        p.use_graph = 0
        p.time_kernels = 1
        g.hisq.hisq_set_solver_params(p)
        g.hisq.hisq_cg_solve(g.fat, g.naik, [bd], [xd], 0.05, TOL)
        stats = g.hisq.hisq_last_stats()
        x = xd.cpu().numpy().view(np.complex128)
        assert g.oracle.true_residual(b, x, 0.05)[0] <= TOL * SLACK
        assert stats.dslash_launches >= 2 * stats.max_iterations and stats.dslash_ms > 0


def test_plain_fp64_cg_on_lower_precision_links():
    """inner_prec FP64 with links packed in FP16 runs on the handle's FP64 copy."""
    dims = (8, 10, 8, 6)
    with gpu(dims, 2) as g:
        b = hi.gaussian_rhs(g.lat, 9)
        x, stats, iters, res = _solve(g, [b], 0.05, inner_prec=0)
        assert g.oracle.true_residual(b, x[0], 0.05)[0] <= TOL * SLACK
        _, it_oracle, _ = g.oracle.cg(b, 0.05, TOL)
        assert abs(int(iters[0]) - it_oracle) <= 2


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("single_reduction", [0, 1])
def test_persistent_matches_graph_iterations(prec, single_reduction):
    """The persistent kernel runs the algorithm of the graph driver -- in Hestenes-Stiefel form,
    or in the single-reduction form that is the same CG in exact arithmetic -- with the same
    iteration counts and reliable updates up to rounding, and meets the FP64 true residual."""
    dims = (8, 10, 8, 6)
    with gpu(dims, prec) as g:
        rhs = [hi.gaussian_rhs(g.lat, 60 + k) for k in range(4)]
        _, s1, it1, _ = _solve(g, rhs, 0.05, inner_prec=prec, use_graph=1, bundle=4)
        x2, s2, it2, _ = _solve(g, rhs, 0.05, inner_prec=prec, use_graph=2, bundle=4,
                                single_reduction=single_reduction)
        # the persistent kernel sums its dots in another block order, and the single-reduction
        # form rounds differently
        slack = 1 if (prec < 2 and not single_reduction) else 3
        assert np.all(np.abs(it1.astype(int) - it2.astype(int)) <= slack), (it1, it2)
        assert abs(s1.reliable_updates - s2.reliable_updates) <= len(rhs) * slack
        assert s2.kernel_launches == 3
        true = g.oracle.true_residual(np.stack(rhs), x2, 0.05)
        assert np.all(true <= TOL * SLACK)


def test_persistent_barrier_timeout_is_reported_and_context_survives():
    """Failure detection without a fault: the test hook makes every grid barrier wait for a block
    that does not exist; the bounded waits run out, the kernel returns, the solve reports
    HISQ_ERR_TIMEOUT, and the same context then solves normally."""
    dims = (8, 8, 8, 4)
    with gpu(dims, 1) as g:
        b = hi.gaussian_rhs(g.lat, 0)
        p = g.hisq.hisq_default_solver_params()
        p.use_graph = 2
        p.debug_barrier_timeout = 1
        g.hisq.hisq_set_solver_params(p)
        x = np.zeros_like(b)
        rc = g.hisq.hisq_cg_solve(g.fat, g.naik, [b], [x], 0.1, TOL, raise_on_error=False)
        assert rc == -6
        x, stats, iters, res = _solve(g, [b], 0.1, inner_prec=1, use_graph=2)
        assert g.oracle.true_residual(b, x[0], 0.1)[0] <= TOL * SLACK


def test_persistent_kernel_timing_and_phases():
    """time_kernels with the persistent driver: one CUDA-event-timed kernel per bundle, and the
    per-phase times from inside the kernel fill most of it without exceeding it."""
    dims = (8, 10, 8, 6)
    with gpu(dims, 2) as g:
        rhs = [hi.gaussian_rhs(g.lat, 70 + k) for k in range(3)]
        x, s, iters, _ = _solve(g, rhs, 0.05, inner_prec=2, use_graph=2, time_kernels=1, bundle=2)
        assert s.bundles == 2 and s.solve_kernel_launches == 2 and s.solve_kernel_ms > 0
        ph = list(s.phase_ms)
        assert all(v >= 0 for v in ph) and ph[0] > 0 and ph[1] > 0 and ph[3] > 0
        assert sum(ph) <= s.solve_kernel_ms * 1.01
        assert np.all(g.oracle.true_residual(np.stack(rhs), x, 0.05) <= TOL * SLACK)


def test_bundle_size_chosen_by_the_autotuner():
    """bundle = 0: the tuner's split of nrhs into bundles; with autotune off, the largest bundle.
    Either way every right-hand side reaches the FP64 true residual."""
    dims = (8, 10, 8, 6)
    with gpu(dims, 2) as g:
        rhs = [hi.gaussian_rhs(g.lat, 90 + k) for k in range(6)]
        x, s, _, res = _solve(g, rhs, 0.05, inner_prec=2, bundle=0)
        assert s.bundle_size in (1, 2, 4, 6) and s.bundles == -(-6 // s.bundle_size)
        assert s.converged == 6 and np.all(res <= TOL)
        x, s, _, res = _solve(g, rhs, 0.05, inner_prec=2, bundle=0, autotune=0)
        assert s.bundle_size == 6 and s.bundles == 1 and s.converged == 6
        assert np.all(g.oracle.true_residual(np.stack(rhs), x, 0.05) <= TOL * SLACK)


def test_graph_reused_after_persistent_solves():
    """Alternating drivers in one context: the captured graph is rebuilt once and then reused
    after persistent-kernel solves have rewritten the host copy of the bundle state (the graph's
    loop ends only through its own conditional handles, which live with the graph)."""
    dims = (8, 10, 8, 6)
    with gpu(dims, 1) as g:
        b = hi.gaussian_rhs(g.lat, 95)
        its = []
        for driver in (1, 2, 1, 2, 1):
            x, s, iters, res = _solve(g, [b], 0.05, inner_prec=1, use_graph=driver, bundle=1)
            assert s.converged == 1 and res[0] <= TOL, driver
            its.append(int(iters[0]))
        assert its[0] == its[2] == its[4]
        assert g.oracle.true_residual(b, x[0], 0.05)[0] <= TOL * SLACK


def test_l2_resident_links_do_not_change_the_solve():
    """With and without the persisting L2 window over the Naik links (32^3 x 8 FP16 fits the
    set-aside): the same iterations and both at the FP64 true residual; repeated solves release
    the window in between."""
    dims = (32, 32, 32, 8)
    with gpu(dims, 2) as g:
        b = hi.gaussian_rhs(g.lat, 77)
        runs = []
        for l2 in (1, 0, 1):
            x, stats, iters, res = _solve(g, [b], 0.01, inner_prec=2, l2_persist_links=l2)
            assert res[0] <= TOL
            runs.append(int(iters[0]))
        assert max(runs) - min(runs) <= 1
        assert g.oracle.true_residual(b, x[0], 0.01)[0] <= TOL * SLACK


def test_reliable_update_threshold_by_precision():
    """delta = 0 (the default) takes the threshold of the inner precision (FP16: 0.03); an explicit
    delta in (0, 1) overrides it; other values are rejected.  Every variant meets the oracle's true
    residual, and the smaller FP16 default recomputes no more often than 0.1."""
    dims = (8, 10, 8, 6)
    mass = 0.05
    with gpu(dims, 2) as g:
        assert g.hisq.hisq_default_solver_params().delta == 0.0
        p = g.hisq.hisq_default_solver_params()
        for bad in (1.0, -0.1, 1.5):
            p.delta = bad
            with pytest.raises(g.hisq.HisqError):
                g.hisq.hisq_set_solver_params(p)
        rhs = [hi.gaussian_rhs(g.lat, k) for k in range(2)]
        updates = {}
        for delta in (0.0, 0.1):
            x, stats, iters, res = _solve(g, rhs, mass, inner_prec=2, delta=delta)
            true = g.oracle.true_residual(np.stack(rhs), x, mass)
            assert np.all(true <= TOL * SLACK), (delta, true)
            assert stats.converged == 2
            updates[delta] = stats.reliable_updates
        assert updates[0.0] <= updates[0.1], updates


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("dims,n", [((4, 4, 4, 4), 1), ((4, 4, 4, 6), 5), ((8, 8, 8, 4), 3), ((8, 10, 8, 6), 9),
                                    ((8, 10, 8, 6), 10)])
def test_four_lanes_per_site_on_small_lattices(prec, dims, n):
    """The persistent solve with four lanes per site and right-hand side: fewer sites than blocks, thread
    positions that are no power of two, the last bundle it takes on 152 SMs (13 sites x 9) and the first
    it does not; both CG forms, uneven norms."""
    with gpu(dims, prec) as g:
        rhs = [hi.gaussian_rhs(g.lat, 60 + k) * 10.0 ** (k % 4 - 2) for k in range(n)]
        for single in (0, 1):
            x, stats, iters, res = _solve(g, rhs, 0.1, inner_prec=prec, bundle=n, single_reduction=single)
            true = g.oracle.true_residual(np.stack(rhs), x, 0.1)
            assert np.all(true <= TOL * SLACK), (single, true)


@pytest.mark.parametrize("prec,dims,n", [(0, (4, 4, 4, 4), 1), (0, (6, 4, 6, 4), 3), (0, (8, 8, 8, 4), 4),
                                         (0, (8, 8, 8, 4), 5), (1, (4, 4, 4, 4), 1), (1, (8, 8, 8, 4), 9),
                                         (1, (8, 8, 8, 4), 10)])
def test_a_lane_per_link_group_on_small_lattices(prec, dims, n):
    """The persistent solve with 16 (FP64) and 8 (FP32) lanes per site and right-hand side: sites and
    right-hand sides whose lanes do not fill the warps, the last bundles taken on 152 SMs (seven sites x 4,
    x 9) and the first that go back to four lanes; both CG forms, uneven norms."""
    with gpu(dims, prec) as g:
        rhs = [hi.gaussian_rhs(g.lat, 80 + k) * 10.0 ** (k % 4 - 2) for k in range(n)]
        for single in (0, 1):
            x, stats, iters, res = _solve(g, rhs, 0.1, inner_prec=prec, bundle=n, single_reduction=single)
            true = g.oracle.true_residual(np.stack(rhs), x, 0.1)
            assert np.all(true <= TOL * SLACK), (single, true)


@pytest.mark.parametrize("prec,n", [(1, 1), (1, 4), (2, 1), (2, 4), (3, 4)])
@pytest.mark.parametrize("single_reduction", [0, 1])
def test_dots_whose_running_sums_pass_the_float_range(prec, n, single_reduction):
    """Right-hand sides of size 4e17: the |A p|^2 and |r|^2 of a site fit a float (1e38), their sums over a
    thread's sites and a warp's lanes do not; they are FP64."""
    dims, mass = (16, 16, 16, 8), 0.1
    with gpu(dims, prec) as g:
        rhs = [4e17 * hi.gaussian_rhs(g.lat, 900 + k) for k in range(n)]
        x, stats, iters, res = _solve(g, rhs, mass, inner_prec=prec, bundle=n, single_reduction=single_reduction)
        assert np.all(g.oracle.true_residual(np.stack(rhs), x, mass) <= TOL * SLACK)
