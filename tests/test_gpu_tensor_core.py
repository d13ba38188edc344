"""The tensor-core Dslash of 16-bit bundles (one warp per site) against the FP64 oracle: operator,
fused dots and the persistent solve, at the edges of its runs, row groups and right-hand-side groups."""
import numpy as np
import pytest

import hisq_inputs as hi
from gpu_util import MMA_PHASES, PREC_TOL, gpu, rel_err

pytestmark = pytest.mark.gpu

LANES = 32  # lanes per site: the shape that selects this kernel


def _rhs(lat, n, seed=0):
    return np.stack([hi.gaussian_rhs(lat, seed + k) for k in range(n)])


# rows of 2, 4, 5, 6 and 8 sites (worked on 2, 4, 1, 2 and 4 at a time); the last group of eight rows short at
# 10 x 6 x 6 x 6 and 12 x 4 x 4 x 6; runs longer than a row, equal to one, and several to a row
@pytest.mark.parametrize("dims,run", [((4, 4, 4, 4), 16), ((8, 10, 8, 4), 4), ((10, 6, 6, 6), 2), ((12, 4, 8, 6), 1),
                                      ((12, 4, 4, 6), 4), ((16, 6, 4, 4), 4)])
@pytest.mark.parametrize("prec,n", [(2, 2), (2, 5), (2, 8), (2, 16), (2, 17), (2, 32), (3, 2), (3, 8), (3, 12), (3, 16), (3, 30)])
def test_operator(dims, run, prec, n):
    mass = 0.2
    with gpu(dims, prec) as g:
        g.hisq.hisq_set_launch_shape(prec, 18, n, 1, 32 * run, LANES)
        v = _rhs(g.lat, n, 700)
        vin, vout = g.pack(v), g.bundle(n)
        for parity in (0, 1):
            vout.zero_()
            g.hisq.hisq_dslash(g.fat, g.naik, vin, vout, n, parity)
            assert rel_err(g.unpack(vout, n), g.oracle.dslash_eo(v, parity)) <= PREC_TOL[prec], parity
        pap = np.zeros(n)
        g.hisq.hisq_aop(g.fat, g.naik, mass, vin, vout, n, pap)
        assert rel_err(g.unpack(vout, n), g.oracle.aop(v, mass)) <= 2 * PREC_TOL[prec]
        vq = g.unpack(vin, n)
        want = np.array([np.vdot(vq[k], g.oracle.aop(vq[k], mass)).real for k in range(n)])
        assert np.max(np.abs(pap - want) / want) <= 4 * PREC_TOL[prec]


@pytest.mark.parametrize("prec,n", [(2, 2), (2, 9), (2, 16), (3, 10), (3, 16)])
@pytest.mark.parametrize("single_reduction", [0, 1])
def test_persistent_solve(prec, n, single_reduction):
    dims, mass, tol = (8, 10, 8, 6), 0.05, 1e-10
    with gpu(dims, prec) as g:
        g.hisq.hisq_set_launch_shape(prec, 18, n, 1, 128, LANES)
        p = g.hisq.hisq_default_solver_params()
        p.inner_prec, p.bundle, p.single_reduction = prec, n, single_reduction
        g.hisq.hisq_set_solver_params(p)
        rhs = list(_rhs(g.lat, n, 720))
        rhs[1] = rhs[1] * 1e-3
        xs = [np.zeros_like(b) for b in rhs]
        g.hisq.hisq_cg_solve(g.fat, g.naik, rhs, xs, mass, tol)
        assert np.all(g.oracle.true_residual(np.stack(rhs), np.stack(xs), mass) <= tol)


# The tensor-core phases of the persistent solve themselves: bundle sizes that take them (test_host_logic.py
# checks that they do), with persistent_threads = 512, so that no small lattice is split over more lanes.
# Rows of 4 and 8 sites (worked on 4 at a time; 16 right-hand sides with a layout known at compile time),
# of 6 (2 at a time) and of 5 (one at a time); the last row group short at 10 x 6 x 6 x 6.
@pytest.mark.parametrize("dims", [(8, 10, 8, 6), (16, 6, 4, 4), (12, 6, 6, 6), (10, 6, 6, 6)])
@pytest.mark.parametrize("prec,n", [(p, n) for p in MMA_PHASES for n in MMA_PHASES[p]])
@pytest.mark.parametrize("single_reduction", [0, 1])
def test_persistent_phases(dims, prec, n, single_reduction):
    mass, tol = 0.05, 1e-10
    with gpu(dims, prec) as g:
        g.hisq.hisq_set_launch_shape(prec, 18, n, 1, 128, LANES)
        p = g.hisq.hisq_default_solver_params()
        p.inner_prec, p.bundle, p.single_reduction, p.persistent_threads = prec, n, single_reduction, 512
        g.hisq.hisq_set_solver_params(p)
        rhs = list(_rhs(g.lat, n, 740))
        rhs[1] = rhs[1] * 1e-3
        rhs[2] = g.oracle.aop(g.oracle.aop(rhs[2], mass), mass)  # converges earlier than the others
        rhs[n - 2] = np.zeros_like(rhs[0])                       # never active
        xs = [np.full_like(b, 7.0) for b in rhs]
        g.hisq.hisq_cg_solve(g.fat, g.naik, rhs, xs, mass, tol)
        some = [k for k in range(n) if k != n - 2]
        res = g.oracle.true_residual(np.stack([rhs[k] for k in some]), np.stack([xs[k] for k in some]), mass)
        assert np.all(res <= tol) and not np.any(xs[n - 2])


# The fused dots of this kernel and of a SIMT one on the same packed input.  Both sum exact products of the
# stored values in FP32 accumulators, 48 per component of D and a few scales, the tensor core with its own
# rounding (towards zero, one unit of 2^-23 for each addition at the most): a component is off by at most
# 48 2^-23 = 6e-6 of its terms' size, a dot by the part of that which all components have in common.  The
# stored intermediate differs where such a difference crosses a rounding boundary of the storage (one component
# in thousands, by one unit in the last place, of random sign).  1e-5 of the dot holds both; the storage
# tolerance above is a thousand times wider.
@pytest.mark.parametrize("dims", [(8, 10, 8, 4), (12, 4, 8, 6), (10, 6, 6, 6)])
@pytest.mark.parametrize("prec,n", [(2, 9), (2, 16), (3, 10), (3, 16)])
def test_fused_dots_agree_with_the_simt_kernel(dims, prec, n):
    mass = 0.1
    with gpu(dims, prec) as g:
        vin, vout = g.pack(_rhs(g.lat, n, 760)), g.bundle(n)
        dots = []
        for shape in ((1, 128, LANES), (1, 128, 1)):
            g.hisq.hisq_set_launch_shape(prec, 18, n, *shape)
            dots.append(np.zeros(n))
            g.hisq.hisq_aop(g.fat, g.naik, mass, vin, vout, n, dots[-1])
        assert np.max(np.abs(dots[0] / dots[1] - 1.0)) <= 1e-5


def test_shape_round_trip_and_validation():
    """The tuner's shape can be pinned again; what the kernel cannot take is refused."""
    from paper_1409_1510_gb300.hisq import HisqError
    with gpu((16, 16, 16, 8), 2) as g:
        h = g.hisq
        for n in (1, 2, 8, 16):
            h.hisq_set_launch_shape(2, 18, n, *h.hisq_autotune(g.fat, g.naik, n))
        for bad in ((1, 18, 16, 1, 128, 32), (2, 13, 16, 1, 128, 32), (2, 18, 16, 2, 128, 32), (2, 18, 1, 1, 128, 32),
                    (2, 18, 33, 1, 128, 32), (3, 18, 9, 1, 128, 32), (2, 18, 16, 1, 2048, 32)):
            with pytest.raises(HisqError):
                h.hisq_set_launch_shape(*bad)
