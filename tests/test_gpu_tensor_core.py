"""The tensor-core Dslash of 16-bit bundles (one warp per site) against the FP64 oracle: operator,
fused dots and the persistent solve, at the edges of its runs, row groups and right-hand-side groups."""
import numpy as np
import pytest

import hisq_inputs as hi
from gpu_util import PREC_TOL, gpu, rel_err

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
