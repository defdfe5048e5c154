"""The one-launch forms of CG and BiCGSTAB on right-hand sides scaled by powers
of two so small or large that the inverse of an inner product leaves the
normal range of FP64 while the quotients that make up beta do not.  Scaling by
a power of two changes no rounding of a solve as long as nothing underflows, so
the scaled solve has to converge wherever the graph form does and to the same
accuracy as the unscaled one.  (BiCGSTAB without a preconditioner at 2^505 is
past the range itself: t.t overflows, and the graph form stops with NaN.)"""
import numpy as np
import pytest

import workloads as W
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


# 64^2: r.z falls below 5.6e-309 in the last iterations at 2^-485; 256^2 at 2^-489
@pytest.mark.parametrize("side,exponent", [(64, -485), (64, -480), (64, 500), (64, 505), (256, -489), (256, 500)])
@pytest.mark.parametrize("kind,prec", [("cg", 0), ("cg", 1), ("bicgstab", 0), ("bicgstab", 1)])
def test_scaled_right_hand_sides(gk, orc, side, exponent, kind, prec):
    A = W.poisson2d(side)
    b = W.uniform_vector(side * side, 3)
    M = gk.Matrix(*[to_dev(a) for a in A])
    P = gk.Precond(M, 1) if prec else None
    scaled = to_dev(np.ldexp(b, exponent))
    out = []
    for check_every in (-1, 0):
        S = gk.Solver(M, P, kind, max_iters=4000, reduction_factor=1e-10, check_every=check_every)
        x = to_dev(np.zeros(b.size))
        st = gk.solve(S, scaled, x)
        out.append(st)
        if out[0].stop_reason == gk.STOP_NAN and (kind, prec, exponent) == ("bicgstab", 0, 505):
            continue
        assert st.stop_reason == gk.STOP_CONVERGED, (check_every, st)
        # scaled back exactly; the bar of the other solver tests
        assert np.linalg.norm(b - orc.spmv(A, np.ldexp(to_np(x), -exponent))) <= 1.5e-10 * np.linalg.norm(b)
    assert out[0].form == gk.FORM_GRAPH and out[1].form == (gk.FORM_CLUSTER if side == 64 else gk.FORM_GRID)
    if out[0].stop_reason == gk.STOP_CONVERGED:
        slack = max(2, out[0].iters * 3 // 100) if kind == "cg" else max(3, out[0].iters // 4)
        assert abs(out[1].iters - out[0].iters) <= slack, (out[1].iters, out[0].iters)
