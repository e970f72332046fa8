"""GPU parity of gauge_force (Wilson and Iwasaki rectangles) and of the action/plaquette."""
import numpy as np
import pytest

import oracle
from gpu_util import dev, host, rel_l2, torch_cuda
from paper_2112_04556_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (5, 3, 4, 7), (3, 4, 3, 6)])
@pytest.mark.parametrize("c1", [0.0, -0.331])
def test_gauge_force_parity(L, c1):
    import paper_2112_04556_gb300 as rm
    U = inputs.random_links(L, eps=0.6, seed=11)
    ref = oracle.gauge_force(L, U, 6.0, c1)
    S_ref, pl_ref = oracle.action(L, U, 6.0, c1)
    with rm.Context(L) as ctx:
        Ud = dev(U)
        F, S, pl = rm.gauge_force(ctx, Ud, 6.0, c1, prec=rm.FP64)
        assert rel_l2(host(F), ref) <= 1e-12
        assert abs(S - S_ref) <= 1e-12 * abs(S_ref) and abs(pl - pl_ref) <= 1e-13
        F32, S32, _ = rm.gauge_force(ctx, None, 6.0, c1, prec=rm.FP32)
        assert rel_l2(host(F32), ref) <= 1e-5
        assert abs(S32 - S_ref) <= 1e-12 * abs(S_ref)     # the action is always float64


def test_gauge_unit_links():
    import paper_2112_04556_gb300 as rm
    L = (4, 4, 4, 6)
    with rm.Context(L) as ctx:
        F, S, pl = rm.gauge_force(ctx, dev(inputs.unit_links(L)), 6.0, -0.331)
        assert np.abs(host(F)).max() == 0.0 and S == 0.0 and abs(pl - 1.0) < 1e-15


@pytest.mark.parametrize("L,c1", [((32, 32, 32, 32), 0.0), ((16, 16, 16, 16), -0.331)])
def test_gauge_force_full_size_sampled(L, c1):
    import paper_2112_04556_gb300 as rm
    U = inputs.random_links(L, eps=0.3, seed=0)
    V = int(np.prod(L))
    rng = np.random.default_rng(3)
    sites = np.unique(np.concatenate([rng.integers(0, V, 600), [0, V - 1]]))
    ref = oracle.gauge_force_sites(L, U, 6.0, c1, sites)
    with rm.Context(L) as ctx:
        F, S, pl = rm.gauge_force(ctx, dev(U), 6.0, c1, prec=rm.FP64)
        assert rel_l2(host(F)[sites], ref) <= 1e-12
        F32, _, _ = rm.gauge_force(ctx, None, 6.0, c1, prec=rm.FP32)
        assert rel_l2(host(F32)[sites], ref) <= 1e-5
    if L == (16, 16, 16, 16):
        S_ref, pl_ref = oracle.action(L, U, 6.0, c1)
        assert abs(S - S_ref) <= 1e-12 * abs(S_ref) and abs(pl - pl_ref) <= 1e-13


@pytest.mark.parametrize("L", [(2, 2, 2, 2), (5, 3, 4, 7), (2, 3, 33, 2)])
@pytest.mark.parametrize("c1", [0.0, -0.331])
def test_staples_and_loops(L, c1):
    """The staples of each link (the form above 2^22 sites and without memory for the loops) and the shared loops
    against the oracle and each other, both precisions, with the bounds of the parity test."""
    import paper_2112_04556_gb300 as rm
    U = inputs.random_links(L, eps=0.6, seed=12)
    ref = oracle.gauge_force(L, U, 6.0, c1)
    S_ref, pl_ref = oracle.action(L, U, 6.0, c1)
    with rm.Context(L) as ctx:
        for loops in (0, 1, 0):
            rm.set_stencil_shape(ctx, rm.SHAPE_LOOPS, rm.FP64, 18, loops, 128)
            rm.counters(ctx, reset=True)
            F, S, pl = rm.gauge_force(ctx, dev(U), 6.0, c1, prec=rm.FP64)
            if not loops:   # links, staples, action
                assert rm.counters(ctx)["launches"] == 3
            assert rel_l2(host(F), ref) <= 1e-12
            assert abs(S - S_ref) <= 1e-12 * abs(S_ref) and abs(pl - pl_ref) <= 1e-13
            F32, S32, _ = rm.gauge_force(ctx, None, 6.0, c1, prec=rm.FP32)
            assert rel_l2(host(F32), ref) <= 1e-5 and abs(S32 - S_ref) <= 1e-12 * abs(S_ref)
        for bad in ((rm.FP32, 18, 1, 128), (rm.FP64, 12, 1, 128), (rm.FP64, 18, 2, 128), (rm.FP64, 18, 1, 64)):
            for kernel in (rm.SHAPE_LOOPS, rm.SHAPE_TABLE):
                with pytest.raises(rm.RmhmcError):
                    rm.set_stencil_shape(ctx, kernel, *bad)


def _single(U):
    return U.astype(np.complex64).astype(np.complex128)


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (5, 3, 4, 7)])
@pytest.mark.parametrize("c1", [0.0, -0.331])
def test_links_that_are_not_unitary(L, c1):
    """float64 force and action of links read from single precision (U U^dag off by 1e-7), of scaled links and, in the same
    context, of SU(3) ones: the derivative of the action of the matrices given, as the oracle's staples have it."""
    import paper_2112_04556_gb300 as rm
    U = inputs.random_links(L, eps=0.6, seed=13)
    with rm.Context(L) as ctx:
        for V in (U, _single(U), 1.001 * U, U):
            ref = oracle.gauge_force(L, V, 6.0, c1)
            S_ref, pl_ref = oracle.action(L, V, 6.0, c1)
            for links in (dev(V), None):   # looked at, and known
                F, S, pl = rm.gauge_force(ctx, links, 6.0, c1, prec=rm.FP64)
                assert rel_l2(host(F), ref) <= 1e-12
                assert abs(S - S_ref) <= 1e-12 * abs(S_ref) and abs(pl - pl_ref) <= 1e-13
            F32, S32, _ = rm.gauge_force(ctx, dev(V), 6.0, c1, prec=rm.FP32)
            assert rel_l2(host(F32), ref) <= 1e-5 and abs(S32 - S_ref) <= 1e-12 * abs(S_ref)


def test_force_alone_of_links_that_are_not_unitary():
    """The same where only the force is asked for (nothing of the call is read back), in the gradient flow and in the
    trajectory's graph, whose forces run on links derived from the caller's."""
    import paper_2112_04556_gb300 as rm
    L = (4, 4, 4, 6)
    U = _single(inputs.random_links(L, eps=0.4, seed=14))
    with rm.Context(L) as ctx:
        F = dev(np.zeros((int(np.prod(L)), 4, 8)))
        ctx.check(rm.lib().gauge_force(ctx.h, dev(U).data_ptr(), 6.0, -0.331, rm.FP64, F.data_ptr(), None, None,
                                       rm._raw_stream()))
        assert rel_l2(host(F), oracle.gauge_force(L, U, 6.0, -0.331)) <= 1e-12
        W, E = oracle.wilson_flow(L, U, 0.02, 3)
        for energies in (True, False):
            Ud = dev(U)
            e = np.zeros(4)
            p = e.ctypes.data_as(rm.ctypes.POINTER(rm.ctypes.c_double)) if energies else None
            ctx.check(rm.lib().wilson_flow(ctx.h, Ud.data_ptr(), 0.02, 3, rm.FP64, p, rm._raw_stream()))
            assert np.abs(host(Ud) - W).max() <= 1e-12
            if energies:
                assert np.abs(e - E).max() <= 1e-11
        P = inputs.gaussian_fields(L, 1, seed=15)[0]
        par = rm.make_params(beta=6.0, c1=-0.331, mass=rm.mass_fit(12, 0.9), tau=0.1, nsteps=2, tol_md=1e-7, tol_h=1e-10,
                             fp_tol=1e-7, fp_maxit=50, maxiter=400, prec=rm.MIXED, fg_fp64=1, metropolis=False)
        out = []
        for loops in (1, 0):   # 1: the default, which has to see that these links need the staples
            rm.set_stencil_shape(ctx, rm.SHAPE_LOOPS, rm.FP64, 18, loops, 128)
            Ud, Pd = dev(U), dev(P)
            rm.md(ctx, Ud, Pd, par)
            out.append((host(Ud), host(Pd)))
        assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("shift,loops", [(2.0 ** -46, True), (2.0 ** -42, False)])
def test_where_links_count_as_unitary(shift, loops):
    """Links scaled by 1 + shift are off by 2 shift; from 2^-43 on they take the staples (two kernels, where the loops of
    the Iwasaki action take four)."""
    import paper_2112_04556_gb300 as rm
    L = (4, 6, 4, 4)
    U = inputs.random_links(L, eps=0.6, seed=16) * (1.0 + shift)
    with rm.Context(L) as ctx:
        rm.gauge_force(ctx, dev(U), 6.0, -0.331)
        rm.counters(ctx, reset=True)
        rm.gauge_force(ctx, None, 6.0, -0.331)
        assert rm.counters(ctx)["launches"] == (4 if loops else 2)


@pytest.mark.parametrize("shift,loops32,loops64", [(0.0, True, True), (2.0 ** -23, True, False), (2.0 ** -19, False, False)])
@pytest.mark.parametrize("first", [0, 1])
def test_where_links_count_as_unitary_in_float32(shift, loops32, loops64, first):
    """The float32 force of links off by 2 shift shares its loops up to 2^-20, whatever was asked before it: a float64
    force (first = 0) or nothing.  The Iwasaki force takes four kernels from loops and one from staples; both are within
    float32 rounding of the oracle's."""
    import paper_2112_04556_gb300 as rm
    L = (4, 6, 4, 4)
    U = inputs.random_links(L, eps=0.6, seed=17) * (1.0 + shift)
    ref = oracle.gauge_force(L, U, 6.0, -0.331)
    S_ref, _ = oracle.action(L, U, 6.0, -0.331)
    with rm.Context(L) as ctx:
        if first == 0:
            F64, S64, _ = rm.gauge_force(ctx, dev(U), 6.0, -0.331, prec=rm.FP64)
            assert rel_l2(host(F64), ref) <= 1e-12
        else:
            rm.set_links(ctx, dev(U))
        F32, S, _ = rm.gauge_force(ctx, None, 6.0, -0.331, prec=rm.FP32)
        assert rel_l2(host(F32), ref) <= 1e-5 and abs(S - S_ref) <= 1e-12 * abs(S_ref)
        for prec, loops in ((rm.FP32, loops32), (rm.FP64, loops64)):
            F = dev(np.zeros((int(np.prod(L)), 4, 8)))
            rm.counters(ctx, reset=True)
            ctx.check(rm.lib().gauge_force(ctx.h, None, 6.0, -0.331, prec, F.data_ptr(), None, None, rm._raw_stream()))
            assert rm.counters(ctx)["launches"] == (4 if loops else 1), prec
            assert rel_l2(host(F), ref) <= (1e-12 if prec == rm.FP64 else 1e-5)
