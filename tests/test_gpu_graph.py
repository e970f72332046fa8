"""The mixed-precision molecular dynamics as one CUDA graph (conditional WHILE nodes for both implicit fixed
points and every Krylov run, decided on the device) against the host-driven path on the same inputs."""
import numpy as np
import pytest

import oracle

from gpu_util import dev, host, rel_l2, torch_cuda
from paper_2112_04556_gb300 import inputs

pytestmark = pytest.mark.gpu


def _params(rm, m, **kw):
    d = dict(beta=6.0, c1=0.0, mass=m, tau=0.2, nsteps=4, tol_md=1e-6, tol_h=1e-12, fp_tol=1e-6, fp_maxit=50,
             maxiter=400, prec=rm.MIXED, seed=5, traj_index=0, metropolis=False)
    d.update(kw)
    return rm.make_params(**d)


@pytest.mark.parametrize("L,c1", [((8, 8, 8, 8), 0.0), ((6, 4, 6, 8), -0.331)])
def test_md_graph_matches_host_driven(L, c1):
    import paper_2112_04556_gb300 as rm
    U = inputs.random_links(L, eps=0.3, seed=71)
    P = inputs.gaussian_fields(L, 1, seed=72)[0]
    m = rm.mass_fit(12, 0.9)
    out = {}
    for graphs in (False, True):
        with rm.Context(L) as ctx:
            rm.set_graphs(ctx, graphs)
            Ud, Pd = dev(U), dev(P)
            r = rm.md(ctx, Ud, Pd, _params(rm, m, c1=c1))
            out[graphs] = (host(Ud), host(Pd), r, rm.tuning(ctx))
    assert "md graph captured" in out[True][3], out[True][3]
    assert np.abs(out[True][0] - out[False][0]).max() <= 1e-9
    assert rel_l2(out[True][1], out[False][1]) <= 1e-8
    assert out[True][2]["fp_iters_p"] == out[False][2]["fp_iters_p"]
    assert out[True][2]["fp_iters_u"] == out[False][2]["fp_iters_u"]
    assert abs(out[True][2]["md_iters"] - out[False][2]["md_iters"]) <= 2


def test_trajectory_graph_reused_and_reversible():
    """The cached graph is reused across trajectories; forward, momentum flip, forward returns to the start."""
    import paper_2112_04556_gb300 as rm
    L = (8, 8, 8, 8)
    U = inputs.random_links(L, eps=0.3, seed=73)
    P = inputs.gaussian_fields(L, 1, seed=74)[0]
    m = rm.mass_fit(12, 0.9)
    with rm.Context(L) as ctx:
        Ud, Pd = dev(U), dev(P)
        p = _params(rm, m, tol_md=1e-7, fp_tol=1e-7)
        rm.md(ctx, Ud, Pd, p)
        Pd.neg_()
        rm.md(ctx, Ud, Pd, p)
        assert "md graph captured" in rm.tuning(ctx)
        assert np.abs(host(Ud) - U).max() <= 1e-5
        for k in range(3):
            r = rm.rmhmc_trajectory(ctx, Ud, _params(rm, m, traj_index=k))
            assert np.isfinite(r["dH"]) and r["md_iters"] > 0


def test_graph_fixed_point_cap_reports_noconv():
    import paper_2112_04556_gb300 as rm
    L = (4, 4, 4, 4)
    U = inputs.random_links(L, eps=0.3, seed=75)
    P = inputs.gaussian_fields(L, 1, seed=76)[0]
    with rm.Context(L) as ctx:
        with pytest.raises(rm.RmhmcError) as e:
            rm.md(ctx, dev(U), dev(P), _params(rm, rm.mass_fit(12, 0.9), fp_maxit=1, fp_tol=1e-15))
        assert e.value.code == rm.ENOCONV


@pytest.mark.parametrize("logdet", [0, 1])
def test_wait_that_runs_out_ends_the_graph(logdet):
    """A Krylov run whose barrier gives up (a wait limit of no polls) ends the captured trajectory: each of the 2 x 4 fixed
    points stops after its first pass, the call returns ETIMEOUT with the links as they were, and with the limit
    back the context gives the trajectory it gave before."""
    import ctypes
    import paper_2112_04556_gb300 as rm
    L = (8, 8, 8, 8)
    U = inputs.random_links(L, eps=0.3, seed=77)
    P = inputs.gaussian_fields(L, 1, seed=78)[0]
    m = rm.mass_fit(12, 0.9)
    p = _params(rm, m, logdet=logdet)
    with rm.Context(L) as ctx:
        def trajectory():
            Ud = dev(U)
            r = rm.rmhmc_trajectory(ctx, Ud, p)
            return host(Ud), r
        want, r = trajectory()
        assert "md graph captured" in rm.tuning(ctx)
        rm.set_wait_limit(ctx, 0)
        Ud, Pd, res = dev(U), dev(P), rm.Result()
        code = rm.lib().rmhmc_md(ctx.h, Ud.data_ptr(), Pd.data_ptr(), ctypes.byref(p), ctypes.byref(res), None)
        assert code == rm.ETIMEOUT
        assert res.fp_iters_p == 4 and res.fp_iters_u == 4
        Ud = dev(U)
        with pytest.raises(rm.RmhmcError) as e:
            rm.rmhmc_trajectory(ctx, Ud, p)
        assert e.value.code == rm.ETIMEOUT and np.array_equal(host(Ud), U)
        rm.set_wait_limit(ctx)
        again, r2 = trajectory()
    assert np.array_equal(again, want) and r2["dH"] == r["dH"]


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (5, 3, 4, 7)])
def test_graph_of_the_callers(L):
    """Calls captured into the caller's own graph read the links of the replay: float64 stencil, link derivative and force,
    with the links set between replays, and with an import in the graph, after which
    the context's other calls see the links of the last replay too.  Bounds of the parity tests."""
    import paper_2112_04556_gb300 as rm
    torch = torch_cuda()
    Us = [inputs.random_links(L, eps=0.5, seed=s) for s in (81, 82)]
    X, Z = inputs.gaussian_fields(L, 2, seed=84)
    m = rm.mass_fit(12, 0.9)
    with rm.Context(L) as ctx:
        Ud, Xd, Zd = dev(Us[0]), dev(X), dev(Z)
        Y, G, F = (torch.empty_like(Xd) for _ in range(3))

        def calls(links=None):
            rm.lap_apply(ctx, links, Xd, Y)
            rm.lap_link_grad(ctx, None, Xd, Zd, [0.7], G=G)
            ctx.check(rm.lib().gauge_force(ctx.h, None, 6.0, -0.331, rm.FP64, F.data_ptr(), None, None, rm._raw_stream()))

        def check(U):
            assert rel_l2(host(Y), oracle.lap(L, U, X)) <= 1e-12
            assert rel_l2(host(G), oracle.lap_link_grad(L, U, X, Z, [0.7])) <= 1e-12
            assert rel_l2(host(F), oracle.gauge_force(L, U, 6.0, -0.331)) <= 1e-12

        calls(Ud)
        check(Us[0])
        held, bringing = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(held):
            calls()
        for U in Us + Us[:1]:
            rm.set_links(ctx, dev(U))
            for t in (Y, G, F):
                t.zero_()
            held.replay()
            torch.cuda.synchronize()
            check(U)
        rm.set_links(ctx, dev(Us[1]))
        calls()                     # outside the graph again: table and loops of the present links
        check(Us[1])
        with torch.cuda.graph(bringing):
            calls(Ud)
        for U in (Us[1], Us[0]):
            Ud.copy_(dev(U))
            bringing.replay()
            torch.cuda.synchronize()
            check(U)
            for t in (Y, G, F):
                t.zero_()
            calls()
            check(U)
            y, _, _, resid = rm.rat_mass_solve(ctx, None, Xd, m, tol=1e-11, prec=rm.MIXED)
            assert np.all(resid <= 1e-11)
            assert rel_l2(host(y), oracle.rational_apply(L, U, X, m, tol=1e-13)[0]) <= 1e-9
