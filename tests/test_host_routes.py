"""The library's host side without a GPU: linked with a stand-in for the CUDA runtime (tests/fake/cudart.cpp: host memory,
kernels recorded but not run), the entry points choose their routes, allocate and report errors as they do on the device.
Allocations, cooperative launches and the device's size are the test's to set."""
import ctypes
import glob
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fake_library(tmp_path_factory):
    import __graft_entry__ as ge
    ge.build_library()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    so = str(tmp_path_factory.mktemp("fake") / "librmhmc_fake.so")
    srcs = {os.path.basename(f) for f in glob.glob(os.path.join(ROOT, "paper_2112_04556_gb300", "csrc", "*.c*"))}
    objs = [o for o in glob.glob(os.path.join(ROOT, "paper_2112_04556_gb300", "_build", "*.o"))
            if os.path.basename(o)[:-2] in srcs]
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I", inc, "-Wl,-Bsymbolic", "-Wl,--no-undefined",
                    "-o", so, os.path.join(ROOT, "tests", "fake", "cudart.cpp")] + objs, check=True)
    return so


@pytest.fixture
def rm(fake_library, monkeypatch):
    import paper_2112_04556_gb300 as rm
    monkeypatch.setattr(rm, "_SO", fake_library)
    monkeypatch.setattr(rm, "_lib", None)
    L = rm.lib()
    L.fake_report.restype = ctypes.c_char_p
    L.fake_watched.restype = L.fake_held.restype = ctypes.c_longlong
    L.fake_device.argtypes = [ctypes.c_int, ctypes.c_longlong]
    L.fake_room.argtypes = [ctypes.c_longlong]
    L.fake_reset()
    return rm


# caller's buffers: the stand-in touches at most the first megabyte of a block
_SPACE = np.zeros((4, (1 << 17) + 2))
LINKS, FIELD, OUT, OUT2 = (a.ctypes.data + -a.ctypes.data % 16 for a in _SPACE)


def launched(rm):
    """Names of the kernels launched since the last call."""
    names = rm.lib().fake_report().decode().split()
    rm.lib().fake_clear_report()
    return names


def context(rm, L):
    ctx = rm.Context(L)
    ctx.check(rm.lib().rmhmc_set_links(ctx.h, LINKS, None))
    rm.lib().fake_poke(b"k_cg_run", 6, 0, 1)     # every Krylov run ends at once, converged with no iteration
    rm.lib().fake_poke(b"k_cg_start", 3, 0, 1)
    launched(rm)
    return ctx


def kinetic(rm, ctx, prec, mass=None):
    m = rm._mass_struct(mass or rm.mass_fit(12, 0.9))
    T = ctypes.c_double()
    return rm.lib().kinetic_force(ctx.h, None, FIELD, ctypes.byref(m), 1e-6, prec, OUT, OUT2, ctypes.byref(T), None)


@pytest.mark.parametrize("prec", [0, 1])
def test_a_failed_allocation_leaves_the_context_usable(rm, prec):
    """Whichever allocation of a kinetic evaluation fails, the call says ENOMEM (or does without the buffer) and the
    next one runs on buffers that exist: the barrier of the cooperative run (arguments 12 and 13) among them."""
    n = 0
    while True:
        n += 1
        with context(rm, (4, 4, 4, 4)) as ctx:
            rm.lib().fake_fail_at(n)
            code = kinetic(rm, ctx, prec)
            reached = not rm.lib().fake_fail_pending()
            rm.lib().fake_fail_at(0)
            assert code in (rm.OK, rm.ENOMEM)
            for arg in (12, 13):
                rm.lib().fake_watch(b"k_cg_run", arg)
                launched(rm)
                assert kinetic(rm, ctx, prec) == rm.OK
                if any("k_cg_run" in k for k in launched(rm)):
                    assert rm.lib().fake_watched() > 0, (n, arg)
        if not reached:
            break
    assert n > 4


SMEM = 232448   # shared memory a block of sm_103 may have


@pytest.mark.parametrize("prec,L", [(1, (64, 64, 8, 8)), (1, (32, 16, 16, 16)), (0, (32, 16, 16, 16))])
def test_cooperative_run_only_where_q_fits(rm, prec, L):
    """On a device of any size a Krylov run on the largest lattices of the cooperative form either fits its shared
    memory or takes the two-kernel form; so does one whose launch the device refuses."""
    seen = set()
    for sms in (152, 148, 147, 146, 145, 144, 132, 76, 38, 19, 1):
        rm.lib().fake_device(sms, SMEM)
        with context(rm, L) as ctx:
            assert kinetic(rm, ctx, prec) == rm.OK, sms
            seen.add((sms, any("k_cg_run" in k for k in launched(rm))))
    assert (152, True) in seen and (1, False) in seen
    rm.lib().fake_device(152, SMEM)
    for error in (720, 801):   # cooperative launch too large, not supported
        with context(rm, L) as ctx:
            rm.lib().fake_coop_error(error)
            assert kinetic(rm, ctx, prec) == rm.OK
            assert any("k_cg_start" in k for k in launched(rm))
            rm.lib().fake_coop_error(0)
            assert kinetic(rm, ctx, prec) == rm.OK   # not asked again
            assert not any("k_cg_run" in k for k in launched(rm))


def krylov_forms(names):
    return {f for f in ("k_cg_run", "k_cg_start", "k_cgg_start") for k in names if f in k}


@pytest.mark.parametrize("prec", [0, 1])
def test_profiling_does_not_outlast_itself(rm, prec):
    """While profiling is on the two-kernel form runs (its stencil launches are what is timed, in a tuned shape); before
    and after it the cooperative one.  A pinned stencil shape selects the two-kernel form for good."""
    with context(rm, (16, 8, 8, 16)) as ctx:
        forms = []
        for on in (0, 1, 0):
            rm.set_profiling(ctx, on)
            assert kinetic(rm, ctx, prec) == rm.OK
            forms.append(krylov_forms(launched(rm)))
        assert forms == [{"k_cg_run"}, {"k_cg_start"}, {"k_cg_run"}]
        rm.set_stencil_shape(ctx, rm.SHAPE_CG, rm.FP64 if prec == 0 else rm.FP32, 18, 1, 128)
        assert kinetic(rm, ctx, prec) == rm.OK
        assert krylov_forms(launched(rm)) == {"k_cg_start"}


def trajectory_md(rm, ctx):
    p = rm.make_params(beta=6.0, mass=rm.mass_fit(12, 0.9), tau=0.1, nsteps=2, prec=rm.MIXED)
    return rm.lib().rmhmc_md(ctx.h, LINKS, FIELD, ctypes.byref(p), None, None)


@pytest.mark.parametrize("L,form", [((4, 4, 4, 4), "k_cg_run"), ((64, 64, 8, 9), "k_cgg_start")])
def test_captured_trajectory_is_kept(rm, L, form):
    """The graph of a trajectory is captured once: profiling in between neither changes it nor what is counted for it,
    and one whose first capture the device refuses (a cooperative run in a conditional node) is captured without."""
    with context(rm, L) as ctx:
        counted = []
        for on in (0, 1, 0):
            rm.set_profiling(ctx, on)
            rm.counters(ctx, reset=True)
            assert trajectory_md(rm, ctx) == rm.OK
            counted.append(rm.counters(ctx)["launches"])
            names = launched(rm)
            assert ("instantiate" in names) == (len(counted) == 1) and "graph" in names
            assert krylov_forms(names) == ({form} if len(counted) == 1 else set())
        assert counted[1] == counted[2] > 0
    rm.lib().fake_instantiate_errors(1)
    with context(rm, L) as ctx:
        assert trajectory_md(rm, ctx) == rm.OK
        if form == "k_cg_run":
            assert krylov_forms(launched(rm)) == {"k_cg_run", "k_cgg_start"}   # two captures
            assert "graphs: on" in rm.tuning(ctx)
            assert trajectory_md(rm, ctx) == rm.OK and "instantiate" not in launched(rm)
        else:
            assert "graphs: off" in rm.tuning(ctx)


@pytest.mark.parametrize("prec,kernel", [(0, "k_link_grad"), (1, "k_link_grad_direct")])
def test_link_derivative_kernel_by_precision(rm, prec, kernel):
    """float64 contracts in the adjoint representation, float32 takes the direct form, which is faster there."""
    with context(rm, (4, 4, 4, 4)) as ctx:
        w = np.ones(3)
        ctx.check(rm.lib().lap_link_grad(ctx.h, None, FIELD, OUT, 3, w.ctypes.data_as(ctypes.POINTER(ctypes.c_double)),
                                         prec, OUT2, None))
        assert "%d%sI" % (len(kernel), kernel) in [k for k in launched(rm) if "k_link_grad" in k][-1]


def test_captured_calls_keep_nothing_derived_from_the_links(rm):
    """Under a capture of the caller's the float64 stencil and link derivative run by 3x3 products and the gauge force on
    staples, nothing is timed or allocated, and the calls after it go on from the table and the loops; a captured import
    ends both for the context."""
    def calls():
        one = np.ones(1).ctypes.data_as(ctypes.POINTER(ctypes.c_double))
        ctx.check(rm.lib().lap_apply(ctx.h, None, FIELD, OUT, 1, rm.FP64, 18, 0, None))
        ctx.check(rm.lib().lap_link_grad(ctx.h, None, FIELD, OUT, 1, one, rm.FP64, OUT2, None))
        ctx.check(rm.lib().gauge_force(ctx.h, None, 6.0, 0.0, rm.FP64, OUT2, None, None, None))
        names = " ".join(launched(rm))
        return ["k_lapIdLi64E" in names, "k_link_gradILi64E" in names, "k_loop_force" in names]
    derived, direct = [True] * 3, [False] * 3
    with context(rm, (4, 4, 4, 4)) as ctx:
        rm.lib().fake_capturing(1)
        held = rm.lib().fake_held()
        assert calls() == direct and rm.lib().fake_held() == held
        rm.lib().fake_capturing(0)
        assert calls() == derived
        rm.lib().fake_capturing(1)
        assert calls() == direct
        rm.lib().fake_capturing(0)
        assert calls() == derived
        rm.lib().fake_capturing(1)
        ctx.check(rm.lib().rmhmc_set_links(ctx.h, LINKS, None))
        rm.lib().fake_capturing(0)
        assert calls() == direct
        assert trajectory_md(rm, ctx) == rm.OK
        assert not any("k_plaquettes" in k for k in launched(rm))


def test_optional_buffers_give_way(rm):
    """The float64 table and the gauge force's loops are given back when another buffer of the context does not fit beside
    them: the call that needs it runs, as it does in a context without them, and the forms that do without them serve
    until the caller asks for the others again."""
    def stencil(ctx):
        ctx.check(rm.lib().lap_apply(ctx.h, None, FIELD, OUT, 1, rm.FP64, 18, 0, None))
        ctx.check(rm.lib().gauge_force(ctx.h, None, 6.0, 0.0, rm.FP64, OUT2, None, None, None))
        names = " ".join(launched(rm))
        return "k_lapIdLi64E" in names, "k_loop_force" in names
    for prec in (rm.FP64, rm.MIXED):
        with context(rm, (4, 4, 4, 4)) as ctx:   # what the evaluation takes without the optional buffers
            for kernel in (rm.SHAPE_TABLE, rm.SHAPE_LOOPS):
                rm.set_stencil_shape(ctx, kernel, rm.FP64, 18, 0, 128)
            held = rm.lib().fake_held()
            assert kinetic(rm, ctx, prec) == rm.OK
            need = rm.lib().fake_held() - held
        with context(rm, (4, 4, 4, 4)) as ctx:
            assert stencil(ctx) == (True, True)
            assert "off" not in rm.tuning(ctx)
            rm.lib().fake_room(need - 1024)
            assert kinetic(rm, ctx, prec) == rm.OK
            assert "float64 table off: no memory" in rm.tuning(ctx) and "gauge loops off" in rm.tuning(ctx)
            assert stencil(ctx) == (False, False)
            rm.lib().fake_room(1 << 40)
            assert stencil(ctx) == (False, False)
            for kernel in (rm.SHAPE_TABLE, rm.SHAPE_LOOPS):
                rm.set_stencil_shape(ctx, kernel, rm.FP64, 18, 1, 128)
            assert stencil(ctx) == (True, True)
        rm.lib().fake_room(1 << 50)


def test_a_trajectory_lets_go_of_its_loops(rm):
    """A captured trajectory whose loops were given back is captured again, on staples."""
    with context(rm, (4, 4, 4, 4)) as ctx:
        assert trajectory_md(rm, ctx) == rm.OK
        assert any("k_loop_force" in k for k in launched(rm))
        rm.lib().fake_room(4096)
        assert kinetic(rm, ctx, rm.FP64) == rm.ENOMEM     # far too large, with or without them
        rm.lib().fake_room(1 << 40)
        launched(rm)
        assert trajectory_md(rm, ctx) == rm.OK
        names = launched(rm)
        assert "instantiate" in names and not any("k_loop_force" in k for k in names)
        assert any("k_gauge_force" in k for k in names)
