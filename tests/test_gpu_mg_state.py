"""What a solve with the coarse-grid correction leaves in its context, and what it does where the correction cannot
be had (csrc/vofp_mg.cu)."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def vofp():
    from paper_1410_1937_gb300 import vofp
    return vofp


def _rebuild(ctx, t, prob):
    ctx.vofp_build_operator(t["F"], t["ax"], t["ay"], t["az"], t["vf"], prob.bc, prob.rho_liquid, prob.rho_gas,
                            prob.merge_threshold, prob.density_smoothing, prob.dt)


def test_kernel_timing_does_not_depend_on_the_last_solve(vofp, monkeypatch):
    """The FP32 red-black kernels are timed on their own vectors: after an FP64 corrected solve, which has no FP32 z,
    and after a corrected mixed solve of an operator with fewer merge groups, whose z is shorter."""
    monkeypatch.setenv("VOFP_MG", "2")
    prob = I.config1(shape=(64, 48, 40))
    ctx, t = vofp.context_for(prob)
    kw = dict(rtol=1e-10, precond=vofp.PRECOND_RBSGS)
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    x, _ = ctx.vofp_solve(b, mode=vofp.MODE_FP64, **kw)
    assert all(ms > 0 for ms in ctx.vofp_time_iteration_kernels(32, reps=2, precond=vofp.PRECOND_RBSGS))
    ctx.vofp_solve(b, mode=vofp.MODE_MIXED, **kw)
    prob.merge_threshold = 0.9
    _rebuild(ctx, t, prob)
    assert all(ms > 0 for ms in ctx.vofp_time_iteration_kernels(32, reps=2, precond=vofp.PRECOND_RBSGS))
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    _, info = ctx.vofp_solve(b, mode=vofp.MODE_MIXED, **kw)
    assert info["status"] == 0 and info["rel_residual"] <= 1e-10
    ctx.close()


def _in_child(tmp_path, code):
    """Run code in a process whose CUDA runtime calls pass through tests/fake_cudart.c (a failing call is made on
    the host); `fake` sets one of its variables, `fakes` reads one."""
    lib = str(tmp_path / "fake.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-Wall", "-o", lib, os.path.join(HERE, "fake_cudart.c"), "-ldl"],
                   check=True)
    head = f"""
import ctypes, sys
sys.path.insert(0, {os.path.dirname(HERE)!r})
import torch
from paper_1410_1937_gb300 import inputs as I, vofp
lib = ctypes.CDLL({lib!r})
TYPES = {{"fake_malloc_limit": ctypes.c_size_t, "fake_drop": ctypes.c_char * 64}}
def fakes(name): return TYPES.get(name, ctypes.c_int).in_dll(lib, name).value
def fake(name, value): TYPES.get(name, ctypes.c_int).in_dll(lib, name).value = value
"""
    r = subprocess.run([sys.executable, "-c", head + textwrap.dedent(code)], env={**os.environ, "LD_PRELOAD": lib},
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]


# bytes above which an allocation is refused: every one, then those after the levels (FP32), then the vectors'
@pytest.mark.parametrize("limit", [0, 100 * 1000, 250 * 1000])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_solve_goes_on_without_the_correction_when_memory_is_refused(tmp_path, mode, limit):
    """The plain iteration's result, bit for bit, no memory kept, and the correction again for the next operator."""
    _in_child(tmp_path, f"""
        import os
        prob = I.config1(shape=(64, 48, 40))
        ctx, t = vofp.context_for(prob)
        kw = dict(rtol=1e-10, precond=vofp.PRECOND_RBSGS, mode=vofp.MODE_{mode.upper()})
        b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
        xs = [torch.zeros_like(b) for _ in range(4)]
        os.environ["VOFP_MG"] = "0"
        plain = ctx.vofp_solve(b, x=xs[0], x0_zero=1, **kw)[1]
        held = ctx.vofp_get_stats()["device_bytes"]
        assert torch.equal(xs[0], xs[0])   # (torch's own memory for it is there)
        os.environ["VOFP_MG"] = "2"
        fake("fake_malloc_limit", {limit})
        for x in xs[1:3]:
            info = ctx.vofp_solve(b, x=x, x0_zero=1, **kw)[1]
            assert info["status"] == 0 and info["iterations"] == plain["iterations"], (info, plain)
            assert torch.equal(x, xs[0])
            assert ctx.vofp_get_stats()["device_bytes"] - held in (0, 8)   # (8: one word, kept)
        assert fakes("fake_refused") == 1
        fake("fake_malloc_limit", 1 << 62)
        ctx.vofp_build_operator(t["F"], t["ax"], t["ay"], t["az"], t["vf"], prob.bc, prob.rho_liquid, prob.rho_gas,
                                prob.merge_threshold, prob.density_smoothing, prob.dt)
        info = ctx.vofp_solve(b, x=xs[3], x0_zero=1, **kw)[1]
        assert info["status"] == 0 and 2 * info["iterations"] < plain["iterations"], (info, plain)
        ctx.close()
    """)


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_growing_merge_groups_leave_no_memory_behind(vofp, monkeypatch, mode):
    """The correction's share of the context's memory (with it less without it) after operators of more and more
    merge groups is at most that of a context which has seen the last one alone: a buffer is of the size that the
    last operator asked for which did not fit, and the last one asks for the most."""
    prob = I.config1(shape=(64, 48, 40))
    open_cells, part = prob.vf == 1.0, np.random.default_rng(8).random(prob.vf.shape)
    kw = dict(rtol=1e-10, precond=vofp.PRECOND_RBSGS, mode=vofp.MODE_MIXED if mode == "mixed" else vofp.MODE_FP64)

    def held(flag, shares):
        monkeypatch.setenv("VOFP_MG", flag)
        ctx, t = vofp.context_for(prob)
        for share in shares:
            t["vf"] = torch.from_numpy(np.where(open_cells & (part < share), 0.05, prob.vf).ravel()).cuda()
            _rebuild(ctx, t, prob)
            b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
            assert ctx.vofp_solve(b, **kw)[1]["status"] == 0
        stats = ctx.vofp_get_stats()
        assert stats["rb_compact"] == (mode == "mixed")
        ctx.close()
        return stats["device_bytes"]

    shares = (0.002, 0.04, 0.13)
    assert held("2", shares) - held("0", shares) <= held("2", shares[-1:]) - held("0", shares[-1:])


# kernel whose launches are dropped: without k_mg_direction r.z stays 0, which ends the first iteration as a lost
# positivity does
@pytest.mark.parametrize("host_loop", [0, 1])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_solve_goes_on_without_the_correction_when_it_breaks_down(tmp_path, mode, host_loop):
    """From 0 and from a starting pressure: converged in the plain iteration's refinement steps (mixed) or intervals
    between convergence tests (FP64) and two more, to its solution (residuals of 1e-10: each within 1e-6); later solves of
    the operator are plain in this precision, corrected in the other, and corrected again for the next operator."""
    other = {"mixed": "FP64", "fp64": "MIXED"}[mode]
    _in_child(tmp_path, f"""
        import os
        prob = I.config1(shape=(64, 48, 40))
        ctx, t = vofp.context_for(prob)
        kw = dict(rtol=1e-10, precond=vofp.PRECOND_RBSGS, mode=vofp.MODE_{mode.upper()}, host_loop={host_loop})
        b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
        os.environ["VOFP_MG"] = "0"
        ref, plain = ctx.vofp_solve(b, **kw)
        _, plain_warm = ctx.vofp_solve(b, x=1.01 * ref, **kw)
        _, plain_other = ctx.vofp_solve(b, **{{**kw, "mode": vofp.MODE_{other}}})
        os.environ["VOFP_MG"] = "2"
        build = lambda: ctx.vofp_build_operator(t["F"], t["ax"], t["ay"], t["az"], t["vf"], prob.bc, prob.rho_liquid,
                                                prob.rho_gas, prob.merge_threshold, prob.density_smoothing, prob.dt)
        for start, want in ((None, plain), (1.01 * ref, plain_warm)):
            build()
            ctx.vofp_solve(b, **{{**kw, "mode": vofp.MODE_{other}}})
            fake("fake_drop", b"k_mg_direction")
            x, info = ctx.vofp_solve(b, x=start, **kw)
            fake("fake_drop", b"")
            assert fakes("fake_dropped") > 0
            assert info["status"] == 0 and info["rel_residual"] <= 1e-10, info
            # (one more step for the pass that broke down, one for the rounding of the pressure it handed over)
            unit, most = ("outer_iterations", 2) if {mode == "mixed"} else ("iterations", 2 * 8)
            assert info[unit] <= want[unit] + most, (info, want)
            assert float((x - ref).norm()) <= 2e-6 * float(ref.norm())
        assert ctx.vofp_solve(b, **kw)[1]["iterations"] == plain["iterations"]
        info = ctx.vofp_solve(b, **{{**kw, "mode": vofp.MODE_{other}}})[1]
        assert info["status"] == 0 and 2 * info["iterations"] < plain_other["iterations"], (info, plain_other)
        build()
        info = ctx.vofp_solve(b, **kw)[1]
        assert info["status"] == 0 and 2 * info["iterations"] < plain["iterations"], (info, plain)
        ctx.close()
    """)


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_solve_that_stagnates_with_the_correction_leaves_it_in_use(vofp, monkeypatch, mode):
    """A residual that neither iteration reaches: in FP64 mode one below rounding (what is reached is a settled solve's,
    1e-14, some thousand roundings); in mixed mode one that inner solves of two restarted iterations do not come to in
    the loop's 200 refinement steps, first the corrected one's and then the plain one's.  The operator's next solve is
    corrected."""
    monkeypatch.setenv("VOFP_MG", "2")
    prob = I.config1(shape=(64, 48, 40))
    ctx, t = vofp.context_for(prob)
    kw = dict(precond=vofp.PRECOND_RBSGS, mode=vofp.MODE_MIXED if mode == "mixed" else vofp.MODE_FP64)
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    before = ctx.vofp_solve(b, rtol=1e-10, **kw)[1]
    short = dict(inner_restart=1, inner_rtol=0.9, check_every=2) if mode == "mixed" else {}
    _, info = ctx.vofp_solve(b, rtol=1e-18, max_iter=20000, raise_on_error=False, **short, **kw)
    assert info["status_name"] in ("STAGNATED", "NOT_CONVERGED"), info
    assert info["rel_residual"] <= 1e-14 if mode == "fp64" else info["outer_iterations"] == 400, info
    assert ctx.vofp_solve(b, rtol=1e-10, **kw)[1]["iterations"] == before["iterations"]
    ctx.close()
