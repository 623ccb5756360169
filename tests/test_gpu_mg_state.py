"""What a solve with the coarse-grid correction leaves in its context, and what it does where the correction cannot
be had (csrc/vofp_mg.cu)."""
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu


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
