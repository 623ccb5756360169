"""Jacobi loops whose stencil and update kernels take the merge groups' rows themselves (k_cg_tma / k_stencil
and k_cg_update), against the oracle: few and many groups, sizes with and without a vector remainder, the
TMA-fed and the register stencil, with the p = 0 exit and in a closed box."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(12, 10, 8), (40, 24, 20), (45, 23, 17)])
@pytest.mark.parametrize("threshold", [0.02, 0.9])
@pytest.mark.parametrize("closed", [False, True])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
@pytest.mark.parametrize("tma", ["1", "0"])
def test_jacobi_with_merge_groups_matches_oracle(monkeypatch, shape, threshold, closed, mode, tma):
    """At a residual of 1e-10 the solution is within the error gate of 1e-6 of the oracle's."""
    from oracle import poisson as oracle
    from paper_1410_1937_gb300 import vofp
    monkeypatch.setenv("VOFP_STENCIL_TMA", tma)
    prob = I.config1(shape=shape)
    prob.merge_threshold = threshold
    if closed:
        prob.bc = (0,) * 6
    ref, _, s = oracle.solve(prob, rtol=1e-12)
    ctx, t = vofp.context_for(prob)
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    kw = dict(rtol=1e-10, mode=vofp.MODE_MIXED if mode == "mixed" else vofp.MODE_FP64, precond=vofp.PRECOND_JACOBI)
    x, info = ctx.vofp_solve(b, **kw)
    y, again = ctx.vofp_solve(b, host_loop=1, **kw)
    ctx.close()
    assert info["status"] == 0 and torch.equal(x, y) and again["iterations"] == info["iterations"]
    got = x.cpu().numpy().reshape(prob.shape)
    assert s.residual(got) <= 1.01e-10
    assert np.linalg.norm(got - ref) <= 1e-6 * np.linalg.norm(ref)
