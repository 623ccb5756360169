"""Red-black solves with the coarse-grid correction (csrc/vofp_mg.cu) from a starting pressure: a time step's
solve starts from the last step's, and a solve that is restarted starts from its iterate.  On full-grid vectors
the red cells, which the iteration does not write, hold rounding errors then."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu

INTERVAL = {"fp64": 8, "mixed": 16}   # iterations between two convergence tests, at most


@pytest.fixture(scope="module")
def vofp():
    from paper_1410_1937_gb300 import vofp
    return vofp


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(64, 48, 40), (45, 23, 18), (125, 61, 47)])
@pytest.mark.parametrize("threshold", [0.0, 0.9])
@pytest.mark.parametrize("closed", [False, True])
def test_warm_start_converges_like_a_cold_one(vofp, monkeypatch, mode, shape, threshold, closed):
    """x0 = 1.01 x has an error parallel to that of x0 = 0 and a hundredth of it: CG's iterates from it are
    those from 0 scaled, so that no more iterations may be needed (one interval for rounding).  From the solution
    of another right-hand side of the same size: converged, within twice the iterations.  max_iter ends a solve
    that does not converge."""
    monkeypatch.setenv("VOFP_MG", "2")
    prob = I.config1(shape=shape)
    prob.merge_threshold = threshold
    if closed:
        prob.bc = (0,) * 6
    kw = dict(rtol=1e-12, mode=vofp.MODE_MIXED if mode == "mixed" else vofp.MODE_FP64, precond=vofp.PRECOND_RBSGS,
              max_iter=3000)
    ctx, t = vofp.context_for(prob)
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    x, cold = ctx.vofp_solve(b, **kw)
    assert cold["status"] == 0, cold
    b2 = ctx.vofp_rhs_from_face_velocity(*(t[k].flip(0).contiguous() for k in "uvw"))
    x2, _ = ctx.vofp_solve(b2, **kw)
    y, warm = ctx.vofp_solve(b, x=1.01 * x, **kw)
    assert warm["status"] == 0 and warm["rel_residual"] <= 1e-12, warm
    assert warm["iterations"] <= cold["iterations"] + INTERVAL[mode], (warm, cold)
    z, other = ctx.vofp_solve(b, x=x2, **kw)
    assert other["status"] == 0 and other["rel_residual"] <= 1e-12, other
    assert other["iterations"] <= 2 * cold["iterations"], (other, cold)
    # two residuals of 1e-12: the errors that the residual gate of 1e-10 holds to 1e-6 are held to 1e-8
    for got in (y, z):
        assert float((got - x).norm()) <= 2e-8 * float(x.norm())
    ctx.close()


def test_two_rk2_steps_with_fp64_red_black_match_oracle(vofp, oracle, monkeypatch):
    """Both solves of a step start from a pressure.  The tolerances of the Jacobi solves' test."""
    from oracle import rk2
    monkeypatch.setenv("VOFP_MG", "2")
    prob = I.tiny_sphere(n=16)
    prob.dt = 0.2 * prob.dx.min() / max(np.abs(prob.u).max(), np.abs(prob.v).max(), np.abs(prob.w).max())
    R = I.momentum_terms(prob)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda()
    Rd = tuple(dev(a) for a in R)
    ctx, t = vofp.context_for(prob)
    p = torch.zeros(prob.n, dtype=torch.float64, device="cuda")
    cur = prob
    for step in range(2):
        i1, i2, _ = ctx.vofp_rk2_step(t["F"], t["ax"], t["ay"], t["az"], t["vf"], t["u"], t["v"], t["w"], cur.bc, p,
                                      order=step % 2, R=Rd, rho_liquid=cur.rho_liquid, rho_gas=cur.rho_gas,
                                      merge_threshold=cur.merge_threshold, dt=cur.dt, mode=vofp.MODE_FP64, rtol=1e-12,
                                      precond=vofp.PRECOND_RBSGS)
        assert i1["status"] == 0 and i2["status"] == 0
        phi, (u, v, w), P2, _, _ = rk2.rk2_step(cur, order=step % 2, R=R)
        assert np.linalg.norm(p.cpu().numpy().reshape(prob.shape) - P2) <= 1e-8 * np.linalg.norm(P2)
        for got, ref in ((t["u"], u), (t["v"], v), (t["w"], w)):
            assert np.abs(got.cpu().numpy().reshape(ref.shape) - ref).max() <= 1e-8 * np.abs(ref).max()
        assert np.abs(t["F"].cpu().numpy().reshape(prob.shape) - phi).max() <= 1e-8
        cur = dataclasses.replace(cur, F=phi, u=u, v=v, w=w)
    ctx.close()
