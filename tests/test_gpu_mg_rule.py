"""Which operators take the coarse-grid correction by default (csrc/vofp_mg.cu, pays): not those whose couplings differ by
more than a hundred between the axes, whose faces are closed by a third, or whose plain iteration is short because
every wall has p = 0; the rule is looked at again for every operator of a context."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _problem(name):
    if name in ("hull", "porous"):
        p = I.config2(shape=(64, 48, 40))
        if name == "porous":
            rng = np.random.default_rng(4)
            for a in ("ax", "ay", "az"):
                v = np.array(getattr(p, a))
                v[rng.random(v.shape) < 0.35] = 0.0
                setattr(p, a, v)
        return p
    p = I.config1(shape=(64, 48, 40))
    p.dx, p.dy, p.dz = (np.full(n, 1.0 / m) for n, m in zip((64, 48, 40), (64, 64, 64)))
    if name == "flat":
        p.dz *= 0.05
    if name == "walls":
        p.bc = (1,) * 6
        p.dy *= 0.5
    return p


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_operators_for_which_it_does_not_pay_keep_the_plain_iteration(monkeypatch, mode):
    from paper_1410_1937_gb300 import vofp
    ctx = None
    for name, corrected in (("hull", True), ("porous", False), ("flat", False), ("cube", True), ("walls", False)):
        p = _problem(name)
        if ctx is None or name in ("hull", "flat", "cube", "walls"):
            ctx, t = vofp.context_for(p)
        else:   # the same grid: the context's next operator
            for k in ("ax", "ay", "az"):
                t[k] = torch.from_numpy(np.ascontiguousarray(getattr(p, k)).ravel()).cuda()
            ctx.vofp_build_operator(t["F"], t["ax"], t["ay"], t["az"], t["vf"], p.bc, p.rho_liquid, p.rho_gas,
                                    p.merge_threshold, p.density_smoothing, p.dt)
        b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
        its, xs = {}, {}
        for flag in (None, "0", "2"):
            monkeypatch.delenv("VOFP_MG", raising=False) if flag is None else monkeypatch.setenv("VOFP_MG", flag)
            xs[flag], info = ctx.vofp_solve(b, rtol=1e-9, precond=vofp.PRECOND_RBSGS,
                                            mode=vofp.MODE_MIXED if mode == "mixed" else vofp.MODE_FP64)
            assert info["status"] == 0
            its[flag] = info["iterations"]
        same = "2" if corrected else "0"
        assert its[None] == its[same] and torch.equal(xs[None], xs[same]), (name, its)
