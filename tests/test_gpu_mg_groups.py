"""The coarse-grid correction with merge groups whose master's aggregate has few couplings of its own (csrc/vofp_mg.cu,
k_mg_groups): cells of less than half their volume merged around a sphere and a hull, open and with every tenth face
closed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
@pytest.mark.parametrize("case", [("sphere", (160, 72, 102), 0.0), ("sphere", (132, 80, 102), 0.0), ("hull", (160, 32, 136), 0.1)])
def test_correction_keeps_its_gain_where_half_full_cells_merge(monkeypatch, mode, case):
    """At most a third of the plain iteration's iterations, as where few cells merge (tests/test_gpu_mg.py)."""
    from paper_1410_1937_gb300 import vofp
    body, shape, closed = case
    prob = I.config1(shape=shape) if body == "sphere" else I.config2(shape=shape)
    prob.merge_threshold = 0.5
    rng = np.random.default_rng(9)
    for name in ("ax", "ay", "az"):
        a = np.array(getattr(prob, name))
        a[rng.random(a.shape) < closed] = 0.0
        setattr(prob, name, a)
    ctx, t = vofp.context_for(prob)
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    its = {}
    for flag in ("0", "2"):
        monkeypatch.setenv("VOFP_MG", flag)
        _, info = ctx.vofp_solve(b, mode=vofp.MODE_MIXED if mode == "mixed" else vofp.MODE_FP64, rtol=1e-9,
                                 precond=vofp.PRECOND_RBSGS)
        assert info["status"] == 0 and info["rel_residual"] <= 1e-9
        its[flag] = info["iterations"]
    assert 3 * its["2"] <= its["0"], its
    ctx.close()
