"""Red-black solves with the coarse-grid correction (csrc/vofp_mg.cu), mixed and FP64, against the plain red-black
iteration and the oracle: grids at the edges of its tiles (16 x 8 x 4 and 32 x 8 x 8 cells per block,
one block from 512 cells down, odd sizes at every level), colour-compact and full-grid vectors, merge
groups with masters of both parities, closed boxes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vofp():
    from paper_1410_1937_gb300 import vofp
    return vofp


def _solve(vofp, prob, flag, monkeypatch, rtol, mode):
    monkeypatch.setenv("VOFP_MG", flag)
    kw = dict(rtol=rtol, mode=vofp.MODE_MIXED if mode == "mixed" else vofp.MODE_FP64, precond=vofp.PRECOND_RBSGS)
    ctx, t = vofp.context_for(prob)
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    x, info = ctx.vofp_solve(b, **kw)
    assert info["status"] == 0, info
    y, again = ctx.vofp_solve(b, host_loop=1, **kw)
    assert torch.equal(x, y) and again["iterations"] == info["iterations"]
    ctx.close()
    return x.cpu().numpy(), info


# (nx, ny, nz): tile edges and remainders, odd at several levels, one cell thick, the large-level kernel
SHAPES = [(16, 16, 16), (17, 16, 16), (33, 17, 9), (40, 24, 20), (72, 33, 17), (63, 65, 31), (520, 9, 1), (4104, 1, 1),
          (1, 70, 90), (136, 70, 41), (256, 160, 128), (251, 163, 127)]


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
@pytest.mark.parametrize("shape", SHAPES)
def test_coarse_grid_correction_matches_plain_red_black(vofp, monkeypatch, shape, mode):
    """Both solves to a residual of 1e-10: their solutions differ by at most twice the error gate of
    1e-6 that such a residual is held to, and the corrected one takes no more iterations."""
    prob = I.config1(shape=shape)
    x1, i1 = _solve(vofp, prob, "2", monkeypatch, 1e-10, mode)
    x0, i0 = _solve(vofp, prob, "0", monkeypatch, 1e-10, mode)
    assert i1["rel_residual"] <= 1e-10 and i0["rel_residual"] <= 1e-10
    assert np.linalg.norm(x1 - x0) <= 2e-6 * np.linalg.norm(x0)
    assert i1["iterations"] <= i0["iterations"] + 16, (i1, i0)
    if prob.n > 100000 and min(shape) > 16:
        # (the plain mixed solve loses some iterations to its refinement steps, the FP64 one none)
        assert (3 if mode == "mixed" else 2) * i1["iterations"] <= i0["iterations"], (i1, i0)


@pytest.mark.parametrize("shape", [(40, 24, 20), (45, 23, 18)])
@pytest.mark.parametrize("threshold", [0.02, 0.9])
@pytest.mark.parametrize("closed", [False, True])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_coarse_grid_correction_with_merge_groups_matches_oracle(vofp, monkeypatch, shape, threshold, closed, mode):
    """Few and many merge groups (with 0.9 nearly every cut cell merges, in chains), with the p = 0 exit
    and in a closed box (singular, zero-mean solution; the right-hand side sums to zero because no
    wall carries flux), against the oracle at the error gate of 1e-6."""
    from oracle import poisson as oracle
    prob = I.config1(shape=shape)
    prob.merge_threshold = threshold
    if closed:
        prob.bc = (0,) * 6
    ref, info_ref, s = oracle.solve(prob, rtol=1e-12)
    x, info = _solve(vofp, prob, "2", monkeypatch, 1e-10, mode)
    got = x.reshape(prob.shape)
    assert s.residual(got) <= 1.01e-10
    assert np.linalg.norm(got - ref) <= 1e-6 * np.linalg.norm(ref)
