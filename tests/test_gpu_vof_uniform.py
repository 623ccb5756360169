"""Volume-fraction step where most cells are full or empty: the stages copy such cells where the slabs stay
within half a donor cell and take the others one by one (csrc/vofp_vof.cu).  A tilted surface on grids
with width ratios of 4 between neighbours, velocities on both sides of that limit (below a whole donor
cell, where a full region stays full), closed faces and body cells, against oracle/vof.py at 1e-11 (two
root searches on the same monotone volume)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _problem(shape, seed):
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    dx, dy, dz = (np.where(rng.uniform(size=n) < 0.3, 0.25, 1.0) for n in shape)
    x, y, z = (np.cumsum(a) - 0.5 * a for a in (dx, dy, dz))
    # every cell's normal is well defined where it matters: a plane through the middle of the box
    surface = 0.5 * dz.sum() + 0.11 * (x[None, None, :] - x.mean()) + 0.07 * (y[None, :, None] - y.mean())
    F = np.clip((surface - (z - 0.5 * dz)[:, None, None]) / dz[:, None, None], 0.0, 1.0)
    sh = ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))
    ax, ay, az = (np.where(rng.uniform(size=s) < 0.9, 1.0, rng.uniform(0.2, 1.0, s)) for s in sh)
    az[:, 0, 0] = 0.0
    vf = np.ones(F.shape)
    vf[0, 0, 0] = 0.0
    u, v, w = (rng.uniform(-0.124, 0.124, s) for s in sh)
    return I.Problem(name="tilted", dx=dx, dy=dy, dz=dz, F=F, vf=vf, ax=ax, ay=ay, az=az, u=u, v=v, w=w)


@pytest.mark.parametrize("shape", [(1, 1, 9), (31, 3, 5), (33, 8, 9), (64, 40, 20), (129, 31, 17)])
@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("dt", [0.3, 1.0])
def test_step_with_full_and_empty_regions_matches_oracle(shape, order, dt):
    from oracle import vof
    from paper_1410_1937_gb300 import vofp
    prob = _problem(shape, 5)
    ctx = vofp.Context(prob.dx, prob.dy, prob.dz)
    t = {k: torch.from_numpy(np.ascontiguousarray(getattr(prob, k)).ravel()).cuda()
         for k in ("F", "vf", "ax", "ay", "az", "u", "v", "w")}
    args = (t["F"], t["ax"], t["ay"], t["az"], t["vf"], t["u"], t["v"], t["w"], dt)
    out = ctx.vofp_vof_advect(*args, order=order)
    ref = vof.advect(prob, dt=dt, order=order)
    got = out.cpu().numpy().reshape(prob.shape)
    # a cell whose neighbourhood is uniform but for rounding has a normal of rounding errors: where the
    # oracle's own result turns on the last place of the velocities (and next to it) there is nothing to
    # compare
    turns = np.zeros(prob.shape)
    u, w = prob.u, prob.w
    for seed in (0, 1):
        rng = np.random.default_rng(seed)
        prob.u = u * (1 + 2.3e-16 * rng.integers(-1, 2, u.shape))
        prob.w = w * (1 + 2.3e-16 * rng.integers(-1, 2, w.shape))
        turns = np.maximum(turns, np.abs(vof.advect(prob, dt=dt, order=order) - ref))
    from scipy.ndimage import maximum_filter
    settled = maximum_filter(turns, size=5) <= 1e-12
    assert settled.mean() > 0.99
    assert np.abs(got - ref)[settled].max() <= 1e-11 * max(1.0, np.abs(ref).max())
    assert torch.equal(ctx.vofp_vof_advect(*args, order=order), out)     # the lists' order does not matter
    ctx.close()
