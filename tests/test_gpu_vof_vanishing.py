"""Volume-fraction step with fractions far below rounding (what a cell is left with after many steps), against
oracle/vof.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _advect(prob, dt, order):
    from paper_1410_1937_gb300 import vofp
    ctx = vofp.Context(prob.dx, prob.dy, prob.dz)
    t = [torch.from_numpy(np.ascontiguousarray(getattr(prob, k)).ravel()).cuda()
         for k in ("F", "ax", "ay", "az", "vf", "u", "v", "w")]
    out = ctx.vofp_vof_advect(*t, dt, order=order).cpu().numpy().reshape(prob.shape)
    ctx.close()
    return out


def _open_box(shape, F, u, v, w):
    nz, ny, nx = shape
    return I.Problem(name="vanishing", dx=np.ones(nx), dy=np.ones(ny), dz=np.ones(nz), F=F, vf=np.ones(shape),
                     ax=np.ones((nz, ny, nx + 1)), ay=np.ones((nz, ny + 1, nx)), az=np.ones((nz + 1, ny, nx)), u=u, v=v, w=w)


@pytest.mark.parametrize("exponent", [100, 152, 155, 158, 162, 200, 300, (50.0, 300.0)])
@pytest.mark.parametrize("order", [0, 1])
def test_blocks_of_vanishing_fractions_stay_finite(exponent, order):
    """Half of the box holds fractions of 10^-exponent (of either of two), up to a surface in the other half: finite,
    and within the 1e-11 of the ordinary test (whose surface this is) wherever the oracle's own result does not turn
    on the last place of the velocities."""
    from oracle import vof
    from scipy.ndimage import maximum_filter
    shape = nz, ny, nx = 18, 11, 13
    rng = np.random.default_rng(3)
    x, y, z = (np.arange(n) + 0.5 for n in (nx, ny, nz))
    surface = 5.0 + 0.11 * (x[None, None, :] - x.mean()) + 0.07 * (y[None, :, None] - y.mean())
    F = np.clip(surface - (z - 0.5)[:, None, None], 0.0, 1.0)
    small = rng.uniform(0.2, 1.0, shape)
    small *= 10.0 ** -rng.choice(exponent, shape) if isinstance(exponent, tuple) else 10.0 ** -exponent
    F = np.where(F == 0.0, small, F)
    vel = [rng.uniform(-0.12, 0.12, s) for s in ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))]
    prob = _open_box(shape, F, *vel)
    got = _advect(prob, 1.0, order)
    assert np.isfinite(got).all()
    ref = vof.advect(prob, dt=1.0, order=order)
    turns = np.zeros(shape)
    for seed in (0, 1):
        r = np.random.default_rng(seed)
        prob.u, prob.w = (a * (1 + 2.3e-16 * r.integers(-1, 2, a.shape)) for a in (vel[0], vel[2]))
        turns = np.maximum(turns, np.abs(vof.advect(prob, dt=1.0, order=order) - ref))
    settled = maximum_filter(turns, size=5) <= 1e-12
    assert settled.mean() > 0.95
    assert np.abs(got - ref)[settled].max() <= 1e-11


@pytest.mark.parametrize("exponent", [20, 36, 40, 43, 46, 50, 60, 100, 155, 200])
def test_vanishing_fraction_keeps_its_fluid(exponent):
    """Fractions of 10^-exponent that fall along every axis, so that each cell's fluid lies in its corner of least
    x, y and z: a shift by 0.3 cells towards -x moves all of it into the neighbour (the box's outer cells, whose
    normals are one-sided, left out).  To 1e-9 of itself: the corner's edge is found to 1e-13 of itself at least, and the
    volume is its cube."""
    shape = nz, ny, nx = 6, 7, 9
    i, j, k = np.arange(nx)[None, None, :], np.arange(ny)[None, :, None], np.arange(nz)[:, None, None]
    F = (1.0 - 0.04 * i - 0.03 * j - 0.02 * k) * 10.0 ** -exponent
    u = np.full((nz, ny, nx + 1), -0.3)
    prob = _open_box(shape, F, u, np.zeros((nz, ny + 1, nx)), np.zeros((nz + 1, ny, nx)))
    got = _advect(prob, 1.0, 0)
    inner = (slice(1, -1),) * 2 + (slice(1, -2),)
    assert np.abs(got[inner] / F[1:-1, 1:-1, 2:-1] - 1.0).max() <= 1e-9
