"""The operator and right-hand side passes that take whole warps of pure, fully open cells a shorter way
(csrc/vofp_assemble.cu), against the oracle: rows of even and odd length, one cell thick, several ranges of planes,
smoothed and sharp density, partly and wholly closed faces with isolated cells, every kind of wall, prescribed and
body fluxes, and time steps of one, a power of two and neither."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1410_1937_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N, D = 0, 1
# (smoothing, dt, walls, cut: random closed faces, prescribed fluxes)
OPTIONS = [(0, 1.0, (N, D, N, N, N, N), False, False), (1, 0.5, (D,) * 6, False, True), (1, 0.013, (N, N, D, N, N, N), True, True),
           (0, 2.0, (N,) * 6, True, False), (1, 1.0, (N, N, N, D, D, N), True, True)]


@pytest.mark.parametrize("option", range(len(OPTIONS)))
@pytest.mark.parametrize("shape", [(16, 16, 16), (45, 23, 18), (64, 6, 70), (33, 1, 40), (1, 40, 33), (96, 80, 60)])
def test_operator_and_right_hand_side_match_oracle(shape, option):
    """Every row within 1e-13 of the largest: a row sums at most a group's faces, each rounded a few times."""
    from oracle import poisson as oracle
    from paper_1410_1937_gb300 import vofp
    smoothing, dt, bc, cut, fluxes = OPTIONS[option]
    rng = np.random.default_rng(11)
    p = I.config1(shape=shape)
    p.bc, p.dt, p.density_smoothing = bc, dt, smoothing
    p.F = np.array(p.F)
    spots = rng.random(p.F.shape) < 0.02
    p.F[spots] = rng.random(int(spots.sum()))
    if cut:
        for name in ("ax", "ay", "az"):
            a = np.array(getattr(p, name))
            a[rng.random(a.shape) < 0.3] = 0.0
            part = rng.random(a.shape) < 0.1
            a[part] = rng.random(int(part.sum()))
            setattr(p, name, a)
        p.vf = np.array(p.vf)
        part = rng.random(p.vf.shape) < 0.05
        p.vf[part] *= rng.random(int(part.sum()))
    nz, ny, nx = p.shape
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda").reshape(-1)
    g = [rng.standard_normal(s) if fluxes and bc[f] == N else None
         for f, s in enumerate([(nz, ny), (nz, ny), (nz, nx), (nz, nx), (ny, nx), (ny, nx)])]
    body = rng.standard_normal(p.shape) if fluxes else None
    ctx = vofp.Context(p.dx, p.dy, p.dz)
    ctx.vofp_build_operator(dev(p.F), dev(p.ax), dev(p.ay), dev(p.az), dev(p.vf), bc, p.rho_liquid, p.rho_gas,
                            p.merge_threshold, smoothing, dt,
                            neumann_flux=[None if a is None else dev(a) for a in g] if fluxes else None)
    s = oracle.System(p, body, g if fluxes else None)
    b = ctx.vofp_rhs_from_face_velocity(dev(p.u), dev(p.v), dev(p.w), body_flux=None if body is None else dev(body))
    assert np.abs(b.cpu().numpy() - s.b).max() <= 1e-13 * np.abs(s.b).max()
    x = rng.uniform(-1, 1, p.n)
    y = ctx.vofp_apply(dev(x)).cpu().numpy()
    ref = s.apply_full(x).ravel()
    assert np.abs(y - ref).max() <= 1e-13 * np.abs(ref).max()
    assert ctx.vofp_get_stats()["inactive"] == int(np.asarray(s.inactive).sum())
    ctx.close()
