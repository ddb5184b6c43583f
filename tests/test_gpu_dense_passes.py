"""The FP32 passes on brick-dense vectors and the cycles that visit only the
needed points, at the edges of their ranges: surfaces and spacings with odd
sizes, no or one sweep on either side, variable c, W-cycles, more levels than
three; the paper-form operator in one pass (FP32, and 2-D)."""
import numpy as np
import pytest

from helpers import oracle_surface, perm_gpu_to_oracle, require_cuda
from oracle.band import build_band
from oracle.mlp import MLP, correction, loss_and_grad, neighbour27
from oracle.multigrid import MGOptions, build_hierarchy, vcycle
from oracle.operators import Operators
import synth

pytestmark = pytest.mark.gpu

EPS32 = float(np.finfo(np.float32).eps)
SURFACES = [("circle", (0.9,), 1 / 25), ("circle", (1.0,), 1 / 130), ("sphere", (1.0,), 1 / 9),
            ("torus", (1.0, 0.45), 1 / 27), ("ellipsoid", (1.1, 0.8, 0.7), 1 / 23)]


def _single_level(pkg, kind, params, dx, **opts):
    import torch
    g = pkg.Band(kind, params, dx)
    H = pkg.Hierarchy(g, coarsest_dx=dx, coarse_sweeps=1, **opts)
    u = torch.from_numpy(synth.random_band_vector(g.nb, 1)).cuda()
    f = torch.from_numpy(synth.random_band_vector(g.nb, 2)).cuda()
    return g, H, u, f


@pytest.mark.parametrize("kind,params,dx", SURFACES)
@pytest.mark.parametrize("op_form", ["mbr", "paper"])
def test_f32_operator_and_sweeps_follow_f64(kind, params, dx, op_form):
    """M u and 0 .. 3 Jacobi sweeps in FP32 against FP64.  Rounding: E u sums 64
    products of weights with sum of magnitudes at most 1.63^3 = 4.4, the stencil
    adds 2d differences and gamma (w - u) of size 2d / dx^2, so an entry of M u
    is off by at most about 20 eps 4d / dx^2 max|u|; a sweep multiplies that by
    omega / diag(A) of about omega dx^2 / 2d."""
    torch, pkg = require_cuda()
    g, H, u, f = _single_level(pkg, kind, params, dx, op_form=op_form)
    d = 2 if kind == "circle" else 3
    umax = float(u.abs().max())
    err = float((H.apply(u.float()).double() - H.apply(u)).abs().max())
    assert err <= 20 * EPS32 * 4 * d / dx ** 2 * umax
    w = H.extend(u, with_ghost=True)
    w32 = H.extend(u.float(), with_ghost=True)
    assert w32.numel() == g.nb + g.ng
    assert float((w32.double() - w).abs().max()) <= 64 * EPS32 * umax
    assert torch.equal(H.extend(u.float()), w32[: g.nb])
    # f scaled like A u, so that the iterates stay of the size of u
    fs = f * (2 * d / dx ** 2)
    for sweeps in range(4):
        a, b = u.clone(), u.float()
        H.smooth(fs, a, sweeps=sweeps)
        H.smooth(fs.float(), b, sweeps=sweeps)
        size = float(a.abs().max())
        assert float((b.double() - a).abs().max()) <= 40 * (sweeps + 1) * EPS32 * size, sweeps


def test_f32_sweeps_with_variable_c_from_any_alignment():
    """Band-order vectors that start at any float of a larger buffer (the passes
    on a caller's vectors use scalar loads), per-point c."""
    torch, pkg = require_cuda()
    g = pkg.Band("sphere", (), 1 / 11)
    c = 1.0 + 0.5 * torch.from_numpy(synth.random_band_vector(g.nb, 3)).cuda()
    H = pkg.Hierarchy(g, coarsest_dx=1 / 11, coarse_sweeps=1, c_device=c)
    u = torch.from_numpy(synth.random_band_vector(g.nb, 4)).cuda().float()
    f = torch.from_numpy(synth.random_band_vector(g.nb, 5)).cuda().float() * 600
    ref = H.smooth(f, u.clone(), sweeps=2)
    for off in (1, 2, 3):
        buf = torch.empty(2 * g.nb + 8, device="cuda")
        ub, fb = buf[off: off + g.nb], buf[g.nb + 4 + off % 3: 2 * g.nb + 4 + off % 3]
        ub.copy_(u)
        fb.copy_(f)
        assert torch.equal(H.smooth(fb, ub, sweeps=2), ref)


@pytest.mark.parametrize("nu1,nu2", [(0, 2), (2, 0), (1, 1), (3, 2)])
@pytest.mark.parametrize("cycle,residual", [(1, "plain"), (1, "extended"), (2, "plain")])
def test_cycles_with_few_sweeps_match_the_oracle(nu1, nu2, cycle, residual):
    """One cycle from a random start on a circle with five levels: FP64 within
    1e-10 of the oracle's cycle (its own tolerance for a V-cycle), FP32 within
    1e-3."""
    torch, pkg = require_cuda()
    dx, cdx = 1 / 128, 1 / 8
    g = pkg.Band("circle", (), dx)
    H = pkg.Hierarchy(g, coarsest_dx=cdx, nu1=nu1, nu2=nu2, cycle=cycle, residual=residual)
    OH = build_hierarchy(oracle_surface("circle", ()), dx, cdx,
                         opts=MGOptions(smoother="jacobi", nu1=nu1, nu2=nu2, omega=0.8,
                                        residual=residual, cycle=cycle))
    assert H.n_levels == len(OH.levels) == 5
    perm = perm_gpu_to_oracle(g, OH.fine.band)
    f = synth.random_band_vector(g.nb, 6)
    u0 = 1e-3 * synth.random_band_vector(g.nb, 7)
    ref = vcycle(OH, u0.copy(), f)[perm]
    ft, ut = torch.from_numpy(f[perm]).cuda(), torch.from_numpy(u0[perm]).cuda()
    u64 = H.vcycle(ft, ut.clone())
    assert np.abs(u64.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
    u32 = H.vcycle(ft.float(), ut.float())
    assert np.abs(u32.double().cpu().numpy() - ref).max() <= 1e-3 * np.abs(ref).max()


@pytest.mark.parametrize("kind,params,dx,cdx", [("sphere", (), 1 / 24, 1 / 6), ("torus", (1.0, 0.5), 1 / 44, 1 / 11)])
def test_needed_points_suffice(kind, params, dx, cdx):
    """A cycle that visits only the needed points equals one of the relative form,
    whose passes run over whole bands: the two differ in rounding alone."""
    torch, pkg = require_cuda()
    g = pkg.Band(kind, params, dx)
    H = pkg.Hierarchy(g, coarsest_dx=cdx, residual="plain")
    Hr = pkg.Hierarchy(g, coarsest_dx=cdx, residual="plain", relative=True)  # whole-band cycles
    f = torch.from_numpy(synth.random_band_vector(g.nb, 8)).cuda()
    for dt, tol in ((torch.float64, 1e-9), (torch.float32, 5e-4)):
        a = H.vcycle(f.to(dt), torch.zeros(g.nb, dtype=dt, device="cuda")).double()
        b = Hr.vcycle(f.to(dt), torch.zeros(g.nb, dtype=dt, device="cuda")).double()
        assert float((a - b).abs().max()) <= tol * float(b.abs().max()), dt


@pytest.mark.parametrize("kind,params,dx", [("sphere", (), 1 / 8), ("sphere", (), 1 / 9),
                                            ("ellipsoid", (1.1, 0.9, 0.8), 1 / 15), ("torus", (1.0, 0.4), 1 / 17)])
def test_network_on_odd_sizes(kind, params, dx):
    """The learned smoother where the last 128 points (backward) and 32 points
    (forward) are partly filled, with the bounds for BF16 features and weights of
    the correction (3e-2), the loss (2e-2) and the gradient (6e-2)."""
    torch, pkg = require_cuda()
    g = pkg.Band(kind, params, dx)
    assert g.nb % 32 and g.nb % 128
    H = pkg.Hierarchy(g, coarsest_dx=dx, coarse_sweeps=1)
    sm = pkg.Smoother(11)
    w = sm.get_params()
    w[2048:2112] += 0.1
    w[6208:6272] += 0.1
    sm.set_params(w)
    H.set_smoother(sm)
    p = np.asarray(w, dtype=np.float64)
    om = MLP(p[0:31 * 64].reshape(31, 64), p[2048:2112], p[2112:6208].reshape(64, 64), p[6208:6272], p[6272:6336],
             float(p[6336]))
    ob = build_band(oracle_surface(kind, params), dx)
    op = Operators(ob)
    perm = perm_gpu_to_oracle(g, ob)
    r = synth.random_band_vector(ob.nb, 12).astype(np.float32).astype(np.float64)
    rt = torch.from_numpy(r[perm]).float().cuda()
    ref, _ = correction(om, ob, r, op.diag_M())
    assert np.abs(H.smoother_correction(rt).double().cpu().numpy() - ref[perm]).max() < 3e-2 * np.abs(ref).max()
    L_ref, grads = loss_and_grad(om, ob, op.A_matrix(1.0), r, op.diag_M(), neighbour27(ob))
    L, gp = H.smoother_loss_grad(rt)
    assert abs(L - L_ref) <= 2e-2 * L_ref
    for a, q in [(0, 0), (2048, 1), (2112, 2), (6208, 3), (6272, 4)]:
        d = grads[q].ravel()
        assert np.linalg.norm(gp[a: a + d.size] - d) < 6e-2 * np.linalg.norm(d), q
