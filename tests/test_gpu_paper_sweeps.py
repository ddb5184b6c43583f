"""Jacobi sweeps of the paper form (one pass over the extension tiles in FP32 and
in 2-D, whose iterate alternates between two vectors) against the oracle's
assembled matrix, with odd and even counts of sweeps."""
import numpy as np
import pytest

from helpers import oracle_surface, perm_gpu_to_oracle, require_cuda
from oracle.band import build_band
from oracle.operators import PaperOperators
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,params,dx", [("circle", (0.9,), 1 / 25), ("circle", (1.0,), 1 / 130),
                                            ("sphere", (), 1 / 9), ("ellipsoid", (1.1, 0.9, 0.8), 1 / 15)])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_paper_form_sweeps(kind, params, dx, prec):
    """Sweeps u += omega / diag(A) (f - A u) with the oracle's assembled matrix.  An
    entry of M u is off by about 20 eps 4d / dx^2 max|u| (rounding) and, as the
    closest points differ in their last digit, by about 8 / dx eps of the weights; a
    sweep multiplies that by about omega dx^2 / 2d."""
    torch, pkg = require_cuda()
    g = pkg.Band(kind, params, dx)
    H = pkg.Hierarchy(g, coarsest_dx=dx, coarse_sweeps=1, op_form="paper")
    ob = build_band(oracle_surface(kind, params), dx)
    A = PaperOperators(ob).A_matrix(1.0)
    perm = perm_gpu_to_oracle(g, ob)
    dt = torch.float64 if prec == "f64" else torch.float32
    eps = float(torch.finfo(dt).eps)
    u = synth.random_band_vector(g.nb, 1)
    f = synth.random_band_vector(g.nb, 2) * (2 * ob.dim / dx ** 2)
    ft, u0 = torch.from_numpy(f[perm]).cuda().to(dt), torch.from_numpy(u[perm]).cuda().to(dt)
    for sweeps in range(1, 5):
        u = u + 0.8 / A.diagonal() * (f - A @ u)
        got = H.smooth(ft, u0.clone(), sweeps=sweeps).double().cpu().numpy()
        tol = (40 * eps + 16 / dx * np.finfo(np.float64).eps) * (sweeps + 1)
        assert np.abs(got - u[perm]).max() <= tol * np.abs(u).max(), sweeps
