"""The explicit inverse of the coarsest level (blocked Gauss-Jordan with sliced
tensor-core products) against a dense FP64 solve.

A hierarchy of one level is its coarsest level, so one V-cycle from zero is the
direct solve u = A^-1 f.  Sizes: fewer rows than two column blocks of 128, a
last block and a last panel of every remainder that comes up, more rows than one
row per thread of the smaller cluster (4096).
"""
import numpy as np
import pytest

from helpers import oracle_surface, perm_gpu_to_oracle, require_cuda
from oracle.band import build_band
from oracle.operators import Operators
import synth

pytestmark = pytest.mark.gpu

CASES = [("circle", (0.8,), 1 / 6), ("circle", (1.0,), 1 / 7), ("circle", (1.0,), 1 / 8),
         ("circle", (0.9,), 1 / 9), ("circle", (1.0,), 1 / 13), ("sphere", (1.0,), 1 / 6), ("sphere", (1.0,), 1 / 9)]


@pytest.mark.parametrize("kind,params,dx", CASES)
def test_direct_solve_matches_dense_solve(kind, params, dx):
    torch, pkg = require_cuda()
    g = pkg.Band(kind, params, dx)
    H = pkg.Hierarchy(g, coarsest_dx=dx)
    assert H.n_levels == 1
    ob = build_band(oracle_surface(kind, params), dx)
    A = Operators(ob).A_matrix(1.0).toarray()
    perm = perm_gpu_to_oracle(g, ob)
    f = synth.random_band_vector(ob.nb, 5)
    ref = np.linalg.solve(A, f)
    u = torch.zeros(ob.nb, dtype=torch.float64, device="cuda")
    H.vcycle(torch.from_numpy(f[perm]).cuda(), u)
    err = np.abs(u.cpu().numpy() - ref[perm]).max() / np.abs(ref).max()
    # backward-stable elimination: a few eps times the condition number, which
    # is at most ||A||_inf ||A^-1||_inf, and ||A^-1||_inf of order 1 / c
    bound = 64 * np.finfo(np.float64).eps * np.abs(A).sum(axis=1).max()
    assert err <= bound, (ob.nb, err, bound)
