"""The precision of the coarsest level's explicit inverse, also where the rows of
the matrix have uneven scales.

A hierarchy of one level is its coarsest level, so one V-cycle from zero is the
direct solve u = A^-1 f.  Its row-wise backward error

    max_i |f - A u|_i / (|A| |u| + |f|)_i

with FP64 elimination is at most 2 n 2^-53 on these systems (textbook
Gauss-Jordan in numpy: 17 to 1256 units at 216 to 712 rows), so the bound is
4 n 2^-53.  Operands of 48 bits miss it by a factor of 7 and more on every system of
constant coefficients, operands of 56 bits below a row's largest entry by 3 to
170 where the diffusion coefficient spans four or six decades.
"""
import numpy as np
import pytest

from helpers import oracle_surface, perm_gpu_to_oracle, require_cuda
from oracle.band import build_band
from oracle.operators import Operators, PaperOperators, VarDiffOperators
import synth

pytestmark = pytest.mark.gpu


def _angle(cp):
    return np.arctan2(cp[:, 1], cp[:, 0])


# (radius, dx, form, decades of a, its wave number, decades of c)
CASES = [(0.8, 1 / 6, "mbr", 0, 0, 0), (1.0, 1 / 8, "mbr", 0, 0, 0), (0.9, 1 / 13, "mbr", 0, 0, 0),
         (1.0, 1 / 16, "mbr", 0, 0, 0), (1.0, 1 / 16, "paper", 0, 0, 0), (1.0, 1 / 16, "mbr", 0, 0, 6),
         (1.0, 1 / 16, "mbr", 0, 0, 12), (0.9, 1 / 13, "vardiff", 4, 5, 0), (0.9, 1 / 13, "vardiff", 6, 3, 0),
         (1.0, 1 / 16, "vardiff", 4, 5, 0), (1.0, 1 / 16, "vardiff", 6, 5, 0), (1.0, 1 / 16, "vardiff", 6, 5, 6)]


@pytest.mark.parametrize("radius,dx,form,da,wave,dc", CASES)
def test_backward_error_of_the_direct_solve(radius, dx, form, da, wave, dc):
    torch, pkg = require_cuda()

    def a_of(cp):
        return 10.0 ** (0.5 * da * np.sin(wave * _angle(cp)))

    def c_of(cp):
        return 10.0 ** (dc * (0.5 + 0.5 * np.sin(7 * _angle(cp))))

    g = pkg.Band("circle", (radius,), dx)
    cp = g.export()[1][: g.nb]
    kw = {"op_form": form, "c_device": torch.from_numpy(c_of(cp)).cuda()}
    if form == "vardiff":
        kw["a_device"] = torch.from_numpy(a_of(cp)).cuda()
    H = pkg.Hierarchy(g, coarsest_dx=dx, **kw)
    assert H.n_levels == 1
    ob = build_band(oracle_surface("circle", (radius,)), dx)
    op = {"mbr": Operators, "paper": PaperOperators,
          "vardiff": lambda b: VarDiffOperators(b, a_of(b.cp[: b.nb]))}[form](ob)
    A = op.A_matrix(c_of(ob.cp[: ob.nb])).toarray()
    perm = perm_gpu_to_oracle(g, ob)
    for seed in (1, 2, 3):
        f = synth.random_band_vector(ob.nb, seed)
        u = torch.zeros(ob.nb, dtype=torch.float64, device="cuda")
        H.vcycle(torch.from_numpy(f[perm]).cuda(), u)
        uo = np.empty(ob.nb)
        uo[perm] = u.cpu().numpy()
        res = np.abs(f.astype(np.longdouble) - A.astype(np.longdouble) @ uo)
        err = float((res / (np.abs(A) @ np.abs(uo) + np.abs(f))).max())
        assert err <= 4 * ob.nb * 2.0 ** -53, (ob.nb, seed, err * 2.0 ** 53)


@pytest.mark.parametrize("kind,dx", [("circle", 1 / 6), ("circle", 1 / 16)])
def test_a_nan_in_the_matrix_is_refused(kind, dx):
    """One NaN in c: the elimination is left with a row of NaNs, which has no
    pivot, whatever the number of column blocks (272 and 712 rows)."""
    torch, pkg = require_cuda()
    g = pkg.Band(kind, (), dx)
    c = torch.ones(g.nb, dtype=torch.float64, device="cuda")
    c[g.nb // 3] = float("nan")
    with pytest.raises(pkg.capi.CpmError, match="singular"):
        pkg.Hierarchy(g, coarsest_dx=dx, c_device=c)
