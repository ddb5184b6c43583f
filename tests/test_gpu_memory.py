"""Device memory of workspaces and of the coarsest level's inverse, as the free
memory of the device shows it (run by itself: other processes on the same device
would be counted too)."""
import threading

import numpy as np
import pytest

from helpers import require_cuda

pytestmark = pytest.mark.gpu


def _free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("opts", [dict(), dict(residual="plain"), dict(smoother="rbgs"), dict(relative=True),
                                  dict(op_form="paper")])
def test_batch_workspace_holds_what_its_cycle_uses(opts):
    """Bytes of one system of a batch, counted per band point from the vectors
    that its passes read: FP64 u, f, r, E u and one more on every level; on the
    finest level u, f, r and the correction, the FP64 form's reference values and,
    but for the paper form, the pair form's 12 bytes per point of B+; FP32
    brick-dense u, f, r and E u where the cycle keeps its vectors so, else the
    band-order vectors.  15 % for allocation granularity and the coarsest levels."""
    torch, pkg = require_cuda()
    g = pkg.Band("sphere", (), 1 / 128)
    H = pkg.Hierarchy(g, coarsest_dx=1 / 8, coarse_sweeps=1, **opts)
    ijk = g.export()[0] // 4
    bricks = len(np.unique(ijk[:, 0] + 1024 * (ijk[:, 1] + 1024 * ijk[:, 2].astype(np.int64))))
    nb, plus, slots = 1.0, 1.0 + g.ng / g.nb, 64 * bricks / g.nb
    levels = sum(H.level_size(l) for l in range(H.n_levels)) / g.nb
    paper, relative, rbgs = "op_form" in opts, "relative" in opts, "smoother" in opts
    per_level = 8 * (4 * nb + plus)
    finest = 8 * 4 * nb + 8 * plus + (0 if paper else 12 * plus)
    if paper:  # L_B u, and E u, in both precisions
        per_level += 8 * nb + 4 * (5 * nb + plus)
    elif relative:  # reference values in both precisions, FP32 E u relative to them, and E u of apply
        per_level += 8 * plus + 4 * (4 * nb + 2 * plus) + 4 * slots
    elif rbgs:
        per_level += 4 * 4 * nb + 4 * slots
    else:
        per_level += 4 * 4 * slots
    if paper or relative or rbgs:
        finest += 2 * 4 * nb  # the scaled residual and its correction, FP32
    expected = (per_level * levels + finest) * g.nb
    pkg.Batch([H], 1).close()
    before, n = _free(torch), 3
    B = pkg.Batch([H], n)
    used = (before - _free(torch)) / n
    B.close()
    assert used <= 1.15 * expected, (used / g.nb, expected / g.nb)


def test_inverse_needs_no_second_matrix():
    """While a hierarchy with an FP64 inverse of 10136 rows (822 MB) is built, the
    device never holds half a matrix more than afterwards."""
    torch, pkg = require_cuda()
    g = pkg.Band("sphere", (0.8,), 1 / 12)
    kw = dict(coarsest_dx=1 / 12)
    pkg.Hierarchy(g, **kw).close()  # (modules and kernels are loaded)
    low, stop = [_free(torch)], threading.Event()

    def watch():
        while not stop.is_set():
            low[0] = min(low[0], torch.cuda.mem_get_info()[0])

    t = threading.Thread(target=watch)
    t.start()
    H = pkg.Hierarchy(g, **kw)
    stop.set()
    t.join()
    assert g.nb > 10000 and H.n_levels == 1
    assert _free(torch) - low[0] <= 4 * g.nb ** 2, (_free(torch) - low[0], g.nb)
