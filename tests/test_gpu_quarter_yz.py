"""The quarter-band y- and z-passes of FP64-data plans.

Where every stick has |k| <= n2/4 (and every plane wave |l| <= n3/4) the
y-passes and the forward z-pass skip the rows outside the band.  Lists that
reach the band's edges, that leave gaps in it, that touch one edge only and
that step over an edge by one (the general passes), at lengths of every
schedule, against the FP64 oracle within the repository's FP64 gate, and the
round trip to real space and back, which returns the coefficients.
"""
import numpy as np
import pytest

from helpers import TOL, oracle_apply, rel_l2_per_band
from paper_1601_07378_gb300 import synth, vloc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1601_07378_gb300.build import build
    build()


def _glist(n, shape):
    q1, q2, q3 = n[0] // 4, n[1] // 4, n[2] // 4
    h, k, l = np.meshgrid(np.arange(-q1, q1 + 1), np.arange(-q2, q2 + 1), np.arange(-q3, q3 + 1), indexing="ij")
    keep = (h / q1) ** 2 + (k / q2) ** 2 + (l / q3) ** 2 <= 1.0
    if shape == "gaps":
        keep &= (k % 3 != 1) & (np.abs(l) != 1)
    elif shape == "edges":
        keep = (k == q2) & (np.abs(l) == q3) | (k == 0) & (np.abs(h) + np.abs(l) < 3)
    g = np.stack([h[keep], k[keep], l[keep]], axis=1).astype(np.int32)
    if shape == "over":
        g = np.concatenate([g, np.array([[0, q2 + 1, 0], [0, 0, -q3 - 1]], dtype=np.int32)])
    return np.ascontiguousarray(g[synth.canonical_order(g, *n)])


@pytest.mark.parametrize("double_float", [False, True])
@pytest.mark.parametrize("n,shape", [((24, 24, 32), "ball"), ((24, 48, 60), "gaps"), ((24, 64, 72), "edges"),
                                     ((24, 80, 96), "over"), ((32, 96, 24), "gaps"), ((24, 100, 120), "ball"),
                                     ((24, 128, 144), "edges"), ((24, 144, 100), "gaps"), ((24, 60, 48), "over")])
def test_quarter_band_fp64_passes(n, shape, double_float):
    g = _glist(n, shape)
    c = synth.coefficients(g, 3, seed=91)
    V = synth.potential(*n, "smooth", 92)[0]
    p = vloc.VlocPlan(n, g, torch.complex128, chunk=2, double_float=double_float, poison=True)
    ct, Vt = torch.from_numpy(c).cuda(), torch.from_numpy(V).cuda()
    ref = oracle_apply(n, g, c, V)
    for adjoint in (False, True):  # A is Hermitian: V is real
        out = p.apply(ct, Vt, adjoint=adjoint).cpu().numpy()
        assert rel_l2_per_band(out, ref).max() < TOL["f64"]
    back = p.to_recip(p.to_real(ct)).cpu().numpy()
    assert rel_l2_per_band(back, c).max() < TOL["f64"]
