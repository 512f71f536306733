"""The line path (csrc/kernels_line.h): the apply of FP32 quarter-band plans as
z-pass, fused y/x pass, z-pass over dense rows, against the FP64 oracle and
against the five-launch chain on the general kernels (a plan made with
VLOC_NO_XQ set, which has no line path).

Tolerances: the FP32 gate against the oracle, and 3e-7 (as for the other
specialised kernels) between the two FP32 paths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from helpers import TOL, make_case, oracle_apply, rel_l2_per_band
from oracle import oracle as O
from paper_1601_07378_gb300 import synth, vloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1601_07378_gb300.build import build
    build()


def _plans(n, g, monkeypatch, **kw):
    p = vloc.VlocPlan(n, g, torch.complex64, **kw)
    monkeypatch.setenv("VLOC_NO_XQ", "1")
    ref = vloc.VlocPlan(n, g, torch.complex64, **kw)
    monkeypatch.delenv("VLOC_NO_XQ")
    return p, ref


def _launches(plan, f):
    l0 = plan.launch_count()
    out = f()
    torch.cuda.synchronize()
    return out, plan.launch_count() - l0


# every size class, lengths 2 mod 4 (no shared rim element), pairs of unequal
# axes, spheres that fill the quarter band and smaller ones, spheres whose rim
# planes are taken off the lines (64, 128), a last group of one line
CASES = [((24, 24, 24), 6.0, 21), ((30, 36, 40), 7.5, 13), ((36, 30, 50), 7.0, 7), ((48, 40, 54), 10.0, 11),
         ((48, 50, 60), 11.9, 9), ((50, 54, 24), 6.0, 20), ((64, 64, 32), 8.0, 17), ((64, 64, 64), 16.0, 9),
         ((72, 90, 30), 7.4, 17), ((80, 64, 36), 9.0, 15), ((96, 80, 48), 12.0, 11), ((90, 96, 100), 3.0, 7),
         ((100, 90, 24), 6.0, 21), ((128, 96, 30), 7.5, 17), ((128, 128, 40), 10.0, 13), ((120, 144, 36), 9.0, 14),
         ((108, 100, 128), 4.5, 5)]


@pytest.mark.parametrize("n,R,nb", CASES)
@pytest.mark.parametrize("order", ["canonical", "shuffled"])
def test_line_path_matches_oracle_and_five_launches(n, R, nb, order, monkeypatch):
    g, c, V = make_case(n, R, nb, seed=201, order=order, prec="f32")
    p, ref = _plans(n, g, monkeypatch, poison=True)
    ct, Vt = torch.from_numpy(c).cuda(), torch.from_numpy(V).cuda()
    h = torch.from_numpy(np.linspace(0.5, 2.0, len(g)).astype(np.float32)).cuda()
    out, launches = _launches(p, lambda: p.apply(ct, Vt))
    assert launches == 4    # V's transpose and three passes: the line path was taken
    want_ref, launches = _launches(ref, lambda: ref.apply(ct, Vt))
    assert launches == 5
    outh = p.apply_h(ct, Vt, h)
    ca = ct.clone()
    p.apply_h(ca, Vt, h, out=ca)
    torch.cuda.synchronize()
    pick = sorted({0, 1, nb - 1})
    want = oracle_apply(n, g, c, V, bands=pick)
    o = out.cpu().numpy()
    assert rel_l2_per_band(o[pick], want).max() < TOL["f32"]
    assert rel_l2_per_band(o, want_ref.cpu().numpy().astype(np.complex128)).max() < 3e-7
    want_h = want + h.cpu().numpy().astype(np.float64)[None, :] * c[pick].astype(np.complex128)
    assert rel_l2_per_band(outh.cpu().numpy()[pick], want_h).max() < TOL["f32"]
    assert torch.equal(ca, outh)


@pytest.mark.parametrize("n,R,nb", [((24, 24, 24), 6.0, 45), ((54, 60, 50), 12.0, 19), ((64, 64, 64), 16.0, 16),
                                    ((96, 90, 30), 7.5, 31), ((128, 120, 36), 8.5, 27)])
@pytest.mark.parametrize("order", ["canonical", "shuffled"])
def test_line_path_gamma_pairs(n, R, nb, order, monkeypatch):
    gh = synth.half_sphere(synth.sphere_glist(*n, R, order=order, seed=5))
    c = synth.coefficients(gh, nb, seed=202).astype(np.complex64)
    zero = np.flatnonzero(~gh.any(axis=1))
    c[:, zero] = c[:, zero].real
    V = synth.potential(*n, "smooth", seed=203)[0].astype(np.float32)
    p, ref = _plans(n, gh, monkeypatch, gamma=True, poison=True)
    ct, Vt = torch.from_numpy(c).cuda(), torch.from_numpy(V).cuda()
    out, launches = _launches(p, lambda: p.apply(ct, Vt))
    assert launches == 4
    want_ref = ref.apply(ct, Vt)
    h = torch.from_numpy(np.linspace(0.5, 2.0, len(gh)).astype(np.float32)).cuda()
    outh, want_h = p.apply_h(ct, Vt, h), ref.apply_h(ct, Vt, h)
    torch.cuda.synchronize()
    pick = [0, 1, nb - 1]
    want = O.gamma_apply(n, gh, c[pick].astype(np.complex128), V.astype(np.float64))
    assert rel_l2_per_band(out.cpu().numpy()[pick], want).max() < TOL["f32"]
    assert rel_l2_per_band(out.cpu().numpy(), want_ref.cpu().numpy().astype(np.complex128)).max() < 3e-7
    assert rel_l2_per_band(outh.cpu().numpy(), want_h.cpu().numpy().astype(np.complex128)).max() < 3e-7


def test_line_path_lists_chunks_and_misaligned_buffers(monkeypatch):
    # a list that is no sphere: planes and plane waves of some sticks missing,
    # every plane's sticks still a range of k around 0; ragged chunks; V and
    # the coefficients at odd offsets of their element size
    n, nb = (48, 60, 72), 29
    g = synth.sphere_glist(*n, 9.7)
    g = g[(g[:, 0] != 3) & (g[:, 0] != -9) & ~((g[:, 2] % 3 == 1) & (g[:, 1] > 2))]
    c = synth.coefficients(g, nb + 1, seed=204).astype(np.complex64)
    V = synth.potential(*n, "smooth", seed=205)[0].astype(np.float32)
    p, ref = _plans(n, g, monkeypatch, chunk=12, poison=True)
    ct = torch.from_numpy(c).cuda()[1:]    # npw odd or even: an 8-byte offset at most
    Vt = torch.empty(V.size + 1, dtype=torch.float32, device="cuda")[1:].reshape(n)
    Vt.copy_(torch.from_numpy(V))
    out, launches = _launches(p, lambda: p.apply(ct, Vt))
    assert launches == 1 + 3 * 3    # 12 + 12 + 5 bands
    want_ref = ref.apply(ct, Vt)
    torch.cuda.synchronize()
    want = oracle_apply(n, g, c[1:], V, bands=[0, 12, nb - 1])
    assert rel_l2_per_band(out.cpu().numpy()[[0, 12, nb - 1]], want).max() < TOL["f32"]
    assert rel_l2_per_band(out.cpu().numpy(), want_ref.cpu().numpy().astype(np.complex128)).max() < 3e-7
    # a gap along k within a plane, or few rows: the five launches
    g2 = g[~((g[:, 0] == 1) & (g[:, 1] == 2))]
    p2 = vloc.VlocPlan(n, g2, torch.complex64)
    assert _launches(p2, lambda: p2.apply(torch.zeros((40, len(g2)), dtype=torch.complex64, device="cuda"), Vt))[1] == 5
    assert _launches(p, lambda: p.apply(ct[:6], Vt))[1] == 5


# lengths with compile-time density kernels on x (the others keep their FP64
# group sums); group sizes 2, 4, 8 and 16, ragged last groups, several chunks
@pytest.mark.parametrize("n,R,nb,chunk,gamma", [((32, 36, 24), 6.0, 23, 0, False), ((48, 40, 36), 9.0, 37, 14, False),
                                                ((64, 64, 64), 16.0, 67, 0, False), ((96, 72, 30), 7.5, 131, 0, False),
                                                ((100, 108, 24), 6.0, 90, 40, False), ((128, 128, 32), 8.0, 33, 0, False),
                                                ((144, 120, 24), 6.0, 20, 0, False), ((60, 64, 48), 12.0, 45, 0, True),
                                                ((96, 96, 24), 6.0, 87, 20, True)])
def test_line_density(n, R, nb, chunk, gamma, monkeypatch):
    g = synth.sphere_glist(*n, R, order="shuffled", seed=6)
    if gamma:
        g = synth.half_sphere(g)
    c = synth.coefficients(g, nb, seed=206).astype(np.complex64)
    if gamma:
        zero = np.flatnonzero(~g.any(axis=1))
        c[:, zero] = c[:, zero].real
    occ = np.linspace(2.0, 0.25, nb).astype(np.float32)
    p, ref = _plans(n, g, monkeypatch, chunk=chunk, gamma=gamma, poison=True)
    ct, ot = torch.from_numpy(c).cuda(), torch.from_numpy(occ).cuda()
    rho, launches = _launches(p, lambda: p.density(ct, ot))
    m = (nb + 1) // 2 if gamma else nb
    assert launches == 3 * (-(-m // chunk) if chunk else 1)    # the line path: three launches a chunk
    rho0 = ref.density(ct, ot)
    ones = p.density(ct)
    assert torch.equal(rho, p.density(ct, ot))
    f = O.gamma_density if gamma else O.density
    want = f(n, g, c.astype(np.complex128), occ.astype(np.float64))
    err = lambda a, b: np.linalg.norm(a.cpu().numpy().astype(np.float64) - b) / np.linalg.norm(b)
    assert err(rho, want) < TOL["f32"]
    assert err(rho, rho0.cpu().numpy().astype(np.float64)) < 3e-7
    assert err(ones, f(n, g, c.astype(np.complex128), np.ones(nb))) < TOL["f32"]


@pytest.mark.parametrize("spec", [
    [(48, 8), (96, 50), (100, 41), (96, 44), (24, 5)],   # 96 twice: a group of two, then 100; the small ones beside them
    [(96, 50), (96, 47)],                                # one kind only: together
    [(90, 60), (108, 40), (120, 0), (90, 3)],            # no bands, and a small instance of a large length
])
def test_batched_groups_bit_identical(spec):
    """Instances of a captured batch that run in turn, in groups and together
    give what single calls give, captured and replayed, also where one plan
    holds two of them."""
    parts = []
    for i, (n, nb) in enumerate(spec):
        g = synth.sphere_glist(n, n, n, n / 4)
        V = torch.from_numpy(synth.potential(n, n, n, "smooth", 70 + i)[0].astype(np.float32)).cuda()
        c = torch.from_numpy(synth.coefficients(g, max(nb, 1), seed=80 + i, dtype=np.complex64)[:nb].copy()).cuda()
        parts.append((vloc.VlocPlan((n,) * 3, g, torch.complex64, graph=True), c, V))
    n, nb = spec[0]
    parts.append((parts[0][0], parts[0][1][: max(1, nb // 2)].contiguous(), parts[0][2]))  # the first plan again
    plans, cs, Vs = zip(*parts)
    ref = [vloc.VlocPlan(p.grid, p.glist, torch.complex64).apply(c, V) for p, c, V in parts]
    outs = [torch.empty_like(c) for c in cs]
    for _ in range(2):
        for o in outs:
            o.fill_(float("nan"))
        vloc.apply_batched(plans, cs, Vs, outs)
        torch.cuda.synchronize()
        for o, r in zip(outs, ref):
            assert torch.equal(o, r)
