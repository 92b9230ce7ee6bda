"""The element, assembly, reduction and projection passes at the sizes where their launch
forms change, against the FP64 oracle and plain sums."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2505_21013_gb300")
from oracle import oracle as O  # noqa: E402
from ppn_inputs import cube_scene, twisting_beam_scene  # noqa: E402


def deformed(spec, seed, amp=0.2):
    x = spec.rest + amp * spec.meta["h"] * np.random.default_rng(seed).standard_normal(spec.rest.shape)
    x[spec.fixed] = spec.rest[spec.fixed]
    return x


# tets 6 (n - 1)^3: FP64 element passes whose Hessian blocks are shared out to 12, 12, 6, 4,
# 2 and 1 CTAs, all but the last two with a ragged warp and a ragged tile
@pytest.mark.parametrize("n", [2, 6, 8, 10, 12, 13])
def test_element_parts(n):
    spec = cube_scene(n, seed=n)
    x = deformed(spec, n)
    sc, o = P.Scene.from_spec(spec, precision=P.PREC_FP64), O.Scene.from_spec(spec, O.default_params())
    _, ge, He = sc.probe_elements(x)
    _, ge_o, He_o = o.element_eval(x)
    v, vo = sc.probe_assemble(x), o.assemble(x)
    sc.close()
    for a, b in ((ge, ge_o), (He, He_o), (v, vo)):  # the FP64 stages' tolerance
        assert np.abs(a - b).max() <= 1e-10 * np.abs(b).max()


# FP32 assembly in one-warp CTAs (149k blocks) and in 8-warp CTAs (173k); the first with
# projected tets, both with ragged ends
@pytest.mark.parametrize("nz,frac", [(5, 0.3), (26, 0.3), (30, 0.0)])
def test_assembly_forms(nz, frac):
    spec = twisting_beam_scene(20, 20, nz, h=0.02, E=1e5, nu=0.45, omega=5.0, dt=1 / 30, seed=nz)
    x = deformed(spec, nz)
    proj = (np.random.default_rng(nz).random(spec.n_tets) < frac).astype(np.uint8)
    sc, o = P.Scene.from_spec(spec, precision=P.PREC_MIXED), O.Scene.from_spec(spec, O.default_params())
    v, vo = sc.probe_assemble(x, proj), o.assemble(x, proj)
    sc.close()
    assert np.abs(v - vo).max() <= 4 * 2e-5 * np.abs(vo).max()  # the mixed stages' tolerance, with projection


# vertex and tet counts at the reductions' edges: one warp, tiles of 256 and one more, and
# more than 256 tiles (several per thread of the finishing CTA)
@pytest.mark.parametrize("dims", [(2, 2, 3), (4, 8, 8), (5, 4, 13), (41, 40, 41)])
@pytest.mark.parametrize("prec", [P.PREC_FP64, P.PREC_MIXED])
def test_gradient_and_energy_reductions(dims, prec):
    spec = twisting_beam_scene(*dims, h=0.02, E=1e5, nu=0.45, omega=5.0, dt=1 / 30, seed=1)
    x = deformed(spec, 3)
    sc = P.Scene.from_spec(spec, precision=prec)
    g, norms, en = sc.probe_gradient(x, x)  # no inertia: the energy is the tets' alone
    psi = sc.probe_elements(x)[0]
    # sums of 64-bit terms by trees of depth < 32 here and in numpy: 64 roundings at most
    s2 = (g * g).sum()
    assert abs(norms[0] ** 2 - s2) <= 80 * 1.2e-16 * s2
    assert norms[1] == np.abs(g).max()
    assert abs(en - psi.sum()) <= 80 * 1.2e-16 * np.abs(psi).sum()
    # a vertex that is not a number spoils the sums, and the maximum is of the others
    y = x.copy()
    y[np.setdiff1d(np.arange(spec.n_verts), spec.fixed)[0]] = np.nan
    g, norms, en = sc.probe_gradient(y, x)
    sc.close()
    assert np.isnan(norms[0]) and np.isnan(en) and norms[1] == np.nanmax(np.abs(g), initial=0.0)


# every CTA's partials, stored by several lanes, are there when the last CTA to count sums them:
# the same bits each time, whichever CTA is the last (794 and 125 tiles)
def test_reductions_repeat():
    spec = twisting_beam_scene(20, 20, 80, h=0.02, E=1e5, nu=0.45, omega=5.0, dt=1 / 30, seed=1)
    x, y = deformed(spec, 3), deformed(spec, 4)
    sc = P.Scene.from_spec(spec, precision=P.PREC_MIXED)
    first = {k: sc.probe_gradient(p, spec.rest) for k, p in enumerate((x, y))}
    for i in range(40):  # in turn, so that a partial left from the call before would show
        g, norms, en = sc.probe_gradient((x, y)[i % 2], spec.rest)
        assert np.array_equal(norms, first[i % 2][1]) and en == first[i % 2][2]
    sc.close()


# state in and out: around one CTA's 128 vertices, the pinned buffer's 16384 (a second piece on
# the way in, the copy engine on the way out), and targets that do not fit the buffer (34848)
@pytest.mark.parametrize("dims", [(2, 2, 2), (4, 4, 8), (3, 43, 1 + 2), (32, 32, 16), (5, 29, 113), (33, 33, 33)])
@pytest.mark.parametrize("prec", [P.PREC_FP64, P.PREC_MIXED])
def test_state_in_and_out(dims, prec):
    import dataclasses
    spec = twisting_beam_scene(*dims, h=0.02, E=1e5, nu=0.45, omega=5.0, dt=1 / 30, seed=2)
    n = spec.n_verts
    fixed = np.arange(n - dims[0] * dims[1], dtype=np.int32)  # all but the last layer
    spec = dataclasses.replace(spec, fixed=fixed, targets=None)
    rng = np.random.default_rng(n)
    u, v, w = (rng.standard_normal((n, 3)) for _ in range(3))
    sc = P.Scene.from_spec(spec, precision=prec)
    sc.set_displacement(u, v)
    a, b = sc.get_displacement()
    assert np.array_equal(a, u) and np.array_equal(b, v)
    X = spec.rest
    a, b = sc.get_state()
    assert np.array_equal(a, X + u) and np.array_equal(b, v)
    sc.set_state(X + w, u)
    a, b = sc.get_displacement()
    assert np.array_equal(a, (X + w) - X) and np.array_equal(b, u)
    # one of the two alone leaves the other as it is
    L, d = P.ppn.lib(), P.ppn._d
    assert L.ppn_set_displacement(sc._h, d(w), None) == 0 and L.ppn_set_state(sc._h, None, d(w)) == 0
    a = np.full((n, 3), 7.0)
    b = np.full((n, 3), 7.0)
    assert L.ppn_get_displacement(sc._h, d(a), None) == 0 and L.ppn_get_state(sc._h, None, d(b)) == 0
    assert np.array_equal(a, w) and np.array_equal(b, w)
    # targets take effect at the step's start: the fixed vertices end on them
    sc.set_displacement(np.zeros((n, 3)), np.zeros((n, 3)))
    t = X[fixed] + 1e-5 * rng.standard_normal((len(fixed), 3))
    sc.set_targets(t)
    sc.step(P.MODE_PPN, 1e-2)
    a = sc.get_displacement()[0]
    sc.close()
    assert np.array_equal(a[fixed], t - X[fixed])


# the one-thread-per-tet projection (forced for the short lists too) at the ends of a warp and
# a CTA, on rest, inverted and clamped tets: the oracle's eigenvalue clamping
@pytest.mark.parametrize("n_sel", [1, 31, 33, 127, 129, 750])
@pytest.mark.parametrize("prec", [P.PREC_FP64, P.PREC_MIXED])
def test_projection_forms(n_sel, prec, monkeypatch):
    spec = cube_scene(6, seed=3)
    x = deformed(spec, 4, amp=0.8)
    x[: spec.n_verts // 3] = spec.rest[: spec.n_verts // 3]  # tets at rest: many zero pairs in the rotations
    sel = np.sort(np.random.default_rng(n_sel).permutation(spec.n_tets)[:n_sel]).astype(np.int32)
    mask = np.zeros(spec.n_tets, np.uint8)
    mask[sel] = 1
    monkeypatch.setenv("PPN_PROJECT_THREAD", "1")
    sc, o = P.Scene.from_spec(spec, precision=prec), O.Scene.from_spec(spec, O.default_params())
    He, dH = sc.probe_elements(x)[2], sc.probe_project(x, sel)
    v, vo = sc.probe_assemble(x, mask), o.assemble(x, mask)
    sc.close()
    tol = 1e-9 if prec == P.PREC_FP64 else 8e-5
    w = np.linalg.eigvalsh(He[sel] + dH)
    assert w.min() >= -tol * np.abs(He).max()  # clamped: no negative eigenvalue is left
    assert np.abs(v - vo).max() <= tol * np.abs(vo).max()
