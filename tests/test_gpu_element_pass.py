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
