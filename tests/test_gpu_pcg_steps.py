"""The streamed layouts of the linear solver with the blocks laid out by step (rebuilt from the
matrix at each solve) against the same layouts reading them row by row (PPN_PCG_NO_STEPS) and,
where it fits, the resident layout: the same sums in the same order, so the same bits."""

import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2505_21013_gb300")
from ppn_inputs import cube_scene, twisting_beam_scene  # noqa: E402


def beam(*dims, omega=4.0, seed=3):
    return twisting_beam_scene(*dims, h=0.02, E=1e5, nu=0.45, omega=omega, dt=1 / 30, seed=seed)


def loose_tets(n):
    """Tets that share no vertex: 16 rows take more step words than their four tets' records have."""
    base = beam(2, 2, 2)
    X = np.concatenate([base.rest[base.tets[0]] + [0.1 * k, 0, 0] for k in range(n)])
    return dataclasses.replace(base, rest=X, tets=np.arange(4 * n, dtype=np.int32).reshape(n, 4),
                               fixed=np.arange(4, dtype=np.int32), targets=None)


def solve(spec, monkeypatch, *env):
    for k in ("PPN_PCG_STREAM", "PPN_PCG_SR_GLOBAL", "PPN_PCG_NO_HALO", "PPN_PCG_NO_STEPS"):
        monkeypatch.delenv(k, raising=False)
    for k in env:
        monkeypatch.setenv(k, "1")
    sc = P.Scene.from_spec(spec, precision=P.PREC_MIXED)
    b = np.random.default_rng(7).standard_normal((spec.n_verts, 3))
    b[spec.fixed] = 0
    x, info = sc.probe_pcg(sc.probe_assemble(spec.rest), b, rel_tol=1e-5, max_iter=60)
    layout = P.PCG_LAYOUTS[sc.info()["pcg_layout"]]
    sc.close()
    return x, info, layout


# rows: 12, 80 without room for the steps, 128, 156, 4864, 32000, and 67240 (526 row tiles: more than
# a thread's one in the reduction of a single scene)
SPECS = {"12": (2, 2, 3), "loose": 20, "128": (4, 4, 8), "156": (3, 4, 13), "4864": (16, 16, 19), "32000": (20, 20, 80),
         "67240": (41, 40, 41)}


@pytest.mark.parametrize("name", list(SPECS))
def test_one_scene(name, monkeypatch):
    d = SPECS[name]
    spec = loose_tets(d) if name == "loose" else beam(*d)
    runs = []
    for form, layout in (("PPN_PCG_STREAM", "streamed"), ("PPN_PCG_SR_GLOBAL", "global")):
        for env in ((form,), (form, "PPN_PCG_NO_STEPS")):
            runs.append(solve(spec, monkeypatch, *env))
            if name != "67240":  # (its vectors may not fit shared memory)
                assert runs[-1][2] == layout
    if spec.n_verts < 5000:
        runs.append(solve(spec, monkeypatch, "PPN_PCG_NO_HALO"))
        assert runs[-1][2] == "resident"
    assert runs[0][1]["iters"] > 0
    for r in runs[1:]:
        assert r[1] == runs[0][1] and np.array_equal(r[0], runs[0][0])


# several scenes in lockstep, two steps from a crumpled state, with retries: the records the steps are kept in are
# overwritten by the projections between two solves
@pytest.mark.parametrize("form", ["PPN_PCG_STREAM", "PPN_PCG_SR_GLOBAL"])
def test_scenes_in_lockstep_with_retries(form, monkeypatch):
    specs = [beam(5, 4, 12, omega=25.0), cube_scene(4, seed=2), beam(7, 6, 13, omega=25.0, seed=5)]
    out = []
    for env in ((form,), (form, "PPN_PCG_NO_STEPS")):
        for k in env:
            monkeypatch.setenv(k, "1")
        scs = [P.Scene.from_spec(s, precision=P.PREC_MIXED) for s in specs]
        for sc, s in zip(scs, specs):
            u = 0.5 * s.meta["h"] * np.random.default_rng(11).standard_normal((s.n_verts, 3))
            u[s.fixed] = 0
            sc.set_displacement(u, np.zeros_like(u))
        tot = []
        for n in range(2):
            for sc, s in zip(scs, specs):
                sc.set_targets(s.targets_at(n))
            rc, st = P.ppn_step_batch(scs, [P.MODE_PPN] * len(scs), 1e-4)
            assert rc == 0
            tot.append([(s["newton_iters"], s["total_cg_iters"], s["total_projections"]) for s in st])
        out.append((tot, [sc.get_displacement()[0] for sc in scs]))
        for sc in scs:
            sc.close()
    assert out[0][0] == out[1][0] and sum(t[2] for step in out[0][0] for t in step) > 0
    assert all(np.array_equal(a, b) for a, b in zip(out[0][1], out[1][1]))


# the halo layout's rows of other CTAs: fewer than threads, one and two a thread, and more than that.
# Vertices numbered at random give a CTA of 128 rows most of a small mesh (896 rows of 1024) or some
# 1700 rows of a larger one as its halo.
@pytest.mark.parametrize("dims,shuffled", [((8, 8, 16), False), ((8, 8, 16), True), ((16, 16, 19), True)])
def test_halo_rows_per_thread(dims, shuffled, monkeypatch):
    spec = beam(*dims)
    if shuffled:
        perm = np.random.default_rng(1).permutation(spec.n_verts)  # new number of each vertex
        rest = np.empty_like(spec.rest)
        rest[perm] = spec.rest
        spec = dataclasses.replace(spec, rest=rest, tets=perm[spec.tets].astype(np.int32),
                                   fixed=np.sort(perm[spec.fixed]).astype(np.int32), targets=None)
    monkeypatch.setenv("PPN_PCG_NO_UNITS", "1")
    a, b = solve(spec, monkeypatch), solve(spec, monkeypatch, "PPN_PCG_NO_HALO")
    assert (a[2], b[2]) == ("halo", "resident") and a[1] == b[1] and a[1]["iters"] > 20
    assert np.array_equal(a[0], b[0])
