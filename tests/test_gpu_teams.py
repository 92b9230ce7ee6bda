"""Team launches of the linear solver: in a batch every scene is solved by a team of
CTAs of its own, instead of all scenes in lockstep over the whole grid.  Each scene's
sums keep their order, so the steps equal those of the lockstep forms bit for bit
(PPN_PCG_NO_HALO keeps the batch on them)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2505_21013_gb300")
from ppn_inputs import cube_scene, twisting_beam_scene  # noqa: E402


def beam(nx, ny, nz, seed, omega=4.0):
    return twisting_beam_scene(nx, ny, nz, h=0.02, E=1e5, nu=0.45, omega=omega, dt=1 / 30, seed=seed)


SETS = {
    # all tiles fit the device at once: one 128-row tile per CTA (rows: 27, 128, 144, 910, 1331)
    "one_tile": [cube_scene(3, seed=1), beam(4, 4, 8, 2), beam(4, 4, 9, 3), beam(7, 10, 13, 4, 20.0), cube_scene(11, seed=5)],
    # more tiles than SMs: two tiles per CTA, teams of 1 to 13 CTAs, some queued behind others
    "two_tiles": [beam(8, 8, 48 + k, 10 + k) for k in range(6)] + [cube_scene(3, seed=20), beam(4, 8, 8, 21)],
    # a scene too large for a team (its rows do not fit two tiles per SM) beside two small ones
    "too_large": [cube_scene(4, seed=30), cube_scene(35, seed=31), beam(5, 5, 12, 32)],
}
# the device has fewer SMs than the second set has tiles
SETS["two_tiles"] += [beam(8, 8, 40, 40 + k) for k in range(4)]


def run(specs, mode):
    scs = [P.Scene.from_spec(s, precision=P.PREC_MIXED) for s in specs]
    for n in range(2):
        for sc, s in zip(scs, specs):
            sc.set_targets(s.targets_at(n))
        rc, st = P.ppn_step_batch(scs, [mode] * len(scs), 1e-4)
        assert rc == 0
    out = [sc.get_displacement()[0] for sc in scs]
    layouts = [P.PCG_LAYOUTS[sc.info()["pcg_layout"]] for sc in scs]
    for sc in scs:
        sc.close()
    return out, layouts, [(x["newton_iters"], x["total_cg_iters"], x["total_projections"]) for x in st]


def test_a_long_solve_before_a_queued_one():
    # 149 CTAs iterate for more than half a second (150,000 iterations of an ill-conditioned system);
    # three members of the second team sit and wait meanwhile for CTAs that only then become free
    params = P.ppn_default_params()
    params.pcg_rel_tol, params.pcg_max_iter, params.newton_max_iter = 1e-30, 200000, 1
    long = twisting_beam_scene(9, 9, 470, h=0.02, E=1e6, nu=0.45, omega=4.0, dt=2.0, seed=3)
    short = twisting_beam_scene(10, 10, 380, h=0.02, E=1e5, nu=0.45, omega=4.0, dt=1 / 30, seed=4)
    assert long.n_verts > short.n_verts  # (the order of the jobs)
    out = []
    for batch in (True, False):
        scs = [P.Scene.from_spec(s, params=params, precision=P.PREC_MIXED) for s in (long, short)]
        for sc, s in zip(scs, (long, short)):
            sc.set_targets(s.targets_at(0))
        if batch:
            rc, st = P.ppn_step_batch(scs, [P.MODE_NEWTON] * 2, 1e-9)
        else:
            st = [sc.step(P.MODE_NEWTON, 1e-9)[2] for sc in scs]
        out.append(([(x["status"], x["total_cg_iters"]) for x in st], [sc.get_displacement()[0] for sc in scs]))
        for sc in scs:
            sc.close()
    assert out[0][0] == out[1][0] and out[0][0][0][1] > 100000
    assert all(np.array_equal(a, b) for a, b in zip(out[0][1], out[1][1]))


def test_team_tables_come_with_the_scene():
    # a scene's device memory is allocated at its creation, and device_bytes counts all of it: a
    # batch's first step, and its later ones, add only the group's own buffers (one dozen)
    torch = pytest.importorskip("torch")
    sizes = []

    def alloc(n):
        sizes.append(n)
        return torch.cuda.caching_allocator_alloc(n, device=0)

    P.ppn.set_allocator(alloc, torch.cuda.caching_allocator_delete)
    try:
        scs = [P.Scene.from_spec(beam(4, 4, 8 + k % 3, k, 10.0 + k), precision=P.PREC_MIXED) for k in range(24)]
        assert sum(sizes) == sum(sc.info()["device_bytes"] for sc in scs)
        created = len(sizes)
        for _ in range(3):
            assert P.ppn_step_batch(scs, [P.MODE_PPN] * len(scs), 1e-4)[0] == 0
        assert len(sizes) - created < len(scs)
        assert sum(sc.info()["device_bytes"] for sc in scs) == sum(sizes[:created])
        for sc in scs:
            sc.close()
    finally:
        P.ppn.set_allocator(None, None)


@pytest.mark.parametrize("name", list(SETS))
def test_teams_equal_the_lockstep_forms(name, monkeypatch):
    u, layouts, st = run(SETS[name], P.MODE_PPN)
    monkeypatch.setenv("PPN_PCG_NO_HALO", "1")
    u0, layouts0, st0 = run(SETS[name], P.MODE_PPN)
    assert st == st0
    assert all(np.array_equal(a, b) for a, b in zip(u, u0))
    assert "halo" not in layouts0
    assert [x for x in layouts if x != "halo"] == ([] if name != "too_large" else [layouts[1]])


def test_team_exits():
    # indefinite systems, the iteration cap and a converged solve beside one another: each scene's
    # step is the one it takes alone (a diagonal block of an elastic energy never fails)
    params = [P.ppn_default_params() for _ in range(4)]
    for p in params:
        p.newton_max_iter = 2
    params[2].pcg_max_iter = 5
    specs = [beam(5, 5, 12, 50), beam(5, 6, 12, 51), beam(6, 6, 12, 52), beam(6, 5, 12, 53)]
    out = []
    for batch in (True, False):
        scs = [P.Scene.from_spec(s, params=p, precision=P.PREC_MIXED) for s, p in zip(specs, params)]
        for sc, s, amp in zip(scs, specs, (3.0, 0.5, 0.0, 0.0)):
            u = amp * s.meta["h"] * np.random.default_rng(9).standard_normal(s.rest.shape)
            u[s.fixed] = 0
            sc.set_displacement(u, np.zeros_like(u))
            sc.set_targets(s.targets_at(0))
        if batch:
            P.ppn_step_batch(scs, [P.MODE_NEWTON] * 4, 1e-9)
            assert [sc.probe_solver() for sc in scs] == ["team"] * 4
        else:
            for sc in scs:
                sc.step(P.MODE_NEWTON, 1e-9)
        out.append(([(sc.iter_stats(), sc.attempts()) for sc in scs], [sc.get_displacement()[0] for sc in scs]))
        for sc in scs:
            sc.close()
    (stats, u), (stats1, u1) = out
    first = [a[0] for _, a in stats]
    assert [bool(a["ind"]) for a in first] == [True, True, False, False]
    assert first[2]["cg_iters"] == 5 and first[3]["cg_iters"] > 5
    assert repr(stats) == repr(stats1)
    assert all(np.array_equal(a, b) for a, b in zip(u, u1))
