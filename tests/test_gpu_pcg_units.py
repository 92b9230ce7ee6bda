"""The unit kernels of the linear solver (32-row units, the halo replicated) against the
kernels whose arithmetic they keep: FP64 scenes against the standard resident kernel,
mixed scenes of at most a tile per SM against the halo layout, the allocation-free solve
against the global-memory kernel.  Same sums in the same order, so the iterates are equal bit for bit at every size: fewer rows than a unit,
exact and ragged units and tiles, one and several units per CTA, more tiles than lanes."""

import dataclasses
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2505_21013_gb300")
from ppn_inputs import kuhn_grid, twisting_beam_scene  # noqa: E402

# rows: 8, 32, 45, 128, 156, 1024, 4864 (152 units), 6480 (two units on some CTAs), 10290 (several)
DIMS = [(2, 2, 2), (2, 4, 4), (3, 3, 5), (4, 4, 8), (3, 4, 13), (8, 8, 16), (16, 16, 19), (12, 12, 45), (14, 15, 49)]


def springs(dims, seed, indefinite=False):
    """An SPD (or, shifted, indefinite) block system on the pattern of a tet grid."""
    X, tets = kuhn_grid(*dims, h=0.1, jitter=0.01, seed=seed)
    n = len(X)
    rng = np.random.default_rng(seed)
    a = np.zeros((n, n), bool) if n < 200 else None
    pairs = np.concatenate([tets[:, [i, j]] for i in range(4) for j in range(4)]).astype(np.int64)
    key = np.unique(np.concatenate([pairs[:, 0] * n + pairs[:, 1], np.arange(n) * (n + 1)]))
    del a
    i, j = key // n, key % n
    d = X[j] - X[i]
    w = np.exp(rng.uniform(-1, 1, len(key)))
    sym = np.minimum(i, j) * n + np.maximum(i, j)  # the same weight both ways
    w = w[np.searchsorted(key, sym)]
    K = -w[:, None, None] * (d[:, :, None] * d[:, None, :] * 100 + 0.1 * np.eye(3))
    K[i == j] = 0
    D = np.zeros((n, 3, 3))
    np.add.at(D, i, -K)
    K[i == j] = D + (-0.6 if indefinite else 0.05) * np.eye(3)
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(i, minlength=n))])
    return X, row_ptr, j.astype(np.int32), K, rng.standard_normal((n, 3))


@pytest.mark.parametrize("indefinite", [False, True])
@pytest.mark.parametrize("dims", DIMS)
def test_fp64_scenes(dims, indefinite, monkeypatch):
    spec = twisting_beam_scene(*dims, h=0.1, seed=3)
    sc = P.Scene.from_spec(spec, precision=P.PREC_FP64)
    rp, col = sc.probe_pattern()
    _, rp2, col2, K, b = springs(dims, 5, indefinite)
    assert np.array_equal(rp, rp2) and np.array_equal(col, col2)
    x, info = sc.probe_pcg(K, b, rel_tol=1e-7)
    sc.close()
    monkeypatch.setenv("PPN_PCG_NO_UNITS", "1")
    sc = P.Scene.from_spec(spec, precision=P.PREC_FP64)
    x0, info0 = sc.probe_pcg(K, b, rel_tol=1e-7)
    sc.close()
    assert info == info0 and (info["ind"] or not indefinite)
    assert np.array_equal(x, x0), (np.abs(x - x0).max(), info)


# 32, 64 and 128 rows per CTA (19456 rows: the most, a tile on each SM), and the size past it
@pytest.mark.parametrize("indefinite", [False, True])
@pytest.mark.parametrize("dims", DIMS + [(16, 19, 32), (16, 16, 76), (16, 16, 77)])
def test_mixed_scenes(dims, indefinite, monkeypatch):
    spec = twisting_beam_scene(*dims, h=0.1, seed=3)
    _, _, _, K, b = springs(dims, 7, indefinite)
    out = []
    for env in (None, "PPN_PCG_NO_UNITS", "PPN_PCG_NO_HALO"):
        if env:
            monkeypatch.setenv(env, "1")
        sc = P.Scene.from_spec(spec, precision=P.PREC_MIXED)
        out.append(sc.probe_pcg(K, b, rel_tol=1e-5))
        if env is None:  # the same scene again: words of the solve before it do not count
            again = sc.probe_pcg(K, b, rel_tol=1e-5)
            assert again[1] == out[0][1] and np.array_equal(again[0], out[0][0])
        sc.close()
    for x, info in out[1:]:
        assert info == out[0][1] and (info["ind"] or not indefinite)
        assert np.array_equal(x, out[0][0]), np.abs(x - out[0][0]).max()


def test_mixed_scene_exits(monkeypatch):
    # a failing diagonal block and a zero right-hand side end the solve alike
    dims = (5, 6, 9)
    spec = twisting_beam_scene(*dims, h=0.1, seed=3)
    _, rp, col, K, b = springs(dims, 8)
    bad = K.copy()
    k = rp[77] + np.nonzero(col[rp[77]:rp[78]] == 77)[0][0]
    bad[k] = np.diag([-1.0, 2.0, 3.0])
    runs = []
    for env in (None, "PPN_PCG_NO_UNITS"):
        if env:
            monkeypatch.setenv(env, "1")
        sc = P.Scene.from_spec(spec, precision=P.PREC_MIXED)
        runs.append((sc.probe_pcg(bad, b)[1], sc.probe_pcg(K, 0 * b)[1], sc.probe_pcg(K, b, max_iter=7)))
        sc.close()
    assert runs[0][:2] == runs[1][:2] and runs[0][0]["precond_fail"] and runs[0][1]["iters"] == 0
    assert runs[0][2][1] == runs[1][2][1] and runs[0][2][1]["hit_max"]
    assert np.array_equal(runs[0][2][0], runs[1][2][0])


@pytest.mark.parametrize("dims", DIMS + [(20, 20, 80), (27, 30, 70), (32, 32, 64)])
def test_allocation_free_solve(dims, monkeypatch):
    # the scene's solve through the global-memory kernel is the reference; 32000 rows keep their
    # blocks in shared memory, 56700 and 65536 (the most that is taken) read them from L2
    spec = twisting_beam_scene(*dims, h=0.1, seed=3)
    _, rp, col, K, b = springs(dims, 6)
    monkeypatch.setenv("PPN_PCG_GLOBAL", "1")
    sc = P.Scene.from_spec(spec, precision=P.PREC_MIXED)
    x0, info0 = sc.probe_pcg(K, b, rel_tol=1e-5)
    sc.close()
    dev = torch.device("cuda", 0)
    n = len(rp) - 1
    b4 = np.zeros((n, 4), np.float32)
    b4[:, :3] = b
    d_rp, d_col = torch.tensor(rp.astype(np.int32), device=dev), torch.tensor(col, device=dev)
    d_val = torch.tensor(np.ascontiguousarray(K.reshape(-1, 9).T.astype(np.float32)), device=dev)
    d_x = torch.tensor(b4, device=dev)  # the solution may take the right-hand side's place
    info = P.ppn.pcg_solve_static(d_rp.data_ptr(), d_col.data_ptr(), d_val.data_ptr(), n, len(col), d_x.data_ptr(),
                                  d_x.data_ptr(), rel_tol=1e-5)
    assert info == info0
    assert np.array_equal(d_x[:, :3].cpu().numpy().astype(np.float64), x0)


# the comparisons above are between kernels only if each of them runs: which one does, at every size
def test_fp64_scenes_run_the_unit_kernel(monkeypatch):
    for env, want in ((None, "rd"), ("PPN_PCG_NO_UNITS", "standard")):
        if env:
            monkeypatch.setenv(env, "1")
        assert [solver(dims, P.PREC_FP64) for dims in DIMS] == [want] * len(DIMS)


def test_mixed_scenes_run_the_unit_kernel(monkeypatch):
    dims = DIMS + [(16, 19, 32), (16, 16, 76)]
    assert [solver(d, P.PREC_MIXED) for d in dims + [(16, 16, 77)]] == ["su"] * len(dims) + ["sr"]
    monkeypatch.setenv("PPN_PCG_NO_UNITS", "1")
    assert [solver(d, P.PREC_MIXED) for d in dims] == ["sr"] * len(dims)


def solver(dims, precision):
    sc = P.Scene.from_spec(twisting_beam_scene(*dims, h=0.1, seed=3), precision=precision)
    assert sc.probe_solver() == "none"
    _, _, _, K, b = springs(dims, 5)
    sc.probe_pcg(K, b, max_iter=2)
    name = sc.probe_solver()
    sc.close()
    return name


def test_allocation_free_solve_runs_the_unit_kernel():
    dev = torch.device("cuda", 0)
    for dims, want in [(d, "rd") for d in DIMS + [(20, 20, 80)]] + [((27, 30, 70), "rd_read"), ((32, 32, 64), "rd_read")]:
        _, rp, col, K, b = springs(dims, 6)
        n = len(rp) - 1
        d_rp, d_col = torch.tensor(rp.astype(np.int32), device=dev), torch.tensor(col, device=dev)
        d_val = torch.tensor(np.ascontiguousarray(K.reshape(-1, 9).T.astype(np.float32)), device=dev)
        d_x = torch.tensor(np.pad(b, ((0, 0), (0, 1))).astype(np.float32), device=dev)
        P.ppn.pcg_solve_static(d_rp.data_ptr(), d_col.data_ptr(), d_val.data_ptr(), n, len(col), d_x.data_ptr(),
                               d_x.data_ptr(), max_iter=2)
        assert P.ppn.pcg_static_solver() == want, dims


def shuffled(dims, seed):
    """A mesh whose vertices are numbered at random: every CTA's halo is spread over all the others."""
    spec = twisting_beam_scene(*dims, h=0.1, seed=3)
    X, rp, col, K, b = springs(dims, seed)
    n = len(X)
    inv = np.random.default_rng(seed).permutation(n)
    i, j = inv[np.repeat(np.arange(n), np.diff(rp))], inv[col]
    order = np.lexsort((j, i))
    rp = np.concatenate([[0], np.cumsum(np.bincount(i, minlength=n))])
    back = np.argsort(inv)
    spec = dataclasses.replace(spec, rest=spec.rest[back], tets=inv[spec.tets].astype(np.int32),
                               fixed=np.sort(inv[spec.fixed]).astype(np.int32), targets=None)
    return spec, rp, j[order].astype(np.int32), K[order], b


def on_device(rp, col, K, b):
    dev = torch.device("cuda", 0)
    return [torch.tensor(a, device=dev) for a in (
        rp.astype(np.int32), col, np.ascontiguousarray(K.reshape(-1, 9).T.astype(np.float32)),
        np.pad(b, ((0, 0), (0, 1))).astype(np.float32), np.zeros((len(b), 4), np.float32))]


def solve_static(t, **kw):
    return P.ppn.pcg_solve_static(t[0].data_ptr(), t[1].data_ptr(), t[2].data_ptr(), len(t[3]), len(t[1]),
                                  t[3].data_ptr(), t[4].data_ptr(), **kw)


# the halo rows' sort: 0, 114, 333 and 420 rows of a CTA, 838 and 1571, 1654, and 2069 and 3191, in the three unit kernels
@pytest.mark.parametrize("dims", [(2, 4, 4), (3, 4, 13), (8, 8, 16), (16, 16, 19), (16, 16, 38), (16, 19, 64), (20, 20, 60)])
def test_meshes_without_an_order(dims, monkeypatch):
    spec, rp, col, K, b = shuffled(dims, 9)
    t = on_device(rp, col, K, b)
    info = solve_static(t, rel_tol=1e-5)
    assert P.ppn.pcg_static_solver() in ("rd", "rd_read")
    runs = []
    for prec, env, tol in ((P.PREC_MIXED, "PPN_PCG_GLOBAL", 1e-5), (P.PREC_MIXED, None, 1e-5), (P.PREC_MIXED, "PPN_PCG_NO_HALO", 1e-5),
                           (P.PREC_FP64, None, 1e-7), (P.PREC_FP64, "PPN_PCG_NO_UNITS", 1e-7)):
        with monkeypatch.context() as m:
            if env:
                m.setenv(env, "1")
            sc = P.Scene.from_spec(spec, precision=prec)
            p_rp, p_col = sc.probe_pattern()
            assert np.array_equal(p_rp, rp) and np.array_equal(p_col, col)
            runs.append((*sc.probe_pcg(K, b, rel_tol=tol), sc.probe_solver()))
            sc.close()
    if len(b) <= 1024:  # (more halo rows than threads take in the mixed scenes, or than fit in FP64)
        assert runs[1][2] == "su" and runs[3][2] == "rd"
    assert info == runs[0][1] and np.array_equal(t[4][:, :3].cpu().numpy().astype(np.float64), runs[0][0])
    for a, c in ((1, 2), (3, 4)):
        assert runs[a][1] == runs[c][1] and np.array_equal(runs[a][0], runs[c][0])


def test_a_mesh_without_an_order_sets_up_as_fast():
    # 24000 rows, some 3300 halo rows per CTA: the set-up and one iteration, against the ordered mesh
    best = []
    for system in (springs((20, 20, 60), 9)[1:], shuffled((20, 20, 60), 9)[1:]):
        t = on_device(*system)
        times = []
        for _ in range(30):
            t0 = time.perf_counter()
            solve_static(t, max_iter=1)
            times.append(time.perf_counter() - t0)
        best.append(min(times))
    assert best[1] < 3 * best[0], best
