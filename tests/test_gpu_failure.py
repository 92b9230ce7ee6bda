"""Failure detection on the GPU without a fault: a bounded wait that nothing
satisfies (the PCG kernels' flag-wait routine, on words no other party writes)
runs out, reports PPN_ERR_TIMEOUT to the host, and leaves the device usable."""

import re
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2505_21013_gb300")
from ppn_inputs import tiny_scene, twisting_beam_scene  # noqa: E402

PPN_ERR_TIMEOUT = 9


def test_wait_that_nothing_satisfies_reports_timeout_and_device_stays_usable():
    assert P.ppn.probe_bounded_wait(152, 4096, preset=True) == 0  # words already at the stamp
    t0 = time.perf_counter()
    assert P.ppn.probe_bounded_wait(152, 4096, preset=False) == PPN_ERR_TIMEOUT
    assert time.perf_counter() - t0 < 10.0
    # the context is intact: a scene steps normally afterwards
    spec = tiny_scene(cells=(2, 2, 2), seed=3)
    sc = P.Scene.from_spec(spec, precision=P.PREC_MIXED)
    rc, x, _ = sc.step(P.MODE_PPN, 1e-6)
    assert rc == 0 and np.isfinite(x).all()


def test_solve_whose_wait_runs_out_says_which(monkeypatch):
    # waits of the small scenes' solver limited to a poll or two run out at once: the error names the
    # wait, and another scene solves as usual afterwards
    spec = twisting_beam_scene(8, 8, 16, h=0.02, E=1e5, nu=0.45, omega=5.0, dt=1 / 30, seed=3)
    sc = P.Scene.from_spec(spec, precision=P.PREC_MIXED)
    sc.set_targets(spec.targets_at(0))
    monkeypatch.setenv("PPN_PCG_WAIT_LIMIT", "0")
    with pytest.raises(P.PPNError) as e:
        sc.step(P.MODE_PPN, 1e-4)
    sc.close()
    assert e.value.status == PPN_ERR_TIMEOUT
    m = re.search(r"wait ([23]) at CG iteration (\d+) in CTA (\d+): word 0/(-?\d+) last seen with stamp (\d+)", str(e.value))
    site, it, cta, index, seen = map(int, m.groups())
    assert cta < 32 and seen <= it
    assert -1 <= index < (32 if site == 2 else spec.n_verts)  # 32 CTAs of 32 rows; -1: the word came meanwhile
    monkeypatch.delenv("PPN_PCG_WAIT_LIMIT")
    sc = P.Scene.from_spec(spec, precision=P.PREC_MIXED)
    sc.set_targets(spec.targets_at(0))
    assert sc.step(P.MODE_PPN, 1e-4)[0] == 0
    sc.close()
