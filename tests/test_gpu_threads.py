"""Scenes of different sizes stepped by several host threads at once, a scene by one thread:
a launch with little shared memory in one thread leaves another's large launch alone."""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2505_21013_gb300")
from ppn_inputs import twisting_beam_scene  # noqa: E402


def beam(*dims):
    return twisting_beam_scene(*dims, h=0.02, E=1e5, nu=0.45, omega=20.0, dt=1 / 30, seed=3)


# the small scenes' solves take the large one's kernel with a fraction of its shared memory
FORMS = {
    "fp64": (beam(2, 2, 3), beam(12, 12, 45), P.PREC_FP64, 1),
    "mixed": (beam(2, 2, 3), beam(8, 8, 16), P.PREC_MIXED, 1),
    "teams": (beam(2, 2, 3), beam(12, 12, 45), P.PREC_MIXED, 2),
}


@pytest.mark.parametrize("form", list(FORMS))
def test_small_and_large_scenes_in_threads(form):
    small, large, prec, batch = FORMS[form]
    stop, failed = threading.Event(), []

    def loop(spec, steps):
        still = np.zeros((spec.n_verts, 3))
        scs = [P.Scene.from_spec(spec, precision=prec) for _ in range(batch)]
        try:
            for _ in range(steps):
                for sc in scs:  # from rest again, so that each step solves
                    sc.set_displacement(still, still)
                    sc.set_targets(spec.targets_at(0))
                rc = P.ppn_step_batch(scs, [P.MODE_PPN] * batch, 1e-2)[0] if batch > 1 else scs[0].step(P.MODE_PPN, 1e-2)[0]
                if rc != 0:
                    failed.append((spec.n_verts, rc))
                if stop.is_set():
                    break
        except P.PPNError as e:
            failed.append((spec.n_verts, str(e)))
        finally:
            for sc in scs:
                sc.close()

    small_ones = [threading.Thread(target=loop, args=(small, 10**6)) for _ in range(4)]
    for t in small_ones:
        t.start()
    loop(large, 150)
    stop.set()
    for t in small_ones:
        t.join()
    assert not failed, failed[:3]
