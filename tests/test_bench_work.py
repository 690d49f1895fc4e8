"""bench.py's algorithmic work of the adjoint: that of its steps, however many launches they take."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PANEL, ENTRIES, STEPS = 1000.0, 50, 3


@pytest.fixture(scope="module")
def work():
    spec = importlib.util.spec_from_file_location("bench", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)

    def call(sched, p, n_probes, back, fp64=False, window=0, n_orb=9):
        n = {"step": STEPS * (p // 2), "backward": STEPS * back, "window": STEPS * window}
        return mod.family_work(sched, p, n, STEPS, PANEL, ENTRIES, 8 if fp64 else 4, n_probes, n_orb, fp64, n_probes)
    return call


# K = 63: 62 adjoint steps and 63 outer products, in 63 launches where fused, 64 .. 125 where they follow 62 .. 1 steps
@pytest.mark.parametrize("n_probes,fp64,back", [(512, False, 63), (128, False, 63), (128, False, 70), (256, False, 94),
                                                (256, False, 125), (64, True, 125)])
def test_backward_flops_follow_from_the_order(work, n_probes, fp64, back):
    alg, products = work("fused", 126, n_probes, back, fp64)
    by, fl, name, prof, src = alg["backward"]
    assert fl == STEPS * (62 + 63) * 2 * ENTRIES * n_probes
    assert products == 63 + 62
    after = back - 62
    steps = 62 * (6 * PANEL + ENTRIES * (8 if fp64 else 4))
    if n_probes == 512:
        assert by == STEPS * (steps + 2 * PANEL + 63 * 16 * ENTRIES) and prof
    else:
        assert by == STEPS * (steps + 63 * 2 * PANEL + after * 16 * ENTRIES) and prof is None
        assert "+" in name


def test_other_schedules_and_the_general_form(work):
    blk = 2 * ENTRIES * 128
    alg, products = work("windowed", 126, 128, 62, window=17)
    assert alg["backward"][1] == STEPS * 62 * blk and alg["window"][1] == STEPS * 63 * blk and products == 125
    alg, products = work("tensor", 126, 128, 63, window=62)
    assert alg["backward"][1] == STEPS * 63 * blk and alg["window"][1] == STEPS * 62 * blk and products == 125
    blk = 2 * ENTRIES * 100
    alg, products = work("fused", 126, 100, 124 + 8)
    assert alg["backward"][1] == STEPS * (124 + 125) * blk
    alg, _ = work("windowed", 20, 64, 19, fp64=True)                   # FP64 has one schedule
    assert alg["backward"][1] == STEPS * (9 + 10) * 2 * ENTRIES * 64
    assert work("fused", 1, 128, 0)[0]["backward"][1] == 0
