"""The push's own launch shape for populations that do not fill the SMs: a block has as many
threads as the population needs, so that several contexts' pushes run side by side, and no
particle is lost or advanced twice at the edges between block sizes."""
import statistics
import threading
import time

import numpy as np
import pytest

from paper_2403_06706_gb300 import synth
from test_gpu_spread import WIND, _run

pytestmark = pytest.mark.gpu
gcpush = pytest.importorskip("paper_2403_06706_gb300.gcpush")
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec,n,mode", [
    (1, 152 * 128 - 1, "steady"), (1, 152 * 128, "steady"), (1, 152 * 128 + 1, "steady"), (1, 152 * 256 + 33, "steady"),
    (1, 152 * 384 + 1, "steady"), (1, 152 * 128 + 1, "time"), (1, 152 * 256 + 1, "time"),
    (0, 152 * 48 + 1, "steady"), (0, 152 * 128 + 1, "steady"), (0, 129, "time"),
])
def test_block_sizes_equal_one_thread_per_particle(prec, n, mode):
    nodes = synth.wind_grid(WIND, dtype=np.float64 if prec == 0 else np.float32)
    a, ta, sa = _run(prec, nodes, n, mode)
    b, tb, sb = _run(prec, nodes, n, mode, grid_waves=0, block=32)
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    for k in ta:
        assert np.array_equal(ta[k], tb[k]), k
    for k in ("collisions", "rebirths", "flags_or", "particle_steps"):
        assert sa[k] == sb[k], k


def test_pushes_of_several_contexts_share_the_sms():
    """Four contexts of 152 x 128 FP32 particles, one warp per scheduler each, on their own
    streams: the four together against one alone. A step of a lone warp is its chain of some
    2400 cycles for 850 instructions, so four on a scheduler take up to 3400, 1.4 times one
    alone; four times where they run one after the other. The line is drawn at 2.5."""
    nodes = synth.wind_grid(WIND, dtype=np.float32)
    steps, ctxs = 20000, []
    for k in range(4):
        c = gcpush.Context(seed=k, stream=torch.cuda.Stream())
        c.field_load(nodes, WIND.r_min_au, WIND.r_max_au)
        c.inject([synth.EnsembleSpec(152 * 128, lam_au=0.5, r_out_au=synth.r_out_default(WIND))])
        c.set_launch(steps_per_launch=steps)
        c.advance(0.5, 100)
        ctxs.append(c)

    def timed(cs):
        th = [threading.Thread(target=c.advance, args=(0.5, steps)) for c in cs]
        t0 = time.perf_counter()
        for t in th:
            t.start()
        for t in th:
            t.join()
        return time.perf_counter() - t0

    one, four = [], []
    for _ in range(4):
        one.append(timed(ctxs[:1]))
        four.append(timed(ctxs))
    for c in ctxs:
        c.close()
    print("one %.1f ms, four %.1f ms" % (1e3 * min(one), 1e3 * min(four)))
    assert min(four) < 2.5 * min(one)


def _push_ms(c, steps=200):
    """Median push time of `steps` steps over a few calls."""
    ms = []
    for _ in range(5):
        m = c.stats()["push_ms"]
        c.advance(0.5, steps)
        ms.append(c.stats()["push_ms"] - m)
    return statistics.median(ms)


def _fp64_4096():
    c = gcpush.Context(precision=gcpush.PREC_FP64, seed=3)
    c.field_load(synth.wind_grid(WIND, dtype=np.float64), WIND.r_min_au, WIND.r_max_au)
    c.inject([synth.EnsembleSpec(4096, lam_au=0.5, r_out_au=synth.r_out_default(WIND))])
    c.advance(0.5, 50)
    return c


def test_the_librarys_own_shape_can_be_asked_for_again():
    """FP64 and 4096 particles: the library's own shape takes four threads per particle, which
    measured 1.6 times as fast as blocks of 64 or 128; after such a block it has to be back."""
    with _fp64_4096() as c:
        own = _push_ms(c)
        c.set_launch(block=64)
        small = _push_ms(c)
        c.set_launch()  # keeps the block
        kept = _push_ms(c)
        c.set_launch(block=gcpush.BLOCK_OWN)
        again = _push_ms(c)
        for bad in (-2, -32, 16, 48 + 1, 160, 512):
            with pytest.raises(gcpush.GcError):
                c.set_launch(block=bad)
        print(own, small, kept, again)
        assert min(small, kept) > 1.3 * own and again < 1.1 * own


def test_autotune_keeps_four_threads_per_particle():
    """FP64 and few particles: no block is as fast as the library's own shape (1.6 times)."""
    with _fp64_4096() as c:
        own = _push_ms(c)
        best = c.autotune(0.5, trial_steps=100)
        tuned = _push_ms(c)
        print(best, own, tuned)
        assert best["own_shape"] == 1 and best["block"] in (64, 128) and best["trials"] == 24
        assert tuned < 1.1 * own


def test_autotunes_choice_is_no_slower_than_the_default():
    """64 uneven ensembles: the choice against a context's own launch shape, in turn, each over
    1000 steps with the sorts they ask for. Two runs of one shape differ by up to 3 %."""
    wl = synth.c3_batched()
    nodes = synth.wind_grid(wl.wind, dtype=np.float32)
    with gcpush.Context(precision=gcpush.PREC_FP32_MIXED, seed=wl.seed) as c:
        c.field_load(nodes, wl.wind.r_min_au, wl.wind.r_max_au)
        c.inject(list(wl.ensembles))
        c.advance(wl.dt, 500)
        best = c.autotune(wl.dt, trial_steps=200)
        block = gcpush.BLOCK_OWN if best["own_shape"] else best["block"]
        ms = {"own": [], "tuned": []}
        for _ in range(5):
            for name, shape in (("own", dict(block=gcpush.BLOCK_OWN)),
                                ("tuned", dict(block=block, sort_every=best["sort_every"], grid_waves=best["grid_waves"]))):
                c.set_launch(steps_per_launch=2000, **shape)
                a = c.stats()
                c.advance(wl.dt, 1000)
                b = c.stats()
                ms[name].append(b["push_ms"] + b["sort_ms"] - a["push_ms"] - a["sort_ms"])
    print(best, ms)
    assert statistics.median(ms["tuned"]) < 1.03 * statistics.median(ms["own"])
