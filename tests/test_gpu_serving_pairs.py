"""The serving kernel of symmetric mu with 3..21 labels: every label count it
is compiled for, tiles cut by the image on either side, single pixels, more
tiles than resident blocks, and slots that retire between two iterations of
one server step while their neighbours run on."""
import numpy as np
import pytest

from paper_1511_06103_gb300 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


def alone(binding, d, iters):
    topo = binding.CRF_GRID8 if d["conn"] == 8 else binding.CRF_GRID4
    with binding.CRF(topo, d["L"], d["H"], d["W"]) as crf:
        crf.use_resident(False)
        crf.set_unary(d["U"])
        crf.set_pairwise(d["mu"], d["w"])
        crf.iterate(iters, eta=0.15)
        return crf.marginals()[0], crf.free_energy_trace(iters)[0][-1]


def serve(binding, reqs, iters, per_step, **kw):
    with binding.Server(1 << 30, **kw) as srv:
        t = [srv.submit(d["U"], d["mu"], d["w"], d["H"], d["W"], d["conn"], eta=0.15, max_iters=n)
             for d, n in zip(reqs, iters)]
        for _ in range(1000):
            srv.step(per_step)
            if all(srv.poll(k)[0] == 2 for k in t):
                break
        srv.sync()
        return [srv.poll(k) for k in t]


SHAPES = [(1, 1), (7, 1), (1, 33), (8, 32), (9, 33), (16, 64), (17, 31), (40, 97), (5, 130), (66, 40)]


@pytest.mark.parametrize("conn", [4, 8])
def test_label_counts_and_cut_tiles(conn):
    from paper_1511_06103_gb300 import binding
    labels = [3, 4, 7, 8, 11, 16, 18, 20, 21, 2]
    reqs = [synth.random_grid(h, w, L, conn, seed=60 + i, symmetric=True)
            for i, (L, (h, w)) in enumerate(zip(labels, SHAPES))]
    iters = [9 + i for i in range(len(reqs))]   # retire at different points of a step of four
    for d, n, (st, F, it, q) in zip(reqs, iters, serve(binding, reqs, iters, 4, max_slots=6)):
        q1, F1 = alone(binding, d, n)
        assert st == 2 and it == n
        assert np.abs(q - q1).max() <= 1e-5, (d["L"], d["H"], d["W"])
        assert H.f_close(F, F1, d["H"] * d["W"])


def test_more_tiles_than_resident_blocks():
    from paper_1511_06103_gb300 import binding
    reqs = [synth.random_grid(203 + 8 * i, 299 - 7 * i, L, 8, seed=90 + i, symmetric=sym)
            for i, (L, sym) in enumerate([(21, True), (8, True), (21, True), (24, True), (5, False), (21, True)])]
    iters = [6, 3, 5, 6, 6, 12]
    for d, n, (st, F, it, q) in zip(reqs, iters, serve(binding, reqs, iters, 2)):
        q1, F1 = alone(binding, d, n)
        assert st == 2 and it == n
        assert np.abs(q - q1).max() <= 1e-5, (d["L"], d["H"], d["W"])
        assert H.f_close(F, F1, d["H"] * d["W"])
