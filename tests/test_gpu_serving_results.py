"""A result that has reached page-locked memory but not yet q_out keeps its
memory: requests admitted in between do not overwrite it."""
import numpy as np
import pytest

from paper_1511_06103_gb300 import synth

pytestmark = pytest.mark.gpu


def run(binding, reqs, iters, slots):
    with binding.Server(1 << 28, max_slots=slots) as srv:
        t = [srv.submit(d["U"], d["mu"], d["w"], d["H"], d["W"], 8, eta=0.15, max_iters=n)
             for d, n in zip(reqs, iters)]
        for _ in range(2000):
            srv.step(4)
            if all(srv.poll(k)[0] == 2 for k in t):
                break
        srv.sync()
        return [srv.poll(k) for k in t]


@pytest.mark.parametrize("slots", [1, 3, 6])
def test_results_survive_later_admissions(slots):
    from paper_1511_06103_gb300 import binding
    reqs = [synth.random_grid(1 + 3 * (i % 5), 1 + 17 * (i % 3), (3, 8, 21, 5)[i % 4], 8, seed=60 + i, symmetric=i % 3 != 0)
            for i in range(24)]
    iters = [5 + i % 7 for i in range(24)]
    want = run(binding, reqs, iters, 64)   # all in flight at once: nothing is admitted after a result leaves
    for a, b in zip(want, run(binding, reqs, iters, slots)):
        assert a[0] == b[0] == 2 and a[2] == b[2] and a[1] == b[1]
        assert np.array_equal(a[3], b[3])
