"""A wait that runs out in a serving launch, reported by setting the word that
the launch would set: nothing that was still under way is delivered."""
import ctypes as C

import numpy as np
import pytest

from paper_1511_06103_gb300 import synth

pytestmark = pytest.mark.gpu

TIMEOUT, STATE = -5, -4


def word(binding, srv):
    f = binding.lib().proxmf_server_status_word
    f.argtypes, f.restype = [C.c_void_p], C.POINTER(C.c_int)
    return f(srv.h)


@pytest.mark.parametrize("L,sym", [(2, True), (8, True), (8, False)])
def test_nothing_is_delivered_after_a_timeout(L, sym):
    import torch
    from paper_1511_06103_gb300 import binding
    d = synth.random_grid(24, 33, L, 8, seed=L, symmetric=sym)

    def submit(srv, n):
        return srv.submit(d["U"], d["mu"], d["w"], 24, 33, 8, eta=0.2, max_iters=n)

    with binding.Server(1 << 26) as srv:
        early = submit(srv, 2)
        for _ in range(3):
            srv.step(4)
            srv.sync()
        st, _, it, q = srv.poll(early)
        assert st == 2 and it == 2
        leaving, running = submit(srv, 3), submit(srv, 100)
        srv.step(4)
        torch.cuda.synchronize()
        srv.step(0)                  # retires `leaving`: its result is on its way
        torch.cuda.synchronize()
        word(binding, srv)[0] = TIMEOUT
        for t in (leaving, running):
            with pytest.raises(binding.ProxMFError) as e:
                srv.poll(t)
            assert e.value.status == TIMEOUT
        assert not np.any(srv._keep[leaving])
        with pytest.raises(binding.ProxMFError) as e:
            srv.step(1)
        assert e.value.status in (TIMEOUT, STATE)
        assert srv.poll(early)[0] == 2 and np.array_equal(srv.poll(early)[3], q)
