"""Label counts whose symmetric mu travels in a parameter of its own (22..28
labels), and the ones beside them, on tiles cut by the image."""
import numpy as np
import pytest

from paper_1511_06103_gb300 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def oracle():
    import oracle
    oracle.build()
    return oracle


@pytest.mark.parametrize("L,conn", [(21, 8), (22, 4), (24, 8), (25, 8), (27, 4), (28, 8), (29, 8)])
def test_steps_against_oracle(oracle, L, conn):
    from paper_1511_06103_gb300 import binding
    d = synth.random_grid(19, 45, L, conn, seed=L, symmetric=True)
    topo = binding.CRF_GRID8 if conn == 8 else binding.CRF_GRID4
    with binding.CRF(topo, L, 19, 45) as crf:
        crf.use_resident(False)
        crf.set_unary(d["U"])
        crf.set_pairwise(d["mu"], d["w"])
        crf.iterate(15, eta=0.1)
        q, tr = crf.marginals()[0], crf.free_energy_trace(15)[0]
    m = oracle.Model.grid(d["U"].astype(np.float64), d["mu"].astype(np.float64), d["w"].astype(np.float64), 19, 45,
                          conn)
    s_ref, F_ref = m.parallel_prox(float(np.float32(0.1)), 15)
    assert np.abs(q - np.exp(s_ref)).max() <= 1e-5
    assert H.f_close(tr[-1], F_ref[-2], 19 * 45)
