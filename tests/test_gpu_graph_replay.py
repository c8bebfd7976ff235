"""Replayed step loops follow the model: after a new mu, one of the other
symmetry, and new weights under the same mu, a handle that replays gives the
same bits as one that launches step by step."""
import numpy as np
import pytest

from paper_1511_06103_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,bf16", [(5, False), (21, False), (22, False), (24, False), (28, False), (32, False),
                                    (24, True), (27, True), (32, True)])
def test_new_model_on_a_handle_that_replays(L, bf16):
    from paper_1511_06103_gb300 import binding
    H, W, conn = 19, 45, 8
    models = [synth.random_grid(H, W, L, conn, seed=L + k, symmetric=sym)
              for k, sym in enumerate((True, True, False, True))]
    steps = [(d["mu"], d["w"]) for d in models]
    steps.insert(2, (models[1]["mu"], models[0]["w"]))   # new weights, the same mu
    got = {}
    for replay in (False, True):
        with binding.CRF(binding.CRF_GRID8, L, H, W,
                         precision=binding.CRF_BF16 if bf16 else binding.CRF_FP32) as crf:
            crf.use_resident(False)
            crf.use_graphs(replay)
            crf.set_unary(models[0]["U"])
            got[replay] = []
            for mu, w in steps:
                crf.set_pairwise(mu, w)
                for _ in range(2):   # recorded, replayed
                    crf.iterate(6, eta=0.1, reset=True, refine_fp32=2 if bf16 else 0)
                got[replay].append((crf.marginals(), crf.free_energy_trace(6)))
    for (q, F), (q2, F2) in zip(got[False], got[True]):
        assert np.array_equal(q, q2) and np.array_equal(F, F2)
