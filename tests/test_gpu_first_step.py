"""The first step of a loop that follows crf_set_unary directly (the library's own
step size, no reset) reads the new unaries: the same bits as with a synchronisation
in between.  The steps request their unaries before they wait for the previous
launch."""
import numpy as np
import pytest

from paper_1511_06103_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,sym,bf16", [(4, True, False), (21, True, False), (21, False, False), (24, True, True)])
@pytest.mark.parametrize("graphs", [False, True])
def test_loop_right_after_new_unaries(L, sym, bf16, graphs):
    import torch
    from paper_1511_06103_gb300 import binding
    H, W = 200, 301
    d = synth.random_grid(H, W, L, 8, seed=L, symmetric=sym)
    g = torch.Generator().manual_seed(L)
    U = [torch.randn((1, H * W, L), generator=g).cuda() for _ in range(3)]
    with binding.CRF(binding.CRF_GRID8, L, H, W,
                     precision=binding.CRF_BF16 if bf16 else binding.CRF_FP32) as crf:
        crf.use_resident(False)
        crf.use_graphs(graphs)
        crf.set_unary(U[0])
        crf.set_pairwise(d["mu"], d["w"])
        crf.lipschitz()
        want = []
        for u in U:
            crf.set_unary(u)
            torch.cuda.synchronize()
            crf.iterate(2)
            want.append(crf.marginals())
        for k in range(30):
            crf.set_unary(U[k % 3])
            crf.iterate(2)
            q = torch.empty((1, H * W, L), device="cuda")
            crf.marginals(q)
            assert np.array_equal(q.cpu().numpy(), want[k % 3]), k
