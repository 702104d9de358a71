"""Loss and gradients of the predictor where the GEMM kernels' blocks end: summed
lengths just below, at and past the 128 terms a block loads at once (batch,
hidden width, features), one sample, one hidden unit, the largest M and s.

The bounds are those of test_gpu_learned.py: both sides sum at most a few hundred
float32 products in different orders behind bfloat16 weights, whose roundings
agree, so sums differ by about sqrt(300) 2^-24 of their terms' size; 1e-4 on the
loss and 1e-3 of the largest entry on each gradient leave the cancellation in
Gram-weighted errors two orders of room."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from test_gpu_learned import _oracle_params, _split, _synthetic_samples

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,s,hidden,B", [(31, 128, 129, 129), (2, 5, 1, 7), (5, 108, 128, 128),
                                          (5, 107, 127, 1), (12, 80, 160, 257)])
def test_loss_and_gradients_at_block_edges(M, s, hidden, B):
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(M + B)
    net = sa.MLP(M, s, hidden=hidden, max_batch=B, seed=3)
    flat, norm = net.get_params()
    S = _synthetic_samples(rng, M, s, B)
    loss, g = net.loss_grad(torch.from_numpy(S).cuda())
    inp = 4 * M + s
    G = S[:, inp + M:inp + M + M * M].reshape(B, M, M)
    l_ref, g_ref = omlp.loss_and_grad(_oracle_params(net, flat, norm), S[:, :inp], S[:, inp:inp + M],
                                      G, S[:, -1], dtype=np.float32, round_bf16=True)
    assert loss == pytest.approx(l_ref, rel=1e-4)
    for got, ref in zip(_split(net, g), g_ref):
        assert np.abs(got - ref).max() <= 1e-3 * np.abs(ref).max() + 1e-12
    net.close()
