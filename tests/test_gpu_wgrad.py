"""The proposal's weight gradients at hit counts around the 128-hit steps and
the splits' ends, against the oracle (the bar of its other gradient test:
relative L2 1e-2, cosine 0.999, for gradients rounded to BF16 once per
factor), and with parameters and features that lie on odd 2-byte addresses:
the same bits."""
import numpy as np
import pytest

from gpu_common import cuda_ok, to_dev
from oracle import mlp
from test_gpu_learned import cosine, gpu_forward, hits, params, rel_l2, to_np_bf16

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("n", [1, 37, 128, 129, 1023, 1025, 2500])
def test_gradients_at_ragged_hit_counts(n):
    import torch
    from paper_1309_6275_gb300 import ht
    p = params(2)
    _, x, y, z, layer = hits(2500, seed=1)
    x, y, z, layer = (a[:n] for a in (x, y, z, layer))
    n = len(x)
    lab = np.random.default_rng(3).integers(-1, 64, n).astype(np.int32)
    lab[0] = 5
    pb, prob, h1, h2, feat = gpu_forward(p, x, y, z, layer)
    ws = torch.empty(ht.ht_mlp_backward_workspace_size(n), dtype=torch.uint8, device="cuda")

    def run(pb_, feat_):
        grad = torch.zeros(mlp.n_params(), dtype=torch.float32, device="cuda")
        ht.ht_mlp_backward(pb_, to_dev(lab), prob, h1, h2, feat_, grad, ws)
        torch.cuda.synchronize()
        return grad.cpu().numpy()

    g = run(pb, feat)
    _, want = mlp.loss_and_grad(p, to_np_bf16(feat)[:, :6], lab)
    k = 0
    for (i, o) in mlp.SIZES:
        for part in (i * o, o):
            a, b = g[k:k + part], want[k:k + part]
            assert rel_l2(a, b) <= 1e-2 and cosine(a, b) >= 0.999, (k, rel_l2(a, b), cosine(a, b))
            k += part

    def odd(t):
        flat = t.reshape(-1)
        b = torch.empty(flat.numel() + 1, dtype=t.dtype, device="cuda")
        b[1:].copy_(flat)
        return b[1:].view(t.shape)

    assert np.array_equal(run(odd(pb), odd(feat)).view(np.int32), g.view(np.int32))
    assert ht.ht_mlp_timeouts() == 0
