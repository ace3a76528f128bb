"""The proposal network's kernels at the edges of their tiles: batches, widths
and outputs that are no multiple of a tile, of a 16-byte chunk or of a batch
slice, and the smallest and largest of each, against the oracle's gradients."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _bf16(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


def _rel_l2(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)


@pytest.mark.parametrize("D,H,O,B", [(1, 8, 1, 1), (128, 8, 256, 33), (65, 37, 5, 31), (63, 129, 67, 200),
                                     (111, 1024, 40, 64), (5, 320, 9, 1025)])
def test_tile_edges_match_oracle(D, H, O, B):
    """The oracle starts from the same BF16 weights and inputs; what differs is
    the BF16 rounding (2^-9) of the two activations and of the output and two
    hidden gradients: five roundings on the longest chain, doubled for what
    they do to the GELU's derivative, so 10 x 2^-9 = 2e-2 in the 2-norm."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_29663_gb300 import build
    build.build()
    import paper_2605_29663_gb300 as ex
    g = np.random.default_rng(D + H + O + B)
    m = ex.MLP(D, H, O, B + 3)
    m.init_params(1)
    W = [_bf16(w) if w.ndim == 2 else w.astype(np.float64) for w in m.unpack(m.get_params().astype(np.float64))]
    x, t = g.normal(size=(B, D)).astype(np.float32), g.normal(0.0, 0.5, size=(B, O)).astype(np.float32)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = m.forward(xd)
    loss, grads = m.loss_grad(xd, td)
    assert _rel_l2(y.cpu().numpy(), oracle.mlp_forward(W, _bf16(x))) <= 2e-2
    lo, go = oracle.mlp_loss_grad(W, _bf16(x), t.astype(np.float64))
    assert abs(loss.item() - lo) <= 2e-2 * lo
    for k, (a, b) in enumerate(zip(m.unpack(grads.cpu().numpy()), go)):
        assert _rel_l2(a, b) <= 2e-2, (k, _rel_l2(a, b))
