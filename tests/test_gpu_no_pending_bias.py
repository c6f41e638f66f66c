"""The last layer's bias is left to the readers of its output where their kernels can add it; buffers that
those kernels cannot take (not 16-byte aligned) have it added first.  Both ways give the same gradients,
to the bit, in any order of forward, backward and graph-replayed training steps."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_10182_gb300.neural import NeuralOperator  # noqa: E402

D, W, B = 16, 32, 2


def _shifted(t):
    """The same values 4 bytes off a 16-byte boundary."""
    buf = torch.empty(t.numel() + 1, device="cuda")
    buf[1:] = t.reshape(-1)
    return buf[1:].view(t.shape)


@pytest.mark.parametrize("replayed", [False, True])
def test_gradients_do_not_depend_on_alignment(replayed):
    gen = torch.Generator(device="cuda").manual_seed(5)
    a = torch.randn((B, 4, D, D, D), generator=gen, device="cuda")
    dout = torch.randn((B, 4, D, D, D), generator=gen, device="cuda")
    net = NeuralOperator(D=D, width=W, modes=4, layers=3, max_batch=B, seed=3)
    if replayed:  # a replayed step in between leaves its own state behind
        for _ in range(3):
            net.train_step(a, dout, 1e-3)
    p = net.get_params()
    p += 0.01 * np.random.default_rng(1).standard_normal(p.size).astype(np.float32)  # non-zero biases
    net.set_params(p)
    grads = []
    for out, g in ((torch.empty_like(a), _shifted(dout)), (_shifted(torch.zeros_like(a)), _shifted(dout)),
                   (torch.empty_like(a), dout), (_shifted(torch.zeros_like(a)), dout)):
        net.forward(a, out)
        net.backward(g)
        net.backward(g)  # again on the same forward
        grads.append((out.clone(), net.get_grads()))
    assert np.array_equal(grads[0][1], grads[1][1])
    assert np.array_equal(grads[2][1], grads[3][1])
    # the aligned and the general kernels add the same products in another order
    scale = np.abs(grads[0][1]).max()
    assert np.abs(grads[0][1] - grads[2][1]).max() <= 1e-5 * scale
    assert torch.equal(grads[0][0], grads[2][0])
