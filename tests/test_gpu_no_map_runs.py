"""The hidden layers' map and activation kernel where a block takes several runs of tiles, short and empty
ones among them (rows of 13.5 and 1.7 chunks of 8,192 positions, more runs than blocks): a batch against its
samples one at a time, where no block takes a second run.

Forward: a sample's values do not depend on the batch it is in, to the bit.  Gradients: the samples' terms
are the same and only summed in another order, in FP32 with about 2^20 positions per sum split over 2^8
and more partial sums; 2^-24 times the square root of the terms of a thread's chain (2^12) times a few is
1e-5 of the largest entry of a block, twice that allowed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from no_params import host_params  # noqa: E402
from oracle import no_oracle as no  # noqa: E402
from paper_1905_10182_gb300.neural import NeuralOperator  # noqa: E402

W, CH, M, L = 32, 4, 4, 3


@pytest.mark.parametrize("D,B", [(48, 4), (24, 24), (8, 48)])
def test_batch_equals_its_samples(D, B):
    chunks = (D ** 3 + 8191) // 8192
    blocks = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert B * chunks * 8 > blocks >= chunks * 8
    lay = no.layout(D, W, M, L, CH, CH)
    net = NeuralOperator(D=D, width=W, modes=M, layers=L, max_batch=B, seed=1)
    net.set_params(host_params(lay, W, 21))
    gen = torch.Generator().manual_seed(D)
    a, dout = (torch.randn((B, CH, D, D, D), generator=gen).cuda() for _ in range(2))
    out = net.forward(a, torch.empty_like(a)).clone()
    net.backward(dout)
    got = net.get_grads().astype(np.float64)
    want = np.zeros_like(got)
    for b in range(B):
        one = net.forward(a[b:b + 1], torch.empty_like(a[b:b + 1]))
        assert torch.equal(one[0], out[b])
        net.backward(dout[b:b + 1])
        want += net.get_grads()
    for name, (off, shape) in lay[0].items():
        n = int(np.prod(shape))
        assert np.abs(got[off:off + n] - want[off:off + n]).max() <= 2e-5 * np.abs(want[off:off + n]).max(), name
