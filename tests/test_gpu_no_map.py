"""The hidden layers' 1x1 map and activation in one kernel (width 32): grids whose rows end inside a chunk of
8,192 positions, inside a run of 1,024 or in the first tile of 128, and one it does not take (D = 12)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from no_params import host_params  # noqa: E402
from oracle import no_oracle as no  # noqa: E402
from paper_1905_10182_gb300.neural import NeuralOperator  # noqa: E402

W, CH = 32, 4


@pytest.mark.parametrize("D,B", [(8, 1), (8, 3), (12, 2), (16, 2), (24, 3), (32, 1)])
def test_map_and_activation(D, B):
    """Mode matrices zero: the network is its dense maps, followed here in FP64 with the operands rounded to
    BF16 as the kernels round them.  FP32 sums may round an activation the other way: 2^-8 of it, through
    one weight and the projection; the bound allows four of them per output."""
    L = 3
    lay, n = no.layout(D, W, 2, L, CH, CH)
    theta = host_params((lay, n), W, 11)
    for k in range(L):
        o, shape = lay["Wm%d" % k]
        theta[o:o + math.prod(shape)] = 0.0
    net = NeuralOperator(D=D, width=W, modes=2, layers=L, max_batch=B, seed=1)
    net.set_params(theta)
    a = torch.randn((B, CH, D, D, D), generator=torch.Generator().manual_seed(D + B))
    out = net.forward(a.cuda(), torch.empty((B, CH, D, D, D), device="cuda")).cpu().double()
    par = {k: torch.from_numpy(theta[o:o + math.prod(s)].reshape(s)).double() for k, (o, s) in lay.items()}

    def bf(t):
        return t.float().to(torch.bfloat16).double()

    def dense(w, h, b):
        return torch.einsum("oc,bczyx->bozyx", w, h) + b[None, :, None, None, None]
    h, most = dense(par["P"], a.double(), par["p"]), 0.0
    for k in range(L):
        z = dense(bf(par["Wc%d" % k]), bf(h), par["b%d" % k])
        most = max(most, float(h.abs().max() * par["Wc%d" % k].abs().max()))
        h = torch.nn.functional.gelu(z) if k < L - 1 else z
    ref = dense(par["Q"], h, par["q"])
    tol = 4 * 2.0 ** -8 * most * float(par["Q"].abs().sum(1).max()) + 1e-5 * float(ref.abs().max())
    assert float((out - ref).abs().max()) <= tol
    assert float((out - ref).abs().mean()) <= 1e-4 * float(ref.abs().mean())  # and nearly all of them round alike


@pytest.mark.parametrize("D,B", [(8, 3), (16, 1), (24, 2)])
def test_whole_network_matches_oracle(D, B):
    """With the mode matrices, which take the row sums of the activations; 3 % as in test_gpu_no."""
    L, m = 3, 3
    lay = no.layout(D, W, m, L, CH, CH)
    theta = host_params(lay, W, 5)
    net = NeuralOperator(D=D, width=W, modes=m, layers=L, max_batch=B, seed=1)
    net.set_params(theta)
    a = np.random.default_rng(D).normal(size=(B, CH, D, D, D)).astype(np.float32)
    out = net.forward(torch.from_numpy(a).cuda(), torch.empty((B, CH, D, D, D), device="cuda"))
    ref = no.forward(torch.tensor(theta.astype(np.float64)), torch.tensor(a.astype(np.float64)), D, W, m, L, CH, CH).numpy()
    assert np.abs(out.cpu().numpy() - ref).max() <= 0.03 * np.abs(ref).max()
