"""The FP32 step with two nodes per thread (periodic, even nx): against the oracle, and to the bit
against the one-node kernel of the batched solver, at the edges of its blocks (128 pairs), of its rows
and of the wrap at a row's start.  Bounds are those of test_gpu_parity."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import test_gpu_parity as par  # noqa: E402

from paper_1905_10182_gb300 import BatchSolver, Solver  # noqa: E402

# a single pair per row; several rows per warp; a block ending inside a row; one row of one block; one node thick
SHAPES = [(2, 5, 3), (20, 13, 11), (66, 5, 4), (256, 2, 3), (300, 4, 1)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("name", ["periodic_uniform", "kolmogorov", "field", "shan_chen"])
def test_pair_steps_match_oracle(orc, name, shape):
    g, kw, okw, force = par._case(name, orc, shape)
    s = Solver(*shape, storage="fp32", **kw)
    if force:
        s.set_force(*force)
    s.set_populations(g)
    og = orc.Grid(*shape, collision=orc.COLL_PAPER, **okw)
    f = par.full(orc, g)
    S = par.scale(orc, f, og)
    for n in (1, 2, 3):
        s.step(1)
        f = og.step(f, 1)
        err = np.abs(s.get_populations().astype(np.float64) - par.dev(orc, f)).max()
        assert err <= n * par.C_STEP * par.EPS32 * S, (name, shape, n, err)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_pair_equals_one_node(shape):
    nx, ny, nz = shape
    rng = np.random.default_rng(7)
    rho = (1 + 0.05 * rng.random((nz, ny, nx))).astype(np.float32)
    u = [(0.05 * rng.standard_normal((nz, ny, nx))).astype(np.float32) for _ in range(3)]
    F = (3e-4, -1e-4, 2e-4)
    s = Solver(nx, ny, nz, nu=0.03)
    s.set_force("uniform", F)
    s.set_state(rho, *u)
    b = BatchSolver([dict(nx=nx, ny=ny, nz=nz, nu=0.03, force=F)])
    b.set_state(0, rho, *u)
    for n in (1, 2, 4):
        s.step(n)
        b.step(n)
        assert np.array_equal(s.get_populations(), b.get_populations(0)), n
