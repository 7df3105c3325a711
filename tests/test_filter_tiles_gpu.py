"""The cone filter's tiles: box extents around its 32 x 8 x 1 blocks, rows that are no multiple of 16 bytes, inputs
that start off a 16-byte boundary, every padding of the half widths (R from below 1 to 12), against the oracle at
the tolerance of test_filter_gpu (1e-5); and non-finite inputs, which reach exactly the outputs whose sphere holds
them."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def N():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_00234_gb300 import build
    build.build()
    from paper_2305_00234_gb300 import _native
    return _native


def rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b))


def filtered(N, x, R, beta=6.0, eta=0.5, shift=0):
    """(rho_t, rho_b) with every array starting `shift` floats after a 16-byte boundary."""
    import torch
    bufs = [torch.empty(x.size + 4, dtype=torch.float32, device="cuda")[shift:shift + x.size].view(x.shape) for _ in range(3)]
    bufs[0].copy_(torch.tensor(x, dtype=torch.float32))
    N.fdtd_filter_project(*bufs, R, beta, eta)
    torch.cuda.synchronize()
    return bufs[1], bufs[2]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("shape,R", [((1, 1, 1), 0.7), ((3, 8, 32), 1.0), ((2, 9, 33), 2.0), ((5, 7, 31), 4.0), ((4, 16, 64), 5.0),
                                     ((6, 17, 36), 5.2), ((1, 40, 65), 8.9), ((12, 8, 28), 9.0), ((25, 15, 40), 11.5),
                                     ((24, 24, 68), 12.0)])
def test_tile_edges(N, shape, R, shift):
    import torch

    from oracle import filter as OF
    rng = np.random.default_rng(int(10 * R) + shift)
    x, gb = rng.uniform(size=shape).astype(np.float32), rng.normal(size=shape).astype(np.float32)
    rt, rb = filtered(N, x, R, shift=shift)
    assert rel(rt.cpu().numpy(), OF.filter_density(x.astype(np.float64), R)) <= 1e-5
    assert rel(rb.cpu().numpy(), OF.project(rt.cpu().numpy().astype(np.float64), 6.0, 0.5)) <= 1e-5
    grad = torch.empty(shape, dtype=torch.float32, device="cuda")
    N.fdtd_filter_project_grad(rt, torch.tensor(gb, device="cuda"), grad, R, 6.0, 0.5)
    go = OF.chain_rule(gb.astype(np.float64), rt.cpu().numpy().astype(np.float64), R, 6.0, 0.5)
    assert rel(grad.cpu().numpy(), go) <= 1e-5


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("R", [1.0, 3.5, 6.0])
def test_non_finite_inputs_stay_in_their_sphere(N, R, value):
    x = np.full((11, 13, 37), 0.5, dtype=np.float32)
    at = (5, 6, 17)
    x[at] = value
    rt, _ = filtered(N, x, R)
    k, j, i = np.meshgrid(*[np.arange(s) for s in x.shape], indexing="ij")
    d2 = (k - at[0]) ** 2 + (j - at[1]) ** 2 + (i - at[2]) ** 2
    hit = np.sqrt(d2.astype(np.float32)) < np.float32(R)
    got = rt.cpu().numpy()
    assert np.array_equal(~np.isfinite(got), hit)
    assert math.isclose(float(got[~hit].min()), 0.5, rel_tol=1e-5) and math.isclose(float(got[~hit].max()), 0.5, rel_tol=1e-5)
