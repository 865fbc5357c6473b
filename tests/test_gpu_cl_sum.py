"""gcamb_cl / gcamb_cl_cross (Eq. 1 on stored transfers) against the FP64 sum
in plain numpy, at the sizes where the split of the k range can go wrong:
fewer k than parts, parts of one k, a ragged last part, multipoles that do
not fill a block of 32, one and several sources."""
import numpy as np
import pytest

from paper_2509_25110_gb300 import build, gcamb, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gcamb.lib()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("nk,nl,M", [(1, 1, 1), (2, 31, 3), (63, 33, 1), (64, 32, 2), (65, 129, 1), (300, 499, 1),
                                     (2049, 65, 1), (700, 1000, 40)])
def test_cl_matches_numpy(nk, nl, M, dtype):
    k = synth.log_grid(1e-4, 0.3, nk) if nk > 1 else np.array([0.01])
    g = gcamb.grid_create(k, synth.uniform_grid(200.0, 14000.0, 8), 14000.0, 2, nl + 1)
    rng = np.random.default_rng(nk + nl)
    X = torch.as_tensor(rng.standard_normal((M, nk, nl)), dtype=dtype, device="cuda")
    Y = torch.as_tensor(rng.standard_normal((M, nk, nl)), dtype=dtype, device="cuda")
    P = torch.as_tensor(rng.uniform(0.0, 2.0, (M, nk)), device="cuda")
    C = gcamb.cl(g, X, P).cpu().numpy()
    Z = gcamb.cl_cross(g, X, Y, P).cpu().numpy()
    gcamb.sync()
    _, wk = gcamb.grid_weights(g)
    w = 4.0 * np.pi * wk[None, :, None] * P.cpu().numpy()[:, :, None]
    x, y = X.cpu().numpy().astype(np.float64), Y.cpu().numpy().astype(np.float64)
    # nk + 3 roundings of 2^-53 each on the sum of magnitudes bounds either side
    tol = 2.0 * (nk + 3) * 2.0 ** -53
    assert (np.abs(C - (w * x * x).sum(1)) <= tol * (w * x * x).sum(1)).all()
    assert (np.abs(Z - (w * x * y).sum(1)) <= tol * (w * np.abs(x * y)).sum(1)).all()
    # the order of the additions does not depend on the batch
    assert np.array_equal(gcamb.cl(g, X[:1].contiguous(), P[:1].contiguous()).cpu().numpy(), C[:1])
    gcamb.sync()


@pytest.mark.parametrize("nk", [1, 2, 7, 8, 9, 40, 63])
def test_cl_of_few_k(nk):
    """Fewer k than parts: most CTAs of a cluster have nothing to sum and reach
    the write into the first one's shared memory at once.  Launched back to
    back, each result against the numpy sum (bound as above) and against one
    another."""
    k = synth.log_grid(1e-4, 0.3, nk) if nk > 1 else np.array([0.01])
    nl = 777
    g = gcamb.grid_create(k, synth.uniform_grid(200.0, 14000.0, 8), 14000.0, 2, nl + 1)
    rng = np.random.default_rng(nk)
    X = rng.standard_normal((1, nk, nl))
    P = rng.uniform(0.5, 2.0, (1, nk))
    d, p = torch.as_tensor(X, device="cuda"), torch.as_tensor(P, device="cuda")
    out = [gcamb.cl(g, d, p) for _ in range(50)]
    gcamb.sync()
    _, wk = gcamb.grid_weights(g)
    ref = 4.0 * np.pi * (wk[None, :, None] * P[:, :, None] * X * X).sum(1)
    assert (np.abs(out[0].cpu().numpy() - ref) <= 2.0 * (nk + 3) * 2.0 ** -53 * ref).all()
    assert all(torch.equal(o, out[0]) for o in out)
