"""The emulator's kernels at the edges of their tiling: widths, output counts
and batches that fill no 128 x 128 tile, more tiles than SMs (persistent
CTAs) and fewer (one tile a CTA), K of one chunk, slices of the
batch sum that are not full, gathered batches; and the fixed-point exponential
of the served spectra over its whole range and beyond it.

Bars of the network: those of test_gpu_emulator.py (its module docstring).
The exponential: y = out sd + mu + shift is rounded three times in the FP64
reference (2^-53 |y| each, relative in exp y), and either side's exp is within
two units in the last place: (2 |y| + 4) 2^-52."""
import numpy as np
import pytest

from oracle import mlp
from paper_2509_25110_gb300 import build, gcamb, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gcamb.lib()


def grid(lmax):
    return gcamb.grid_create(synth.log_grid(1e-4, 0.3, 16), synth.uniform_grid(200.0, 14000.0, 32), 14000.0, 2, lmax)


def frob_rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("width,depth,lmax,B,gather", [
    (16, 1, 9, 40, False), (33, 2, 130, 127, True), (64, 3, 129, 128, False), (130, 2, 131, 129, True),
    (128, 1, 300, 257, False), (200, 2, 2500, 1153, True), (512, 2, 40, 2500, False),
    (32, 1, 40, 20000, False), (1100, 2, 2500, 130, False)])
def test_network_at_tile_edges(width, depth, lmax, B, gather):
    g = grid(lmax)
    e = gcamb.emu_create(g, width=width, depth=depth, max_batch=B, seed=1)
    Ws, bs = mlp.init_params([9] + [width] * depth + [g.nl], seed=5)
    flat = gcamb.flatten(Ws, bs)
    gcamb.emu_params(e, flat)
    Ws32, bs32 = gcamb.unflatten(e, flat)
    rng = np.random.default_rng(6)
    n = B + 17 if gather else B
    X = rng.normal(size=(n, 9)).astype(np.float32)
    Y = rng.normal(size=(n, g.nl)).astype(np.float32)
    idx = rng.integers(0, n, B).astype(np.int32) if gather else np.arange(B, dtype=np.int32)
    Xd, Yd = torch.as_tensor(X, device="cuda"), torch.as_tensor(Y, device="cuda")
    out = gcamb.emu_forward(e, Xd[idx.astype(np.int64)].contiguous()).cpu().numpy()
    ref, cache = mlp.forward(Ws32, bs32, X[idx].astype(np.float64), rounding=True)
    assert frob_rel(out, ref) <= 1e-3
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    gcamb.emu_train_step(e, Xd, Yd, torch.as_tensor(idx, device="cuda") if gather else None, B, 1e-3, loss)
    gcamb.sync()
    Lr, dW, db = mlp.backward(Ws32, bs32, cache, Y[idx].astype(np.float64), rounding=True)
    assert abs(float(loss.item()) - Lr) <= 1e-4 * Lr
    gW, gb = gcamb.unflatten(e, gcamb.emu_grads(e))
    for l in range(len(Ws)):
        assert frob_rel(gW[l], dW[l]) <= 3e-3, ("W", l, frob_rel(gW[l], dW[l]))
        assert frob_rel(gb[l], db[l]) <= 3e-3, ("b", l, frob_rel(gb[l], db[l]))
    # the forward pass after the step runs on the updated weights' bf16 copies
    p1 = gcamb.emu_params(e)
    assert not np.array_equal(p1, flat)
    out1 = gcamb.emu_forward(e, Xd[:min(n, 64)].contiguous())
    e2 = gcamb.emu_create(g, width=width, depth=depth, max_batch=64, seed=2)
    gcamb.emu_params(e2, p1)
    out2 = gcamb.emu_forward(e2, Xd[:min(n, 64)].contiguous())
    gcamb.sync()
    assert torch.equal(out1, out2)


@pytest.mark.parametrize("B", [1, 31, 160])
def test_served_exponential(B):
    lmax = 301
    g = grid(lmax)
    e = gcamb.emu_create(g, width=32, depth=1, max_batch=256, seed=3)
    n_out = g.nl
    mu_y = np.linspace(-705.0, 705.0, n_out).astype(np.float32)  # beyond +-690: the FP64 path
    mu_y[::3] = np.linspace(-40.0, 5.0, mu_y[::3].size)
    sd_y = np.geomspace(1e-6, 2.0, n_out).astype(np.float32)
    sd_y[5], sd_y[6], sd_y[7] = 0.0, 1e-39, 1.0  # zero counts as one; subnormal: the FP64 path
    gcamb.emu_norm(e, np.zeros(9, np.float32), np.ones(9, np.float32), mu_y, sd_y)
    rng = np.random.default_rng(9)
    X = rng.normal(size=(256, 9)).astype(np.float32)
    Xd = torch.as_tensor(X, device="cuda")

    def spectra(x):
        y = gcamb.emu_forward(e, x).cpu().numpy().astype(np.float64)
        y = y * np.where(sd_y > 0, sd_y, 1.0).astype(np.float64) + mu_y.astype(np.float64)
        y = y + x[:, 8:9].cpu().numpy().astype(np.float64)
        return y, np.exp(y)

    gcamb.emu_check(e, Xd, torch.as_tensor(spectra(Xd)[1], device="cuda"), tol=1e-9, min_count=1)
    C, fb = gcamb.emulate(e, Xd[:B].contiguous())
    gcamb.sync()
    assert int(fb.sum().item()) == 0
    y, ref = spectra(Xd[:B].contiguous())
    err = np.abs(C.cpu().numpy() / ref - 1.0)
    assert (err <= (2.0 * np.abs(y) + 4.0) * 2.0 ** -52).all(), np.max(err / ((2.0 * np.abs(y) + 4.0) * 2.0 ** -52))


@pytest.mark.parametrize("lmax,B,step", [(301, 6600, 2000), (2500, 1025, 128)])
def test_persistent_ctas_give_the_same_rows(lmax, B, step):
    """Every row of a batch whose tiles outnumber the SMs against the same rows
    in batches of one tile a CTA: a row's sums know nothing of the others."""
    g = grid(lmax)
    e = gcamb.emu_create(g, width=48, depth=2, max_batch=B, seed=4)
    rng = np.random.default_rng(10)
    X = torch.as_tensor(rng.normal(size=(B, 9)).astype(np.float32), device="cuda")
    out = gcamb.emu_forward(e, X)
    parts = [gcamb.emu_forward(e, X[i:i + step].contiguous()) for i in range(0, B, step)]
    gcamb.emu_check(e, X, torch.exp(out.double() + X[:, 8:9].double()), tol=1e-9, min_count=1)
    C, fb = gcamb.emulate(e, X)
    Cp = [gcamb.emulate(e, X[i:i + step].contiguous())[0] for i in range(0, B, step)]
    gcamb.sync()
    assert int(fb.sum().item()) == 0
    assert torch.equal(out, torch.cat(parts))
    assert torch.equal(C, torch.cat(Cp))


@pytest.mark.parametrize("lmax,B", [(130, 64), (2500, 1100)])
def test_served_spectra_do_not_depend_on_the_batch(lmax, B):
    """Requests beside ones whose exponent is out of the fixed-point range, in
    amplitude (rows) and in network output (single elements): the bits they have
    among others; the ones out of range have theirs alone."""
    g = grid(lmax)
    e = gcamb.emu_create(g, width=32, depth=1, max_batch=2048, seed=3)
    sd = np.geomspace(0.05, 3.0, g.nl).astype(np.float32)
    gcamb.emu_norm(e, np.zeros(9, np.float32), np.ones(9, np.float32), np.linspace(-30.0, 5.0, g.nl).astype(np.float32), sd)
    rng = np.random.default_rng(11)
    X = rng.normal(size=(B, 9)).astype(np.float32)
    odd = np.arange(5, B, 32)
    X[odd[::2], 8] = 350.0         # amplitude
    X[odd[1::2], :8] *= 1e3        # outputs of hundreds: some of its elements
    Xd = torch.as_tensor(X, device="cuda")
    ones = torch.ones((B, g.nl), dtype=torch.float64, device="cuda")
    gcamb.emu_check(e, Xd, ones, tol=float("inf"), min_count=1)
    C, fb = gcamb.emulate(e, Xd)
    plain = torch.as_tensor(np.setdiff1d(np.arange(B), odd), device="cuda")
    Cp, _ = gcamb.emulate(e, Xd[plain].contiguous())
    Co = [gcamb.emulate(e, Xd[i:i + 1].contiguous())[0] for i in odd[:4]]
    y = gcamb.emu_forward(e, Xd).double().cpu().numpy() * sd
    gcamb.sync()
    assert int(fb.sum().item()) == 0
    assert (np.abs(y[odd[1::2]]) >= 100.0).any() and (np.abs(y[odd[1::2]]) < 100.0).any()
    assert torch.equal(C[plain], Cp)
    for i, c in zip(odd, Co):
        assert torch.equal(C[int(i)], c[0])
