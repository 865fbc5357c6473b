"""The integer recurrences of the Bessel tables where they change branch: x at
and around 1 and whole numbers, the match at ls or ls - 1, orders cut below,
at and above x, x beyond every order, lanes of one warp whose orders lie far
apart (each then keeps its own Miller start) or close together, tables of
sampled multipoles, and activity thresholds down to the smallest the grid
takes.  Against the FP64 oracle with the bars of the other parity tests:
1e-11 of the order's envelope (sph_bessel), of the largest |Delta| (tables)."""
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


def check_rows(orc, x, lmax):
    out = gcamb.sph_bessel(torch.as_tensor(x, device="cuda"), lmax).cpu().numpy()
    gcamb.sync()
    ref = orc.sph_bessel(lmax, x)
    l = np.arange(lmax + 1)[None, :]
    env = np.where(l > x[:, None], np.abs(ref), np.maximum(np.abs(ref), 1.0 / np.maximum(x[:, None], 1e-300)))
    err = np.abs(out - ref)
    ok = err <= 1e-11 * env + 1e-40
    assert ok.all(), (np.argwhere(~ok)[:5], x[np.argwhere(~ok)[:5, 0]], err[~ok][:5], ref[~ok][:5])


@pytest.mark.parametrize("lmax", [0, 1, 2, 3, 7, 64, 700])
def test_orders_at_branch_points(orc, lmax):
    n = np.array([1.0, 2.0, 3.0, 4.0, 7.0, 8.0, 31.0, 63.0, 64.0, 65.0, 700.0, 701.0])
    x = np.concatenate([[0.0, 1e-300, 1e-20, 1e-3, 0.5, np.nextafter(1.0, 0.0), np.pi, 2 * np.pi, 4.4934094579],
                        n, np.nextafter(n, 0.0), np.nextafter(n, 1e9), n + 0.5, [5000.0, 20000.0, 3.0e5]])
    check_rows(orc, x, lmax)
    # the same nodes one to a warp neighbourhood of their own
    check_rows(orc, np.repeat(x, 32)[:32 * 12], lmax)


def test_orders_of_neighbouring_nodes(orc):
    # as in a table: x falls along the lanes, in small and in large steps
    for step in (0.01, 1.3, 4.1, 40.0):
        x = np.maximum(1900.0 - step * np.arange(160), 0.3)
        check_rows(orc, x, 2200)


@pytest.mark.parametrize("ntau,eps_cut,boost", [(40, 0.0, 1.0), (40, 1e-200, 1.0), (300, 1e-200, 3.0), (300, 0.0, 50.0)])
@pytest.mark.parametrize("mode", [gcamb.PLAIN64, gcamb.PLAIN32])
def test_tables(orc, ntau, eps_cut, boost, mode):
    k = synth.log_grid(1e-4, 0.1, 23)
    tau = synth.uniform_grid(200.0, 14000.0, ntau)
    lmax = 500
    rows = gcamb.l_sampling(2, lmax, boost)
    S = np.random.default_rng(ntau).standard_normal((2, k.size, ntau))
    g = gcamb.grid_create_lsampled(k, tau, 14000.0, rows, eps_cut=eps_cut)
    gcamb.bessel_table(g, mode)
    dt = torch.float64 if mode == gcamb.PLAIN64 else torch.float32
    D = gcamb.los_transfer(g, torch.as_tensor(S, dtype=dt, device="cuda"), mode).cpu().numpy()
    gcamb.sync()
    ref = orc.los_cl(k, tau, 14000.0, 2, lmax, S, want_cl=False)[0][:, :, rows - 2]
    scale = np.abs(ref).reshape(2, -1).max(axis=1)[:, None, None]
    assert (np.abs(D - ref) <= (1e-11 if mode == gcamb.PLAIN64 else 1e-5) * scale).all()


@pytest.mark.parametrize("lmax,hi", [(40, 60.0), (700, 900.0), (2200, 2300.0)])
def test_values_do_not_depend_on_neighbours(lmax, hi):
    """j_l of a node is the same bits alone and among others, in any order."""
    rng = np.random.default_rng(lmax)
    x = torch.as_tensor(rng.uniform(0.2, hi, 300), device="cuda")
    all_ = gcamb.sph_bessel(x, lmax)
    p = torch.as_tensor(rng.permutation(300), device="cuda")
    assert torch.equal(gcamb.sph_bessel(x[p].contiguous(), lmax), all_[p])
    for i in (0, 17, 299):
        assert torch.equal(gcamb.sph_bessel(x[i:i + 1].contiguous(), lmax), all_[i:i + 1])
    gcamb.sync()


@pytest.mark.parametrize("lmax", [0, 1, 2, 7, 300])
def test_infinite_and_nan_arguments(lmax):
    """No finite j_l: every order is NaN, and the values beside them are theirs."""
    x = np.array([0.5, np.nan, 3.0, np.inf, 400.0, -np.nan, 0.0])
    out = gcamb.sph_bessel(torch.as_tensor(x, device="cuda"), lmax).cpu().numpy()
    fin = gcamb.sph_bessel(torch.as_tensor(x[[0, 2, 4, 6]], device="cuda"), lmax).cpu().numpy()
    gcamb.sync()
    assert np.isnan(out[[1, 3, 5]]).all()
    assert np.array_equal(out[[0, 2, 4, 6]], fin)


@pytest.mark.parametrize("x", [1e20, 1e100, 1e285, 1e290, 1e295, 8e299])
def test_huge_arguments(x):
    """x far beyond every order: j_l(x) = sin(x - l pi / 2) / x but for l (l+1) / (2x),
    within 1e-11 of 1/x, up to the documented 1e-300."""
    lmax = 50
    out = gcamb.sph_bessel(torch.as_tensor([x], dtype=torch.float64, device="cuda"), lmax).cpu().numpy()[0]
    gcamb.sync()
    s, c = np.sin(x), np.cos(x)
    ref = np.array([(s, -c, -s, c)[l % 4] for l in range(lmax + 1)]) / x
    assert (np.abs(out - ref) <= 1e-11 / x + 1e-300 * (np.abs(ref) < 1e-300)).all(), (out, ref)


def test_arguments_below_zero():
    """Outside the documented range, as ever: j_0 = 1, j_1 = x/3, the others 0."""
    x = np.array([-1e-160, -0.25, -5.0])
    out = gcamb.sph_bessel(torch.as_tensor(x, device="cuda"), 4).cpu().numpy()
    gcamb.sync()
    ref = np.zeros((3, 5))
    ref[:, 0], ref[:, 1] = 1.0, x / 3.0
    assert np.array_equal(out, ref)


@pytest.mark.parametrize("x0", [11900.0, 14990.0, 19900.0])
def test_highest_orders(orc, x0):
    """Orders up to the highest, at x where x j_l(x) comes closest to the limit of
    the fixed-point numbers (4.41 of 8 at x = 20000)."""
    x = np.concatenate([x0 + np.linspace(0.0, 200.0, 41), [x0 + 97.3]])
    out = gcamb.sph_bessel(torch.as_tensor(x, device="cuda"), 20000).cpu().numpy()
    gcamb.sync()
    assert np.abs(out[:, :int(x0)] * x[:, None]).max() > 4.0
    check_rows(orc, x, 20000)
