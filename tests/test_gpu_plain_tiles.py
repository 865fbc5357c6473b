"""The plain transfers at the edges of their tiling: multipole tiles and row
sets that are not full, tau grids of one node, around a step, a block and the
staged chunk, the batch sizes of every sources-per-CTA variant, and both row
splits (64 rows where the grid is small, 128 where it is large), against the
FP64 oracle.

Bounds.  FP64: 1e-11 of the model's largest |Delta| (the recurrences of the
table, as in the other parity tests).  FP32, per element: table, source and
product roundings plus at most ntau / 32 + 12 additions in sequence, each
2^-24 of A = sum_i w_i |S_i| |kernel_l(x_i)|, and the terms the grid's activity
threshold leaves out, each below eps_cut = 1e-30 times w_i |S_i| (E-mode: times
c_l, the kernel's prefactor)."""
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


def make(nk, ntau, lmax, M, seed):
    k = synth.log_grid(1e-3, 0.08, nk)
    tau = synth.uniform_grid(200.0, 14000.0, ntau) if ntau > 1 else np.array([300.0])
    rng = np.random.default_rng(seed)
    S = rng.standard_normal((2, M, nk, ntau)) * (1.0 + 10.0 * rng.random((2, M, 1, 1)))
    g = gcamb.grid_create(k, tau, 14000.0, 2, lmax)
    return k, tau, S, g


CASES = [  # nk, ntau, lmax, M
    (3, 1, 2, 1), (3, 15, 3, 2), (4, 16, 33, 3), (4, 17, 34, 4), (3, 63, 65, 5), (3, 64, 128, 6), (3, 65, 129, 7),
    (2, 129, 130, 8), (2, 300, 257, 9), (2, 2049, 200, 2), (2, 2113, 70, 1), (1300, 40, 131, 1), (1300, 70, 190, 5),
]


@pytest.mark.parametrize("nk,ntau,lmax,M", CASES)
def test_fp64_fields(orc, nk, ntau, lmax, M):
    k, tau, S, g = make(nk, ntau, lmax, M, seed=nk + ntau)
    gcamb.bessel_table(g, gcamb.PLAIN64)
    d = [torch.as_tensor(s, device="cuda") for s in S]
    got = [gcamb.los_transfer(g, d[0], gcamb.PLAIN64), gcamb.los_transfer_e(g, d[1], gcamb.PLAIN64)]
    ref = [orc.los_cl(k, tau, 14000.0, 2, lmax, S[0], want_cl=False)[0], orc.los_e(k, tau, 14000.0, 2, lmax, S[1])]
    if lmax > 2:
        got += gcamb.los_transfer_tensor(g, d[0], d[1], gcamb.PLAIN64)
        ref += orc.los_tensor(k, tau, 14000.0, 2, lmax, S[0], S[1])
    gcamb.sync()
    for a, r in zip(got, ref):
        scale = np.abs(r).reshape(M, -1).max(axis=1)[:, None, None] + 1e-300
        assert (np.abs(a.cpu().numpy() - r) <= 1e-11 * scale).all(), np.max(np.abs(a.cpu().numpy() - r) / scale)
    # a source's sums do not depend on the batch it came in
    one = gcamb.los_transfer(g, d[0][M - 1:].contiguous(), gcamb.PLAIN64)
    gcamb.sync()
    assert torch.equal(one[0], got[0][M - 1])


@pytest.mark.parametrize("nk,ntau,lmax,M", CASES)
def test_fp32_fields(orc, nk, ntau, lmax, M):
    k, tau, S, g = make(nk, ntau, lmax, M, seed=nk + ntau + 1)
    S = S.astype(np.float32).astype(np.float64)
    gcamb.bessel_table(g, gcamb.PLAIN32)
    d = [torch.as_tensor(s, dtype=torch.float32, device="cuda") for s in S]
    got = [gcamb.los_transfer(g, d[0], gcamb.PLAIN32), gcamb.los_transfer_e(g, d[1], gcamb.PLAIN32)]
    gcamb.sync()
    x = k[:, None] * (14000.0 - tau)[None, :]
    j = orc.sph_bessel(lmax, x.ravel()).reshape(nk, ntau, -1)[:, :, 2:]
    l = np.arange(2, lmax + 1)[None, None, :]
    xs = np.maximum(x, 1e-3)[:, :, None]
    e = np.where(x[:, :, None] < 1e-3, np.where(l == 2, np.sqrt(24.0) / 15.0, 0.0),
                 np.sqrt((l + 2.0) * (l + 1.0) * l * (l - 1.0)) * j / xs ** 2)
    w = orc.trapz_weights(tau)
    c = np.sqrt((l + 2.0) * (l + 1.0) * l * (l - 1.0))
    for s, kern, pre, a in ((S[0], j, 1.0, got[0]), (S[1], e, c, got[1])):
        r = np.einsum("mqt,qtl->mql", s * w, kern)
        A = np.einsum("mqt,qtl->mql", np.abs(s) * w, np.abs(kern))
        tol = (ntau / 32.0 + 12.0) * 2.0 ** -24
        err = np.abs(a.cpu().numpy() - r)
        left_out = 1e-30 * pre * (np.abs(s) * w).sum(2)[:, :, None]
        assert (err <= tol * A + left_out).all(), np.max(err / (tol * A + left_out + 1e-300))


@pytest.mark.parametrize("mode,M,ntau", [(m, M, n) for m, Ms in ((gcamb.PLAIN64, (2, 3, 4, 7)), (gcamb.PLAIN32, (2, 3, 5, 8, 13)))
                                         for M in Ms for n in (2048, 2113, 4200)])
def test_long_tau_grids_of_a_batch(mode, M, ntau):
    """A source's sums are the same bits alone and in a batch, also where its
    prefix is longer than the chunk of a batch that is staged at a time:
    temperature, E-mode and tensor fields."""
    k, tau, S, g = make(4, ntau, 150, M, seed=M + ntau)
    gcamb.bessel_table(g, mode)
    d = [torch.as_tensor(s, dtype=torch.float64 if mode == gcamb.PLAIN64 else torch.float32, device="cuda") for s in S]

    def calls(a, b):
        return [gcamb.los_transfer(g, a, mode), gcamb.los_transfer_e(g, b, mode), *gcamb.los_transfer_tensor(g, a, b, mode)]

    batch = calls(*d)
    for m in (0, M - 1):
        one = calls(*(s[m:m + 1].contiguous() for s in d))
        gcamb.sync()
        for a, b in zip(one, batch):
            assert torch.equal(a[0], b[m])


@pytest.mark.parametrize("M", [1, 3, 8])
def test_fp32_lane_sums_are_rounded_once(M):
    """FP32 sums over lanes, warps and groups of tau are carried as two floats
    and rounded once.  Sources at one node per lane (every 4th of two steps, a
    warp each, and of the second group of 2048), so that what a lane adds up
    is one rounded product t s, with t read back by unit sources: the result is
    within 2^-24 of the sum of those products, and 2^-44 of their magnitudes
    (about 20 additions of pairs, each within 2^-47)."""
    k, tau, S, g = make(3, 2113, 70, M, seed=M)
    gcamb.bessel_table(g, gcamb.PLAIN32)
    nodes = np.concatenate([np.arange(0, 64, 4), 2048 + np.arange(0, 64, 4)])
    U = torch.zeros((nodes.size, k.size, tau.size), dtype=torch.float32, device="cuda")
    U[torch.arange(nodes.size), :, torch.as_tensor(nodes)] = 1.0
    t = gcamb.los_transfer(g, U, gcamb.PLAIN32).cpu().numpy()  # [node][q][l]
    s = np.random.default_rng(M).standard_normal((M, k.size, nodes.size)).astype(np.float32)
    d = torch.zeros((M, k.size, tau.size), dtype=torch.float32, device="cuda")
    d[:, :, torch.as_tensor(nodes)] = torch.as_tensor(s, device="cuda")
    got = gcamb.los_transfer(g, d, gcamb.PLAIN32).cpu().numpy().astype(np.float64)
    gcamb.sync()
    p = (t[None] * s.transpose(0, 2, 1)[:, :, :, None]).astype(np.float64)  # [m][node][q][l], products rounded to FP32
    ref = p.sum(1)
    assert (np.abs(got - ref) <= 2.0 ** -24 * np.abs(ref) + 2.0 ** -44 * np.abs(p).sum(1) + 1e-40).all()


@pytest.mark.parametrize("mode,bar", [(gcamb.PLAIN64, 1e-11), (gcamb.PLAIN32, 1e-6)])
@pytest.mark.parametrize("eps_cut", [1e-12, 1e-6, 1e-4])
def test_polarisation_rows_at_large_eps_cut(mode, bar, eps_cut):
    """Polarisation and tensor rows take their tile's whole prefix at a large
    eps_cut: only its lowest rows lose terms (a node left out has |j_l| < eps_cut at
    the lowest multipole, where x < l, and j_l falls by more than a factor of two
    every few orders above: by 2^-40 and more over 40 orders).  Rows 40.. of every
    tile against the grid of default eps_cut, within the bars of the other tests of
    the largest |Delta|."""
    k, tau, S, _ = make(60, 500, 400, 2, seed=12)
    d = [torch.as_tensor(s, dtype=torch.float64 if mode == gcamb.PLAIN64 else torch.float32, device="cuda") for s in S]

    def fields(eps):
        g = gcamb.grid_create(k, tau, 14000.0, 2, 400, eps_cut=eps)
        gcamb.bessel_table(g, mode)
        return [gcamb.los_transfer_e(g, d[1], mode), *gcamb.los_transfer_tensor(g, d[0], d[1], mode)]

    rows = torch.arange(399, device="cuda")
    rows = rows[rows % 128 >= 40]
    got, ref = fields(eps_cut), fields(0.0)
    gcamb.sync()
    for a, r in zip(got, ref):
        assert ((a - r).abs()[:, :, rows] <= bar * r.abs().max()).all(), float(((a - r).abs()[:, :, rows] / r.abs().max()).max())


@pytest.mark.parametrize("mode,bar", [(gcamb.PLAIN64, 1e-11), (gcamb.PLAIN32, 1e-6)])
@pytest.mark.parametrize("eps_cut", [1e-6, 1e-3])
def test_temperature_rows_at_large_eps_cut(mode, bar, eps_cut):
    """Temperature rows take whole blocks of 64 nodes at a large eps_cut: a grid of
    one block, whose first node has x above every multipole, loses nothing."""
    k = np.array([0.0036, 0.005, 0.02])
    tau = synth.uniform_grid(200.0, 13990.0, 64)
    S = np.random.default_rng(5).standard_normal((3, 3, 64))
    d = torch.as_tensor(S, dtype=torch.float64 if mode == gcamb.PLAIN64 else torch.float32, device="cuda")

    def field(eps):
        g = gcamb.grid_create(k, tau, 14000.0, 2, 48, eps_cut=eps)
        gcamb.bessel_table(g, mode)
        return gcamb.los_transfer(g, d, mode)

    got, ref = field(eps_cut), field(0.0)
    gcamb.sync()
    assert ((got - ref).abs() <= bar * ref.abs().max()).all(), float((got - ref).abs().max() / ref.abs().max())


def test_threads_with_grids_of_different_sizes():
    """Two host threads whose plain transfers take different amounts of shared
    memory, on their own streams: every launch succeeds and gives the bits it
    gives alone."""
    import threading
    work = []
    for ntau in (40, 7000):  # 1 KB and 60 KB
        k, tau, S, g = make(4, ntau, 40, 1, seed=ntau)
        gcamb.bessel_table(g, gcamb.PLAIN64)
        d = torch.as_tensor(S[0], device="cuda")
        work.append((g, d, gcamb.los_transfer(g, d, gcamb.PLAIN64)))
    torch.cuda.synchronize()
    bad = []

    def run(g, d, ref):
        s = torch.cuda.Stream()
        out = torch.empty_like(ref)
        try:
            for _ in range(3000):
                gcamb.los_transfer(g, d, gcamb.PLAIN64, out, stream=s)
            s.synchronize()
            if not torch.equal(out, ref):
                bad.append("values")
        except Exception as e:  # reported below, on the main thread
            bad.append(repr(e))

    ts = [threading.Thread(target=run, args=w) for w in work]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad
