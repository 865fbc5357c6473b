"""Calls whose kernels are launched programmatically behind one another, in a
caller's CUDA graph: captured behind a copy (no kernel to be behind), replayed
on changed inputs, against the same calls made directly: the same bits."""
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


def replayed(call, src, dst):
    """call(stream) reads dst, which the graph fills from src first."""
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        dst.copy_(src)
        call(st)  # plans and tensor maps exist before the capture
    st.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        dst.copy_(src)
        call(torch.cuda.current_stream())
    return graph


@pytest.mark.parametrize("M", [1, 70])
def test_projection_calls(M):
    k, tau = synth.log_grid(1e-4, 0.3, 40), synth.uniform_grid(200.0, 14000.0, 128)
    p = synth.model_params(M, seed=3)
    S = torch.as_tensor(synth.sources(k, tau, p).astype(np.float32), device="cuda")
    P = torch.as_tensor(synth.primordial(k, p), device="cuda")
    g = gcamb.grid_create(k, tau, 14000.0, 2, 300)
    for mode in (gcamb.PLAIN32, gcamb.F16X3, gcamb.BF16X3):
        gcamb.bessel_table(g, mode)
    D = gcamb.los_transfer(g, S, gcamb.PLAIN32)
    src, Sd, Dd = S.clone(), torch.empty_like(S), torch.empty_like(D)
    out = [torch.empty((M, g.nl), dtype=torch.float64, device="cuda") for _ in range(4)]
    ws = torch.empty(max(gcamb.los_cl_workspace(g, M, m) for m in (gcamb.F16X3, gcamb.BF16X3)), dtype=torch.uint8,
                     device="cuda")

    def call(st):
        gcamb.cl(g, D, P, out[0], stream=st)  # behind the copy
        gcamb.los_transfer(g, Sd, gcamb.PLAIN32, Dd, stream=st)
        gcamb.cl(g, Dd, P, out[1], stream=st)
        gcamb.los_cl(g, Sd, P, gcamb.F16X3, out[2], ws, stream=st)
        gcamb.los_cl(g, Sd, P, gcamb.BF16X3, out[3], ws, stream=st)

    graph = replayed(call, src, Sd)
    for scale in (1.0, -0.5):
        src.copy_(S * scale)
        for o in out:
            o.fill_(-1.0)
        graph.replay()
        torch.cuda.synchronize()
        got = [o.clone() for o in out]
        ref = [gcamb.cl(g, D, P), gcamb.cl(g, gcamb.los_transfer(g, src, gcamb.PLAIN32), P),
               gcamb.los_cl(g, src, P, gcamb.F16X3), gcamb.los_cl(g, src, P, gcamb.BF16X3)]
        gcamb.sync()
        for a, b in zip(got, ref):
            assert torch.equal(a, b)


@pytest.mark.parametrize("B", [40, 700])
def test_emulator_calls(B):
    g = gcamb.grid_create(synth.log_grid(1e-4, 0.3, 16), synth.uniform_grid(200.0, 14000.0, 32), 14000.0, 2, 4000)
    e, f = [gcamb.emu_create(g, width=64, depth=2, max_batch=B, seed=4) for _ in range(2)]
    rng = np.random.default_rng(1)
    X = torch.as_tensor(rng.normal(size=(B, 9)).astype(np.float32), device="cuda")
    Y = torch.as_tensor(rng.normal(size=(B, g.nl)).astype(np.float32), device="cuda")
    src, Xd = X.clone(), torch.empty_like(X)
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    out = torch.empty((B, g.nl), dtype=torch.float32, device="cuda")

    def call(st):
        gcamb.emu_train_step(e, Xd, Y, None, B, 1e-3, loss, stream=st)
        gcamb.emu_forward(e, Xd, out, stream=st)

    p0 = gcamb.emu_params(e)
    graph = replayed(call, src, Xd)
    assert np.array_equal(p0, gcamb.emu_params(f))
    for _ in range(2):  # the direct step and the replay: both with their step's own bias correction
        gcamb.emu_train_step(f, X, Y, None, B, 1e-3, loss)
        if _ == 0:
            torch.cuda.synchronize()
            assert np.array_equal(gcamb.emu_params(e), gcamb.emu_params(f))
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(gcamb.emu_params(e), gcamb.emu_params(f))
    assert torch.equal(out, gcamb.emu_forward(f, X))
    gcamb.sync()
