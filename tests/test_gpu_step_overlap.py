"""Consecutive steps overlap on the stream (a step starts while the one before it drains): the
fields must be those of steps that are waited for one by one, and of captured steps replayed."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2101_11107_gb300 import inputs as I  # noqa: E402
from paper_2101_11107_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("config", [0, 2, 4, 5, 7])
@pytest.mark.parametrize("scheme,storage", [("esoteric", "fp32"), ("ab", "fp32"), ("ab", "bf16"), ("esoteric", "fp16")])
@pytest.mark.parametrize("edge", [48, 96])
def test_overlapped_steps_equal_waited_steps(edge, scheme, storage, config):
    g = I.aneurysm(7, edge=edge, period=200.0, reynolds=40.0)
    a, b = (lbm.Domain.from_geometry(g, scheme=scheme, storage=storage) for _ in range(2))
    for d in (a, b):
        d.set_launch_config(config)
    a.step(60)
    for _ in range(60):
        b.step(1)
        b.sync()
    (ra, ua), (rb, ub) = a.macroscopic(), b.macroscopic()
    assert np.isfinite(ua).all() and np.abs(ua).max() > 0
    assert np.array_equal(ra, rb) and np.array_equal(ua, ub)


@pytest.mark.parametrize("scheme", ["esoteric", "ab"])
def test_captured_steps_replay(scheme):
    """Two steps captured in a CUDA graph on the domain's stream, replayed ten times."""
    g = I.pipe(20, 20, 16, 8.0, tau=0.6, g0=(0.0, 0.0, 1e-5), bouzidi=True)
    s = torch.cuda.Stream()
    a = lbm.Domain.from_geometry(g, scheme=scheme, stream=s)
    b = lbm.Domain.from_geometry(g, scheme=scheme)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        a.step(2)
    with torch.cuda.stream(s):
        for _ in range(10):
            graph.replay()
    s.synchronize()
    b.step(20)
    (ra, ua), (rb, ub) = a.macroscopic(), b.macroscopic()
    assert np.abs(ua).max() > 0
    assert np.array_equal(ra, rb) and np.array_equal(ua, ub)


@pytest.mark.parametrize("graph_steps", [1, 2, 5])
def test_batch_chunks_in_flight(graph_steps):
    """Many short batch chunks enqueued without waiting, each with its own level arguments (pulsatile inflow and
    force): the fields of the domains stepped alone."""
    gs = [I.aneurysm(20 + k, edge=e, period=37.0 + 5 * k, reynolds=40.0, wave_seed=50 + k) for k, e in enumerate((48, 64))]
    doms, alone = ([lbm.Domain.from_geometry(g, storage="fp32") for g in gs] for _ in range(2))
    batch = lbm.Batch(doms, graph_steps=graph_steps)
    for n in (graph_steps, 23, 1, 16):
        batch.step(n)
    batch.sync()
    for d, a in zip(doms, alone):
        a.step(graph_steps + 40)
        assert d.time == a.time
        (r1, u1), (r2, u2) = d.macroscopic(), a.macroscopic()
        assert np.abs(u1).max() > 0 and np.array_equal(r1, r2) and np.array_equal(u1, u2)
    batch.close()


def test_queued_training_steps_equal_waited_ones():
    """Training steps without a loss are only enqueued: each one's weight update has to be seen by the weight copies
    of the next one's convolutions, which run ahead of the kernels before them."""
    g = I.aneurysm(5, edge=64)
    mask = (g.mask > 0).astype(np.uint8)
    fluid = torch.from_numpy(mask).cuda()
    gen = torch.Generator("cuda").manual_seed(2)
    rho = 1.0 + 0.01 * torch.randn(mask.shape, device="cuda", generator=gen) * fluid
    u, target = (0.03 * torch.randn((3, *mask.shape), device="cuda", generator=gen) * fluid for _ in range(2))
    nets = [lbm.Corrector(mask, I.corrector_init_params(4), 0.05, 0.01, 0.005) for _ in range(2)]
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    for _ in range(12):
        assert lbm.load_library().lbm_corrector_train_step(nets[0]._h, None, None, p(rho), p(u), p(target), 1e-3, None) == 0
    for _ in range(12):
        nets[1].train_step(rho, u, target, 1e-3)
        torch.cuda.synchronize()
    queued, waited = (n.params() for n in nets)
    assert np.abs(waited - lbm.flatten_params(I.corrector_init_params(4))).max() > 1e-3
    assert np.array_equal(queued, waited)
    assert torch.equal(nets[0].forward(rho, u), nets[1].forward(rho, u))
