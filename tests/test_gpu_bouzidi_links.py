"""The Bouzidi links of a warp's cells are shared out among its lanes in rounds of 32.  A random porous
box drives that at its edges: half-bricks with no link, a few, and several hundred (more rounds than a
warp holds in registers), cells walled on both sides of a direction, wall links without a q, q on both
sides of 1/2 and exactly 1/2."""
import dataclasses
import functools
import os

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2101_11107_gb300 import inputs as I  # noqa: E402
from paper_2101_11107_gb300 import lbm  # noqa: E402

oracle.set_threads(min(16, os.cpu_count() or 1))


def porous(fluid_fraction, seed, shape=(16, 20, 24)):
    rng = np.random.default_rng(seed)
    mask = (rng.random(shape) < fluid_fraction).astype(np.uint8)
    mask[:, 8:12, :] = 1  # an open channel: bricks without a wall
    mask[4:8] = 1
    links = I.wall_links(mask, lambda p: np.ones(p.shape[:-1]), periodic=(1, 1, 1), iters=1)
    cell, beta, _ = links
    q = rng.uniform(0.02, 1.0, len(cell))
    q[rng.random(len(q)) < 0.1] = 0.5
    keep = rng.random(len(q)) < 0.9  # the others: halfway bounce-back
    return I.Geometry(mask=mask, periodic=(1, 1, 1), links=(cell[keep], beta[keep], q[keep]), tau=0.8,
                      g0=(2e-6, 1e-6, 3e-6))


@pytest.mark.parametrize("scheme", ["esoteric", "ab"])
@pytest.mark.parametrize("fluid_fraction", [0.45, 0.8, 0.99])
def test_porous_box_against_the_oracle(fluid_fraction, scheme):
    g = porous(fluid_fraction, 11)
    ref = oracle.Case(g.mask, periodic=g.periodic, links=g.links, inlet_center=g.inlet_center,
                      inlet_radius=g.inlet_radius, tau=g.tau, g0=g.g0, gamp=g.gamp, gomega=g.gomega, tau_cell=None)
    ref.step(41)
    rho_r, u_r = ref.macroscopic()
    # the library's tolerance for FP32 populations (1e-5 of the largest velocity), any configuration
    for config in range(lbm.N_LAUNCH_CONFIGS):
        d = lbm.Domain.from_geometry(g, scheme=scheme)
        d.set_launch_config(config)
        d.step(41)
        rho, u = d.macroscopic()
        assert np.abs(u - u_r).max() <= 1e-5 * np.abs(u_r).max(), config
        assert np.abs(rho - rho_r).max() <= 1e-5, config
        d.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("collision", ["chm", "trt2"])
def test_every_configuration_gives_the_same_bits(storage, collision):
    """The two-cell kernels and A-B handle a cell's links in other ways: same fields, bit for bit."""
    g = porous(0.6, 12)
    out = []
    for scheme in ("esoteric", "ab"):
        for config in range(lbm.N_LAUNCH_CONFIGS):
            d = lbm.Domain.from_geometry(g, scheme=scheme, storage=storage, collision=collision)
            d.set_launch_config(config)
            d.step(30)
            out.append(d.macroscopic())
            d.close()
    assert np.abs(out[0][1]).max() > 0
    for rho, u in out[1:]:
        assert np.array_equal(rho, out[0][0]) and np.array_equal(u, out[0][1])


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_large_domain_gives_the_same_bits(storage):
    """A domain of more than 8192 bricks runs kernels of its own (fewer links held in registers, another default
    register budget), and a state of more than 64 MB is swept backwards on odd levels; the two-cell kernels,
    A-B and, in FP16, the twist (40 MB, one order) are the comparison."""
    g = porous(0.6, 13, shape=(64, 84, 128))
    out = []
    for scheme, configs in (("esoteric", (6, 0, 1, 2, 3, 4)), ("ab", (0, 2, 4))):
        for config in configs:
            d = lbm.Domain.from_geometry(g, scheme=scheme, storage=storage)
            assert d.info()["n_bricks"] > 8192
            d.set_launch_config(config)
            d.step(7)
            out.append(d.macroscopic(dense=False))
            d.close()
    assert np.abs(out[0][1]).max() > 0
    for rho, u in out[1:]:
        assert np.array_equal(rho, out[0][0]) and np.array_equal(u, out[0][1])


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_batches_of_porous_boxes(storage, persistent):
    """The batched kernels run the links in instances of their own: the fields of the boxes stepped alone."""
    gs = [porous(f, 20 + k) for k, f in enumerate((0.45, 0.8))]
    doms, alone = ([lbm.Domain.from_geometry(g, storage=storage) for g in gs] for _ in range(2))
    batch = lbm.Batch(doms, graph_steps=10)
    batch.set_persistent(persistent)
    for n in (10, 7, 10):
        batch.step(n)
    batch.sync()
    for d, a in zip(doms, alone):
        a.step(27)
        (r1, u1), (r2, u2) = d.macroscopic(), a.macroscopic()
        assert np.abs(u1).max() > 0 and np.array_equal(r1, r2) and np.array_equal(u1, u2)
    batch.close()


@pytest.mark.parametrize("persistent", [False, True])
def test_batch_of_more_than_8192_bricks(persistent):
    gs = [porous(0.6, 30, shape=(64, 84, 64)), porous(0.99, 31, shape=(64, 64, 64))]
    doms, alone = ([lbm.Domain.from_geometry(g) for g in gs] for _ in range(2))
    assert sum(d.info()["n_bricks"] for d in doms) > 8192
    batch = lbm.Batch(doms, graph_steps=4)
    batch.set_persistent(persistent)
    batch.step(11)
    batch.sync()
    for d, a in zip(doms, alone):
        a.step(11)
        (r1, u1), (r2, u2) = d.macroscopic(dense=False), a.macroscopic(dense=False)
        assert np.abs(u1).max() > 0 and np.array_equal(r1, r2) and np.array_equal(u1, u2)
    batch.close()


@functools.lru_cache(maxsize=1)
def _large_box():
    return porous(0.6, 14, shape=(64, 84, 128))


@pytest.mark.parametrize("storage", ["fp32", "bf16"])
@pytest.mark.parametrize("collision", ["srt2", "trt2"])
@pytest.mark.parametrize("bouzidi", [True, False])
def test_large_domain_of_the_other_operators(bouzidi, collision, storage):
    """Their kernels without links and with three rounds, against the pipelined one and A-B, bit for bit."""
    g = _large_box()
    if not bouzidi:
        g = dataclasses.replace(g, links=None)
    out = []
    for scheme, configs in (("esoteric", (0, 1, 2, 3, 4, 5)), ("ab", (2, 3))):
        for config in configs:
            d = lbm.Domain.from_geometry(g, scheme=scheme, storage=storage, collision=collision)
            d.set_launch_config(config)
            d.step(7)
            out.append(d.macroscopic(dense=False))
            d.close()
    assert np.abs(out[0][1]).max() > 0
    for rho, u in out[1:]:
        assert np.array_equal(rho, out[0][0]) and np.array_equal(u, out[0][1])
