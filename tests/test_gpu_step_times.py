"""Times that must stand in a known relation to one another, whatever the GPU's clock: a step that moves half
the bytes of another, or does less arithmetic, is not the slower one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2101_11107_gb300 import inputs as I  # noqa: E402
from paper_2101_11107_gb300 import lbm  # noqa: E402


def gpu_us(fn, n=1, repeats=7):
    """Median device time of one of the n things that fn does."""
    fn()
    out = []
    for _ in range(repeats):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        out.append(a.elapsed_time(b) * 1e3 / n)
    return float(np.median(out))


@pytest.fixture(scope="module")
def large_pipe():
    """19 k bricks, 1.2 M cells, interpolated walls: larger than L2 in every storage with two arrays."""
    return I.pipe(96, 96, 192, 44.3, tau=0.55, gamp=(0.0, 0.0, 1e-5), gomega=0.001, bouzidi=True)


@pytest.mark.parametrize("storage", ["fp16", "bf16"])
@pytest.mark.parametrize("collision", ["chm", "trt2"])
def test_16_bit_ab_step_is_no_slower_than_fp32(large_pipe, collision, storage):
    """Half the bytes and the same number of loads (5% for the spread of the times)."""
    t = {}
    for st in ("fp32", storage):
        d = lbm.Domain.from_geometry(large_pipe, storage=st, scheme="ab", collision=collision)
        t[st] = gpu_us(lambda: d.step(40), 40)
        d.close()
    assert t[storage] <= 1.05 * t["fp32"], t


@pytest.mark.parametrize("scheme", ["esoteric", "ab"])
@pytest.mark.parametrize("case", ["default", "rates", "srt2", "trt2"])
def test_default_configuration_is_a_fast_one(large_pipe, case, scheme):
    """The configuration that a large domain starts with is within 8% of the best of the one-cell kernels."""
    kw = dict(default={}, rates=dict(omega_hi=(1.2, 1.1, 1.05, 0.95))).get(case, dict(collision=case))
    d = lbm.Domain.from_geometry(large_pipe, scheme=scheme, **kw)
    first = d.info()["launch_config"]
    t = gpu_us(lambda: d.step(40), 40)
    times = {}
    for c in range(5):
        d.set_launch_config(c)
        assert d.info()["launch_config"] == c
        times[lbm.LAUNCH_CONFIG_NAMES[c]] = gpu_us(lambda: d.step(40), 40)
    d.close()
    assert t <= 1.08 * min(times.values()), (lbm.LAUNCH_CONFIG_NAMES[first], t, times)
    # the name is that of the kernel that runs
    assert abs(t - times[lbm.LAUNCH_CONFIG_NAMES[first]]) <= 0.05 * t, (lbm.LAUNCH_CONFIG_NAMES[first], t, times)


def test_default_configuration_by_size():
    """6 CTAs per SM up to 8192 bricks; 8 above, but for the twist of TRT2 with links."""
    small = I.pipe(32, 32, 64, 12.0, tau=0.6, g0=(0.0, 0.0, 1e-6))
    large = I.pipe(64, 64, 256, 28.0, tau=0.6, g0=(0.0, 0.0, 1e-6))
    linked = I.pipe(64, 64, 256, 28.0, tau=0.6, g0=(0.0, 0.0, 1e-6), bouzidi=True)
    for g, kw, want in ((small, {}, "128x6"), (large, {}, "128x8"), (large, dict(collision="trt2"), "128x8"),
                        (linked, {}, "128x8"), (linked, dict(collision="trt2"), "128x6"),
                        (linked, dict(collision="trt2", scheme="ab"), "128x8")):
        d = lbm.Domain.from_geometry(g, **kw)
        assert lbm.LAUNCH_CONFIG_NAMES[d.info()["launch_config"]] == want
        d.set_launch_config(2)
        assert d.info()["launch_config"] == 2
        d.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_persistent_batch_with_default_rates_is_the_fastest(storage):
    """The default rates leave out the higher moments, which general rates compute on top (5% for the spread of
    the times; nothing else differs)."""
    gs = [I.aneurysm(300 + k, edge=e) for k, e in enumerate((96, 112))]
    t = {}
    for rates in ((1.0, 1.0, 1.0, 1.0), (1.2, 1.1, 1.05, 0.95)):
        doms = [lbm.Domain.from_geometry(g, storage=storage, omega_hi=rates) for g in gs]
        batch = lbm.Batch(doms, graph_steps=50)
        batch.set_persistent(True, 1.0)
        t[rates] = gpu_us(lambda: batch.step(50), 50)
        batch.sync()
        batch.close()
        for d in doms:
            d.close()
    assert t[(1.0, 1.0, 1.0, 1.0)] <= 1.05 * t[(1.2, 1.1, 1.05, 0.95)], t


def test_restriction_of_a_full_box_is_no_slower_than_a_copy():
    """It reads the fine fields and a mask byte per cell and writes an eighth: 0.6 of a copy's bytes."""
    n = 256
    rho, u = torch.rand((n, n, n), device="cuda"), torch.rand((3, n, n, n), device="cuda")
    mask = torch.ones((n, n, n), dtype=torch.uint8, device="cuda")
    rho2, u2 = torch.empty_like(rho), torch.empty_like(u)
    t = gpu_us(lambda: [lbm.restrict(rho, u, mask) for _ in range(10)], 10)
    copy = gpu_us(lambda: [(rho2.copy_(rho), u2.copy_(u)) for _ in range(10)], 10)
    assert t <= copy, (t, copy)


def test_forward_on_a_nearly_empty_box_costs_its_clear():
    """One tile of fluid in a 256^3 box: the pass on a small box with the same tile, and a clear of the correction
    (1.5 for the spread and the clear's own launch)."""
    def forward(n):
        mask = np.zeros((n, n, n), np.uint8)
        mask[n // 2:n // 2 + 4, n // 2:n // 2 + 4, n // 2:n // 2 + 4] = 1
        net = lbm.Corrector(mask, I.corrector_init_params(1), 0.05, 0.01, 0.005)
        rho, u = torch.ones(mask.shape, device="cuda"), torch.zeros((3, *mask.shape), device="cuda")
        t = gpu_us(lambda: [net.forward(rho, u) for _ in range(10)], 10)
        clear = gpu_us(lambda: [u.zero_() for _ in range(10)], 10)
        net.close()
        return t, clear

    (small, _), (large, clear) = forward(64), forward(256)
    assert large <= 1.5 * (small + clear), (small, large, clear)
