"""Restriction and the correction's zero fill at the edges of their wide accesses: rows that are not whole
groups of four coarse cells, arrays off the 8- and 16-byte boundaries."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2101_11107_gb300 import inputs as I  # noqa: E402
from paper_2101_11107_gb300 import lbm  # noqa: E402


def _at(n, dtype, offset):
    """n values that start `offset` elements into an allocation."""
    return torch.empty(n + offset, dtype=dtype, device="cuda")[offset:]


@pytest.mark.parametrize("offsets", [(0, 0, 0, 0), (1, 0, 0, 0), (4, 1, 0, 0), (0, 0, 1, 0), (8, 3, 0, 2)])
@pytest.mark.parametrize("shape", [(2, 2, 2), (4, 6, 8), (6, 10, 12), (8, 2, 24), (34, 18, 40)])
def test_restrict(shape, offsets):
    nz, ny, nx = shape
    rng = np.random.default_rng(nx)
    m = (rng.random(shape) < 0.3).astype(np.uint8)
    m[: nz // 2, :, nx // 2:] = 0
    f = [rng.normal(0.3, 1.0, shape).astype(np.float32) for _ in range(4)]
    mo, fo, ro, uo = offsets
    mask = _at(m.size, torch.uint8, mo)
    mask.copy_(torch.from_numpy(m.reshape(-1)))
    rho, u = _at(m.size, torch.float32, fo), _at(3 * m.size, torch.float32, fo)
    rho.copy_(torch.from_numpy(f[0].reshape(-1)))
    u.copy_(torch.from_numpy(np.stack(f[1:]).reshape(-1)))
    n = m.size // 8
    crho, cu = _at(n, torch.float32, ro), _at(3 * n, torch.float32, uo)
    crho.fill_(7.0)
    cu.fill_(7.0)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = lbm.load_library().lbm_restrict(p(rho), p(u), p(mask), nx, ny, nz, p(crho), p(cu),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    torch.cuda.synchronize()
    k = m.astype(np.float64).reshape(nz // 2, 2, ny // 2, 2, nx // 2, 2).sum((1, 3, 5))
    for q, got in enumerate([crho] + list(cu.reshape(3, n))):
        v = (f[q] * m).astype(np.float64).reshape(nz // 2, 2, ny // 2, 2, nx // 2, 2)
        want = v.sum((1, 3, 5)) / np.maximum(k, 1)
        # at most 7 additions, one reciprocal and one product, each rounded to 2^-24
        bound = 9 * 2.0 ** -24 * np.abs(v).sum((1, 3, 5)) + 1e-30
        assert np.all(np.abs(got.cpu().numpy().reshape(want.shape) - want) <= bound)


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_forward_clears_the_box(offset):
    """The correction outside the fluid cells is 0 whatever the caller's array held and wherever it starts."""
    g = I.aneurysm(5, edge=48)
    net = lbm.Corrector(g.mask, I.corrector_init_params(1), 0.05, 0.01, 0.005)
    fluid = torch.from_numpy((g.mask > 0).astype(np.uint8)).cuda()
    rng = torch.Generator("cuda").manual_seed(1)
    rho = 1.0 + 0.01 * torch.randn(g.mask.shape, device="cuda", generator=rng) * fluid
    u = 0.03 * torch.randn((3, *g.mask.shape), device="cuda", generator=rng) * fluid
    want = net.forward(rho, u)
    du = _at(3 * fluid.numel(), torch.float32, offset)
    du.fill_(float("nan"))
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lbm.load_library().lbm_corrector_forward(net._h, None, None, p(rho), p(u), p(du)) == 0
    torch.cuda.synchronize()
    du = du.reshape(want.shape)
    assert torch.equal(du, want) and float(want.abs().max()) > 0
    assert not bool(du[:, fluid == 0].any())


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("fill", [0.03, 0.6, 1.0])
def test_restrict_large_enough_for_four_cells_a_thread(fill, offset):
    """The wide form, and with fields off the 16-byte boundary the form that reads the children one by one; what
    solid cells hold is not read into a sum."""
    shape = (66, 178, 192)  # 281,952 coarse cells, rows of whole groups
    rng = torch.Generator("cuda").manual_seed(3)
    m = (torch.rand(shape, device="cuda", generator=rng) < fill).to(torch.uint8)
    f = torch.randn((4, *shape), device="cuda", generator=rng)
    nan = torch.where(m.bool(), f, torch.full_like(f, float("nan")))
    rho, u = _at(m.numel(), torch.float32, offset), _at(3 * m.numel(), torch.float32, offset)
    rho.copy_(nan[0].reshape(-1))
    u.copy_(nan[1:].reshape(-1))
    crho, cu = lbm.restrict(rho.reshape(shape), u.reshape(3, *shape), m)
    split = lambda t: t.double().reshape(33, 2, 89, 2, 96, 2)  # noqa: E731
    k = split(m).sum((1, 3, 5))
    for q, got in enumerate([crho, *cu]):
        v = split(f[q] * m)
        bound = 9 * 2.0 ** -24 * v.abs().sum((1, 3, 5)) + 1e-30  # as above
        assert bool(((got.double() - v.sum((1, 3, 5)) / k.clamp(min=1)).abs() <= bound).all())
