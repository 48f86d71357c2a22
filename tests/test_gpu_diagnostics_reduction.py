"""The FP64 diagnostics at the edges of their reduction: no cell, one cell, a partial warp and block, more blocks
than the last stage has threads, no or some open cells, non-finite cells."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2101_11107_gb300 import inputs as I  # noqa: E402
from paper_2101_11107_gb300 import lbm  # noqa: E402


def _check(d, dg):
    rho, u = d.macroscopic(dense=False)
    rho, u = rho.astype(np.float64), u.astype(np.float64)
    # at most n additions in FP64
    assert abs(dg["mass"] - rho.sum()) <= 1e-13 * max(rho.size, 1) ** 0.5 * max(rho.sum(), 1.0)
    want = np.sqrt((u * u).sum(0)).max() if rho.size else 0.0
    assert abs(dg["max_u"] - want) <= 1e-15 + 4 * 2.0 ** -52 * want
    assert dg["n_nonfinite"] == 0 and dg["time"] == d.time


@pytest.mark.parametrize("scheme", ["esoteric", "ab"])
@pytest.mark.parametrize("n", [0, 1, 31, 33, 255, 257, 70001])
def test_cell_counts(n, scheme):
    mask = np.zeros(44 * 40 * 40, np.uint8)
    mask[np.random.default_rng(n).permutation(mask.size)[:n]] = 1
    d = lbm.Domain(mask.reshape(40, 40, 44), periodic=(1, 1, 1), tau=0.8, force=(1e-5, 2e-5, -1e-5), scheme=scheme)
    d.step(7)
    _check(d, d.diagnostics())
    _check(d, d.diagnostics_noalloc())


@pytest.mark.parametrize("storage", ["fp32", "bf16"])
def test_open_faces(storage):
    g = I.inlet_pipe(24, 20, 20, 7.5, u_peak=0.02, tau=0.7)
    d = lbm.Domain.from_geometry(g, storage=storage)
    d.step(40)
    dg = d.diagnostics()
    _check(d, dg)
    rho, u = (x.astype(np.float64) for x in d.macroscopic())
    for key, face, sign in (("flux_in", 2, 1.0), ("flux_out", 3, 1.0)):
        sel = g.mask == face
        want = sign * (rho[sel] * u[0][sel]).sum()
        assert want != 0.0 and abs(dg[key] - want) <= 1e-12 * abs(want) + 1e-15


def test_non_finite_cells_are_counted():
    """NaN density in a block of cells: the cells they reach in one step are counted, all others summed."""
    mask = np.ones((16, 16, 16), np.uint8)
    d = lbm.Domain(mask, periodic=(1, 1, 1), tau=0.8)
    rho, u = np.ones(mask.shape), np.zeros((3, *mask.shape))
    rho[4:6, 4:6, 4:6] = np.nan
    d.init_equilibrium(rho, u)
    dg = d.diagnostics(raise_unstable=False)
    assert dg["n_nonfinite"] == 4 ** 3
    assert abs(dg["mass"] - (mask.size - 64)) <= 1e-4 and dg["max_u"] <= 1e-6
