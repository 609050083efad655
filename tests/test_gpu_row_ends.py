"""FP32 grids: rows that end inside a tile of 64 x 8 cells, at its edge and one
pair after it, on the tiled kernels and in the linear order, bit for bit: odd
and even lengths, every kind of x face, viscous and Euler steps, both lattices
and the 2-D reduction, with the previous level."""
import numpy as np
import pytest

from paper_1302_1125_gb300 import rlb
from paper_1302_1125_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
P, O, I = 0, 1, 2


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1302_1125_gb300 import build
    build.build()


def state(dims, lo, hi, mapping, **kw):
    w = W.periodic_box(*dims, seed=dims[0], amp=0.1)
    fields = list(w.fields())
    if kw.get("symmetry_2d"):
        fields[4] = 0.0 * fields[4]
    g = rlb.Grid(*dims, bc_lo=(lo, O, P), bc_hi=(hi, O, P), inlet=(2.0, 1.1, (0.1, 0.0, 0.0)), dt_over_dx=0.1,
                 eta_over_s=0.1, alpha_override=0.1, precision=rlb.FP32_STORAGE, thread_mapping=mapping, **kw)
    return g.init(*fields).step(3), g.step_kernel


@pytest.mark.parametrize("nx", [1, 2, 3, 5, 63, 64, 65, 66, 67, 127, 128, 129, 131])
@pytest.mark.parametrize("lo,hi", [(P, P), (O, O), (I, I), (P, O), (O, P), (I, P), (P, I), (I, O)])
@pytest.mark.parametrize("ny,nz,kw", [(17, 1, {}), (9, 3, {}), (17, 1, {"euler_mode": 1}), (9, 3, {"euler_mode": 1}),
                                      (9, 3, {"model": 1}), (17, 1, {"symmetry_2d": 1})])
def test_tiles_and_linear_order_agree(nx, lo, hi, ny, nz, kw):
    tiles, name = state((nx, ny, nz), lo, hi, rlb.MAPPING_TILES, **kw)
    linear, other = state((nx, ny, nz), lo, hi, rlb.MAPPING_LINEAR, **kw)
    assert (name, other) == ("fp32_tiles", "fp32_linear")
    for a, b in zip(tiles.get_state(), linear.get_state()):
        assert np.array_equal(a, b)
