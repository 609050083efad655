"""A launch that the runtime refuses fails that call only: a grid of more
planes than a launch has in z (65535) cannot run the tiled kernels, and says
so; the error is not left behind for the next call of this or another grid,
or of the caller's own CUDA code."""
import numpy as np
import pytest

from paper_1302_1125_gb300 import rlb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1302_1125_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", [rlb.FP64, rlb.FP32_STORAGE])
def test_a_refused_launch_leaves_no_error_behind(precision):
    kw = dict(dt_over_dx=0.1, alpha_override=0.1, precision=precision)
    g = rlb.Grid(2, 2, 65536, thread_mapping=rlb.MAPPING_TILES, **kw).init(1.0, 1.0, 0.0, 0.0, 0.0)
    before = g.get_state()
    with pytest.raises(rlb.RLBError) as e:
        g.step(1)
    assert e.value.status == rlb.RLB_E_CUDA
    small = rlb.Grid(33, 3, 2, **kw).init(1.0, 1.0, 0.0, 0.0, 0.0).step(1)   # raises if the error were kept
    assert np.isfinite(small.totals()).all()
    assert float(torch.ones(4, device="cuda").sum()) == 4.0
    for a, b in zip(before, g.get_state()):
        assert np.array_equal(a, b)
