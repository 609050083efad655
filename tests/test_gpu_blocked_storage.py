"""FP32 grids store populations in blocks of 32 cells with rows padded to even
length: rows that end inside a pair, inside a block and at a block's edge, with
every kind of x face, against the FP64 form of the same run (a few float
roundings a step), and the state through host, device and misaligned buffers."""
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


def grid(nx, ny, nz, lo, hi, precision, **kw):
    w = W.periodic_box(nx, ny, nz, seed=nx, amp=0.1, tau_override=0.9, alpha_override=0.1, dt_over_dx=0.1)
    g = rlb.Grid(nx, ny, nz, bc_lo=(lo, O, P), bc_hi=(hi, O, P), inlet=(2.0, 1.1, (0.1, 0.0, 0.0)), dt_over_dx=0.1,
                 tau_override=0.9, alpha_override=0.1, precision=precision, **kw)
    return g.init(*w.fields())


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 5, 31, 32, 33, 63, 64, 65, 127, 129])
@pytest.mark.parametrize("lo,hi", [(P, P), (O, O), (I, I), (P, O), (O, P), (I, P), (P, I), (I, O)])
@pytest.mark.parametrize("ny,nz", [(1, 1), (3, 1), (2, 3)])
def test_rows_of_every_length(nx, lo, hi, ny, nz):
    steps = 3
    a = grid(nx, ny, nz, lo, hi, rlb.FP32_STORAGE).step(steps).get_state()
    b = grid(nx, ny, nz, lo, hi, rlb.FP64).step(steps).get_state()
    for x, y in zip(a[:2], b[:2]):
        # each step rounds a population a few times, at the scale of the cell's
        # largest one: 64 float roundings of the grid's largest value
        assert np.abs(x - y).max() <= 64 * 2.0 ** -24 * np.abs(y).max()


@pytest.mark.parametrize("nx", [32, 33])
def test_state_buffers(nx):
    g = grid(nx, 3, 2, O, O, rlb.FP32_STORAGE).step(2)
    host = np.concatenate([np.ravel(a) for a in g.get_state()])
    dev = torch.empty(host.size, dtype=torch.float32, device="cuda")
    rlb.rlb_get_state(g.ctx, dev, 1)
    assert np.array_equal(dev.cpu().numpy(), host)
    odd = torch.empty(host.nbytes + 1, dtype=torch.uint8, device="cuda")[1:]   # not aligned to a float
    rlb.rlb_get_state(g.ctx, odd, 1)
    assert np.array_equal(odd.cpu().numpy().view(np.float32) if odd.data_ptr() % 4 == 0
                          else np.frombuffer(odd.cpu().numpy().tobytes(), np.float32), host)
    g.step(2)
    want = np.concatenate([np.ravel(a) for a in g.get_state()])
    for buf in (host, dev, odd):
        rlb.rlb_set_state(g.ctx, buf, int(hasattr(buf, "is_cuda")))
        g.step(2)
        assert np.array_equal(np.concatenate([np.ravel(a) for a in g.get_state()]), want)
