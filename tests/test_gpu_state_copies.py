"""The state of FP32 grids through every kind of buffer, small and large (from
32 MB on, 4 MB of pinned memory, the copies run beside the kernels): host memory, pinned host memory
(reached by a kernel), device memory at any 4-byte offset, and a few bytes off."""
import numpy as np
import pytest

from paper_1302_1125_gb300 import rlb
from paper_1302_1125_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1302_1125_gb300 import build
    build.build()


def grid(dims):
    w = W.periodic_box(*dims, seed=4, dt_over_dx=0.1)
    g = rlb.Grid(*dims, bc_lo=(1, 0, 1), bc_hi=(1, 0, 1), dt_over_dx=0.1, alpha_override=0.1, precision=rlb.FP32_STORAGE)
    return g.init(*w.fields()).step(2)


def buffers(count):
    yield "host", np.zeros(count, np.float32)
    yield "pinned", torch.zeros(count, dtype=torch.float32).pin_memory()
    yield "pinned, inside", torch.zeros(count + 9, dtype=torch.float32).pin_memory()[5:count + 5]
    yield "device", torch.zeros(count, dtype=torch.float32, device="cuda")
    yield "device, inside", torch.zeros(count + 9, dtype=torch.float32, device="cuda")[3:count + 3]
    yield "device, off", torch.zeros(4 * count + 8, dtype=torch.uint8, device="cuda")[2:4 * count + 2]


# 43 values of 4 bytes a cell: 0.1 MB, on both sides of 1, 4 and 32 MB
@pytest.mark.parametrize("dims", [(801, 1, 1), (2016, 3, 1), (6112, 1, 1), (24352, 1, 1), (24401, 1, 1), (151, 23, 7), (64, 64, 47), (65, 61, 49), (129, 65, 40)])
def test_every_buffer_holds_the_same_state(dims):
    g = grid(dims)
    want = np.concatenate([np.ravel(a) for a in g.get_state()])
    g.step(2)
    ahead = np.concatenate([np.ravel(a) for a in g.get_state()])
    assert not np.array_equal(want, ahead)
    for name, buf in buffers(want.size):
        rlb.rlb_set_state(g.ctx, want, 0)
        rlb.rlb_get_state(g.ctx, buf, 0)
        got = buf if isinstance(buf, np.ndarray) else np.frombuffer(buf.cpu().contiguous().numpy().tobytes(), np.float32)
        assert np.array_equal(got, want), name
        g.step(2)                      # another state in the way
        rlb.rlb_set_state(g.ctx, buf, 0)
        g.step(2)
        assert np.array_equal(np.concatenate([np.ravel(a) for a in g.get_state()]), ahead), name
