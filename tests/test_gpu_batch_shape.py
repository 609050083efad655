"""The launch shape that a batch takes when nobody tuned it."""
import time

import numpy as np
import pytest

from paper_1302_1125_gb300 import rlb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1302_1125_gb300 import build
    build.build()


def batch(nx, sym=0):
    b = rlb.Batch(np.asarray(nx, np.int32), 0.1, 0.0, dt_over_dx=0.1, alpha_override=0.1, symmetry_1d=sym)
    rng = np.random.default_rng(5)
    return b.init(1.6 * (1.0 + 0.3 * rng.random(b.total)), np.ones(b.total), np.zeros(b.total))


def ms(b, steps):
    b.step(steps)
    best = float("inf")
    for _ in range(5):
        s, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        s.record()
        b.step(steps)
        e.record()
        torch.cuda.synchronize()
        best = min(best, s.elapsed_time(e))
    return best


def shape(b):
    t, _ = b.tuning()
    return t.threads, t.bound, t.cluster, t.pairs_per_thread


@pytest.mark.parametrize("count,nx", [(4, 256), (16, 1024), (64, 256), (64, 1024), (200, 256)])
@pytest.mark.parametrize("sym", [0, 1])
def test_small_batches_take_a_shape_near_the_best(count, nx, sym):
    """within a third of the best of a few shapes (a pass with one, two and
    four warps per scheduler takes 4.3, 5.2 and 9.1 us, so a shape that puts
    too many blocks on an SM loses more)"""
    steps = 200
    b = batch([nx] * count, sym)
    got = ms(b, steps)
    best = float("inf")
    for t in ((128, 256, 1), (128, 256, 4), (256, 256, 1), (256, 256, 2), (512, 512, 1), (512, 512, 2)):
        b.set_tuning(*t)
        best = min(best, ms(b, steps))
    assert got <= 4.0 / 3.0 * best


def test_the_choice_costs_little_of_the_first_call():
    """beside the second call of the same batch: 2048 tubes take 0.3 ms to
    sort, to lay out and to choose a shape for, 1.8 ms when every shape's plan
    is made"""
    nx = np.full(2048, 256)
    batch(nx[:64]).step(4).close()     # what the first batch of a process pays
    extra = []
    for _ in range(3):
        b = batch(nx)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        b.step(16)
        t1 = time.perf_counter()
        b.step(16)
        extra.append((t1 - t0) - (time.perf_counter() - t1))
        b.close()
    assert min(extra) < 1.0e-3


def test_the_shape_follows_the_step_counts():
    """a call that advances one tube, or a few steps, leaves no shape behind;
    the results do not depend on the shape"""
    rng = np.random.default_rng(2)
    nx = np.exp(rng.uniform(np.log(256), np.log(8192), 200)).astype(np.int32)
    one, steps = np.zeros(200, np.int64), (nx // 64).astype(np.int64)
    one[7] = 3
    fresh, other = batch(nx).step(steps), batch(nx).step(one)
    assert shape(other) != shape(fresh)
    other.step(steps)
    assert shape(other) == shape(fresh)
    fresh.step(one)
    assert shape(fresh) != shape(other)
    a, c = fresh.macroscopic(device=False), other.macroscopic(device=False)
    keep = np.ones(fresh.total, bool)
    keep[fresh.offsets[7]:fresh.offsets[8]] = False      # tube 7 took its steps in another order: alike too
    assert np.array_equal(a[:, keep], c[:, keep]) and np.array_equal(a, c)


def test_a_shape_set_by_hand_or_tuned_stays():
    nx = np.array([300, 64, 5000, 128], np.int32)
    b = batch(nx)
    b.set_tuning(64, 512, 2, 2)
    b.step(8).step([1, 0, 0, 0])
    assert shape(b) == (64, 512, 2, 2)
    best, _ = b.autotune(8, divisor=1)
    b.step(8).step([0, 0, 9, 1])
    assert shape(b) == (best.threads, best.bound, best.cluster, best.pairs_per_thread)
