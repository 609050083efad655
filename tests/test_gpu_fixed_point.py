"""FP64 step: the streaming stencils in 64-bit fixed point against the oracle's
floating-point form, population by population, on states whose neighbouring
values lie apart by more and less than the spread the fixed-point form takes
exactly (2^6), with zeros, signs and far smaller values among them; and the two
FP64 kernels (four warps to 32 cells on small grids, tiles) bit for bit.

The increment is formed exactly and rounded twice (conversion, fused
multiply-add per prefactor), so a population is within a few roundings of the
largest value of its stencil: 2^-50 of the plane's largest value.
"""
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


@pytest.mark.parametrize("dims", [(67, 1, 1), (33, 5, 1), (18, 7, 5)])
@pytest.mark.parametrize("spread", [0, 5, 6, 7, 40])
@pytest.mark.parametrize("limiter,alpha", [(0, 0.1), (0, 0.0), (1, 0.1)])
def test_one_step_with_spread_values(orc, dims, spread, limiter, alpha):
    w = W.periodic_box(*dims, seed=3, tau_override=0.9, alpha_override=alpha, dt_over_dx=0.1)
    g = rlb.Grid(*dims, bc_lo=w.bc_lo, bc_hi=w.bc_hi, limiter=limiter, dt_over_dx=0.1, tau_override=0.9,
                 alpha_override=alpha, precision=rlb.FP64)
    g.init(*w.fields())
    f, h, prev = g.get_state()
    rng = np.random.default_rng(spread)
    # scale single cells' populations by up to 2^-spread; E stays far above |M|
    # because the rest population is left alone; a few exact zeros
    scale = np.exp2(-rng.uniform(0.0, spread, f[1:].shape))
    f[1:] *= scale
    h[1:] *= np.exp2(-rng.uniform(0.0, spread, h[1:].shape))
    f[0] = np.abs(f[0]) + 8.0 * np.abs(f[1:]).sum(0)
    if spread:
        h[5, ::7] = 0.0
        f[9, ::11] = 0.0
        f[12, ::5] *= -1.0
    g.set_state(f, h, prev).step(1)
    f1, h1, p1 = g.get_state()
    p = orc.Params(nx=dims[0], ny=dims[1], nz=dims[2], bc_lo=w.bc_lo, bc_hi=w.bc_hi, dt=0.1, tau_override=0.9,
                   alpha_override=alpha, limiter=limiter)
    fo, ho, mo, bad = orc.step_cells(p, f, h, prev, np.arange(g.N))
    assert bad == 0
    for a, b in ((f1, fo.T), (h1, ho.T), (p1, mo.T)):
        for k in range(a.shape[0]):
            s = np.abs(b[k]).max()
            assert np.abs(a[k] - b[k]).max() <= 2.0 ** -44 * max(s, np.abs(f).max() if a is not h1 else np.abs(h).max())


DIMS = [(1, 1, 1), (31, 1, 1), (33, 1, 1), (32, 4, 1), (29, 3, 1), (32, 4, 3), (17, 9, 7)]
FORMS = [(d, {}) for d in DIMS] + [(d, {"model": 1}) for d in DIMS] + \
    [(d, {"symmetry_1d": 1}) for d in DIMS[:3]] + [(d, {"symmetry_2d": 1}) for d in DIMS[3:5]]


@pytest.mark.parametrize("dims,kw", FORMS)
def test_split_blocks_agree_with_tiles(dims, kw):
    w = W.periodic_box(*dims, seed=8, tau_override=0.0, alpha_override=0.1, dt_over_dx=0.1)
    states = []
    for mapping in (rlb.MAPPING_TILES, rlb.MAPPING_AUTO):
        g = rlb.Grid(*dims, bc_lo=(1, 0, 1), bc_hi=(1, 0, 1), dt_over_dx=0.1, eta_over_s=0.05, alpha_override=0.1,
                     precision=rlb.FP64, thread_mapping=mapping, **kw)
        g.init(*w.fields()).step(12)
        states.append(g.get_state())
        assert (g.step_kernel == "fp64_small") == (mapping == rlb.MAPPING_AUTO)
    for a, b in zip(*states):
        assert np.array_equal(a, b)
