"""FP64 step: the streaming alone, population by population, against extended
precision, and the kernel of small grids against the tiles at inlet faces.

With tau = 1e30 a step returns the explicit part (Eqs. 47-53 and the bulk term)
and kappa = 2.5e-31 of the equilibrium's distance, less than 1e-29 of the largest
population (a term that counts where values lie 2^80 apart).  M: the largest value of a population's stencil.  |D| <= 2 M
per axis, so the increments are below 0.56 M (0.139 a diagonal's two axes) and
0.3 M (bulk).  In fixed point they are exact up to one conversion each, a
rounded prefactor, two fused sums and the relaxation's: 7 roundings of 2^-53 M
at most, 2^-50 M.  Stencils whose values lie further apart than 2^6 round every
difference: 24, 2^-48 M.  An inlet's ghost values may differ by two roundings
between the library and the oracle: 2^-49 M where all else is fixed point."""
import math

import numpy as np
import pytest

from paper_1302_1125_gb300 import rlb
from paper_1302_1125_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
P, O, I = 0, 1, 2
LD = np.longdouble
INLET = (2.0, 1.1, (0.1, 0.0, 0.0))


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1302_1125_gb300 import build
    build.build()


def neighbour(q, axis, d, lo, hi, ghost):
    """q (z, y, x) at distance d along the axis (0: x) through its faces"""
    a, n = 2 - axis, q.shape[2 - axis]
    c = np.arange(n) + d
    src = np.where((c < 0) & (lo == P) | (c >= n) & (hi == P), c % n, np.clip(c, 0, n - 1))
    out = np.take(q, src, axis=a)
    g = (c < 0) & (lo == I) | (c >= n) & (hi == I)
    shape = [1, 1, 1]
    shape[a] = n
    return np.where(g.reshape(shape), LD(ghost), out)


def explicit(q, c, bulk, k, kb, limited, lo, hi, ghost):
    """the explicit part and the stencil's largest magnitude, in extended precision"""
    def mm(a, b):
        return np.where(a * b > 0, np.sign(a) * np.minimum(abs(a), abs(b)), LD(0)) if limited else LD(0) * a
    out, big = q.copy(), abs(q)
    for a in range(3):
        if q.shape[2 - a] == 1 or not (c[a] or bulk):
            continue
        v = {d: neighbour(q, a, d, lo[a], hi[a], ghost) for d in (-2, -1, 1, 2)}
        used = [-1, 1] + ([-2] if c[a] > 0 else [2] if c[a] < 0 else [])
        big = np.maximum.reduce([big] + [abs(v[d]) for d in used])
        if c[a] > 0:
            out -= k * c[a] * (q + mm(v[1] - q, q - v[-1]) / 2 - v[-1] - mm(q - v[-1], v[-1] - v[-2]) / 2)
        elif c[a] < 0:
            out -= k * c[a] * (v[1] - mm(v[1] - q, v[2] - v[1]) / 2 - q + mm(q - v[-1], v[1] - q) / 2)
        if bulk:
            out += kb * (v[1] - 2 * q + v[-1])
    return out, big


FACES = [((P, P, P), (P, P, P)), ((O, O, O), (O, O, O)), ((I, P, O), (O, P, O)), ((P, O, P), (I, O, P))]


@pytest.mark.parametrize("dims", [(67, 1, 1), (33, 5, 1), (18, 7, 5)])
@pytest.mark.parametrize("lo,hi", FACES)
@pytest.mark.parametrize("spread", [0.0, 2.5, 40.0])
@pytest.mark.parametrize("limiter,alpha", [(0, 0.1), (0, 0.0), (1, 0.1)])
@pytest.mark.parametrize("mapping", [rlb.MAPPING_AUTO, rlb.MAPPING_TILES])
def test_streaming_alone(orc, dims, lo, hi, spread, limiter, alpha, mapping):
    dt = 0.1
    w = W.periodic_box(*dims, seed=3, amp=0.1)
    g = rlb.Grid(*dims, bc_lo=lo, bc_hi=hi, inlet=INLET, limiter=limiter, dt_over_dx=dt, tau_override=1e30,
                 alpha_override=alpha, precision=rlb.FP64, thread_mapping=mapping)
    f, h, prev = g.init(*w.fields()).get_state()
    inlet = I in lo or I in hi
    n, T, u = INLET
    gam = 1.0 / math.sqrt(1.0 - u[0] ** 2)
    gf = orc.feq(n * T, [gam * x for x in u])
    gh = orc.heq(n, [gam * x for x in u])
    # values within 2^spread of one magnitude per population (its ghost's where
    # there is an inlet); the rest population keeps E far above |M|
    rng = np.random.default_rng(int(spread))
    for q, ghost in ((f, gf), (h, gh)):
        for i in range(1, 19):
            size = abs(ghost[i]) if inlet else abs(q[i]).mean()
            q[i] = math.copysign(size, q[i].mean()) * np.exp2(rng.uniform(-spread, spread, q[i].shape))
    f[0] = 50.0 * np.abs(f[1:]).sum(0).max()
    if spread > 6.0:
        f[9, ::11] = 0.0
        h[5, ::7] = 0.0
        f[12, ::5] *= -1.0
    g.set_state(f, h, prev).step(1)
    f1, h1, _ = g.get_state()
    vec = np.rint(orc.lattice(0)[1]).astype(int)
    k = LD(dt) * np.sqrt(LD(13) / LD(27))
    kb = LD(13) / np.sqrt(LD(27)) * LD(dt) * LD(alpha)
    eps = 2.0 ** (-48 if spread > 6.0 else -49 if inlet else -50)
    shape = (dims[2], dims[1], dims[0])
    for q, q1, ghost, is_f in ((f, f1, gf, True), (h, h1, gh, False)):
        for i in range(19):
            want, big = explicit(q[i].reshape(shape).astype(LD), vec[i], is_f and i > 0, k, kb, limiter == 0, lo, hi, ghost[i])
            assert (abs(q1[i].reshape(shape) - want) <= eps * big + 1e-29 * abs(q).max()).all(), (is_f, i)


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 1, 1), (33, 1, 1), (29, 3, 1), (32, 4, 3), (17, 9, 7)])
@pytest.mark.parametrize("lo,hi", [(I, O), (O, I), (I, I), (P, I)])
@pytest.mark.parametrize("model", [0, 1])
def test_small_grid_kernel_agrees_with_tiles_at_inlets(dims, lo, hi, model):
    w = W.periodic_box(*dims, seed=8, amp=0.1)
    states = []
    for mapping in (rlb.MAPPING_TILES, rlb.MAPPING_AUTO):
        g = rlb.Grid(*dims, bc_lo=(lo, O, P), bc_hi=(hi, O, P), inlet=INLET, dt_over_dx=0.1, eta_over_s=0.05,
                     alpha_override=0.1, precision=rlb.FP64, thread_mapping=mapping, model=model)
        states.append(g.init(*w.fields()).step(12).get_state())
    for a, b in zip(*states):
        assert np.array_equal(a, b)
