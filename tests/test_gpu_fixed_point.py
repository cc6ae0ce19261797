"""The fixed-point form of the FP64 stencil (wilson_apply) against the
double-precision kernel (wilson_apply_noalloc) on the same inputs: tile edges
(V below, at and off multiples of 32), both tile shapes (lattices below and
above two tiles per SM), and inputs that fixed point hands to double precision
(NaN, Inf, scales near the ends of the exponent range, links that are not
unitary).

Tolerance: a component is a sum of 48 products and the diagonal; either kernel
rounds at most 61 times by 2^-53 of the largest input component around the site
times the sum of the link moduli (8 x sqrt 3 / 2) or the diagonal, so two results
differ by less than 2 x 61 x 2^-53 x 11 = 1.5e-13 of that component."""
import numpy as np
import pytest

import lattice_inputs as li
from tests.gpu_util import lib, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

M0 = -0.35


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    return torch, lib()


def _around(x, dims):
    """max |x| over each site and its eight neighbours."""
    m = np.abs(x).reshape(-1, 12).max(1).reshape(tuple(reversed(dims)))
    out = m.copy()
    for ax in range(4):
        out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
    return out.reshape(-1, 1)


def _both(env, dims, U, x):
    torch, gs = env
    ctx = gs.Context(dims, M0, torch.cuda.current_stream().cuda_stream)
    Ud, xd = to_dev(U, torch), to_dev(x, torch)
    ctx.set_gauge(Ud)
    y, ref = torch.empty_like(xd), torch.empty_like(xd)
    ctx.wilson_apply(xd, y)
    assert gs.wilson_apply_noalloc(dims, M0, Ud, xd, ref, torch.cuda.current_stream().cuda_stream) == gs.GS_OK
    torch.cuda.synchronize()
    y, ref = y.cpu().numpy().reshape(-1, 12), ref.cpu().numpy().reshape(-1, 12)
    ctx.close()
    return y, ref


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 2, 7), (4, 4, 2, 1 + 1), (8, 4, 4, 8), (5, 7, 9, 11), (8, 8, 8, 16)])
@pytest.mark.parametrize("scale", ["plain", "by site", "by component", "tiny", "huge", "zero"])
def test_equals_double_precision(env, dims, scale):
    rng = np.random.default_rng(3)
    V = li.volume(dims)
    U = li.random_gauge(dims, 0.3, 1)
    x = rng.standard_normal((V, 12)) + 1j * rng.standard_normal((V, 12))
    if scale == "by site":
        x *= 10.0 ** rng.uniform(-12, 3, (V, 1))
    elif scale == "by component":
        x *= 10.0 ** rng.uniform(-12, 3, (V, 12))
    elif scale == "tiny":
        x *= 1e-306
    elif scale == "huge":
        x *= 1e300
    elif scale == "zero":
        x[rng.random(V) < 0.7] = 0.0
    y, ref = _both(env, dims, U, x)
    if scale in ("tiny", "huge"):        # every tile is done in double precision
        assert np.array_equal(y, ref)
    assert np.all(np.abs(y - ref) <= 1.5e-13 * _around(x, dims))


@pytest.mark.parametrize("dims", [(2, 3, 4, 3), (6, 5, 7, 9), (8, 8, 8, 16)])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 1e308, 5e-324])
def test_values_out_of_range(env, dims, value):
    """One odd component: its tiles hold exactly what double precision gives, the others a number as close as ever."""
    rng = np.random.default_rng(4)
    V = li.volume(dims)
    U = li.random_gauge(dims, 0.3, 2)
    x = rng.standard_normal((V, 12)) + 1j * rng.standard_normal((V, 12))
    if value == 5e-324:
        x[V // 3] = 0.0
    x[V // 3, 7] = complex(1.0 if value != 5e-324 else 0.0, value)
    y, ref = _both(env, dims, U, x)
    yr, rr = y.view(np.float64), ref.view(np.float64)
    assert np.array_equal(np.isnan(yr), np.isnan(rr)) and np.array_equal(np.isinf(yr), np.isinf(rr))
    near = _around(np.where(np.isfinite(x), x, 0.0), dims)
    fine = np.isfinite(yr) & np.isfinite(rr)
    assert np.all((np.abs(np.where(fine, yr, 0) - np.where(fine, rr, 0)) <= 1.5e-13 * np.repeat(near, 24, 1)))


@pytest.mark.parametrize("which", ["one entry", "all", "nan"])
def test_links_out_of_range(env, which):
    """A link outside fixed point's range sends the whole field to double precision, entry for entry."""
    rng = np.random.default_rng(5)
    dims = (4, 6, 5, 8)
    V = li.volume(dims)
    U = li.random_gauge(dims, 0.3, 3)
    if which == "one entry":
        U[17, 2, 1, 0] = 1.02 + 0.1j
    elif which == "all":
        U = U * 7.5
    else:
        U[3, 0, 0, 0] = np.nan
    x = rng.standard_normal((V, 12)) + 1j * rng.standard_normal((V, 12))
    y, ref = _both(env, dims, U, x)
    assert np.array_equal(y, ref, equal_nan=True)
