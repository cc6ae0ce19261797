"""Inputs at the limits of the fixed-point FP64 kernels, where their range or their
resolution ends and double precision takes over, against the double-precision
kernel (wilson_apply_noalloc) or one launch per phase on the same inputs."""
import numpy as np
import pytest

import lattice_inputs as li
from oracle import dirac
from tests.gpu_util import lib, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    return torch, lib()


def _ctx(gs, torch, dims, m0, U):
    ctx = gs.Context(dims, m0, torch.cuda.current_stream().cuda_stream)
    ctx.set_gauge(to_dev(U, torch))
    return ctx


def _both(env, dims, m0, U, x):
    """D x by the context and by the double-precision kernel, or above that one's 8192
    sites by the oracle's matrix; complex128 [V][12]."""
    torch, gs = env
    ctx = _ctx(gs, torch, dims, m0, U)
    xd = to_dev(x, torch)
    y, ref = torch.empty_like(xd), torch.empty_like(xd)
    ctx.wilson_apply(xd, y)
    if li.volume(dims) > 8192:
        torch.cuda.synchronize()
        ctx.close()
        return y.cpu().numpy().reshape(-1, 12), (dirac.wilson_matrix(U, dims, m0) @ x.ravel()).reshape(-1, 12)
    assert gs.wilson_apply_noalloc(dims, m0, to_dev(U, torch), xd, ref,
                                   torch.cuda.current_stream().cuda_stream) == gs.GS_OK
    torch.cuda.synchronize()
    ctx.close()
    return y.cpu().numpy().reshape(-1, 12), ref.cpu().numpy().reshape(-1, 12)


# A component sums 48 products and the diagonal and either kernel rounds at most 61
# times by 2^-53 of the sum of the terms' moduli: at most 8 hops x 2 spin components x
# 3 x sqrt 2 / 2 x 1.01 and |diagonal| < 4, together 38.3, times sqrt 2 for the largest modulus here.
@pytest.mark.parametrize("entries", ["all", "at the limit", "row", "column"])
def test_links_with_large_rows(env, entries):
    """Links that are not unitary, entry by entry within fixed point's range: a row's
    sum of products leaves 63 bits unless the whole row is looked at."""
    rng = np.random.default_rng(11)
    dims = (8, 8, 8, 16)
    V = li.volume(dims)
    a = (1 + 1j) * rng.uniform(0.99, 1.01, (V, 4, 1, 1))
    U = np.zeros((V, 4, 3, 3), complex)
    if entries == "all":
        U[:] = a
    elif entries == "at the limit":
        U[:] = a * 0.625
    elif entries == "row":
        U[:, :, 1:2, :] = a
    else:
        U[:, :, :, 1:2] = a
    x = np.repeat((1 + 1j) * 0.9 * rng.uniform(0.99, 1.01, (V, 1)), 12, 1)
    y, ref = _both(env, dims, -0.35, U, x)
    assert np.abs(y - ref).max() <= 2 * 61 * 2.0 ** -53 * 38.3 * np.sqrt(2) * np.abs(x).max()


def test_a_dot_that_cancels_is_not_a_breakdown(env):
    """<b, D_rr b> of terms -1/2, -1/2, 1/2, 1/2 and 124 of 0.9 x 2^-55: the small ones vanish
    beside the large ones in the fixed-point sums, but the dot is not zero.  m0 = -4 takes
    the diagonal away; the only links join the pairs x3 = 0, 1 and 2, 3."""
    torch, gs = env
    dims = (4, 4, 4, 4)
    V = li.volume(dims)
    s = np.arange(V)
    x0, x3, first = s % 4, s // 64, (s % 64) == 1        # `first`: the line of the large terms
    U = np.zeros((V, 4, 3, 3), complex)
    up = x3 % 2 == 0
    U[up, 3] = -np.eye(3)
    U[first & (x3 == 0), 3] = np.eye(3)
    full = np.zeros((V, 12), complex)
    full[:, 0] = np.where(first, 1.0, np.where(up, 1.0, 0.9) * 2.0 ** -27)
    b = to_dev(full[x0 % 2 == 1], torch)                 # Type II, direction 0: the rest set, in order
    ctx = _ctx(gs, torch, dims, -4.0, U)
    z = torch.empty_like(b)
    st = ctx.solve_rr(2, 0, 0, b, z, gs.gs_default_opts(inner_max_iter=1), allow=(gs.GS_MAXITER,))
    assert st.status == gs.GS_MAXITER and st.inner_iters == 1
    ctx.close()


# Powers of two change no rounding: the solve is the same, step by step, and its result the scaled one.
@pytest.mark.parametrize("dims,t", [((4, 4, 4, 2), 1), ((8, 8, 8, 10), 1), ((9, 10, 11, 12), 2)])
@pytest.mark.parametrize("power", [-200, -130, -100, 100, 130, 200])
def test_rest_solve_at_any_scale(env, dims, t, power):
    torch, gs = env
    rng = np.random.default_rng(12)
    mu = 1 if dims[0] % 2 else 0
    V = li.volume(dims)
    nr = V - (V // 16 if t == 1 else V // 2)
    b = to_dev(rng.standard_normal((nr, 12)) + 1j * rng.standard_normal((nr, 12)), torch)
    ctx = _ctx(gs, torch, dims, 0.1, li.random_gauge(dims, 0.3, 13))
    o = gs.gs_default_opts(inner_tol=1e-13)
    z1, z2 = torch.empty_like(b), torch.empty_like(b)
    one = ctx.solve_rr(t, mu, 0, b, z1, o)
    two = ctx.solve_rr(t, mu, 0, b * 2.0 ** power, z2, o)
    assert two.inner_iters == one.inner_iters
    assert torch.equal(z2, z1 * 2.0 ** power)
    ctx.close()


@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (8, 10, 8, 24)])
def test_applications_back_to_back(env, dims):
    """The conversion of an input and the stencil overlap at the edges: in a row of
    applications to inputs of different scale each result is that of its own input."""
    torch, gs = env
    rng = np.random.default_rng(14)
    V = li.volume(dims)
    ctx = _ctx(gs, torch, dims, -0.35, li.random_gauge(dims, 0.3, 15))
    xs = [to_dev(s * (rng.standard_normal((V, 12)) + 1j * rng.standard_normal((V, 12))), torch)
          for s in (1.0, 1e-9, 1e9)]
    alone = []
    for x in xs:
        y = torch.empty_like(x)
        ctx.wilson_apply(x, y)
        torch.cuda.synchronize()
        alone.append(y)
    ys = [torch.full_like(xs[0], float("nan")) for _ in range(60)]
    for k, y in enumerate(ys):
        ctx.wilson_apply(xs[k % 3], y)
    torch.cuda.synchronize()
    assert all(torch.equal(y, alone[k % 3]) for k, y in enumerate(ys))
    ctx.close()


def _terms(U, dims, m0, x):
    """Sum of the moduli of the terms of each component of D x: hops of moduli of links and spinors."""
    shape = tuple(reversed(dims))
    A = np.abs(U).reshape(*shape, 4, 3, 3)
    v = np.abs(x).reshape(*shape, 4, 3)
    out = abs(m0 + 4) * v
    for mu in range(4):
        ax, g = 3 - mu, (3, 2, 1, 0) if mu < 2 else (2, 3, 0, 1)    # |gamma_mu| exchanges these spins
        h = v + v[..., g, :]
        out += 0.5 * np.einsum("...ab,...sb->...sa", A[..., mu, :, :], np.roll(h, -1, ax))
        out += 0.5 * np.roll(np.einsum("...ba,...sb->...sa", A[..., mu, :, :], h), 1, ax)
    return out.reshape(-1, 12)


# Either kernel is off by a few units of the terms' moduli: double precision by at most 61 x 2^-53; fixed
# point, where a hop contributes at least 2^-8 of the scale, by 21 units of 2^-57 of it (per hop: six dropped
# products of a quarter unit, two roundings of half a unit, 0.15 for the input): together below 2^-44.
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 6, 5, 8), (8, 10, 8, 24)])
@pytest.mark.parametrize("links", ["rough", "near the identity", "identity"])
@pytest.mark.parametrize("uneven", ["spin", "colour", "spin and colour", "one spin only", "sites", "mild"])
def test_weak_components_keep_their_digits(env, dims, links, uneven):
    rng = np.random.default_rng(16)
    V = li.volume(dims)
    U = li.random_gauge(dims, {"rough": 0.4, "near the identity": 1e-7, "identity": 0.0}[links], 17)
    x = rng.standard_normal((V, 4, 3)) + 1j * rng.standard_normal((V, 4, 3))
    if "spin" in uneven:
        x *= np.array([1.0, 1e-6, 1e-12, 1e-25]).reshape(4, 1)
    if "colour" in uneven:
        x *= np.array([1e-9, 1.0, 1e-30])
    if uneven == "one spin only":
        x[:, 1:] = 0.0
    if uneven == "sites":
        x *= 10.0 ** rng.uniform(-12, 3, (V, 1, 1))
    if uneven == "mild":
        x *= np.array([1.0, 2.0 ** -7, 2.0 ** -9, 2.0 ** -14]).reshape(4, 1)
    y, ref = _both(env, dims, -0.35, U, x.reshape(V, 12))
    assert np.all(np.abs(y - ref) <= 2.0 ** -44 * _terms(U, dims, -0.35, x))
