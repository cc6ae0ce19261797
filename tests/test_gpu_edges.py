"""Kernels at the sizes where they change form.

* The FP64 rest solve in one launch: rest sets off the tile size, both shapes
  (below and above 32 sites per SM), a field that fixed point cannot hold (one link
  not unitary: the double-precision kernel), right-hand sides near the ends of
  the range and with a NaN.
* The block-sparse levels of the V-cycle: more rest rows than blocks of a
  product with dots, rows of more blocks than one pass of the row loop.
* A training step with batches below, at and above the samples per launch, on
  lattices off the row and site tiles.
* The tensor-core layer with a last tile that is full, and of one site.
"""
import numpy as np
import pytest

import lattice_inputs as li
from oracle import dirac, permute, vcycle
from oracle import net as onet
from tests.gpu_util import close, lib, maxrel, rel, to_dev, torch_cuda
from tests.test_gpu_net import test_tensor_core_layer_matches_cuda_cores_and_oracle as _tensor_core_layer

pytestmark = pytest.mark.gpu

I, II = permute.TYPE_I, permute.TYPE_II


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    return torch, lib()


def _ctx(gs, torch, dims, m0, U):
    ctx = gs.Context(dims, m0, torch.cuda.current_stream().cuda_stream)
    ctx.set_gauge(to_dev(U, torch))
    return ctx


def _rest_residual(torch, ctx, perm, nb, t, z):
    """||t - D_rr z|| / ||t|| from the double-precision D of the whole lattice."""
    x = np.zeros((len(perm), 12), complex)
    x[perm[nb:]] = z
    xd = to_dev(x, torch)
    yd = torch.empty_like(xd)
    ctx.wilson_apply(xd, yd)
    torch.cuda.synchronize()
    y = yd.cpu().numpy().reshape(-1, 12)
    scale = np.abs(t).max()
    return np.linalg.norm((t - y[perm[nb:]]) / scale) / np.linalg.norm(t / scale)


# The recurred residual stops at 1e-9 of ||t||; it drifts from the true one by at most
# some 2^-53 ||D|| max ||x_i|| an iteration (200 iterations x 10 x 12 x 1e-16 x a
# hundredfold overshoot of x_i = 2.7e-11), so 1.1e-9 bounds the true one.
@pytest.mark.parametrize("dims,t", [((2, 2, 2, 2), 1), ((4, 3, 5, 3), 2), ((4, 2, 6, 10), 1), ((8, 8, 8, 10), 1),
                                    ((8, 10, 8, 10), 1), ((9, 10, 11, 12), 2)])
@pytest.mark.parametrize("kind", ["plain", "tiny", "huge", "by component", "link"])
def test_rest_solve_fp64(env, dims, t, kind):
    torch, gs = env
    V = li.volume(dims)
    U = li.random_gauge(dims, 0.3, 4)
    if kind == "link":
        U[V // 2, 1, 0, 2] += 0.2
    mu = 1 if dims[0] % 2 else 0
    perm, nb = permute.permutation(dims, t, mu)
    ctx = _ctx(gs, torch, dims, 0.1, U)
    rng = np.random.default_rng(6)
    b = rng.standard_normal((V - nb, 12)) + 1j * rng.standard_normal((V - nb, 12))
    if kind == "tiny":
        b *= 1e-140
    elif kind == "huge":
        b *= 1e140
    elif kind == "by component":
        b *= 10.0 ** rng.uniform(-12, 3, b.shape)
    bd = to_dev(b, torch)
    z = torch.empty_like(bd)
    st = ctx.solve_rr(t, mu, 0, bd, z, gs.gs_default_opts(inner_tol=1e-9), allow=(gs.GS_OK, gs.GS_NONFINITE))
    assert st.inner_solves == 1
    if st.status != gs.GS_OK:
        # the scalar algebra's |<r, v>|^2 leaves the range of a double: one launch per
        # phase answers the same
        assert kind in ("tiny", "huge")
        ctx.set_option(gs.GS_OPT_INNER_KERNEL, 1)
        st = ctx.solve_rr(t, mu, 0, bd, z, gs.gs_default_opts(inner_tol=1e-9), allow=(gs.GS_OK, gs.GS_NONFINITE))
        assert st.status == gs.GS_NONFINITE
        ctx.close()
        return
    assert st.inner_residual <= 1e-9
    assert _rest_residual(torch, ctx, perm, nb, b, z.cpu().numpy().reshape(-1, 12)) <= 1.1e-9
    ctx.close()


@pytest.mark.parametrize("dims", [(4, 4, 4, 2), (8, 10, 8, 10)])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_rest_solve_refuses_what_is_not_finite(env, dims, value):
    torch, gs = env
    ctx = _ctx(gs, torch, dims, 0.1, li.random_gauge(dims, 0.3, 4))
    perm, nb = permute.permutation(dims, 1)
    b = np.ones((len(perm) - nb, 12), complex)
    b[7, 3] = value
    bd = to_dev(b, torch)
    z = torch.empty_like(bd)
    with pytest.raises(gs.GschurError, match="NONFINITE"):
        ctx.solve_rr(1, 0, 0, bd, z, gs.gs_default_opts(inner_tol=1e-9))
    b[7, 3] = 0.0                      # the context stays usable
    bd = to_dev(b, torch)
    ctx.solve_rr(1, 0, 0, bd, z, gs.gs_default_opts(inner_tol=1e-9))
    assert _rest_residual(torch, ctx, perm, nb, b, z.cpu().numpy().reshape(-1, 12)) <= 1.1e-9
    ctx.close()


# Both sides solve the rest sets to 1e-13; the result differs by that times the
# condition of the blocks (hundreds at this mass), per level: 1e-10.
@pytest.mark.parametrize("dims,levels,order", [((8, 8, 8, 8), [(II, 0, True), (I, 0, True)], 1),
                                               ((6, 6, 6, 6), [(II, 0, True), (II, 1, True), (II, 2, True), (II, 3, True)], 2)])
def test_vcycle_wide_levels(env, dims, levels, order):
    torch, gs = env
    m0 = 0.2
    U = li.random_gauge(dims, 0.35, 7)
    ovc = vcycle.VCycle(dirac.wilson_matrix(U, dims, m0), dims, levels, schur={2: "reusken", 1: "first"}[order],
                        inner=1e-13)
    f = li.gaussian_source(dims, 41).ravel()
    ref = ovc.apply(f)
    ctx = _ctx(gs, torch, dims, m0, U)
    vc = gs.VCycle(ctx, levels, order=order, rest_tol=1e-13)
    fd = to_dev(f, torch)
    xd = torch.empty_like(fd)
    vc.apply(fd, xd)
    got = xd.cpu().numpy()
    assert close(got, ref, 1e-10), (rel(got, ref), maxrel(got, ref))
    fd[5] = float("nan")
    with pytest.raises(gs.GschurError, match="NONFINITE"):
        vc.apply(fd, xd)
    fd.zero_()
    vc.apply(fd, xd)
    assert not xd.cpu().numpy().any()
    vc.close()
    ctx.close()


# FP32 sums of up to 96 x 3 x V products: the bound of the one-sample test, 1e-4.
@pytest.mark.parametrize("dims,t", [((2, 2, 2, 2), 1), ((4, 3, 5, 3), 2), ((4, 5, 4, 6), 2)])
@pytest.mark.parametrize("batch", [1, 3, 4, 5])
def test_training_gradient_of_a_batch(env, dims, t, batch):
    torch, gs = env
    V = li.volume(dims)
    U = li.random_gauge(dims, 0.4, 2)
    ctx = _ctx(gs, torch, dims, 0.1, U)
    perm, nb = permute.permutation(dims, t)
    nr = V - nb
    Ws = [w.astype(np.complex64) for w in onet.init_weights(24, 5, scale=0.25)]
    nt = gs.Net(24)
    for l, w in enumerate(Ws):
        nt.set_weights(l, w)
    rng = np.random.default_rng(1)
    T, Z = ((rng.standard_normal((batch, nr, 12)) + 1j * rng.standard_normal((batch, nr, 12))).astype(np.complex64)
            for _ in range(2))
    W64, tr = [w.astype(np.complex128) for w in Ws], onet.transports(U, dims)
    L, G = 0.0, [0.0, 0.0, 0.0]
    for b in range(batch):
        tfull = np.zeros((V, 12), complex)
        tfull[perm[nb:]] = T[b]
        acts = onet.forward(W64, tfull.reshape(V, 4, 3), tr)
        y, z = acts[-1].reshape(V, 12), Z[b].astype(np.complex128)
        L += onet.loss(y[perm[nb:]], z) / batch
        gy = np.zeros((V, 12), complex)
        gy[perm[nb:]] = 2.0 * (y[perm[nb:]] - z) / np.vdot(z, z).real / batch
        G = [a + g for a, g in zip(G, onet.backward(W64, acts, gy.reshape(V, 1, 4, 3), tr))]
    td, zd = torch.from_numpy(T).to("cuda:0"), torch.from_numpy(Z).to("cuda:0")
    loss = nt.train_step(ctx.handle, t, 0, 0, batch, td, zd, 0.0, update=False)
    assert abs(loss - L) <= 1e-4 * L
    for l in range(3):
        assert close(nt.get(1, l).astype(np.complex128), G[l], 1e-4), l
    nt.close()
    ctx.close()


# V = 256 = 3 x 85 + 1, 16 (one tile, part full), 1360 = 16 x 85; that test's own bounds.
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (2, 2, 2, 2), (2, 10, 34, 2)])
def test_tensor_core_layer_last_tile(env, dims):
    _tensor_core_layer(env, dims)
