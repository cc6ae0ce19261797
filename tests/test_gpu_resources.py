"""What calls hold and share between them: a network's buffers on several
lattices, memory, the blocks of batched solves, and the routes of fields that
fixed point cannot hold."""
import numpy as np
import pytest

import lattice_inputs as li
from oracle import net as onet
from tests.gpu_util import lib, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    return torch, lib()


def _ctx(gs, torch, dims, m0, U, stream=None):
    ctx = gs.Context(dims, m0, torch.cuda.current_stream().cuda_stream if stream is None else stream)
    ctx.set_gauge(to_dev(U, torch))
    return ctx


def _net(gs, seed):
    nt = gs.Net(24)
    for l, w in enumerate(onet.init_weights(24, seed, scale=0.25)):
        nt.set_weights(l, w.astype(np.complex64))
    return nt


def test_network_on_two_lattices_keeps_its_buffers(env):
    """Training in groups of samples on a small lattice and applying on a large one in
    turn: nothing is allocated or freed once both have been seen."""
    torch, gs = env
    small, large = (4, 4, 4, 4), (8, 8, 8, 32)
    cs, cl = (_ctx(gs, torch, d, 0.1, li.random_gauge(d, 0.3, 1)) for d in (small, large))
    rng = np.random.default_rng(2)
    t, z = (to_dev((rng.standard_normal((4, 240, 12)) + 1j * rng.standard_normal((4, 240, 12))).astype(np.complex64),
                   torch) for _ in range(2))
    x = to_dev(rng.standard_normal((8192, 12)) + 0j, torch)
    ys = [torch.empty_like(x) for _ in range(2)]
    nt = _net(gs, 3)
    losses, free = [], []
    for k in range(2):
        losses.append(nt.train_step(cs.handle, 1, 0, 0, 4, t, z, 0.0, update=False))
        free.append(torch.cuda.mem_get_info()[0])
        nt.apply(cl.handle, 2, 0, 0, x, ys[k])
        free.append(torch.cuda.mem_get_info()[0])
    assert free[1] == free[2] == free[3]
    assert losses[0] == losses[1] and torch.equal(ys[0], ys[1])
    nt.close()
    cs.close()
    cl.close()


def test_two_networks_follow_a_new_field(env):
    """Each network of a context copies the new field's links, whichever is used first."""
    torch, gs = env
    dims = (4, 4, 4, 4)
    U1, U2 = li.random_gauge(dims, 0.3, 4), li.random_gauge(dims, 0.4, 5)
    x = to_dev(np.random.default_rng(6).standard_normal((128, 12)) + 0j, torch)

    def apply(ctx, nt):
        y = torch.empty_like(x)
        nt.apply(ctx.handle, 2, 0, 0, x, y)
        return y

    ctx, fresh = _ctx(gs, torch, dims, 0.1, U1), _ctx(gs, torch, dims, 0.1, U2)
    a, b, c = _net(gs, 7), _net(gs, 7), _net(gs, 7)
    apply(ctx, a)
    apply(ctx, b)
    ctx.set_gauge(to_dev(U2, torch))
    want = apply(fresh, c)
    assert torch.equal(apply(ctx, a), want) and torch.equal(apply(ctx, b), want)
    for n in (a, b, c):
        n.close()
    ctx.close()
    fresh.close()


@pytest.mark.parametrize("inner", [0, 1])
def test_field_beyond_fixed_point_goes_straight_to_double_precision(env, inner):
    """One link far from unitary: no conversion, no attempt of the fixed-point solver.
    S_bb x = two stencils and an inner solve, as kernels: 3 in one cooperative launch,
    and with one launch per phase the two stencils an iteration are single ones."""
    torch, gs = env
    dims, V = (4, 6, 4, 8), 768
    U = li.random_gauge(dims, 0.3, 8)
    bad = U.copy()
    bad[V // 2, 1, 0, 2] = 1.5            # an entry above 1.01
    rng = np.random.default_rng(9)
    x = to_dev(rng.standard_normal((V // 16, 12)) + 1j * rng.standard_normal((V // 16, 12)), torch)
    y, ref = torch.empty_like(x), torch.empty_like(x)
    o = gs.gs_default_opts(inner_tol=1e-12)
    ctx = _ctx(gs, torch, dims, 0.1, bad)
    ctx.set_option(gs.GS_OPT_INNER_KERNEL, inner)
    ctx.schur_apply(1, 0, 0, x, y, o)
    st = ctx.schur_apply(1, 0, 0, x, y, o)
    if inner == 0:
        assert st.kernel_launches == 3
    else:      # init, then five launches an iteration, at most two iterations queued past the last
        assert st.kernel_launches <= 3 + 5 * (st.inner_iters + 2)
    # the fixed-point route of a field within its range, a rounding away from the same operator
    good = bad.copy()
    good[V // 2, 1] *= 0.5
    ctx.set_gauge(to_dev(good, torch))
    ctx.schur_apply(1, 0, 0, x, ref, o)
    ctx.set_gauge(to_dev(bad, torch))
    ctx.schur_apply(1, 0, 0, x, ref, o)
    assert torch.equal(y, ref)
    ctx.close()


@pytest.mark.parametrize("dims,fields", [((8, 8, 8, 12), "within"), ((8, 8, 8, 12), "beyond"), ((4, 4, 4, 8), "beyond"),
                                         ((8, 8, 8, 8), "both"), ((8, 8, 8, 12), "both")])
def test_batched_fp64_solves(env, dims, fields):
    """Six FP64 solves at once: rest sets above 32 sites per SM (5760: the solves share the
    co-resident blocks, a part of their tiles each) and below, fields within and beyond fixed
    point's range, and the two solvers' blocks side by side.  Every inner solve stays one
    cooperative launch and the solutions are those of one solve at a time."""
    torch, gs = env
    streams = [torch.cuda.Stream() for _ in range(6)]
    V, o = li.volume(dims), gs.gs_default_opts()
    ctxs, probs = [], []
    for k, s in enumerate(streams):
        U = li.random_gauge(dims, 0.3, 40 + k)
        if fields == "beyond" or (fields == "both" and k % 2):
            U[V // 3, 2, 1, 1] = 1.2
        ctxs.append(_ctx(gs, torch, dims, 0.0, U, s.cuda_stream))
        f = to_dev(li.gaussian_source(dims, 50 + k), torch)
        probs.append(dict(ctx=ctxs[-1].handle, type=1 + k % 2, dir=0, inverse=k // 4, nrhs=1, f=f, x=torch.zeros_like(f)))
    ctxs[0].set_option(gs.GS_OPT_BATCH_LANES, 6)
    torch.cuda.synchronize()
    for _ in range(2):
        status, stats = gs.schur_solve_batched(probs, o)
        assert status == gs.GS_OK
    for c, pr, st in zip(ctxs, probs, stats):
        x1 = torch.zeros_like(pr["f"])
        one = c.schur_solve(pr["type"], 0, pr["inverse"], pr["f"], x1, o)
        assert st.true_residual <= 1e-10 and one.true_residual <= 1e-10
        assert (pr["x"] - x1).norm() <= 1e-8 * x1.norm()
        # as many launches as alone, up to an outer iteration or two (19 launches at most)
        assert st.kernel_launches <= one.kernel_launches + 40
        c.close()


def test_lattice_that_just_fits(env):
    """The fixed-point copies are there for speed only: with room for what double
    precision needs (1768 bytes a site) and not for them, the calls run in double
    precision."""
    torch, gs = env
    dims, m0 = (16, 16, 16, 32), 0.1
    V = li.volume(dims)
    rng = np.random.default_rng(10)
    U = to_dev(li.random_gauge(dims, 0.3, 60), torch)
    x = to_dev(rng.standard_normal((V, 12)) + 1j * rng.standard_normal((V, 12)), torch)
    xb = x[:V // 16].clone()
    out = []
    torch.cuda.synchronize()
    for tight in (False, True):
        torch.cuda.empty_cache()
        y, yb = torch.empty_like(x), torch.empty_like(xb)
        hog = None
        if tight:
            hog = torch.empty(torch.cuda.mem_get_info()[0] - (1768 * V + (32 << 20)), dtype=torch.uint8, device="cuda:0")
        ctx = gs.Context(dims, m0, torch.cuda.current_stream().cuda_stream)
        ctx.set_gauge(U)
        ctx.wilson_apply(x, y)
        del hog
        torch.cuda.empty_cache()
        ctx.schur_apply(1, 0, 0, xb, yb, gs.gs_default_opts(inner_tol=1e-12))
        torch.cuda.synchronize()
        ctx.close()
        out.append((y, yb))
    (y1, b1), (y2, b2) = out
    assert (y1 - y2).abs().max() <= 1.5e-13 * x.abs().max()
    assert (b1 - b2).norm() <= 1e-10 * b1.norm()


def test_block_counts_that_fill_the_gpu(env):
    """GS_OPT_COOP_BLOCKS: four FP64 solves with a quarter of 3 blocks per SM each, which is what
    the GPU holds by the option's description, run together."""
    torch, gs = env
    dims = (8, 8, 8, 8)
    blocks = 3 * torch.cuda.get_device_properties(0).multi_processor_count // 4
    streams = [torch.cuda.Stream() for _ in range(4)]
    ctxs = [_ctx(gs, torch, dims, 0.0, li.random_gauge(dims, 0.3, 70 + k), s.cuda_stream) for k, s in enumerate(streams)]
    probs = []
    for k, c in enumerate(ctxs):
        c.set_option(gs.GS_OPT_COOP_BLOCKS, blocks)
        f = to_dev(li.gaussian_source(dims, 80 + k), torch)
        probs.append(dict(ctx=c.handle, type=1 + k % 2, dir=0, inverse=0, nrhs=1, f=f, x=torch.zeros_like(f)))
    torch.cuda.synchronize()
    status, stats = gs.schur_solve_batched(probs, gs.gs_default_opts())
    assert status == gs.GS_OK and max(st.true_residual for st in stats) <= 1e-10
    for c in ctxs:
        c.close()


def test_waiting_for_blocks_is_no_timeout(env):
    """24 FP64 solves at once on 8^4 wait tens of milliseconds for their turn; the wait limit of
    the kernels (1 ms here) has nothing to do with it."""
    torch, gs = env
    dims, N = (8, 8, 8, 8), 24
    U = li.random_gauge(dims, 0.3, 90)
    streams = [torch.cuda.Stream() for _ in range(N)]
    ctxs = [_ctx(gs, torch, dims, 0.0, U, s.cuda_stream) for s in streams]
    ctxs[0].set_option(gs.GS_OPT_BATCH_LANES, N)
    probs = []
    for k, c in enumerate(ctxs):
        c.set_option(gs.GS_OPT_WAIT_LIMIT_US, 1000)
        f = to_dev(li.gaussian_source(dims, 100 + k), torch)
        probs.append(dict(ctx=c.handle, type=1, dir=0, inverse=k % 2, nrhs=1, f=f, x=torch.zeros_like(f)))
    torch.cuda.synchronize()
    status, stats = gs.schur_solve_batched(probs, gs.gs_default_opts())
    assert status == gs.GS_OK and max(st.true_residual for st in stats) <= 1e-10
    for c in ctxs:
        c.close()
