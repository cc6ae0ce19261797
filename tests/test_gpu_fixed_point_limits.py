"""Inputs at the limits of the fixed-point FP64 kernels, where their range or their
resolution ends and double precision takes over, against the double-precision
kernel (wilson_apply_noalloc) or one launch per phase on the same inputs."""
import numpy as np
import pytest

import lattice_inputs as li
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
    """D x by the context and by the double-precision kernel, complex128 [V][12]."""
    torch, gs = env
    ctx = _ctx(gs, torch, dims, m0, U)
    xd = to_dev(x, torch)
    y, ref = torch.empty_like(xd), torch.empty_like(xd)
    ctx.wilson_apply(xd, y)
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
