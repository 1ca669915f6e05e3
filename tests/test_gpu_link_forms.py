"""Which links the FP64 passes sum in fixed point: unitary ones, whatever their
determinant, whose entries couple the colours; the others keep the FP64 form,
componentwise.
A small FP64 solve shows the form that was taken: only with limbs does it run
in the cooperative iterations, which take no timing samples."""
import numpy as np
import pytest

import oracle
from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    msc.load()
    c = msc.msc_create(0, torch.cuda.current_stream())
    yield c
    msc.msc_destroy(c)


def solve_samples(ctx, U, dims, nc, seed, flags=0):
    n = inputs.volume(dims) * nc
    b = inputs.gaussian_source(n, seed)
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(U).cuda(), 0.2, flags)
    x, info = msc.solve(ctx, op, torch.from_numpy(b).cuda(), [0.01, 0.2], tol=1e-10, precision=msc.MSC_FP64)
    out = np.empty_like(b)
    msc.msc_op_apply(ctx, op, 0.0, b, out, msc.MSC_FP64)
    want = oracle.staggered_apply(U, dims, nc, 0.2, b)
    assert np.linalg.norm(out - want) <= 1e-14 * np.linalg.norm(want)
    rho = oracle.true_residual_staggered(U, dims, nc, 0.2, b, np.array([0.01, 0.2]),
                                         x.cpu().numpy().reshape(2, -1))
    assert info.status == 0 and np.all(rho <= 1.01e-10)
    msc.msc_op_destroy(op)
    return info.prof_samples


@pytest.mark.parametrize("nc,dims", [(2, (6, 4, 4, 8)), (3, (4, 4, 6, 8))])
def test_determinant_is_free(ctx, nc, dims):
    U = inputs.su_n_links(dims, nc, 0.8, 700 + nc)
    assert solve_samples(ctx, U, dims, nc, 701) == 0
    # antiperiodic in the last direction
    W = U.copy()
    W[3, inputs.volume(dims) - inputs.volume(dims) // dims[3]:] *= -1.0
    assert solve_samples(ctx, W, dims, nc, 702) == 0
    # a U(1) phase on every link
    th = inputs.rng(703).uniform(0, 2 * np.pi, U.shape[:2])
    assert solve_samples(ctx, np.exp(1j * th)[:, :, None, None] * U, dims, nc, 704) == 0
    # not unitary
    assert solve_samples(ctx, U * 1.001, dims, nc, 705, msc.MSC_LINKS_FULL) > 0


def dslash_ext(U, dims, nc, v):
    """D v in extended precision, and sum |U| |v| of each output."""
    V = inputs.volume(dims)
    U = U.astype(np.clongdouble)
    w = v.reshape(V, nc).astype(np.clongdouble)
    y, big = np.zeros((V, nc), np.clongdouble), np.zeros((V, nc), np.longdouble)
    x = np.arange(V)
    stride, par = 1, np.zeros(V, int)
    for mu, L in enumerate(dims):
        c = (x // stride) % L
        f, b = np.where(c == L - 1, x - (L - 1) * stride, x + stride), np.where(c == 0, x + (L - 1) * stride, x - stride)
        eta = np.where(par % 2 == 0, 0.5, -0.5).astype(np.longdouble)[:, None]
        y += eta * (np.einsum("xab,xb->xa", U[mu], w[f]) - np.einsum("xba,xb->xa", np.conj(U[mu][b]), w[b]))
        big += 0.5 * (np.einsum("xab,xb->xa", abs(U[mu]), abs(w[f])) + np.einsum("xba,xb->xa", abs(U[mu][b]), abs(w[b])))
        stride, par = stride * L, par + c
    return y.reshape(-1), big.reshape(-1)


@pytest.mark.parametrize("nc", [2, 3])
# four lanes and one lane per site
@pytest.mark.parametrize("dims", [(4, 6, 2, 8), (16, 16, 12, 10)])
@pytest.mark.parametrize("form", ["unit", "phases", "nearly unit", "one link"])
def test_links_that_do_not_couple_the_colours(ctx, nc, dims, form):
    """Colours that are systems of their own keep their own precision, and so do
    entries far below 1. FP64 rounds 8 nc complex products of a sum to below
    2 * 25 * 2^-52 < 2^-46 of the sum of their moduli."""
    V = inputs.volume(dims)
    U = np.zeros((4, V, nc, nc), complex)
    g = inputs.rng(710)
    for a in range(nc):
        U[:, :, a, a] = np.exp(1j * g.uniform(0, 2 * np.pi, (4, V))) if form == "phases" else 1.0
    if form == "nearly unit":
        U[:, :, 0, 1], U[:, :, 1, 0] = 1.2e-14 + 0.7e-14j, -1.2e-14 + 0.7e-14j
    if form == "one link":
        U = inputs.su_n_links(dims, nc, 0.8, 711)
        U[2, V // 2] = np.eye(nc)
    v = inputs.gaussian_source(V * nc, 712)
    if form != "one link":
        v = v * np.tile(10.0 ** -np.linspace(0, 20, nc), V) if form != "nearly unit" else v * np.tile(np.arange(nc) == 0, V)
    else:
        v = v * np.repeat(np.arange(V) == (V // 2 + dims[0] * dims[1]) % V, nc) * np.tile(10.0 ** -np.linspace(0, 20, nc), V)
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(U).cuda(), 0.1)
    out = np.empty_like(v)
    msc.msc_op_dslash(ctx, op, v, out)
    msc.msc_op_destroy(op)
    want, big = dslash_ext(U, dims, nc, v)
    assert np.all(np.abs(out - want) <= 2.0 ** -46 * big)
