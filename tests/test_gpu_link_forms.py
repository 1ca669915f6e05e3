"""Which links the FP64 passes sum in fixed point: unitary ones, whatever their
determinant, whose entries couple the colours; the others keep the FP64 form.
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
