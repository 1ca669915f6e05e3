"""Small staggered systems through the cooperative iterations (csrc/persist.cu)
at the edges of their blocks: one block and a part of one, sites that do not
fill 256-site blocks, the parity-reduced operator, several right-hand sides,
links without row reconstruction, one and many shifts, FP64 and mixed, an
iteration cap, and the largest stage the path takes next to the first that it
leaves to the per-pass kernels.

Tolerances as in the parity tests: the FP64 true residual of every shift (the
oracle's, of the solution returned) at most tol, x within 1e-8 of the oracle's
solution (solved to 1e-13)."""
import numpy as np
import pytest

import oracle
from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available()
    c = msc.msc_create(0, torch.cuda.current_stream())
    yield c
    msc.msc_destroy(c)


CASES = [((2, 2, 2, 2), 3, 1, 1), ((4, 4, 4, 4), 2, 3, 8), ((6, 4, 10, 2), 3, 2, 5), ((6, 10, 6, 14), 3, 1, 37),
         ((8, 8, 6, 12), 2, 4, 3)]


@pytest.mark.parametrize("dims,nc,nrhs,S", CASES)
@pytest.mark.parametrize("prec", [msc.MSC_FP64, msc.MSC_MIXED])
@pytest.mark.parametrize("flags", [0, msc.MSC_LINKS_FULL])
def test_small_solves(ctx, dims, nc, nrhs, S, prec, flags):
    p = inputs.staggered_problem(dims, nc, 0.1, 0.7, inputs.log_shifts(1e-3, 2.0, S), nrhs, 1e-10, 7700)
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(p.links).cuda(), p.mass, flags)
    x, info = msc.solve(ctx, op, torch.from_numpy(p.b).cuda(), p.sigma, tol=p.tol, precision=prec)
    assert info.status == 0 and info.kernel_launches > 0
    xs = x.cpu().numpy()
    for r in range(nrhs):
        rho = oracle.true_residual_staggered(p.links, dims, nc, p.mass, p.b[r], p.sigma, xs[r])
        assert np.all(rho <= p.tol), (r, rho.max())
        ref = oracle.cgm_staggered(p.links, dims, nc, p.mass, p.b[r], p.sigma, 1e-13)
        for s in range(S):
            assert np.linalg.norm(xs[r, s] - ref.x[s]) <= 1e-8 * np.linalg.norm(ref.x[s])
    # a cap inside a launch, and one that falls on its end
    for cap in (7, 50):
        y, i2 = msc.solve(ctx, op, torch.from_numpy(p.b).cuda(), p.sigma, tol=1e-14, precision=prec, max_iter=cap,
                          refine=0)
        assert i2.iters <= cap
    msc.msc_op_destroy(op)


@pytest.mark.parametrize("parity", [0, 1])
def test_parity_view(ctx, parity):
    dims, nc = (6, 4, 8, 10), 3
    p = inputs.staggered_problem(dims, nc, 0.1, 0.7, inputs.log_shifts(1e-3, 2.0, 6), 1, 1e-10, 7800)
    V = inputs.volume(dims)
    x = np.arange(V)
    par = sum((x // int(np.prod(dims[:mu]))) % dims[mu] for mu in range(4)) % 2
    sites = np.flatnonzero(par == parity)
    b = np.zeros((V, nc), complex)
    b[sites] = p.b[0].reshape(V, nc)[sites]
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(p.links).cuda(), p.mass)
    half = np.ascontiguousarray(b[sites].reshape(-1))
    for prec in (msc.MSC_FP64, msc.MSC_MIXED):
        y, info = msc.solve_parity(ctx, op, parity, half, p.sigma, tol=p.tol, precision=prec)
        assert info.status == 0
        full = np.zeros((len(p.sigma), V, nc), complex)
        full[:, sites] = y.reshape(len(p.sigma), -1, nc)
        rho = oracle.true_residual_staggered(p.links, dims, nc, p.mass, b.reshape(-1), p.sigma,
                                             full.reshape(len(p.sigma), -1))
        assert np.all(rho <= 1.01 * p.tol)
    msc.msc_op_destroy(op)


def test_both_sides_of_the_line(ctx):
    """16^4 (256 blocks of sites): 16 right-hand sides are the last on the
    cooperative path, 17 the first off it; each column solves its system."""
    dims, nc = (16, 16, 16, 16), 3
    p = inputs.staggered_problem(dims, nc, 0.3, 0.6, np.array([0.05, 0.5]), 17, 1e-10, 7900)
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(p.links).cuda(), p.mass)
    b = torch.from_numpy(p.b).cuda()
    x17, i17 = msc.solve(ctx, op, b, p.sigma, tol=p.tol)
    x16, i16 = msc.solve(ctx, op, b[:16].contiguous(), p.sigma, tol=p.tol)
    assert i17.status == 0 and i16.status == 0
    assert i16.prof_samples == 0 and i17.prof_samples > 0
    assert float((x17[:16] - x16).norm() / x16.norm()) <= 1e-8
    msc.msc_op_destroy(op)
