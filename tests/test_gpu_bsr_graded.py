"""Block-CSR matrices whose blocks hold entries of very different sizes
(unknowns in different units): FP64 applies keep every entry, componentwise,
and the true residual that a solve reports is that of the matrix given.

Tolerances: an output is at most 8 blocks of 3 entries, 24 complex products, so
its FP64 rounding is below 2 * 25 * 2^-52 < 2^-46 of sum |A_ab| |x_b|. The
residual is recomputed from the original entries; the two evaluations differ by
such roundings, below 1e-12 of |b| here."""
import numpy as np
import pytest

from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402


def dense(rp, ci, va, bd):
    n = len(rp) - 1
    A = np.zeros((n * bd, n * bd), np.clongdouble)
    for i in range(n):
        for k in range(rp[i], rp[i + 1]):
            A[i * bd:(i + 1) * bd, ci[k] * bd:(ci[k] + 1) * bd] += va[k].astype(np.clongdouble)
    return A


def check_apply(c, rp, ci, va, bd, v):
    nbr = len(rp) - 1
    op = msc.msc_op_bsr(c, nbr, bd, rp, ci, va)
    out = np.empty_like(v)
    msc.msc_op_apply(c, op, 0.0, v, out, msc.MSC_FP64)
    msc.msc_op_destroy(op)
    A = dense(rp, ci, va, bd)
    err = np.abs(out - A @ v.astype(np.clongdouble))
    big = np.abs(A) @ np.abs(v)
    return float(np.max(err / big))


@pytest.fixture(scope="module")
def ctx():
    msc.load()
    c = msc.msc_create(0, torch.cuda.current_stream())
    yield c
    msc.msc_destroy(c)


@pytest.mark.parametrize("bd", [2, 3])
@pytest.mark.parametrize("decades", [8, 12, 18])
@pytest.mark.parametrize("form", ["rows and columns", "rows", "columns"])
def test_graded_components(ctx, bd, decades, form):
    nbr = 35
    rp, ci, va, _ = inputs.random_hpd_bsr(nbr, bd, 5, 0.5, 500 + bd)
    s = 10.0 ** -np.linspace(0, decades, bd)
    left = s if form != "columns" else np.ones(bd)
    right = s if form != "rows" else np.ones(bd)
    va = va * left[None, :, None] * right[None, None, :]
    v = inputs.gaussian_source(nbr * bd, 501)
    assert check_apply(ctx, rp, ci, va, bd, v / np.tile(right, nbr)) <= 2.0 ** -46
    assert check_apply(ctx, rp, ci, va, bd, v) <= 2.0 ** -46


@pytest.mark.parametrize("bd", [2, 3])
def test_one_graded_row_among_even_ones(ctx, bd):
    """The block rows but one are of like sizes; the one has a small row."""
    nbr = 70
    rp, ci, va, _ = inputs.random_hpd_bsr(nbr, bd, 5, 0.5, 510 + bd)
    va[rp[41]:rp[42], bd - 1, :] *= 1e-13
    v = inputs.gaussian_source(nbr * bd, 511)
    assert check_apply(ctx, rp, ci, va, bd, v) <= 2.0 ** -46


@pytest.mark.parametrize("bd", [2, 3])
def test_decoupled_components(ctx, bd):
    """Blocks that are multiples of the identity, a source whose components
    differ by 20 decades: each component is a system of its own."""
    nbr = 33
    rp, ci, va, _ = inputs.random_hpd_bsr(nbr, bd, 5, 0.5, 520 + bd)
    va = va[:, :1, :1] * np.eye(bd)[None]
    v = inputs.gaussian_source(nbr * bd, 521) * np.tile(10.0 ** -np.linspace(0, 20, bd), nbr)
    assert check_apply(ctx, rp, ci, va, bd, v) <= 2.0 ** -46


@pytest.mark.parametrize("big", [1e8, 1e10, 1e12])
def test_reported_residual_is_the_given_matrix(ctx, big):
    nbr, bd = 40, 2
    rp = np.arange(nbr + 1, dtype=np.int64)
    ci = np.arange(nbr, dtype=np.int32)
    d = np.array([big, np.pi])
    va = np.ascontiguousarray(np.broadcast_to(np.diag(d), (nbr, bd, bd))).astype(complex)
    b = inputs.gaussian_source(nbr * bd, 530)
    sig = np.array([0.0, 1.0])
    op = msc.msc_op_bsr(ctx, nbr, bd, rp, ci, va)
    x, info = msc.solve(ctx, op, torch.from_numpy(b).cuda(), sig, tol=1e-10, precision=msc.MSC_FP64)
    msc.msc_op_destroy(op)
    x = x.cpu().numpy().reshape(len(sig), -1)
    rep = np.asarray(info.true_rel_resid).reshape(-1)
    for s, sg in enumerate(sig):
        r = b - (np.tile(d, nbr) + sg) * x[s]
        rho = np.linalg.norm(r) / np.linalg.norm(b)
        assert abs(rho - rep[s]) <= 1e-12, (sg, rho, rep[s])
        if info.status == 0:
            assert rho <= 1.01e-10


def test_bad_column_behind_a_graded_row_is_refused(ctx):
    """A column out of range in the last row, with a first row that sends the
    matrix to FP64 before the last is looked at."""
    bd, nbr = 2, 200000
    rp = np.arange(nbr + 1, dtype=np.int64)
    ci = np.arange(nbr, dtype=np.int32)
    va = np.tile(np.array([[2.0, 1.0], [1.0, 2.0]], complex), (nbr, 1, 1))
    va[0] = np.diag([1e12, 1.0])
    op = msc.msc_op_bsr(ctx, nbr, bd, rp, ci, va)
    msc.msc_op_destroy(op)
    ci[-1] = nbr
    with pytest.raises(msc.MscError) as e:
        msc.msc_op_bsr(ctx, nbr, bd, rp, ci, va)
    assert e.value.code == msc.MSC_ERR_ARG
