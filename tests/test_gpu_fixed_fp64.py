"""FP64 operator passes by fixed-point sums (csrc/fixed.cuh) against the same
sums in extended precision.

Tolerances, from the arithmetic: an output of D is at most 96 products of a
link part (quantised to 2^-57) and an entry part (truncated at 2^-56 of twice
the largest of the output's own 48 neighbour parts), the product of the low
limbs dropped (2^-56), halved: below 96 * 2^-55 * vmax = 2^-48.4 vmax, elementwise; the FP64
form of the oracle must not have a smaller 2-norm error. Entries outside the
fixed-point range (Inf, NaN, subnormal or near the ends of the exponent range)
take FP64 arithmetic and give what the oracle gives.
"""
import numpy as np
import pytest

import oracle
from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402

DIMS = [(3, (2, 4, 6, 2)), (2, (6, 4, 2, 8)), (3, (10, 6, 4, 12))]


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available()
    c = msc.msc_create(0, torch.cuda.current_stream())
    yield c
    msc.msc_destroy(c)


def hops(dims):
    V = inputs.volume(dims)
    x = np.arange(V)
    out, stride, par = [], 1, np.zeros(V, int)
    for L in dims:
        c = (x // stride) % L
        out.append((np.where(c == L - 1, x - (L - 1) * stride, x + stride),
                    np.where(c == 0, x + (L - 1) * stride, x - stride), np.where(par % 2 == 0, 0.5, -0.5)))
        stride, par = stride * L, par + c
    return out


def dslash_ext(U, dims, nc, v):
    """D v in extended precision, and the largest neighbour part of each output."""
    V = inputs.volume(dims)
    U = U.astype(np.clongdouble)
    w = v.reshape(V, nc).astype(np.clongdouble)
    y = np.zeros((V, nc), np.clongdouble)
    big = np.zeros(V)
    part = np.maximum(np.abs(v.real), np.abs(v.imag)).reshape(V, nc).max(1)
    for mu, (f, b, eta) in enumerate(hops(dims)):
        e = eta[:, None].astype(np.longdouble)
        y += e * np.einsum("xab,xb->xa", U[mu], w[f])
        y -= e * np.einsum("xba,xb->xa", np.conj(U[mu][b]), w[b])
        big = np.maximum(big, np.maximum(part[f], part[b]))
    return y.reshape(-1), np.repeat(big, nc)


def vectors(n, seed):
    g = inputs.rng(seed)
    v = inputs.gaussian_source(n, seed)
    point = np.zeros(n, complex)
    point[n // 3] = 1.0 - 0.5j
    return {"gaussian": v, "tiny": v * 1e-200, "huge": v * 1e200, "point": point,
            "spread": v * np.exp(g.uniform(-60, 60, n)), "zero": np.zeros(n, complex)}


@pytest.mark.parametrize("nc,dims", DIMS)
def test_dslash_against_extended_precision(ctx, nc, dims):
    U = inputs.su_n_links(dims, nc, 0.9, 40 + nc)
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(U).cuda(), 0.1)
    n = inputs.volume(dims) * nc
    for name, v in vectors(n, 50).items():
        out = np.empty_like(v)
        msc.msc_op_dslash(ctx, op, v, out)
        want, big = dslash_ext(U, dims, nc, v)
        err = np.abs(out.astype(np.clongdouble) - want)
        assert np.all(err <= 2.0 ** -48.4 * big), (name, float(np.max(err / np.maximum(big, 1e-300))))
        scale = 1.0 / max(np.abs(v).max(), 1e-300)
        here = np.linalg.norm((err * scale).astype(float))
        fp64 = np.linalg.norm((np.abs(oracle.dslash(U, dims, nc, v) - want) * scale).astype(float))
        if name in ("gaussian", "tiny", "huge"):
            assert here <= fp64, (name, here, fp64)
    msc.msc_op_destroy(op)


@pytest.mark.parametrize("nc,dims", DIMS)
def test_out_of_range_entries_take_fp64(ctx, nc, dims):
    U = inputs.su_n_links(dims, nc, 0.9, 60 + nc)
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(U).cuda(), 0.1)
    n = inputs.volume(dims) * nc
    v = inputs.gaussian_source(n, 61)
    for bad in (np.inf, -np.inf, np.nan):
        w = v.copy()
        w[n // 2] = bad
        out = np.empty_like(w)
        msc.msc_op_dslash(ctx, op, w, out)
        want = oracle.dslash(U, dims, nc, w)
        assert np.array_equal(np.isfinite(out), np.isfinite(want))
        ok = np.isfinite(want)
        assert np.linalg.norm(out[ok] - want[ok]) <= 1e-13 * np.linalg.norm(want[ok])
    for scale in (1e-318, 1e-300, 1e307):
        w = v * scale
        out = np.empty_like(w)
        msc.msc_op_dslash(ctx, op, w, out)
        want = oracle.dslash(U, dims, nc, w)
        assert np.max(np.abs(out - want) / scale) <= max(1e-12, 16 * 5e-324 / scale)
    msc.msc_op_destroy(op)


def test_non_unitary_links_stay_on_the_fp64_form(ctx):
    dims, nc = (4, 6, 4, 2), 3
    U = 3.0 * inputs.su_n_links(dims, nc, 0.9, 70)
    U[0, 3] *= 1e5
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(U).cuda(), 0.1)
    n = inputs.volume(dims) * nc
    v = inputs.gaussian_source(n, 71)
    out = np.empty_like(v)
    msc.msc_op_apply(ctx, op, 0.2, v, out, msc.MSC_FP64)
    want = oracle.staggered_apply(U, dims, nc, 0.1, v, sigma=0.2)
    assert np.linalg.norm(out - want) <= 1e-13 * np.linalg.norm(want)
    msc.msc_op_destroy(op)


def bsr_ext(rp, ci, va, v, nbr, bd):
    """A v in extended precision and, per row, the largest block part times
    entry part summed over its blocks."""
    w = v.reshape(nbr, bd).astype(np.clongdouble)
    y = np.zeros((nbr, bd), np.clongdouble)
    big = np.zeros(nbr)
    part = np.maximum(np.abs(v.real), np.abs(v.imag)).reshape(nbr, bd).max(1)
    for i in range(nbr):
        for k in range(rp[i], rp[i + 1]):
            y[i] += va[k].astype(np.clongdouble) @ w[ci[k]]
            big[i] += max(np.abs(va[k].real).max(), np.abs(va[k].imag).max()) * part[ci[k]]
    return y.reshape(-1), np.repeat(big, bd)


@pytest.mark.parametrize("bd,nbr", [(2, 37), (3, 33), (3, 70)])
@pytest.mark.parametrize("scaled", [False, True])
def test_bsr_against_extended_precision(ctx, bd, nbr, scaled):
    """Ragged rows; `scaled`: A -> S A S with S spread over 12 decades and
    entries over its inverse (products of like size from unlike factors). A
    group of blocks is summed to 2^-56 of its largest product: an output is
    within 18 products * 4 * 2^-56 of the sum of the blocks' bounds, plus
    FP64 roundings of the row sum, below 2^-49 of it."""
    rp, ci, va, A = inputs.random_hpd_bsr(nbr, bd, 5, 0.5, 80 + nbr)
    g = inputs.rng(81)
    s = 10.0 ** g.uniform(-6, 6, nbr) if scaled else np.ones(nbr)
    for i in range(nbr):
        for k in range(rp[i], rp[i + 1]):
            va[k] = va[k] * (s[i] * s[ci[k]])
    op = msc.msc_op_bsr(ctx, nbr, bd, rp, ci, va)
    n = nbr * bd
    v = inputs.gaussian_source(n, 82) / np.repeat(s, bd)
    for scale in (1.0, 1e-150, 1e150):
        w = v * scale
        out = np.empty_like(w)
        msc.msc_op_apply(ctx, op, 0.0, w, out, msc.MSC_FP64)
        want, big = bsr_ext(rp, ci, va, w, nbr, bd)
        err = np.abs(out - want)
        assert np.all(err <= 2.0 ** -49 * big), float(np.max(err / big))
        rel = (1.0 / np.repeat(s, bd)) / np.abs(v).max() / scale
        here = np.linalg.norm((err * rel).astype(float))
        fp64 = np.linalg.norm((np.abs(oracle.bsr_apply(rp, ci, va, w) - want) * rel).astype(float))
        assert here <= fp64, (scale, here, fp64)
    msc.msc_op_destroy(op)


@pytest.mark.parametrize("bd", [2, 3])
def test_bsr_out_of_range_takes_fp64(ctx, bd):
    nbr = 41
    rp, ci, va, A = inputs.random_hpd_bsr(nbr, bd, 4, 0.5, 90)
    n = nbr * bd
    v = inputs.gaussian_source(n, 91)

    def apply(vals, w):
        op = msc.msc_op_bsr(ctx, nbr, bd, rp, ci, vals)
        out = np.empty_like(w)
        msc.msc_op_apply(ctx, op, 0.0, w, out, msc.MSC_FP64)
        msc.msc_op_destroy(op)
        return out
    w = v.copy()
    w[n // 2] = np.nan
    out, want = apply(va, w), oracle.bsr_apply(rp, ci, va, w)
    # padding blocks read column 0: the others' rows are finite in both
    assert np.array_equal(np.isfinite(out), np.isfinite(want))
    for scale_a, scale_v in ((1e250, 1e-310), (1e-250, 1e250), (1e-280, 1.0), (1e290, 1e-5), (1.0, 1e-305)):
        out, want = apply(va * scale_a, v * scale_v), oracle.bsr_apply(rp, ci, va * scale_a, v * scale_v)
        tiny = 64 * 5e-324 * max(scale_a, 1.0)
        assert np.linalg.norm((out - want) / (scale_a * scale_v)) <= \
            1e-13 * np.linalg.norm(want / (scale_a * scale_v)) + tiny / (scale_a * scale_v), (scale_a, scale_v)
    b = va.copy()
    b[3, 0, 0] = np.inf
    out, want = apply(b, v), oracle.bsr_apply(rp, ci, b, v)
    assert np.array_equal(np.isfinite(out), np.isfinite(want))


@pytest.mark.parametrize("bsr", [False, True])
def test_apply_in_place_overlapping_and_unaligned(ctx, bsr):
    """msc_op_apply on the caller's vectors in place: the same results whether
    input and output are the same vector, overlap by part, start between
    16-byte boundaries, or lie on the host. Exact: the kernels are the same."""
    dims, nc = (4, 6, 2, 4), 3
    U = inputs.su_n_links(dims, nc, 0.9, 95)
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(U).cuda(), 0.1)
    if bsr:
        nbr, nnzb, bd = msc.msc_op_bsr_size(op)
        rp = torch.empty(nbr + 1, dtype=torch.int64, device="cuda")
        ci = torch.empty(nnzb, dtype=torch.int32, device="cuda")
        va = torch.empty((nnzb, bd, bd), dtype=torch.complex128, device="cuda")
        msc.msc_staggered_export_bsr(ctx, op, rp, ci, va)
        op = msc.msc_op_bsr(ctx, nbr, bd, rp, ci, va)
    n = inputs.volume(dims) * nc
    v = inputs.gaussian_source(n, 96)
    x = torch.from_numpy(v).cuda()
    want = torch.empty_like(x)
    msc.msc_op_apply(ctx, op, 0.2, x, want, msc.MSC_FP64)
    assert torch.equal(x, torch.from_numpy(v).cuda())
    host = np.empty_like(v)
    msc.msc_op_apply(ctx, op, 0.2, v, host, msc.MSC_FP64)
    assert np.array_equal(host, want.cpu().numpy())
    same = x.clone()
    msc.msc_op_apply(ctx, op, 0.2, same, same, msc.MSC_FP64)
    assert torch.equal(same, want)
    buf = torch.zeros(2 * (n + 64), dtype=torch.float64, device="cuda")
    for at_in, at_out in ((0, 34), (34, 0), (1, 1), (3, 0), (0, 5)):
        i = buf[at_in:at_in + 2 * n]
        i.copy_(torch.view_as_real(x).reshape(-1))
        base = buf.data_ptr()
        msc.msc_op_apply(ctx, op, 0.2, base + 8 * at_in, base + 8 * at_out, msc.MSC_FP64)
        assert torch.equal(buf[at_out:at_out + 2 * n], torch.view_as_real(want).reshape(-1)), (at_in, at_out)
    if not bsr:
        d = torch.empty_like(x)
        msc.msc_op_dslash(ctx, op, x, d)
        y = x.clone()
        msc.msc_op_dslash(ctx, op, y, y)
        assert torch.equal(y, d)


def test_real_1x1_rows_equal_complex_rows(ctx):
    """A matrix of real 1 x 1 entries (ragged, with padding) against the oracle
    in FP64 (1e-13: rounding order only), with an Inf among the entries of x as
    the complex form has it, and one imaginary entry, which leaves the path."""
    n = 77
    rp, ci, va, _ = inputs.random_hpd_bsr(n, 1, 5, 0.5, 97)
    va = np.ascontiguousarray(va.real.astype(complex))
    v = inputs.gaussian_source(n, 98)
    for imag in (0.0, 0.25):
        w = va.copy()
        w[3, 0, 0] += 1j * imag
        op = msc.msc_op_bsr(ctx, n, 1, rp, ci, w)
        for x in (v, np.where(np.arange(n) == 40, np.inf + 1j, v)):
            out = np.empty_like(v)
            msc.msc_op_apply(ctx, op, 0.3, x, out, msc.MSC_FP64)
            want = oracle.bsr_apply(rp, ci, w, x, 0.3)
            ok = np.isfinite(want)
            # rows shorter than their slice's longest are padded with zeros on column 0
            assert np.array_equal(ok, np.isfinite(out))
            assert np.linalg.norm(out[ok] - want[ok]) <= 1e-13 * np.linalg.norm(want[ok])
        msc.msc_op_destroy(op)
