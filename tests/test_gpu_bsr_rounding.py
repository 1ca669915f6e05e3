"""FP64 block-CSR rows by fixed-point sums are rounded, not floored: their
errors have no mean.

One block a row, parts of block and entries in +-[0.5, 1): every product is in
the same unit, 2^-56. An output is then a sum of 2 bd products of at most 2 bd
in size, rounded to FP64 with an error spread over at most 64 units (19 units
rms), quantisation and dropped terms below a unit each with the products' signs;
the mean of 240,000 of them is within 5 x 19 / sqrt(240,000) = 0.2 units of
zero, a floor's is at -0.5."""
import numpy as np
import pytest

from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402


@pytest.mark.parametrize("bd,nbr", [(2, 60000), (3, 40000)])
def test_errors_have_no_mean(bd, nbr):
    g = inputs.rng(900 + bd)

    def parts(*shape):
        def one():
            return g.uniform(0.5, 1.0, shape) * np.where(g.random(shape) < 0.5, -1.0, 1.0)
        return one() + 1j * one()
    va, x = parts(nbr, bd, bd), parts(nbr, bd)
    c = msc.msc_create(0, torch.cuda.current_stream())
    op = msc.msc_op_bsr(c, nbr, bd, np.arange(nbr + 1, dtype=np.int64), np.arange(nbr, dtype=np.int32), va)
    out = np.empty(nbr * bd, complex)
    msc.msc_op_apply(c, op, 0.0, x.reshape(-1), out, msc.MSC_FP64)
    msc.msc_op_destroy(op)
    msc.msc_destroy(c)

    # exact sums: each product of two doubles as a pair of doubles (numpy's
    # extended precision is only FP64 on some machines)
    def split(a):
        t = a * 134217729.0
        hi = t - (t - a)
        return hi, a - hi

    def two_prod(a, b):
        p = a * b
        (ah, al), (bh, bl) = split(a), split(b)
        return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl

    def two_sum(a, b):
        s = a + b
        t = s - a
        return s, (a - (s - t)) + (b - t)
    y = out.reshape(nbr, bd)
    err = []
    for a in range(bd):
        for part in ("re", "im"):
            s, e = -(y[:, a].real if part == "re" else y[:, a].imag), 0.0
            for b in range(bd):
                u, v = va[:, a, b], x[:, b]
                for p, q in ((u.real, v.real), (-u.imag, v.imag)) if part == "re" else ((u.real, v.imag), (u.imag, v.real)):
                    h, l = two_prod(p, q)
                    s, r = two_sum(s, h)
                    e = e + (r + l)
            err.append(-(s + e))
    err = np.concatenate(err) * 2.0 ** 56
    assert len(err) == 240000 and np.abs(err).max() <= 80
    assert abs(err.mean()) <= 0.2, err.mean()
