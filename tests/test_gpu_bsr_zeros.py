"""FP64 block-CSR rows in which a block meets exact zeros: it adds nothing,
whatever the sizes of the row's other products (powers of two far apart, for
which the FP64 sum is one block's product alone).

Tolerance: one block's 2 bd products per part in FP64 or in fixed point below
2^-50 of the sum of their moduli."""
import numpy as np
import pytest

from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402


@pytest.mark.parametrize("bd", [2, 3])
@pytest.mark.parametrize("big,small", [(100, -900), (200, -820), (40, -880), (0, -880), (300, -700)])
@pytest.mark.parametrize("neg", [False, True])
def test_block_times_zero_adds_nothing(bd, big, small, neg):
    c = msc.msc_create(0, torch.cuda.current_stream())
    g = inputs.rng(30 + bd)
    M = g.standard_normal((3, bd, bd)) + 1j * g.standard_normal((3, bd, bd))
    # row 0: a large block on zeros, a block of size 1 on entries of 2^small;
    # rows 1 and 2: the identity
    va = np.stack([M[0] * 2.0 ** big, M[1], M[2] * 2.0 ** big, np.eye(bd), np.eye(bd)]).astype(complex)
    rp = np.array([0, 3, 4, 5], dtype=np.int64)
    ci = np.array([0, 1, 2, 1, 2], dtype=np.int32)
    z = g.standard_normal(bd) + 1j * g.standard_normal(bd)
    zero = np.full(bd, -0.0 - 0.0j if neg else 0j)
    x = np.concatenate([zero, z * 2.0 ** small, zero])
    op = msc.msc_op_bsr(c, 3, bd, rp, ci, va)
    out = np.empty_like(x)
    msc.msc_op_apply(c, op, 0.0, x, out, msc.MSC_FP64)
    want, scale = M[1] @ z, np.abs(M[1]) @ np.abs(z)
    assert np.all(np.abs(out[:bd] * 2.0 ** -small - want) <= 2.0 ** -50 * scale)
    msc.msc_op_destroy(op)
    msc.msc_destroy(c)
