"""Creating an operator where the device has room for the data that it cannot do
without but not for the copy that serves speed alone (the fixed-point links of a
staggered operator, the real parts of a real 1 x 1 block matrix): it is created
without the copy and applies as before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402


def test_operator_fits_without_the_fixed_point_copy():
    dims, nc = (32, 32, 32, 32), 2
    V = int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(9)
    q = torch.randn((4 * V, 4), generator=g, device="cuda", dtype=torch.float64)
    q = q / q.norm(dim=1, keepdim=True)
    a, b = torch.complex(q[:, 0], q[:, 1]), torch.complex(q[:, 2], q[:, 3])
    U = torch.stack([a, b, -b.conj(), a.conj()], 1).reshape(4, V, nc, nc).contiguous()
    n = V * nc
    x = torch.complex(torch.randn(n, generator=g, device="cuda", dtype=torch.float64),
                      torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
    del q, a, b
    c = msc.msc_create(0, torch.cuda.current_stream())
    op = msc.msc_op_staggered(c, nc, dims, U, 0.1)
    want, out = torch.empty_like(x), torch.empty_like(x)
    msc.msc_op_apply(c, op, 0.3, x, want, msc.MSC_FP64)
    # the FP64 form of the same links, for its workspace
    full = msc.msc_op_staggered(c, nc, dims, U * 1.5, 0.1, msc.MSC_LINKS_FULL)
    msc.msc_op_apply(c, full, 0.3, x, out, msc.MSC_FP64)
    msc.msc_op_destroy(full)
    msc.msc_op_destroy(op)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # FP64 268 MB and FP32 67 MB, fixed-point copy 268 MB
    free, _ = torch.cuda.mem_get_info()
    filler = torch.empty(free - (420 << 20), dtype=torch.uint8, device="cuda")
    try:
        op = msc.msc_op_staggered(c, nc, dims, U, 0.1)
        msc.msc_op_apply(c, op, 0.3, x, out, msc.MSC_FP64)
        msc.msc_op_destroy(op)
    finally:
        del filler
        torch.cuda.empty_cache()
    # the two forms differ by roundings of 32 products per part and pass
    assert float((out - want).norm() / want.norm()) <= 1e-15
    msc.msc_destroy(c)


def test_real_matrix_fits_without_its_real_parts():
    n, per = 4 << 20, 5
    g = torch.Generator(device="cuda").manual_seed(10)
    rp = torch.arange(0, per * n + 1, per, dtype=torch.int64, device="cuda")
    ci = torch.randint(0, n, (per * n,), generator=g, device="cuda", dtype=torch.int32)
    va = torch.randn(per * n, generator=g, device="cuda", dtype=torch.float64).to(torch.complex128)
    x = torch.complex(torch.randn(n, generator=g, device="cuda", dtype=torch.float64),
                      torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
    c = msc.msc_create(0, torch.cuda.current_stream())
    op = msc.msc_op_bsr(c, n, 1, rp, ci, va)
    want, out = torch.empty_like(x), torch.empty_like(x)
    msc.msc_op_apply(c, op, 0.3, x, want, msc.MSC_FP64)
    msc.msc_op_destroy(op)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # FP64 336 MB, FP32 168, columns 84 and (while packing) row starts 34; real parts 168
    free, _ = torch.cuda.mem_get_info()
    filler = torch.empty(free - (700 << 20), dtype=torch.uint8, device="cuda")
    try:
        op = msc.msc_op_bsr(c, n, 1, rp, ci, va)
        msc.msc_op_apply(c, op, 0.3, x, out, msc.MSC_FP64)
        msc.msc_op_destroy(op)
    finally:
        del filler
        torch.cuda.empty_cache()
    # the same sums, with products by zero beside them
    assert float((out - want).norm() / want.norm()) <= 1e-15
    msc.msc_destroy(c)
