"""A NaN or an Inf among the gauge links is no unitary link: an operator made
of them applies as the FP64 form does (non-finite where a link with the bad
entry is used, the oracle's numbers elsewhere), and a solve ends in
MSC_ERR_NONFINITE."""
import numpy as np
import pytest

import oracle
from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402


@pytest.mark.parametrize("nc", [2, 3])
@pytest.mark.parametrize("bad", [np.nan, 1j * np.nan, np.inf, -1j * np.inf])
def test_nonfinite_link_entry_is_seen(nc, bad):
    dims = (4, 6, 2, 4)
    c = msc.msc_create(0, torch.cuda.current_stream())
    U = inputs.su_n_links(dims, nc, 0.7, 20 + nc)
    n = inputs.volume(dims) * nc
    v = inputs.gaussian_source(n, 21)
    # every row and column: each sits elsewhere in U U^dagger and the determinant
    for a in range(nc):
        for b in range(nc):
            W = U.copy()
            W[1, 17, a, b] = bad
            op = msc.msc_op_staggered(c, nc, dims, torch.from_numpy(W).cuda(), 0.1)
            out = np.empty_like(v)
            msc.msc_op_apply(c, op, 0.2, v, out, msc.MSC_FP64)
            want = oracle.staggered_apply(W, dims, nc, 0.1, v, sigma=0.2)
            ok = np.isfinite(want)
            assert not ok.all() and ok.any()
            assert np.array_equal(np.isfinite(out), ok)
            assert np.linalg.norm(out[ok] - want[ok]) <= 1e-13 * np.linalg.norm(want[ok])
            for prec in (msc.MSC_FP64, msc.MSC_MIXED):
                with pytest.raises(msc.MscError) as e:
                    msc.solve(c, op, torch.from_numpy(v).cuda(), [0.1, 0.5], tol=1e-10, precision=prec)
                assert e.value.code == msc.MSC_ERR_NONFINITE
            msc.msc_op_destroy(op)
    msc.msc_destroy(c)
