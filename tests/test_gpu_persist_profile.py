"""A context created with MSC_PERSIST=0 runs the per-pass kernels on small
staggered systems too and reports their times; the solutions are those of the
cooperative iterations to 1e-8 (both meet the tolerance in FP64)."""
import os

import numpy as np
import pytest

from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("prec", [msc.MSC_FP64, msc.MSC_MIXED])
def test_small_solve_is_profiled(monkeypatch, prec, nrhs):
    p = inputs.staggered_problem((8, 4, 6, 8), 3, 0.1, 0.7, inputs.log_shifts(1e-3, 2.0, 5), nrhs, 1e-10, 7420)
    xs = []
    for on in ("1", "0"):
        monkeypatch.setenv("MSC_PERSIST", on)
        c = msc.msc_create(0, torch.cuda.current_stream())
        op = msc.msc_op_staggered(c, p.nc, p.dims, torch.from_numpy(p.links).cuda(), p.mass)
        x, info = msc.solve(c, op, torch.from_numpy(p.b).cuda(), p.sigma, tol=p.tol, precision=prec)
        assert info.status == 0 and np.all(info.true_rel_resid <= p.tol)
        if on == "0":
            assert info.prof_samples > 0 and info.prof_active > 0
            assert min(info.op_ms, info.rupdate_ms, info.update_ms) > 0
        else:
            assert info.prof_samples == 0
        xs.append(x.cpu().numpy())
        msc.msc_op_destroy(op)
        msc.msc_destroy(c)
    assert np.linalg.norm(xs[0] - xs[1]) <= 1e-8 * np.linalg.norm(xs[1])
