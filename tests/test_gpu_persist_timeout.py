"""The grid barrier of the cooperative iterations (csrc/persist.cu) is bounded
in time. With MSC_TEST_ABSENT=1 it waits for one arrival more than there are
blocks, so that every wait runs out (after MSC_WAIT_NS): the solve returns
MSC_ERR_TIMEOUT, the launches already queued behind the first do not wait again
(a mixed solve queues four), and a new context solves normally afterwards."""
import os
import time

import numpy as np
import pytest

from paper_1102_2143_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1102_2143_gb300 as msc  # noqa: E402

LIMIT = 0.25  # seconds


def _ctx(env):
    old = {k: os.environ.get(k) for k in env}
    os.environ.update(env)
    try:
        return msc.msc_create(0, torch.cuda.current_stream())
    finally:
        for k, v in old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v


def _solve(p, prec, env):
    c = _ctx(env)
    op = msc.msc_op_staggered(c, p.nc, p.dims, torch.from_numpy(p.links).cuda(), p.mass)
    b = torch.from_numpy(p.b).cuda()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    try:
        x, info = msc.solve(c, op, b, p.sigma, tol=p.tol, precision=prec)
        return x, info, None, time.perf_counter() - t0
    except msc.MscError as e:
        return None, None, e.code, time.perf_counter() - t0
    finally:
        msc.msc_op_destroy(op)
        msc.msc_destroy(c)


@pytest.mark.parametrize("prec", [msc.MSC_FP64, msc.MSC_MIXED])
def test_barrier_wait_that_runs_out_reports_timeout_once(prec):
    msc.load()
    p = inputs.staggered_problem((8, 8, 8, 8), 3, 0.2, 0.6, [0.01, 0.1], 1, 1e-10, 7410)
    _solve(p, prec, {})  # loads the kernels
    x, info, code, dt = _solve(p, prec, {"MSC_TEST_ABSENT": "1", "MSC_WAIT_NS": str(int(LIMIT * 1e9))})
    assert code == msc.MSC_ERR_TIMEOUT
    assert LIMIT <= dt < 2 * LIMIT
    x, info, code, _ = _solve(p, prec, {})
    assert code is None and info.status == 0 and np.all(info.true_rel_resid <= p.tol)
