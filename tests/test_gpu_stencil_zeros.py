"""FP64 stencil passes on sources with exact zeros: sums without a term are 0."""
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


def unit_links(dims, nc):
    U = np.zeros((4, inputs.volume(dims), nc, nc), complex)
    U[...] = np.eye(nc)
    return U


# below and above 24,576 sites: four lanes and one lane per site
@pytest.mark.parametrize("dims", [(4, 6, 8, 4), (16, 16, 12, 10)])
@pytest.mark.parametrize("nc", [2, 3])
def test_sums_without_a_term_are_exactly_zero(ctx, nc, dims):
    """Zeros of both signs everywhere but at one site, which holds one colour:
    on unit links every other colour of D x is exactly 0, at the sites whose
    first direction has only zeros among them."""
    V = inputs.volume(dims)
    g = inputs.rng(600)
    x = (np.where(g.random(V * nc) < 0.5, -0.0, 0.0) + 1j * np.where(g.random(V * nc) < 0.5, -0.0, 0.0)).reshape(V, nc)
    x[V // 2 + 1, 0] = 0.7 - 0.4j
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(unit_links(dims, nc)).cuda(), 0.1)
    out = np.empty(V * nc, complex)
    msc.msc_op_dslash(ctx, op, x.reshape(-1), out)
    want = oracle.dslash(unit_links(dims, nc), dims, nc, x.reshape(-1))
    assert np.count_nonzero(want) == 8
    assert np.array_equal(out, want)
    msc.msc_op_destroy(op)


@pytest.mark.parametrize("dims", [(4, 6, 8, 4), (16, 16, 12, 10)])
@pytest.mark.parametrize("nc", [2, 3])
def test_real_fields_stay_real(ctx, nc, dims):
    """The same on links that are summed in fixed point (real orthogonal ones
    without a zero): no imaginary part has a term, so every one is exactly 0."""
    V = inputs.volume(dims)
    g = inputs.rng(610)
    q = np.linalg.qr(g.standard_normal((nc, nc)))[0]
    U = np.zeros((4, V, nc, nc), complex)
    U[...] = q
    assert np.abs(q).min() > 1e-3
    x = (np.where(g.random(V * nc) < 0.5, -0.0, 0.0) + 1j * np.where(g.random(V * nc) < 0.5, -0.0, 0.0)).reshape(V, nc)
    x[V // 2 + 1, 0] = 0.7
    op = msc.msc_op_staggered(ctx, nc, dims, torch.from_numpy(U).cuda(), 0.1)
    out = np.empty(V * nc, complex)
    msc.msc_op_dslash(ctx, op, x.reshape(-1), out)
    msc.msc_op_destroy(op)
    want = oracle.dslash(U, dims, nc, x.reshape(-1))
    assert np.count_nonzero(want.imag) == 0 and np.count_nonzero(out.imag) == 0
    assert np.array_equal(out != 0, want != 0) and np.max(np.abs(out - want)) <= 1e-15
