"""Which kernel runs a filter, and that it makes no difference: the staged steps, the resident filter and the block
kernel for several weight tables against the launch shapes (autotune = 0), bit for bit, each asserted to have run.
The matrices are larger than the resident filter takes unless they test that line."""
import numpy as np
import pytest
import scipy.sparse as sp

import paper_2402_08515_gb300 as K
from fe_inputs import Problem, box_grid, flared_tube, square_grid, start_vectors

pytestmark = pytest.mark.gpu


def _from_csr(name, S, m):
    S = sp.csr_matrix(S)
    S.sort_indices()
    return Problem(name, S.shape[0], S.indptr.astype(np.int64), S.indices.astype(np.int32), S.data.copy(), m)


def _gaps():
    """A box of 45 thousand rows with every seventh coupling pair dropped (uneven rows) and some diagonals missing."""
    p = box_grid((47, 33, 32))
    S = p.to_scipy().tocoo()
    lo, hi = np.minimum(S.row, S.col), np.maximum(S.row, S.col)
    keep = ((lo * 7919 + hi) % 7 != 0) & ~((S.row == S.col) & (S.row % 41 == 3))
    return _from_csr("gaps", sp.csr_matrix((S.data[keep] + 0.01, (S.row[keep], S.col[keep])), shape=S.shape), p.m)


def _lattice(n, reach):
    """A line of n rows coupled to the `reach` next ones on each side: 2 reach + 1 entries a row."""
    I = np.repeat(np.arange(n), reach)
    J = I + np.tile(np.arange(1, reach + 1), n)
    I, J = I[J < n], J[J < n]
    w = 0.5 + np.random.default_rng(4).random(len(I))
    S = sp.csr_matrix((np.r_[-w, -w], (np.r_[I, J], np.r_[J, I])), shape=(n, n))
    return _from_csr("lattice", S + sp.diags(0.01 - np.asarray(S.sum(axis=1)).ravel()),
                     1.0 + np.random.default_rng(5).random(n))


MATRICES = {
    "box": lambda: box_grid((43, 31, 29)),
    "plane": lambda: box_grid((260, 40, 5)),
    "tube": lambda: flared_tube(0.013),                      # lines of every length: stored places
    "batch": lambda: [square_grid(100), box_grid((37, 29, 23)), flared_tube(0.02)],
    "gaps": _gaps,                                           # no folded diagonal
}


def _apply(c, n, b, F, L, tau, columns=False):
    nm = K.kes_mesh_count(c.handle)
    lo = [5.0 + 3 * f for f in range(F)]
    K.kes_set_filters_batch(c.handle, [lo] * nm, [[a + 2.0 for a in lo]] * nm, [tau] * nm, L)
    R = start_vectors(n, b, 11)
    out = np.zeros((b, n) if columns else (F, b, n))
    (K.kes_filter_apply_columns if columns else K.kes_filter_apply)(c.handle, R, out, b)
    assert np.isfinite(out).all()
    return out, K.kes_filter_kernel(c.handle)


def _both(p, b, F, L, columns=False, tau=0.004, **opts):
    n = sum(q.n for q in p) if isinstance(p, list) else p.n
    res = []
    for autotune in (True, False):
        with K.Context(p, block_b=b, autotune=autotune, **opts) as c:
            assert K.kes_filter_kernel(c.handle) == K.KES_KERNEL_NONE
            res.append(_apply(c, n, b, F, L, tau, columns))
    (got, kernel), (ref, plain) = res
    assert plain == K.KES_KERNEL_SHAPES
    np.testing.assert_array_equal(got, ref)
    return kernel


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("b,F,L", [(1, 1, 7), (1, 4, 5), (1, 8, 3), (2, 1, 1), (2, 3, 8), (3, 2, 6), (4, 4, 7), (8, 1, 9)])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_staged_filter_equals_the_launch_shapes(name, b, F, L, precision):
    assert _both(MATRICES[name](), b, F, L, precision=precision) == K.KES_KERNEL_STAGED


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("opts", [dict(stepper="leapfrog4"), dict(sell_sigma=256), dict(use_graph=False)])
@pytest.mark.parametrize("b", [1, 2, 4])
def test_staged_filter_equals_the_launch_shapes_with_options(opts, b, precision):
    kernel = _both(MATRICES["batch"](), b, 1, 8, precision=precision, **opts)
    assert kernel == K.KES_KERNEL_STAGED or "sell_sigma" in opts


@pytest.mark.parametrize("b,F", [(2, 2), (6, 3), (8, 4)])
def test_staged_columns_equal_the_launch_shapes(b, F):
    assert _both(MATRICES["tube"](), b, F, 10, columns=True, precision="fp32") == K.KES_KERNEL_STAGED


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("b", [5, 8])
def test_eight_columns_with_several_tables(b, use_graph):
    """Eight FP32 columns leave the staged steps for several tables, in one context that goes from one table to
    several and back with another time step each time."""
    p = box_grid((53, 43, 39))
    got, ref = [], []
    for out, autotune in ((got, True), (ref, False)):
        with K.Context(p, block_b=b, precision="fp32", autotune=autotune, use_graph=use_graph) as c:
            for F, tau in ((1, 0.004), (4, 0.003), (2, 0.0045), (1, 0.0035)):
                out.append(_apply(c, p.n, b, F, 8, tau))
    for (a, ka), (r, _), F in zip(got, ref, (1, 4, 2, 1)):
        np.testing.assert_array_equal(a, r)
        assert ka == (K.KES_KERNEL_STAGED if F == 1 else K.KES_KERNEL_SHAPES)


# stored entries a block: a matrix of s slices with w entries a row has ceil(s / 16) * 32 w
@pytest.mark.parametrize("precision,b,F,n,reach,kernel", [
    ("fp64", 1, 1, 32 * 16 * 14, 7, "RESIDENT"),             # 6,720 entries (the limit is 7,000),
    ("fp64", 1, 1, 32 * 16 * 15, 7, "STAGED"),               # 7,200
    ("fp64", 1, 4, 32 * 16 * 14, 7, "RESIDENT"),
    ("fp64", 8, 2, 32 * 16 * 14, 7, "RESIDENT"),
    ("fp32", 1, 1, 32 * 16 * 50 - 7, 7, "RESIDENT"),         # 24,000
    ("fp32", 1, 1, 32 * 16 * 51, 7, "STAGED"),               # 24,480
    ("fp32", 4, 4, 32 * 16 * 50, 7, "RESIDENT"),
    ("fp32", 8, 1, 32 * 16 * 14, 7, "RESIDENT"),
    ("fp32", 8, 1, 32 * 16 * 15, 7, "STAGED"),
])
def test_the_lines_between_the_kernels(precision, b, F, n, reach, kernel):
    p = _lattice(n, reach)
    assert _both(p, b, F, 6, precision=precision, tau=0.3) == getattr(K, f"KES_KERNEL_{kernel}")


@pytest.mark.parametrize("precision,b,opts", [("fp64", 1, {}), ("fp32", 8, {}), ("fp32", 2, dict(use_graph=False)),
                                              ("fp64", 4, dict(stepper="leapfrog4"))])
def test_a_wait_that_runs_out_is_an_error_and_the_context_stays_usable(precision, b, opts):
    """With a limit of no polls every wait of the staged steps gives up: the copies under way still land, the call says
    KES_ERR_TIMEOUT, and with the default limit the same context filters as if nothing had been."""
    p = box_grid((43, 31, 29))
    R = start_vectors(p.n, b, 11)
    with K.Context(p, precision=precision, block_b=b, **opts) as c:
        ref, kernel = _apply(c, p.n, b, 1, 8, 0.004)
        assert kernel == K.KES_KERNEL_STAGED
        K.kes_set_wait_limit(c.handle, 0)
        with pytest.raises(K.KesError) as e:
            K.kes_filter_apply(c.handle, R, np.zeros((1, b, p.n)), b)
        assert e.value.status == -6
        with pytest.raises(K.KesError) as e:
            K.kes_set_wait_limit(c.handle, -2)
        assert e.value.status == -1
        K.kes_set_wait_limit(c.handle, -1)
        out = np.zeros((1, b, p.n))
        K.kes_filter_apply(c.handle, R, out, b)
        np.testing.assert_array_equal(out, ref)
