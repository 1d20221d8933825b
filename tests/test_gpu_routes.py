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
    # sorted rows gather from all over their window: too few of them fit the FP64 stages of several columns
    scattered = "sell_sigma" in opts and precision == "fp64" and b > 1
    assert kernel == (K.KES_KERNEL_SHAPES if scattered else K.KES_KERNEL_STAGED)


@pytest.mark.parametrize("b,F", [(2, 2), (6, 3), (8, 4)])
def test_staged_columns_equal_the_launch_shapes(b, F):
    assert _both(MATRICES["tube"](), b, F, 10, columns=True, precision="fp32") == K.KES_KERNEL_STAGED


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("cells,kernel", [((43, 31, 29), "STAGED"), ((53, 43, 39), "SHAPES")])
@pytest.mark.parametrize("b", [5, 8])
def test_eight_columns_with_several_tables(b, cells, kernel, use_graph):
    """Eight FP32 columns leave the staged steps for several tables from 56 thousand rows on (83 thousand here), in
    one context that goes from one table to several and back with another time step each time."""
    p = box_grid(cells)
    got, ref = [], []
    for out, autotune in ((got, True), (ref, False)):
        with K.Context(p, block_b=b, precision="fp32", autotune=autotune, use_graph=use_graph) as c:
            for F, tau in ((1, 0.004), (4, 0.003), (2, 0.0045), (1, 0.0035)):
                out.append(_apply(c, p.n, b, F, 8, tau))
    want = {1: K.KES_KERNEL_STAGED, 2: getattr(K, f"KES_KERNEL_{kernel}"), 4: getattr(K, f"KES_KERNEL_{kernel}")}
    for (a, ka), (r, _), F in zip(got, ref, (1, 4, 2, 1)):
        np.testing.assert_array_equal(a, r)
        assert ka == want[F]


# stored entries a block: a matrix of s slices with w entries a row has ceil(s / 16) * 32 w
@pytest.mark.parametrize("precision,b,F,n,reach,kernel", [
    ("fp64", 1, 1, 32 * 16 * 14, 7, "RESIDENT"),             # 6,720 entries (the limit is 7,000),
    ("fp64", 1, 1, 32 * 16 * 15, 7, "STAGED"),               # 7,200
    ("fp64", 1, 4, 32 * 16 * 14, 7, "RESIDENT"),             # 6,720 and 448 rows for each further table,
    ("fp64", 1, 8, 32 * 16 * 40, 2, "STAGED"),               # 6,400 and 1,280 for each of seven
    ("fp64", 8, 2, 32 * 16 * 14, 7, "RESIDENT"),
    ("fp32", 1, 1, 32 * 16 * 50 - 7, 7, "RESIDENT"),         # 24,000
    ("fp32", 1, 1, 32 * 16 * 51, 7, "STAGED"),               # 24,480
    ("fp32", 4, 4, 32 * 16 * 50, 7, "RESIDENT"),
    ("fp32", 8, 1, 32 * 16 * 14, 7, "RESIDENT"),
    ("fp32", 8, 2, 32 * 16 * 15, 7, "STAGED"),
    # five entries a row: from 20,480 rows on the alternative is a launch shape
    ("fp32", 1, 1, 32 * 16 * 78, 2, "RESIDENT"),             # 12,480 entries and 2,496 rows,
    ("fp32", 1, 8, 32 * 16 * 78, 2, "SHAPES"),               # with seven further tables,
    ("fp32", 8, 1, 32 * 16 * 42, 2, "SHAPES"),               # 6,720 and 1,344 in eight columns
    ("fp32", 2, 1, 32 * 2500, 2, "SHAPES"),
    ("fp32", 1, 1, 32 * 8191, 2, "SHAPES"),                  # one column up to 262,144 rows
    ("fp32", 1, 1, 32 * 8192, 2, "STAGED"),
    ("fp32", 1, 1, 32 * 8192, 1, "SHAPES"),                  # but not with three entries
    ("fp64", 1, 1, 32 * 2500, 2, "STAGED"),
])
def test_the_lines_between_the_kernels(precision, b, F, n, reach, kernel):
    p = _lattice(n, reach)
    assert _both(p, b, F, 6, precision=precision, tau=0.3) == getattr(K, f"KES_KERNEL_{kernel}")


@pytest.mark.parametrize("slices,kernel", [(1300, "STAGED"), (1800, "SHAPES")])
def test_columns_of_narrow_rows(slices, kernel):
    """With a table each, columns of narrow rows stay staged to 57 thousand rows; in one context with a filter that does
    not, with another time step."""
    p = _lattice(32 * slices, 2)
    got, ref = [], []
    for out, autotune in ((got, True), (ref, False)):
        with K.Context(p, block_b=8, precision="fp32", autotune=autotune) as c:
            for F, tau, columns in ((2, 0.3, True), (1, 0.25, False), (2, 0.35, True)):
                out.append(_apply(c, p.n, 8, F, 6, tau, columns))
    for (a, ka), (r, _), columns in zip(got, ref, (True, False, True)):
        np.testing.assert_array_equal(a, r)
        assert ka == (getattr(K, f"KES_KERNEL_{kernel}") if columns else K.KES_KERNEL_SHAPES)


@pytest.mark.parametrize("precision,b,kernel", [("fp64", 1, "SHAPES"), ("fp64", 2, "SHAPES"), ("fp32", 4, "SHAPES"),
                                                ("fp32", 1, "STAGED")])
def test_wide_rows_are_staged_where_enough_of_them_fit(precision, b, kernel):
    """125 entries a row, all over a box of 46^3 nodes: few rows fit a stage."""
    m = 46
    at = np.arange(m ** 3).reshape(m, m, m)
    I, J = [], []
    for dz in range(-2, 3):
        for dy in range(-2, 3):
            for dx in range(-2, 3):
                sl = [slice(max(0, -d), m - max(0, d)) for d in (dz, dy, dx)]
                to = [slice(max(0, d), m - max(0, -d)) for d in (dz, dy, dx)]
                I.append(at[tuple(sl)].ravel())
                J.append(at[tuple(to)].ravel())
    I, J = np.concatenate(I), np.concatenate(J)
    S = sp.csr_matrix((np.where(I == J, 125.0, -1.0), (I, J)), shape=(m ** 3, m ** 3))
    p = _from_csr("wide", S, 1.0 + np.random.default_rng(6).random(m ** 3))
    assert _both(p, b, 1, 4, precision=precision, tau=0.05) == getattr(K, f"KES_KERNEL_{kernel}")


@pytest.mark.parametrize("precision,b,opts", [("fp64", 1, {}), ("fp32", 8, {}), ("fp32", 1, dict(use_graph=False)),
                                              ("fp64", 4, dict(stepper="leapfrog4"))])
def test_a_wait_that_runs_out_is_an_error_and_the_context_stays_usable(precision, b, opts):
    """The copying warps give up once the ring is full: the copies under way still land, the computing warps' waits run
    out (1.5 seconds), the call says KES_ERR_TIMEOUT, and afterwards the same context filters as if nothing had been."""
    p = box_grid((73, 65, 64))                                   # 290 thousand rows: more tiles a block than stages
    R = start_vectors(p.n, b, 11)
    with K.Context(p, precision=precision, block_b=b, **opts) as c:
        ref, kernel = _apply(c, p.n, b, 1, 1, 0.004)
        assert kernel == K.KES_KERNEL_STAGED
        K.kes_fail_waits(c.handle, True)
        with pytest.raises(K.KesError) as e:
            K.kes_filter_apply(c.handle, R, np.zeros((1, b, p.n)), b)
        assert e.value.status == -6
        with pytest.raises(K.KesError) as e:
            K.kes_fail_waits(c.handle, 2)
        assert e.value.status == -1
        K.kes_fail_waits(c.handle, False)
        out = np.zeros((1, b, p.n))
        K.kes_filter_apply(c.handle, R, out, b)
        np.testing.assert_array_equal(out, ref)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kernel", ["RESIDENT", "STAGED", "SHAPES"])
@pytest.mark.parametrize("b", [1, 3])
def test_a_value_that_is_not_finite_stays_in_its_mesh_and_column(b, kernel, precision):
    """An infinite start value is reported, and the other meshes' and the other columns' results are the bits that they
    are without it (the staged steps hold zeros for couplings that a row lacks, but none out of its mesh)."""
    p = [square_grid(20), box_grid((9, 8, 7))] if kernel == "RESIDENT" else MATRICES["batch"]()
    n, n0 = sum(q.n for q in p), p[0].n
    with K.Context(p, block_b=b, precision=precision, autotune=kernel != "SHAPES") as c:
        ref, ran = _apply(c, n, b, 1, 6, 0.004)
        assert ran == getattr(K, f"KES_KERNEL_{kernel}")
        R, out = start_vectors(n, b, 11), np.zeros((1, b, n))
        R[b - 1, n0 - 1] = np.inf                                # the last row of the first mesh
        with pytest.raises(K.KesError) as e:
            K.kes_filter_apply(c.handle, R, out, b)
        assert e.value.status == -3
        assert not np.isfinite(out[0, b - 1, :n0]).all()
        np.testing.assert_array_equal(out[..., n0:], ref[..., n0:])
        np.testing.assert_array_equal(out[:, :b - 1], ref[:, :b - 1])
