"""The staged step kernels against the register-staged ones, bit for bit, over the matrices and options they take:
both form every row and column as one FMA chain in entry order (a zero entry adds nothing to a finite sum)."""
import numpy as np
import pytest

import paper_2402_08515_gb300 as K
from fe_inputs import Problem, box_grid, flared_tube, square_grid, start_vectors

pytestmark = pytest.mark.gpu


def _gap_rows():
    """A box with every seventh coupling pair dropped (uneven rows) and diagonals missing from some rows."""
    p = box_grid((19, 17, 13))
    S = p.to_scipy().tocoo()
    lo, hi = np.minimum(S.row, S.col), np.maximum(S.row, S.col)
    keep = ((lo * 7919 + hi) % 7 != 0) & ~((S.row == S.col) & (S.row % 41 == 3))
    S.data = S.data + 0.01
    import scipy.sparse as sp
    S = sp.csr_matrix((S.data[keep], (S.row[keep], S.col[keep])), shape=S.shape)
    S.sort_indices()
    return Problem("gaps", p.n, S.indptr.astype(np.int64), S.indices.astype(np.int32), S.data.copy(), p.m.copy())


MATRICES = {
    "one_tile": lambda: square_grid(5),                          # 16 rows
    "square": lambda: square_grid(64),                           # ragged last tile, 7 entries a row
    "ragged_box": lambda: box_grid((37, 29, 23)),                # lines shorter than a slice's 32 rows and longer
    "plane": lambda: box_grid((130, 40, 4)),                     # lines longer than half a tile
    "tube": lambda: flared_tube(0.02),                           # lines of every length: stored places
    "batch": lambda: [square_grid(40), box_grid((23, 19, 17)), flared_tube(0.03, length=1.0, r0=0.06, growth=1.2)],
    "gaps": _gap_rows,                                           # rows without a diagonal, uneven rows
}


def _filter(problem, autotune, L, b, F=1, columns=False, **opts):
    n = sum(p.n for p in problem) if isinstance(problem, list) else problem.n
    R = start_vectors(n, b, 11)
    with K.Context(problem, block_b=b, autotune=autotune, **opts) as c:
        nm = K.kes_mesh_count(c.handle)
        lo = [5.0 + 3 * f for f in range(F)]
        K.kes_set_filters_batch(c.handle, [lo] * nm, [[a + 2.0 for a in lo]] * nm, [0.004] * nm, L)
        staged = K.kes_get_stats(c.handle)["step_variant"] == -1
        if columns:
            out = np.zeros((b, n))
            K.kes_filter_apply_columns(c.handle, R, out, b)
        else:
            out = np.zeros((F, b, n))
            K.kes_filter_apply(c.handle, R, out, b)
    assert np.isfinite(out).all()
    return out, staged


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("b,F,L", [(1, 1, 1), (1, 3, 7), (2, 1, 8), (3, 2, 6), (8, 1, 9)])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_staged_filter_equals_the_launch_shapes(name, b, F, L, precision):
    p = MATRICES[name]()
    got, staged = _filter(p, True, L, b, F, precision=precision)
    ref, plain = _filter(p, False, L, b, F, precision=precision)
    assert staged and not plain
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("b", [1, 4])
@pytest.mark.parametrize("opts", [dict(stepper="leapfrog4"), dict(sell_sigma=256), dict(use_graph=False)])
def test_staged_filter_equals_the_launch_shapes_with_options(opts, b, precision):
    p = MATRICES["batch"]()
    got, _ = _filter(p, True, 10, b, precision=precision, **opts)
    ref, _ = _filter(p, False, 10, b, precision=precision, **opts)
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("b,F", [(2, 2), (6, 3), (8, 4)])
def test_staged_columns_equal_the_launch_shapes(b, F, precision):
    p = MATRICES["tube"]()
    got, staged = _filter(p, True, 10, b, F, columns=True, precision=precision)
    ref, _ = _filter(p, False, 10, b, F, columns=True, precision=precision)
    assert staged
    np.testing.assert_array_equal(got, ref)


def test_scattered_columns_are_not_staged():
    """A tile of 32 rows already gathers from all over the matrix (22,176 rows): the launch shapes take it."""
    p = box_grid((37, 29, 23))
    perm = np.random.default_rng(3).permutation(p.n)
    S = p.to_scipy()[perm][:, perm].tocsr()
    S.sort_indices()
    q = Problem("scattered", p.n, S.indptr.astype(np.int64), S.indices.astype(np.int32), S.data.copy(), p.m[perm])
    got, staged = _filter(q, True, 12, 1)
    ref, _ = _filter(q, False, 12, 1)
    assert not staged
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("b,F,L", [(1, 1, 1), (1, 4, 5), (3, 2, 6), (8, 1, 9)])
@pytest.mark.parametrize("cells", [(3, 2), (17, 33), (60, 70), (11, 12, 13), (24, 21, 24)])
def test_resident_filter_equals_the_launch_shapes(cells, b, F, L, precision):
    """Small matrices run a filter in one kernel (one slice up to the largest that FP64 and eight columns take): same bits."""
    p = box_grid(cells, extent=tuple(c / 16.0 for c in cells))
    got, _ = _filter(p, True, L, b, F, precision=precision)
    ref, _ = _filter(p, False, L, b, F, precision=precision)
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_resident_columns_and_meshes_equal_the_launch_shapes(precision):
    p = [square_grid(20), box_grid((9, 8, 7)), flared_tube(0.05, length=1.0, r0=0.1, growth=1.0)]
    got, _ = _filter(p, True, 12, 6, 3, columns=True, precision=precision)
    ref, _ = _filter(p, False, 12, 6, 3, columns=True, precision=precision)
    np.testing.assert_array_equal(got, ref)
