"""Rows of the stacked form whose ratio y / (A f + r) is infinite or NaN: they
reach the columns that they hold a nonzero in and no other, as a product over the
nonzeros alone does. Counts on rows without nonzeros and no background, images
that are zero along a row, and images past FP32's range, in tiles that hold
ordinary rows too; in a batch, tiles that hold rows of two scans.

Reference: the FP64 oracle on all columns outside the rows in question. Tolerances
are the FP32 mode's: relative L2 1e-5 and, element by element with a floor of
1e-2 of the largest, 1e-3 (tests/test_gpu_parity.py)."""
import dataclasses

import numpy as np
import pytest
import scipy.sparse as sparse

import oracle as O
from paper_1601_08201_gb300 import sgtv, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

SP, TUNE = sgtv.FLAG_SINGLE_PASS, sgtv.FLAG_NO_AUTOTUNE
FORMS = pytest.mark.parametrize("flags", [SP, 0])
PRECISIONS = pytest.mark.parametrize("precision", ["fp32", "bf16"])
# (3, 4, 8): 32-bit records; (5, 8, 12): 64-bit ones; odd row counts, several tiles
SHAPES = pytest.mark.parametrize("shape,I", [((3, 4, 8), 71), ((5, 8, 12), 203)])


def problem(shape, I, seed, b=0.3, empty=()):
    """Rows of 5 to 40 nonzeros, those of `empty` without any; rho small, so that the update's B stays positive."""
    rng = np.random.default_rng(seed)
    J = int(np.prod(shape))
    per_row = [np.sort(rng.choice(J, 0 if i in empty else rng.integers(5, 41), replace=False)) for i in range(I)]
    idx = np.concatenate(per_row)
    rows = np.repeat(np.arange(I), [len(p) for p in per_row])
    A = sparse.csr_matrix((rng.uniform(0.1, 1.0, rows.size).astype(np.float32), (rows, idx)), shape=(I, J))
    A.sort_indices()
    C = A.tocsc()
    C.sort_indices()
    f = rng.uniform(0.5, 2.0, J)
    y = rng.poisson(A @ f + b).astype(np.float32)
    y[list(empty)] = 0.0
    return synth.Problem(Nx=shape[0], Nz=shape[1], Nq=shape[2], I=I, J=J, nnz=A.nnz,
                         csc_colptr=C.indptr.astype(np.int64), csc_row=C.indices.astype(np.int32),
                         csc_val=C.data.astype(np.float32), csr_rowptr=A.indptr.astype(np.int64),
                         csr_col=A.indices.astype(np.int32), csr_val=A.data.astype(np.float32), y=y,
                         b=np.array([b], np.float32), beta=0.01, rho=0.01, f_true=f.astype(np.float32), seed=seed)


def oracle_of(P, precision, **kw):
    if precision == "bf16":
        kw.update(csr_val=synth.round_to_bf16(P.csr_val), csc_val=synth.round_to_bf16(P.csc_val))
    return O.from_problem(P, **kw)


def stacked(problem, flags, precision, **kw):
    h = sgtv.Handle(problem, flags=flags | TUNE, precision=precision, **kw)
    names = h.variant_names()
    if flags & SP:
        h.set_variant(sgtv.K_SCATTER, names["k_scatter"].index("stack"))
    else:
        h.set_variants(names["k_forward"].index("stack_v4"), names["k_back_update"].index("stack_v4"))
    return h


def row(P, i):
    return P.csr_col[P.csr_rowptr[i]:P.csr_rowptr[i + 1]]


def close(a, b):
    assert np.isfinite(a).all() and np.isfinite(b).all()
    assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)
    assert (np.abs(a - b) / np.maximum(np.abs(b), 1e-2 * np.abs(b).max())).max() <= 1e-3


@FORMS
@PRECISIONS
@SHAPES
def test_counts_on_empty_rows_without_background(flags, precision, shape, I):
    empty = (0, 9, 40, 63, I - 1)
    P = problem(shape, I, seed=I, b=0.0, empty=empty)
    Q = dataclasses.replace(P, y=P.y.copy())
    Q.y[list(empty)] = 3.0
    op = oracle_of(Q, precision)
    with stacked(P, flags, precision) as h:
        h.set_data(Q.y, Q.b, Q.beta)
        h.iterate(5)
        f = h.get_state_f64()[0]
    close(f, O.iterate(op, O.init_state(op), 5)[0])


@FORMS
@PRECISIONS
@SHAPES
def test_images_that_are_zero_along_rows(flags, precision, shape, I):
    # one row of a pair, both rows of a pair, the last row; the image is otherwise positive
    P = problem(shape, I, seed=I + 1, b=0.0)
    zero = np.unique(np.concatenate([row(P, i) for i in (3, 36, 37, I - 1)]))
    for i in (3, 36, 37, I - 1):
        P.y[i] = 4.0
    start = np.random.default_rng(1).uniform(0.5, 2.0, P.J)
    start[zero] = 0.0
    op = oracle_of(P, precision)
    st = O.init_state(op)
    s = start.astype(np.float32).astype(np.float64)
    d = O.wgrad(op, s)
    ref = O.iterate(op, (s, d, np.zeros_like(d)), 1)[0]
    rest = np.setdiff1d(np.arange(P.J), zero)
    assert rest.size > P.J // 4 and len(st) == 3
    with stacked(P, flags, precision) as h:
        h.set_state_f64(start)
        h.iterate(1)
        f = h.get_state_f64()[0]
    close(f[rest], ref[rest])
    assert (f[zero] == 0.0).all()


@FORMS
@PRECISIONS
def test_a_scan_leaves_its_neighbours_in_a_batch_alone(flags, precision):
    scans = [problem((3, 4, 8), 33, seed=5, b=0.0), problem((5, 3, 7), 45, seed=6), problem((3, 4, 8), 31, seed=7)]
    zero = row(scans[0], 32)  # the last row of the first scan shares its tile with the second
    scans[0].y[32] = 4.0
    ops = [oracle_of(P, precision) for P in scans]
    starts = [np.ones(P.J) for P in scans]
    starts[0][zero] = 0.0
    with stacked(scans, flags, precision) as h:
        off = h.batch_info()["vox_off"]
        h.set_state_f64(np.concatenate(starts))
        h.iterate(1)
        f = h.get_state_f64()[0]
    for k, (P, op) in enumerate(zip(scans, ops)):
        d = O.wgrad(op, starts[k])
        ref = O.iterate(op, (starts[k], d, np.zeros_like(d)), 1)[0]
        rest = np.setdiff1d(np.arange(P.J), zero) if k == 0 else np.arange(P.J)
        close(f[off[k]:off[k + 1]][rest], ref[rest])


@FORMS
@PRECISIONS
@SHAPES
def test_an_image_value_past_fp32_reaches_its_rows_only(flags, precision, shape, I):
    # one MLEM step: the rows that hold column 11 have an infinite forecast, so a ratio of 0
    P = problem(shape, I, seed=I + 2)
    start = np.random.default_rng(2).uniform(0.5, 2.0, P.J).astype(np.float32).astype(np.float64)
    start[11] = 1e39
    op = oracle_of(P, precision, rho=0.0)
    d = O.wgrad(op, start)
    ref = O.iterate(op, (start, d, np.zeros_like(d)), 1)[0]
    rest = np.setdiff1d(np.arange(P.J), [11])
    with stacked(P, flags | sgtv.FLAG_ALLOW_RHO0, precision, rho=0.0) as h:
        h.set_state_f64(start)
        h.iterate(1)
        f = h.get_state_f64()[0]
    close(f[rest], ref[rest])
