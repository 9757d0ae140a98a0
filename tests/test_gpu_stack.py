"""The stacked row form (variants "stack" of the single-pass scatter and
"stack_v4" of the two-pass products) against the FP64 oracle, at the sizes where
it can go wrong: columns of a tile at a word's edge, up to the most it takes
and past it, odd row counts, empty rows, rows as long as the tile, backgrounds
per measurement, images with few q-bins (the per-voxel f-update), batches whose
scans end inside a tile, and every option of the iteration.

Tolerances are the FP32 mode's: relative L2 1e-5 and, element by element with a
floor of 1e-2 of the largest, 1e-3 (tests/test_gpu_parity.py)."""
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


def problem(shape, I, lengths, seed=0, cols=None, per_row_b=False):
    """A scan with row i holding lengths[i % len(lengths)] nonzeros among the first `cols` hyper-voxels."""
    rng = np.random.default_rng(seed)
    J = int(np.prod(shape))
    cols = J if cols is None else cols
    rows, idx = [], []
    for i in range(I):
        k = min(lengths[i % len(lengths)], cols)
        idx.append(np.sort(rng.choice(cols, k, replace=False)))
        rows.append(np.full(k, i))
    rows, idx = np.concatenate(rows), np.concatenate(idx)
    val = rng.uniform(0.1, 1.0, rows.size).astype(np.float32)
    A = sparse.csr_matrix((val, (rows, idx)), shape=(I, J))
    A.sort_indices()
    C = A.tocsc()
    C.sort_indices()
    f = rng.uniform(0.0, 2.0, J) * (rng.random(J) < 0.7)
    b = rng.uniform(0.2, 0.6, I).astype(np.float32) if per_row_b else np.array([0.3], np.float32)
    y = rng.poisson(A @ f + b).astype(np.float32)
    return synth.Problem(Nx=shape[0], Nz=shape[1], Nq=shape[2], I=I, J=J, nnz=A.nnz,
                         csc_colptr=C.indptr.astype(np.int64), csc_row=C.indices.astype(np.int32),
                         csc_val=C.data.astype(np.float32), csr_rowptr=A.indptr.astype(np.int64),
                         csr_col=A.indices.astype(np.int32), csr_val=A.data.astype(np.float32), y=y, b=b, beta=0.4,
                         rho=2.0, f_true=f.astype(np.float32), seed=seed)


def close(a, b, what):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    n = np.linalg.norm(b)
    assert np.linalg.norm(a - b) <= 1e-5 * (n if n > 0 else 1.0), (what, np.linalg.norm(a - b), n)
    m = np.abs(b).max()
    if m > 0:
        assert (np.abs(a - b) / np.maximum(np.abs(b), 1e-2 * m)).max() <= 1e-3, what


def pick(h, flags):
    names = h.variant_names()
    if flags & SP:
        h.set_variant(sgtv.K_SCATTER, names["k_scatter"].index("stack"))
    else:
        h.set_variants(names["k_forward"].index("stack_v4"), names["k_back_update"].index("stack_v4"))


def oracle_of(P, precision="fp32", **kw):
    if precision == "bf16":
        kw.update(csr_val=synth.round_to_bf16(P.csr_val), csc_val=synth.round_to_bf16(P.csc_val))
    return O.from_problem(P, **kw)


@pytest.mark.parametrize("flags", [SP, 0])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("shape,I,lengths,cols", [
    ((4, 4, 8), 70, [20], 128),            # 4 words full
    ((3, 43, 1), 71, [129, 3], 129),       # one column past 4 words; one q-bin; odd rows
    ((5, 8, 8), 200, [0, 320, 1, 0, 77], 320),   # 10 words full (the last of the 32-bit records), empty rows
    ((7, 3, 16), 131, [321, 2], 321),      # one past it
    ((6, 8, 16), 257, [768, 5, 0, 300], 768),    # the most columns of a tile, rows of that length
    ((2, 8, 48), 1, [400], 640),           # a single row
    ((9, 5, 17), 3000, [3, 40, 11, 64, 9], None),  # many short rows, nothing aligned
])
def test_edges_match_oracle(flags, precision, shape, I, lengths, cols):
    P = problem(shape, I, lengths, seed=I, cols=cols, per_row_b=bool(I % 2))
    op = oracle_of(P, precision)
    st = O.iterate(op, O.init_state(op), 6)
    with sgtv.Handle(P, precision=precision, flags=flags | TUNE) as h:
        pick(h, flags)
        h.iterate(6)
        for a, b, what in zip(h.get_state_f64(), st, "fdc"):
            close(a, b, what)
        # the accumulator and the partial sums are as the next step needs them
        h.residuals()
        h.objective()
        h.iterate(1)
        close(h.get_state_f64()[0], O.iterate(op, st, 1)[0], "f after the measures")


def test_refused_where_it_does_not_apply():
    # 769 columns in every tile of 8 rows; FP64 vectors; a pair with one stacked product
    wide = problem((7, 11, 10), 24, [769], cols=769)
    with sgtv.Handle(wide, flags=SP | TUNE) as h:
        with pytest.raises(sgtv.SgtvError):
            pick(h, SP)
        h.iterate(2)  # not sticky
        h.sync()
    P = problem((5, 8, 8), 100, [40])
    with sgtv.Handle(P, precision="fp64", flags=TUNE) as h:
        assert "stack_v4" not in h.variant_names()["k_forward"]
    with sgtv.Handle(P, flags=TUNE) as h:
        v = h.variant_names()["k_forward"].index("stack_v4")
        with pytest.raises(sgtv.SgtvError):
            h.set_variants(v, 0)
        with pytest.raises(sgtv.SgtvError):
            h.set_variants(0, h.variant_names()["k_back_update"].index("stack_v4"))
        h.iterate(1)
        h.sync()


@pytest.mark.parametrize("flags", [SP, SP | sgtv.FLAG_GRAPH, 0, sgtv.FLAG_GRAPH, sgtv.FLAG_STANDARD_TV])
def test_options_and_switching_forms(flags):
    # two directions with weights, two surrogate steps; the stacked form chosen, left and chosen again
    P = problem((9, 6, 20), 301, [50, 90, 7], per_row_b=True)
    kw = dict(n_dirs=2, w=[0.7, 1.4])
    op = O.from_problem(P, per_bin=True, **kw) if flags & sgtv.FLAG_STANDARD_TV else O.from_problem(P, **kw)
    st = O.iterate(op, O.init_state(op), 27, 2)
    with sgtv.Handle(P, n_inner=2, flags=flags | TUNE, **kw) as h:
        for n, stacked in ((10, True), (7, False), (10, True)):
            if stacked:
                pick(h, flags)
            elif flags & SP:
                h.set_variant(sgtv.K_SCATTER, 0)
            else:
                h.set_variants(1, 1)
            h.iterate(n)
        for a, b, what in zip(h.get_state_f64(), st, "fdc"):
            close(a, b, what)


def test_two_pass_is_deterministic_and_survives_new_states():
    P = problem((9, 6, 20), 301, [50, 90, 7])
    out = []
    for _ in range(2):
        with sgtv.Handle(P, flags=TUNE) as h:
            pick(h, 0)
            h.iterate(9)
            s = h.get_state_f64()
            h.set_state_f64(*s)
            h.iterate(3)
            h.set_data(P.y, P.b, P.beta)
            h.iterate(3)
            h.warm_start(s[0].astype(np.float32), 0.5)
            h.iterate(3)
            out.append(h.get_state_f64())
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    with sgtv.Handle(P, flags=TUNE) as h:  # the same calls in the plain form
        h.iterate(9)
        h.warm_start(h.get_state_f64()[0].astype(np.float32), 0.5)
        h.iterate(3)
        close(out[0][0], h.get_state_f64()[0], "f")


@pytest.mark.parametrize("flags", [SP, 0])
def test_batch_with_scans_ending_inside_a_tile(flags):
    scans = [dataclasses.replace(problem(sh, I, ln, seed=I), rho=r)
             for sh, I, ln, r in [((5, 4, 7), 90, [12, 30], 0.5), ((8, 3, 16), 33, [20], 1.0),
                                  ((4, 4, 32), 201, [24, 0, 60], 3.0)]]
    with sgtv.Handle(scans, flags=flags | TUNE) as h:
        pick(h, flags)
        h.iterate(12)
        f, off = h.get_state_f64()[0], h.batch_info()["vox_off"]
    for k, P in enumerate(scans):
        op = O.from_problem(P)
        close(f[off[k]:off[k + 1]], O.iterate(op, O.init_state(op), 12)[0], k)


def test_no_penalty_is_mlem():
    P = problem((6, 5, 16), 120, [30, 0, 64])
    op = O.from_problem(P, rho=0.0)
    st = O.iterate(op, O.init_state(op), 4)
    for flags in (SP, 0):
        with sgtv.Handle(P, rho=0.0, flags=flags | TUNE | sgtv.FLAG_ALLOW_RHO0) as h:
            pick(h, flags)
            h.iterate(4)
            close(h.get_state_f64()[0], st[0], flags)
