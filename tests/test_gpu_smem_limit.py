"""Tiles whose dynamic shared memory comes to exactly the 48 KB that a block has
without asking: with the kernel's own barriers it is more. Windows of that size for
three and four pipeline stages, for one staged tile and for the scatter's two
buffers, in rows and in columns; and one element less and more.

Tolerances are those of tests/test_gpu_parity.py (FP32 1e-5, FP64 1e-11)."""
import numpy as np
import pytest
import scipy.sparse as sparse

import oracle as O
from paper_1601_08201_gb300 import sgtv, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def problem(w, by_rows):
    """64 columns (or rows) of 8 nonzeros that span w rows (columns)."""
    rng = np.random.default_rng(w)
    seg = np.concatenate([np.sort(np.r_[0, w - 1, 1 + rng.choice(w - 2, 6, replace=False)]) for _ in range(64)])
    val = rng.uniform(0.1, 1.0, 512).astype(np.float32)
    A = sparse.csr_matrix((val, seg, np.arange(0, 513, 8)), shape=(64, w))
    A = A if by_rows else A.T.tocsr()
    A.sort_indices()
    C = A.tocsc()
    C.sort_indices()
    I, J = A.shape
    y = rng.poisson(3.0, I).astype(np.float32)
    return synth.Problem(Nx=1, Nz=J, Nq=1, I=I, J=J, nnz=512, csc_colptr=C.indptr.astype(np.int64),
                         csc_row=C.indices.astype(np.int32), csc_val=C.data, csr_rowptr=A.indptr.astype(np.int64),
                         csr_col=A.indices.astype(np.int32), csr_val=A.data, y=y, b=np.array([0.3], np.float32),
                         beta=0.1, rho=1.0, f_true=None, seed=0)


def check(h, ref, s0, tol, what):
    h.set_state_f64(*s0)
    h.iterate(2)
    f = h.get_state_f64()[0]
    assert np.linalg.norm(f - ref) <= tol * np.linalg.norm(ref), what


@pytest.mark.parametrize("by_rows", [False, True])
@pytest.mark.parametrize("precision,widths", [("fp32", (3100, 2076, 12287, 12288, 12289)),
                                              ("bf16", (3350, 2330, 12288)), ("fp64", (1290, 780, 6143, 6144, 6145))])
def test_every_tiled_form_runs(precision, widths, by_rows):
    for w in widths:
        P = problem(w, by_rows)
        kw = dict(csr_val=synth.round_to_bf16(P.csr_val), csc_val=synth.round_to_bf16(P.csc_val)) if precision == "bf16" else {}
        op = O.from_problem(P, **kw)
        ref = O.iterate(op, O.init_state(op), 2)[0]
        with sgtv.Handle(P, precision=precision) as h:  # the timing of every form
            s0 = None
            names = h.variant_names()
            kernel, name = (sgtv.K_FORWARD, "k_forward") if by_rows else (sgtv.K_BACK_UPDATE, "k_back_update")
            ran = 0
            for v, n in enumerate(names[name]):
                try:
                    h.set_variant(kernel, v)
                except sgtv.SgtvError:
                    continue
                s0 = h.get_state_f64() if s0 is None else s0
                check(h, ref, s0, 1e-11 if precision == "fp64" else 1e-5, (w, n))
                ran += 1
            assert ran >= 8


@pytest.mark.parametrize("precision,w", [("fp32", 6143), ("fp32", 6144), ("fp32", 6145), ("fp64", 3072)])
def test_every_scatter_form_runs(precision, w):
    P = problem(w, True)
    op = O.from_problem(P)
    ref = O.iterate(op, O.init_state(op), 2)[0]
    with sgtv.Handle(P, precision=precision, flags=sgtv.FLAG_SINGLE_PASS) as h:
        s0 = h.get_state_f64()
        for v, n in enumerate(h.variant_names()["k_scatter"]):
            try:
                h.set_variant(sgtv.K_SCATTER, v)
            except sgtv.SgtvError:
                continue
            check(h, ref, s0, 1e-11 if precision == "fp64" else 1e-5, n)
