"""The FP64 products with eight lanes per segment against the oracle, at the
edges of a warp (4 segments), a block (8) and a lane group's loads (64 nonzeros):
scans of one voxel, of one bin, batches whose scans end inside a block.

Tolerance: both sides form every sum in FP64 with relative errors of some 1e-15
per product (up to some hundred terms), over 12 iterations that contract or
keep such errors: 1e-11, the bound the FP64 form is held to elsewhere."""
import numpy as np
import pytest

import oracle as O
from paper_1601_08201_gb300 import sgtv, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def scan(shape, I, nnz_col, seed=0):
    return synth.make_problem(*shape, I, nnz_col, n_regions=2, mean_counts=5.0, seed=seed)


def lanes8(problem, **kw):
    h = sgtv.Handle(problem, precision="fp64", flags=sgtv.FLAG_NO_AUTOTUNE, **kw)
    names = h.variant_names()
    h.set_variants(names["k_forward"].index("lanes8"), names["k_back_update"].index("lanes8"))
    return h


def rel(a, b):
    return np.linalg.norm(a - b) / max(1e-300, np.linalg.norm(b))


# (3, 5, 31) with 700 rows: rows of less than a nonzero per lane, some empty; with 15: rows of several rounds
@pytest.mark.parametrize("n_dirs,w", [(2, [0.7, 1.4]), (4, [0.5, 1.3, 2.0, 0.7])])
@pytest.mark.parametrize("shape,I,nnz_col", [((1, 1, 1), 4, 1), ((1, 7, 1), 9, 3), ((3, 5, 31), 15, 5),
                                             ((3, 5, 31), 24, 8), ((3, 5, 31), 700, 3), ((13, 7, 37), 3001, 50),
                                             ((8, 6, 16), 193, 63), ((8, 6, 16), 200, 65)])
def test_one_scan(shape, I, nnz_col, n_dirs, w):
    P = scan(shape, I, nnz_col)
    op = O.from_problem(P, n_dirs=n_dirs, w=w)
    ref = O.iterate(op, O.init_state(op), 12)
    with lanes8(P, n_dirs=n_dirs, w=w) as h:
        h.iterate(12)
        f = h.get_state_f64()[0]
    assert rel(f, ref[0]) <= 1e-11


def test_batch_of_scans_that_end_inside_a_block():
    scans = [scan(s, I, k, seed=n) for n, (s, I, k) in
             enumerate([((3, 5, 31), 30, 9), ((1, 3, 5), 11, 4), ((8, 6, 16), 190, 40)])]
    with lanes8(scans) as h:
        h.iterate(12)
        f = h.get_state_f64()[0]
        off = h.batch_info()["vox_off"]
    for k, P in enumerate(scans):
        op = O.from_problem(P)
        ref = O.iterate(op, O.init_state(op), 12)
        assert rel(f[off[k]:off[k + 1]], ref[0]) <= 1e-11, k
