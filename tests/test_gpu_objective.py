"""The deviance reduction's tiled and plain forms against the FP64 oracle at
the GPU's own iterate, at the edges of its tiles (64 rows), its row chunks (256
nonzeros) and its ranges (scans of a batch that end inside a tile).

Tolerance: each side forms every ybar and term in FP64 with relative errors of
a few 1e-16 times the row length's square root, and sums at most some thousand
nonnegative terms: 1e-12 relative is two orders above both."""
import numpy as np
import pytest

import oracle as O
from paper_1601_08201_gb300 import sgtv, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def scan(I, nnz_col, shape=(8, 6, 16), seed=0):
    P = synth.make_problem(*shape, I, nnz_col, n_regions=2, mean_counts=3.0, seed=seed)
    P.y[::7] = 0.0  # terms without a logarithm
    return P


def oracle_of(P, precision):
    if precision == "bf16":
        return O.from_problem(P, csr_val=synth.round_to_bf16(P.csr_val), csc_val=synth.round_to_bf16(P.csc_val))
    return O.from_problem(P)


# rows of about nnz_col * 768 / I nonzeros: 256 and more, short ones, none at all in part of the rows;
# tiles of 64 rows and one row more or less; (20, 1, 200): windows too wide for the FP64 staging
@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp64"])
@pytest.mark.parametrize("I,nnz_col,shape", [(63, 24, (8, 6, 16)), (64, 22, (8, 6, 16)), (65, 20, (8, 6, 16)),
                                             (129, 43, (8, 6, 16)), (700, 3, (8, 6, 16)), (2000, 1, (8, 6, 16)),
                                             (200, 70, (20, 1, 200))])
def test_objective_at_tile_and_row_edges(precision, I, nnz_col, shape):
    P = scan(I, nnz_col, shape)
    op = oracle_of(P, precision)
    with sgtv.Handle(P, precision=precision, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        h.iterate(2)
        f = h.get_state_f64()[0]
        phi, dev, tv = h.objective()
    ophi, odev, otv = O.objective(op, f)
    assert dev == pytest.approx(odev, rel=1e-12)
    assert phi == pytest.approx(ophi, rel=1e-12)


def test_objective_of_scans_that_end_inside_a_tile():
    scans = [scan(I, nc, seed=k) for k, (I, nc) in enumerate([(30, 9), (100, 20), (64, 16), (7, 2), (190, 40)])]
    with sgtv.Handle(scans, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        h.iterate(2)
        f = h.get_state_f64()[0]
        off = h.batch_info()["vox_off"]
        each = [h.objective_scan(k) for k in range(len(scans))]
        total = h.objective()
    for k, P in enumerate(scans):
        ref = O.objective(O.from_problem(P), np.ascontiguousarray(f[off[k]:off[k + 1]]))
        assert each[k] == pytest.approx(ref, rel=1e-12), k
    assert total[1] == pytest.approx(sum(e[1] for e in each), rel=1e-12)


# sites of one bin, of a warp's 32 less and more one, with edges on every side; fewer and more sites than
# a block's warps. The TV terms are FP64 sums of one differenced value each: the same 1e-12.
@pytest.mark.parametrize("per_bin", [False, True])
@pytest.mark.parametrize("n_dirs,w", [(2, [0.7, 1.4]), (4, [0.5, 1.3, 2.0, 0.7])])
@pytest.mark.parametrize("shape", [(1, 3, 1), (3, 5, 31), (9, 7, 33), (40, 33, 65)])
def test_tv_terms_at_site_and_bin_edges(shape, n_dirs, w, per_bin):
    J = shape[0] * shape[1] * shape[2]
    P = scan(max(4, J // 3), 3, shape)
    op = O.from_problem(P, n_dirs=n_dirs, w=w, per_bin=per_bin)
    flags = sgtv.FLAG_NO_AUTOTUNE | (sgtv.FLAG_STANDARD_TV if per_bin else 0)
    with sgtv.Handle(P, n_dirs=n_dirs, w=w, flags=flags) as h:
        h.iterate(3)
        f, d, c = h.get_state_f64()
        tv = h.objective()[2]
        primal = h.residuals()[0]
    assert tv == pytest.approx(O.objective(op, f)[2], rel=1e-12)
    assert primal == pytest.approx(O.residuals(op, f, d, c)[0], rel=1e-12)


# one window that is the image: 3913 columns still staged as FP64, 4004 not
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("Nq", [43, 44])
def test_objective_at_the_staging_limit(Nq, precision):
    P = scan(2000, 40, (13, 7, Nq))
    with sgtv.Handle(P, precision=precision, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        h.iterate(2)
        f = h.get_state_f64()[0]
        dev = h.objective()[1]
    assert dev == pytest.approx(O.objective(oracle_of(P, precision), f)[1], rel=1e-12)


# images whose products with A leave FP32's range (some rows, or all), or are subnormal, and ordinary ones;
# odd numbers of rows per warp and rows of more than 128 nonzeros
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("scale", [1e-44, 1e-38, 1e-22, 1.0, 1e28, 1e36])
@pytest.mark.parametrize("mixed", [False, True])
def test_deviance_of_images_at_the_ends_of_fp32(scale, mixed, precision):
    P = scan(331, 90, (8, 6, 16))
    rng = np.random.default_rng(3)
    f = (rng.uniform(0.5, 2.0, P.J) * scale).astype(np.float32)
    if mixed:
        f[::2] = rng.uniform(0.5, 2.0, f[::2].size)
    f = f.astype(np.float64)
    with sgtv.Handle(P, precision=precision, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        h.set_state_f64(f)
        dev = h.objective()[1]
    assert dev == pytest.approx(O.objective(oracle_of(P, precision), f)[1], rel=1e-12)
