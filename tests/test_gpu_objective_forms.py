"""The deviance's tiled form at the edges of its tiles (64 rows), warps' row pairs,
row chunks (128 nonzeros) and ranges, on scans of more rows than the plain form
takes (16 a multiprocessor), and both forms at the row counts where the choice
changes, against the FP64 oracle at the GPU's own iterate.

Tolerance: as tests/test_gpu_objective.py, 1e-12 (FP64 terms and sums of some
thousand nonnegative ones)."""
import numpy as np
import pytest

import oracle as O
from paper_1601_08201_gb300 import sgtv, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

SMS = torch.cuda.get_device_properties(0).multi_processor_count
MANY = 16 * SMS  # plain up to MANY rows, tiled from more on


def scan(I, lengths, shape=(8, 6, 16), seed=0):
    """Rows of lengths[i % len] nonzeros; every seventh count 0."""
    rng = np.random.default_rng(seed)
    J = int(np.prod(shape))
    n = np.minimum(np.array([lengths[i % len(lengths)] for i in range(I)]), J)
    rowptr = np.zeros(I + 1, np.int64)
    np.cumsum(n, out=rowptr[1:])
    col = np.concatenate([np.sort(rng.choice(J, k, replace=False)) for k in n]).astype(np.int32)
    val = rng.uniform(0.1, 1.0, col.size).astype(np.float32)
    rows = np.repeat(np.arange(I), n)
    order = np.argsort(col, kind="stable")
    colptr = np.zeros(J + 1, np.int64)
    np.cumsum(np.bincount(col, minlength=J), out=colptr[1:])
    y = rng.poisson(3.0, I).astype(np.float32)
    y[::7] = 0.0
    return synth.Problem(Nx=shape[0], Nz=shape[1], Nq=shape[2], I=I, J=J, nnz=col.size, csc_colptr=colptr,
                         csc_row=rows[order].astype(np.int32), csc_val=val[order], csr_rowptr=rowptr, csr_col=col,
                         csr_val=val, y=y, b=np.array([0.3], np.float32), beta=0.1, rho=1.0, f_true=None, seed=seed)


def oracle_of(P, precision):
    if precision == "bf16":
        return O.from_problem(P, csr_val=synth.round_to_bf16(P.csr_val), csc_val=synth.round_to_bf16(P.csc_val))
    return O.from_problem(P)


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp64"])
@pytest.mark.parametrize("I,lengths", [(MANY - 1, [20, 3]), (MANY, [1, 64]), (MANY, [300, 260]),
                                       (MANY + 1, [300, 257]), (MANY + 1, [129, 127, 128, 0, 1, 31, 33]),
                                       (MANY + 64, [5]), (MANY + 127, [257, 0, 0, 2]), (2 * MANY + 7, [32, 9])])
def test_objective_at_the_lines_between_the_forms(precision, I, lengths):
    P = scan(I, lengths)
    with sgtv.Handle(P, precision=precision, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        h.iterate(2)
        f = h.get_state_f64()[0]
        phi, dev, _ = h.objective()
    ophi, odev, _ = O.objective(oracle_of(P, precision), f)
    assert dev == pytest.approx(odev, rel=1e-12)
    assert phi == pytest.approx(ophi, rel=1e-12)


@pytest.mark.parametrize("rows,mean", [(MANY + 5, 40), (8 * MANY + 3, 3), (MANY + 5, 600)])
def test_plain_form_takes_several_rows_in_turn(rows, mean):
    # windows too wide for the tiled form: rows spread over 6000 columns
    P = scan(rows, [mean, mean - 1, 0, mean + 2], shape=(20, 10, 30))
    with sgtv.Handle(P, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        assert h.tli_info()["csr"]["max_stage"] > 3968
        h.iterate(1)
        f = h.get_state_f64()[0]
        dev = h.objective()[1]
    assert dev == pytest.approx(O.objective(oracle_of(P, "fp32"), f)[1], rel=1e-12)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_scans_of_many_rows_that_end_inside_a_tile(precision):
    scans = [scan(I, ln, seed=k) for k, (I, ln) in enumerate([(MANY + 30, [9, 4]), (MANY + 5, [20]), (70, [16, 0])])]
    with sgtv.Handle(scans, precision=precision, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        h.iterate(2)
        f = h.get_state_f64()[0]
        off = h.batch_info()["vox_off"]
        each = [h.objective_scan(k) for k in range(len(scans))]
        total = h.objective()
    for k, P in enumerate(scans):
        ref = O.objective(O.from_problem(P), np.ascontiguousarray(f[off[k]:off[k + 1]]))
        assert each[k] == pytest.approx(ref, rel=1e-12), k
    assert total[1] == pytest.approx(sum(e[1] for e in each), rel=1e-12)


# images whose products with A leave FP32's range (some rows, or all), or are subnormal, and ordinary ones
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("scale", [1e-44, 1e-38, 1e-22, 1.0, 1e28, 1e36])
@pytest.mark.parametrize("mixed", [False, True])
def test_tiled_deviance_of_images_at_the_ends_of_fp32(scale, mixed, precision):
    P = scan(MANY + 75, [90, 140, 7])
    rng = np.random.default_rng(3)
    f = (rng.uniform(0.5, 2.0, P.J) * scale).astype(np.float32)
    if mixed:
        f[::2] = rng.uniform(0.5, 2.0, f[::2].size)
    f = f.astype(np.float64)
    with sgtv.Handle(P, precision=precision, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        h.set_state_f64(f)
        dev = h.objective()[1]
    assert dev == pytest.approx(O.objective(oracle_of(P, precision), f)[1], rel=1e-12)
