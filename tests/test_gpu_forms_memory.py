"""The forms of A beside the CSR, CSC and tiled ones are held only while a chosen
variant reads them: not by a handle that pins nothing, not the ones that lost the
set-up's choice; pinning a variant brings its form back, with the same result."""
import numpy as np
import pytest

from paper_1601_08201_gb300 import sgtv, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

SP, TUNE = sgtv.FLAG_SINGLE_PASS, sgtv.FLAG_NO_AUTOTUNE


def held(h):
    return sgtv.info(h.h)["device_bytes"]


def scatter(h, name):
    h.set_variant(sgtv.K_SCATTER, h.variant_names()["k_scatter"].index(name))


def pair(h):
    n = h.variant_names()
    h.set_variants(n["k_forward"].index("stack_v4"), n["k_back_update"].index("stack_v4"))


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp64"])
def test_single_pass_holds_the_form_in_use(precision):
    P = synth.preset("wide_64x16x32")
    V = {"fp32": 4, "bf16": 2, "fp64": 8}[precision]
    with sgtv.Handle(P, precision=precision, flags=SP | TUNE) as h:
        bare = held(h)
        scatter(h, "sp_v4x2_atomic_min4")
        stream = held(h) - bare
        assert stream >= P.nnz * (V + 2)
    stacked = None
    if precision != "fp64":
        with sgtv.Handle(P, precision=precision, flags=SP | TUNE) as h:
            assert held(h) == bare
            scatter(h, "stack")
            stacked = held(h) - bare
            assert stacked >= P.nnz * V
    with sgtv.Handle(P, precision=precision, flags=SP) as h:
        chosen = h.variant_names()["k_scatter"][h.get_variant(sgtv.K_SCATTER)]
        form = stream if chosen.startswith("sp_") else (stacked if chosen == "stack" else 0)
        assert held(h) == bare + form


def test_two_passes_hold_the_form_in_use():
    P = synth.preset("wide_64x16x32")
    with sgtv.Handle(P, flags=TUNE) as h:
        bare = held(h)
        pair(h)
        stacked = held(h) - bare
        assert stacked >= 4 * P.nnz
        h.set_variants(0, 0)
        h.iterate(2)
        ref = h.get_state_f64()
    with sgtv.Handle(P) as h:
        name = h.variant_names()["k_forward"][h.get_variants()[0]]
        assert held(h) == bare + (stacked if name == "stack_v4" else 0)
    with sgtv.Handle(P, flags=TUNE) as h:  # entered, left, tuned (the iterate under way), entered again
        pair(h)
        h.iterate(1)
        h.autotune()
        pair(h)
        assert held(h) == bare + stacked
        h.iterate(1)
        assert np.linalg.norm(h.get_state_f64()[0] - ref[0]) <= 1e-5 * np.linalg.norm(ref[0])


def test_a_refused_pin_builds_nothing():
    P = synth.preset("wide_64x16x32")
    with sgtv.Handle(P, flags=SP | TUNE) as h:  # its products serve the KKT measure only
        bare = held(h)
        with pytest.raises(sgtv.SgtvError):
            pair(h)
        assert held(h) == bare
    with sgtv.Handle(P, flags=TUNE) as h:
        bare = held(h)
        with pytest.raises(sgtv.SgtvError):
            scatter(h, "stack")
        with pytest.raises(sgtv.SgtvError):
            h.set_variants(h.variant_names()["k_forward"].index("stack_v4"), 0)
        assert held(h) == bare


@pytest.mark.parametrize("flags", [0, sgtv.FLAG_GRAPH])
def test_a_form_given_back_and_pinned_again_gives_the_same(flags):
    P = synth.preset("ragged_13x7x37")
    out = []
    for tuned in (False, True):
        with sgtv.Handle(P, flags=flags | TUNE) as h:
            pair(h)
            h.iterate(9)
            if tuned:
                h.autotune()
                pair(h)
            h.iterate(9)
            out.append(h.get_state_f64())
    for a, b in zip(*out):
        assert np.array_equal(a, b)
