"""sgtv_set_variant one product at a time on handles that run the stacked pair:
every form that fits can be pinned from it, and the pair entered from any form;
saved choices come back in either order."""
import numpy as np
import pytest

import oracle as O
from paper_1601_08201_gb300 import sgtv, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

KERNELS = ((sgtv.K_FORWARD, "k_forward"), (sgtv.K_BACK_UPDATE, "k_back_update"))


def stacked(h):
    names = h.variant_names()
    pair = tuple(names[n].index("stack_v4") for _, n in KERNELS)
    h.set_variants(*pair)
    return names, pair


@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("which", [0, 1])
def test_every_fitting_form_is_reached_from_the_pair_alone(which, tuned):
    P = synth.preset("ragged_13x7x37")
    op = O.from_problem(P)
    ref = O.iterate(op, O.init_state(op), 3)[0]
    kernel, name = KERNELS[which]
    with sgtv.Handle(P, flags=0 if tuned else sgtv.FLAG_NO_AUTOTUNE) as h:
        names, pair = stacked(h)
        f0, d0, c0 = h.get_state_f64()
        for v in range(len(names[name])):
            h.set_variants(*pair)
            h.set_variant(kernel, v)  # this scan's tiled forms all fit
            got = h.get_variants()
            assert got[which] == v
            assert (got == pair) if v == pair[which] else (pair[1 - which] != got[1 - which])
            h.set_state_f64(f0, d0, c0)
            h.iterate(3)
            f = h.get_state_f64()[0]
            assert np.linalg.norm(f - ref) <= 1e-5 * np.linalg.norm(ref), names[name][v]
            h.set_variant(KERNELS[1 - which][0], pair[1 - which])  # and back, by the other product
            assert h.get_variants() == pair


@pytest.mark.parametrize("order", [(0, 1), (1, 0)])
def test_saved_choices_come_back(order):
    P = synth.preset("ragged_13x7x37")
    with sgtv.Handle(P, flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        names, pair = stacked(h)
        for saved in (pair, (1, 2), pair, (0, 0)):
            for k in order:
                h.set_variant(KERNELS[k][0], saved[k])
            assert h.get_variants() == saved


def test_what_does_not_fit_stays_refused():
    rng = np.random.default_rng(0)
    # FP64 vectors have no stacked pair; out of range
    P = synth.preset("ragged_13x7x37")
    with sgtv.Handle(P, precision="fp64", flags=sgtv.FLAG_NO_AUTOTUNE) as h:
        for kernel, name in KERNELS:
            n = len(h.variant_names()[name])
            for v in (-1, n, int(rng.integers(n, 1000))):
                with pytest.raises(sgtv.SgtvError):
                    h.set_variant(kernel, v)
        assert h.get_variants() == (0, 0)
    # the persistent launch fuses two tiled forms only
    with sgtv.Handle(P, flags=sgtv.FLAG_PERSISTENT | sgtv.FLAG_NO_AUTOTUNE) as h:
        before = h.get_variants()
        for kernel, name in KERNELS:
            with pytest.raises(sgtv.SgtvError):
                h.set_variant(kernel, h.variant_names()[name].index("stack_v4"))
        assert h.get_variants() == before
