"""The benchmark's byte count of the stacked row form is what the form holds: the
levels of its stacks, the records (64 bits from 11 words on), the copies' control
words, the tiles' columns and, in two passes, the partial sums and their places."""
import pytest

import bench
from paper_1601_08201_gb300 import sgtv, synth


@pytest.mark.parametrize("precision,V", [("fp32", 4), ("bf16", 2)])
@pytest.mark.parametrize("words,rec", [(10, 4), (12, 8), (20, 8)])
def test_bytes_of_the_stacked_form(precision, V, words, rec):
    P = synth.preset("ragged_13x7x37")  # an odd number of rows
    I, J, pairs = P.I, P.J, (P.I + 1) // 2
    st = dict(words=words, tile_rows=64, tiles=47, levels=9000, partials=12345)
    tli = {"csr": {"list_entries": 0}, "csc": {"list_entries": 0}, "stack": st}
    a = 32 * V * 9000 + pairs * (32 * rec + 4) + 8 * 48 + 4 * 32 * 47 * words
    one = bench.algorithmic_bytes(P, precision, {"k_scatter": "stack"}, tli)
    assert one["k_scatter"] == a + 4 * (2 * J + I) + 4 * P.b.size
    two = bench.algorithmic_bytes(P, precision, {"k_forward": "stack_v4", "k_back_update": "stack_v4"}, tli)
    assert two["k_forward"] == a + 4 * 32 * 47 * words + 4 * 12345 + 4 * (J + 2 * I) + 4 * P.b.size
    assert two["k_back_update"] == 4 * 12345 + 4 * (J + 1) + 4 * 7 * J
    assert one["k_shrink"] == two["k_shrink"] == 4 * J * 17
    rows = bench.batch_bytes_by_kernel([P], precision, "single_pass", tli, {"k_scatter": "stack"})["k_scatter"]
    assert rows == a + 4 * (2 * J + 2 * I)


@pytest.mark.gpu
@pytest.mark.parametrize("flags", [sgtv.FLAG_SINGLE_PASS, 0])
def test_the_handle_says_what_it_holds(flags):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():  # pragma: no cover
        pytest.skip("needs a CUDA GPU")
    P = synth.preset("ragged_13x7x37")
    with sgtv.Handle(P, flags=flags | sgtv.FLAG_NO_AUTOTUNE) as h:
        assert not any(h.stack_info().values())
        n = h.variant_names()
        if flags:
            h.set_variant(sgtv.K_SCATTER, n["k_scatter"].index("stack"))
        else:
            h.set_variants(n["k_forward"].index("stack_v4"), n["k_back_update"].index("stack_v4"))
        s = h.stack_info()
        held = sgtv.info(h.h)["device_bytes"]
    assert s["tiles"] == -(-P.I // s["tile_rows"]) and 4 <= s["words"] <= 24 and s["levels"] * 32 >= P.nnz
    assert (P.J <= s["partials"] <= s["tiles"] * s["words"] * 32) if not flags else s["partials"] == 0
    assert held >= bench.stacked_bytes(P.nnz, P.I, 4, s)
