"""The two forms of the row GEMMs (tokens or weights on the M side): the rule that chooses, and the weights-on-M form
at the edges of its units in shapes for which it is chosen."""
import pytest

from test_gpu_kernel_edges import test_expert_ffn_at_the_edges_of_its_units as check_units

pytestmark = pytest.mark.gpu

PHASES = ("expert_fwd_gu", "expert_fwd_down", "dgrad_down", "dgrad_gu")


def on_weights(d, f, experts, k, T, sizes_known=True, pool=None):
    from paper_2605_06665_b200 import binding as B
    ctx = B.Context(B.make_config(d, f, pool or experts, k, 1, T, B.BF16, 1e-6, 2.0))
    names = [ctx.gemm_kernel(p, experts, sizes_known) for p in PHASES]
    assert ctx.gemm_kernel("wgrad_gu", experts) == "wgrad_pair_kernel" and ctx.gemm_kernel("combine", experts) == ""
    ctx.close()
    assert set(names) <= {"wm_kernel", "row_pair_kernel", "grouped_gemm_tc_kernel"}
    return "".join("W" if n == "wm_kernel" else "T" for n in names)


@pytest.mark.parametrize("sizes,d,f,forms,forms_padded", [
    # one chunk of <= 192 tokens at gate/up on average, up to three in the largest groups
    ([0, 1, 15, 16, 17, 31, 33, 191, 192, 193, 255, 256, 257, 383, 384, 385], 1024, 4864, "WWWW", "WWWW"),
    ([301, 383, 384, 385, 193, 192, 290] * 2, 768, 3008, "WTWT", "WTWT"),  # two chunks; a partial weight tile
    ([383, 384, 385, 401, 512, 450, 397], 1280, 3840, "WWWW", "WWWW"),     # two MMAs, three chunks
    ([48, 1, 0, 33, 64, 65, 17] * 3, 768, 1600, "TWWW", "TTTT"),           # few rows; an odd number of k-blocks
])
@pytest.mark.parametrize("with_rows", [True, False])
def test_weights_on_m_where_it_is_chosen(sizes, d, f, forms, forms_padded, with_rows):
    n = len(sizes)
    assert on_weights(d, f, n, 1, sum(sizes), with_rows, pool=n + 2) == (forms if with_rows else forms_padded)
    check_units(sizes, d, f, with_rows)


@pytest.mark.parametrize("shape,forms", [
    ((768, 2048, 96, 2, 16384), "WWWW"), ((768, 2048, 96, 2, 1501), "TWWW"), ((768, 2048, 96, 2, 33), "TWWW"),
    ((1536, 4096, 192, 2, 32768), "WWWW"),
    ((768, 512, 384, 8, 16384), "WTWT"),               # narrow experts
    ((768, 320, 300, 6, 8000), "TTWT"),                # ... and a half-empty last weight tile
    ((768, 2048, 96, 2, 11000), "WWWW"),               # 229 rows: two half-empty chunks at gate/up, in many deals
    ((768, 2048, 29, 2, 464), "TTWT"),                 # few rows, and units for 1.2 rounds
    ((384, 768, 24, 2, 4000), "TTTT"),
    ((768, 2048, 40, 2, 16384), "TTWT"), ((768, 2048, 8, 2, 16384), "TTTT"),
    ((768, 2048, 480, 2, 8192), "TTTT"),               # more experts than the unit list holds
])
def test_the_form_follows_what_was_measured_faster(shape, forms):
    assert on_weights(*shape) == forms
