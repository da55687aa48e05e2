"""Register budgets of the kernels chosen for few tiles and small steps (nvcc -Xptxas -v, no GPU needed): the
four-candidate blend forward two 256-thread CTAs per SM (<= 128 registers), the binning cluster's CTA of 1024
threads (<= 64), the passes over 8-byte words and the large steps' scan two 512-thread CTAs (<= 64); none
spills."""
import pytest

from test_register_budgets import ptxas_report

BUDGETS = {"k_blend.cu": [("k_blend_forward_few", 128)],
           "k_sort.cu": [("k_bin_small", 64), ("k_sort_pass_words", 64), ("k_scan", 64)]}


@pytest.mark.parametrize("src", sorted(BUDGETS))
def test_budgets(src, tmp_path):
    rep = ptxas_report(src, tmp_path)
    for frag, most in BUDGETS[src]:
        hits = {k: v for k, v in rep.items() if frag in k and "regs" in v}
        assert hits, frag
        for name, v in hits.items():
            assert v["regs"] <= most and v.get("spill", 0) == 0, (name, v)
