"""What plan creation falls back to, read from its source (no GPU): a failure of the CUDA driver cannot be had
on demand."""
import os
import re

CAPI = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_14780_gb300", "csrc",
                    "ptycho_capi.cu")


def test_no_plan_is_refused_for_want_of_a_tensor_map():
    """Without the driver's tensor-map encoder (an older driver) plans run the one-field passes with plain
    loads; the pair passes, which need a map, are no reason to refuse the plan."""
    text = re.sub(r"//[^\n]*", "", open(CAPI).read())
    failed = text[text.index("!make_pair_map("):]
    code = re.search(r"return (\w+);", failed).group(1)
    assert not code.startswith("PTYCHO_")
    create = re.search(r"int create_plan\([^)]*\) \{(.*?)\n\}", text, re.S).group(1)
    assert re.search(r"rc == %s \? make_plan\([^)]*false[^)]*\)" % code, create)
    pick = re.search(r"if \(([^{]*)\{[^{}]*PairSizes z = pair_sizes\(F, g->M, 1\);\s*int rpb", text, re.S).group(1)
    assert pick.startswith("pairs && ")                        # the second attempt asks for none
