"""A warp that issues MMAs waits for them before the tensor memory is freed, also
where it has issued all of its own and another warp's wait ran out: the drain must
not hang on the issuing warp's own success. No wait can be made to run out in these
kernels without a GPU fault, so the sources are read."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2412_02413_gb300" / "csrc"


@pytest.mark.parametrize("name,barrier", [("pam_wgrad.cu", r"&dbar\[v\]"), ("pam_conv_tc.cu", "dbar")])
def test_issuing_warps_drain_whoever_gave_up(name, barrier):
    src = (CSRC / name).read_text()
    m = re.search(r"if \(([^)]*)\) \{[^}]*umma_commit_elect\(" + barrier + r"\);\s*mbar_wait\(" + barrier + r", 0\);", src)
    assert m and m[1] == "any"
    free = max(src.find("tmem_dealloc(tmem"), src.find("tcgen05.dealloc"))
    assert m.end() < free
