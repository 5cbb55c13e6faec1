"""The roles of the tensor-core kernels that run as whole warps (no GPU; reads the sources): every wait of
theirs combines the lanes' answers.  A lane that decided for itself, say because the time ran out for it
alone, would leave the others at an elect.sync or a __syncwarp of all 32 lanes without an end."""
import os
import re

import pytest

from tests.conftest import ROOT


@pytest.mark.parametrize("source,start,end,wait", [
    ("fused_tc.cu", "if (warp == TMA_WARP) {", "epilogue (warps 0..15)", "mbar_wait"),
    ("layer_tc.cu", "if (warp == RL::TMA_W) {", "} else if (!TA && warp >= RL::GATHER0) {", "lt_wait"),
])
def test_whole_warp_roles_wait_together(source, start, end, wait):
    with open(os.path.join(ROOT, "paper_2103_06624_gb300", "csrc", source)) as f:
        text = f.read()
    roles = text[text.index(start):text.index(end)]
    calls = re.findall(r"\b(%s\w*)\(" % wait, roles)
    assert len(calls) >= 3 and set(calls) == {wait + "_all"}
    assert re.search(r"%s_all\([^)]*\) \{\s*return mbar_wait_together\(" % wait, text)
