"""The bounded barrier waits of the tensor-core kernels, where whole warps wait."""
import os
import re

import pytest

from paper_2411_05799_gb300 import build, npx


@pytest.mark.parametrize("source", ["npx_gemm.cu", "npx_mlp_fused.cu"])
def test_epilogue_warps_wait_as_one(source):
    """The accumulators' barriers, and the one that frees the activations' memory, are waited for by
    whole warps that then read tensor memory together: never lane by lane."""
    text = open(os.path.join(build.CSRC, source)).read()
    epilogue = text[text.index("// ---- epilogue"):]
    epilogue = epilogue[:epilogue.index("\n}\n")]
    waits = re.findall(r"\b(mbar_wait\w*)\(&?(tfull|freed|full|staged)\b", epilogue)
    assert ("mbar_wait_warp", "tfull") in waits
    assert not [w for w in waits if w[0] == "mbar_wait" and w[1] in ("tfull", "freed")], waits


@pytest.mark.gpu
def test_a_warp_goes_on_or_gives_up_as_one():
    assert npx.gemm_warp_wait_selftest() == (0, 32)
