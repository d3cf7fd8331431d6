"""What the compiler says of the kernels (no GPU)."""
import re

import pytest

from paper_2609_34054_b200 import build


@pytest.mark.parametrize("src", ["api_prefill64.cu", "api_prefill128.cu"])
def test_tensor_memory_prefill_kernels_do_not_spill(src):
    """Their step loop holds a row's 128 scores and 64 packed weights per thread: a spill there is paid at every step."""
    build.build()
    found = re.findall(r"Compiling entry function '(\S*lr_attend_prefill_tc_kernel\S*)'.*?(\d+) bytes stack frame, (\d+) bytes spill stores,"
                       r" (\d+) bytes spill loads", open(build.resource_log(src)).read(), re.S)
    assert len(found) >= 18                             # nine pairs of ranks, with and without helper blocks
    assert [f for f in found if f[2:] != ("0", "0")] == []
