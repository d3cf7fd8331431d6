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
    # nine pairs of ranks, each for a whole context (0, 0), a context split over a cluster (0, 1) and with helper blocks (1, 0)
    forms = [re.search(r"ILi(\d+)ELi(\d+)ELi(\d+)ELb(\d)ELb\d+ELb(\d)E", f[0]).groups() for f in found]
    for form in (("0", "0"), ("0", "1"), ("1", "0")):
        assert len({f[:3] for f in forms if f[3:] == form}) == 9, form
    assert [f for f in found if f[2:] != ("0", "0")] == []
