"""The product kernel starts while the digits' kernel still writes its inputs
(programmatic launch): it may read nothing through the read-only path, which asks that
nobody writes the data as long as the kernel lives (no GPU)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1306_4161_gb300", "csrc")


def test_no_read_only_loads_in_the_product_kernel():
    text = open(os.path.join(CSRC, "split_fused.cuh")).read()
    assert "wait_for_primary();" in text
    code = re.sub(r"//.*", "", text)
    assert not re.search(r"__ldg\b|ld\.global\.nc|__restrict__", code)
