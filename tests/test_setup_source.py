"""The set-up kernel may run in place: host buffers land in the residual, and
clean_hogbom_noalloc takes a residual that is the dirty image."""
import os
import re

import paper_2501_01461_gb300 as cg


def test_set_up_reads_the_dirty_image_with_coherent_loads():
    src = open(os.path.join(os.path.dirname(cg.__file__), "csrc", "aux_kernels.cu")).read()
    body = re.search(r"\n    init_kernel\((.*?)\n}\n", src, re.S).group(1)
    assert "dirty" in body
    assert not re.search(r"ld_nc|__ldg|const float\* __restrict__ dirty", body)
