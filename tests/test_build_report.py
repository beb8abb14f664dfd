"""What ptxas said when the library was built: registers that do not fit go to memory ("spills"), in kernels
that are bound by their instructions or by a chain of steps.  The bounds are what the present kernels need;
a change that exceeds one has to show by measurement that it is worth it."""
import os
import re

import pytest

from paper_2404_14469_b200 import build


def _spills(source, kernel):
    """{mangled name: bytes of spill stores} of the kernel's instantiations."""
    path = os.path.join(build.OBJ, source + ".ptxas")
    if not os.path.exists(path):
        pytest.skip("the library was not built here")
    found, name = {}, None
    for line in open(path):
        m = re.search(r"Compiling entry function '(\S+)'", line)
        if m:
            name = m.group(1)
        m = re.search(r"(\d+) bytes spill stores", line)
        if m and kernel in name:
            found[name] = int(m.group(1))
    return found


@pytest.mark.parametrize("rows,most", [("OneLength", 0), ("GroupedRows", 0), ("RaggedRows", 24)])
def test_select_kernels_keep_their_keys_in_registers(rows, most):
    # five shapes times the three radii of the paper for both pooling types, and any radius
    kernels = {k: v for k, v in _spills("snapkv_select_cluster.cu", "pool_topk_cluster_kernel").items() if rows in k}
    assert len(kernels) == 35
    assert max(kernels.values()) <= most, {k: v for k, v in kernels.items() if v > most}


def test_scoring_kernels_do_not_spill():
    kernels = _spills("snapkv_score.cu", "score_kernel")
    assert len(kernels) == 10 and not any(kernels.values())
    # the split kernels of ragged batches with 128 columns are three registers short
    kernels = _spills("snapkv_score_ragged.cu", "score_kernel")
    assert len(kernels) == 20 and max(kernels.values()) <= 12
    assert all("Li4ELb1E" in k for k, v in kernels.items() if v)
