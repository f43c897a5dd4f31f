"""Grid sizes that bah_create takes before it touches a device: the 3-D level kernels reach a
block's vector through 32-bit byte offsets, so an FP64 grid has at most 2^28 cells.  Without a
device an accepted grid stops at the stream's creation (BAH_ERR_CUDA); the medium arrays are not
read before that."""
import numpy as np
import pytest

import paper_2411_15897_gb300 as bah
from paper_2411_15897_gb300 import _build


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if torch.cuda.is_available():
        pytest.skip("an accepted grid would be built")
    try:
        _build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    _build.build()


@pytest.mark.parametrize("n,precision,refused", [
    ((1024, 512, 768), bah.BAH_FP64, True), ((1024, 512, 768), bah.BAH_MIXED, False),
    ((1024, 512, 512), bah.BAH_FP64, False), ((1024, 1024, 512), bah.BAH_MIXED, True),
])
def test_3d_cells_fit_the_kernels_offsets(n, precision, refused):
    one = np.ones(1)
    o = bah.bah_default_opts(precision=precision, intergrid=bah.BAH_INTERGRID_MIXED)
    with pytest.raises(bah.BahError) as e:
        bah.bah_create(n, (1.0, 1.0, 1.0), one, one, one, one, 1.0, o)
    assert e.value.status == (bah.BAH_ERR_ARG if refused else bah.BAH_ERR_CUDA), str(e.value)
    assert ("too large" in str(e.value)) == refused
