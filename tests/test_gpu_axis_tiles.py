"""Strided passes whose blocks take the columns of several planes (planes of fewer
column pairs than a tile is wide, csrc/qhd_kernels.cu), with a last block that is
partly empty, against the FP64 oracle.  Tolerance per amplitude: the short-run
bound of tests/test_gpu_parity.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_packed import run_and_compare


# every line length along axis 0, and lines of several lengths along axis 1
@pytest.mark.parametrize("shape,batch", [((2, 2), 33), ((4, 4), 37), ((8, 2), 65), ((16, 4), 19), ((32, 8), 5), ((64, 2), 17),
                                         ((128, 4), 7), ((256, 8), 3), ((512, 2), 5), ((1024, 2), 3), ((2, 8, 2), 35),
                                         ((4, 4, 4), 9), ((2, 16, 8), 5), ((2, 128, 2), 7), ((1024, 8, 8), 1),
                                         ((4, 1024, 2), 3), ((1024, 2), 515), ((8, 1024, 2), 67)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
@pytest.mark.parametrize("own_phi", [False, True], ids=["shared-kinetic", "own-kinetic"])
def test_columns_of_several_planes_match_oracle(shape, batch, own_phi):
    run_and_compare(shape, batch, sorted({0, batch // 2, batch - 1}), own_phi)
