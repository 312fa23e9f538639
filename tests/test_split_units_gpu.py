"""The warp-per-pixel kernel's units: geometry in double-float for one or two
units per pixel and in FP64 for more, and batches of pixels whose size follows
from the launch.  Against the oracle with the mixed form's tolerance, and
pixel by pixel bitwise between launches of different sizes."""
import numpy as np
import pytest

import oracle
from paper_2205_07976_gb300 import nbgb
from paper_2205_07976_gb300 import workloads as W
from tests.test_parity_gpu import check_mixed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("interp", [W.INTERP_NEAREST, W.INTERP_TRICUBIC])
@pytest.mark.parametrize("os,T", [(1, 1), (1, 2), (2, 1), (1, 3)])
def test_units_and_batches(os, T, interp):
    s = W.large_shot(n_src=3, n_mosaic=9)
    s.oversample, s.n_layers, s.interp = os, T, interp
    if T == 1:
        s.thickness_m = 0.0
    s = W.shrink(s, 517, 509, 2200, 600)  # several pixels per batch
    full = nbgb.simulate(s, "mixed", variant="warp")
    rows = np.concatenate([np.arange(r * 517, (r + 1) * 517)
                           for r in (0, 200, 290, 508)])
    check_mixed(full[rows], oracle.image(s, rows))
    sub = np.concatenate([rows[::97], [517 * 509 - 1]])
    one = nbgb.simulate(s, "mixed", pixels=sub, variant="warp")
    np.testing.assert_array_equal(one, full[sub])
