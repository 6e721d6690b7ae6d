"""The bilateral filter and Eq. 5's z-slice kernel at the sizes where their
launches change form, every voxel against the FP64 oracle: the filter's blocks
inside the volume (all of their windows in it; from 65 voxels a side at radius
1) beside blocks at its faces, every radius, and every number of planes a block
walks (one below about 100 a side, 16 above); Eq. 5 on both sides of the
line between 8 and 32 planes a block, with scalar and 16-byte staging and a
ragged last chunk.  Bounds: those of the operators' own tests."""
import numpy as np
import pytest

import oracle as O
from paper_2103_10329_gb300 import mgct, synth
from tests.helpers import cuda, gpu_geom, scan_desc, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_10329_gb300 import build
    build.build()
    O.build()


@pytest.mark.parametrize("n,ss,sr,r", [(17, 1.0, 0.2, 4), (70, 1.5, 0.1, 2), (88, 1.2, 0.2, 3), (75, 2.0, 0.5, 4),
                                       (101, 1.0, 0.2, 1), (101, 1.5, 0.3, 2), (260, 1.0, 0.2, 1)])
def test_bilateral_filter_blocks(n, ss, sr, r):
    x = synth.random_volume(n, 90 + r).astype(np.float32)
    ref = O.bilateral_filter(x.astype(np.float64), ss, sr, r)
    got = to_np(mgct.bilateral(cuda(x), ss, sr, r))
    assert np.abs(got - ref).max() <= 1e-5 * (x.max() - x.min())


@pytest.mark.parametrize("n", [157, 160, 161, 172])
def test_precondition_z_chunks(n):
    g = gpu_geom(scan_desc(n, 12, 12, 4, 1, levels=1, slice_axis=2))
    x = synth.random_volume(n, 18).astype(np.float32) - 0.5
    ref = O.precondition(x.astype(np.float64), 2)
    assert np.abs(to_np(mgct.precondition(g, cuda(x))) - ref).max() <= 1e-6 * np.abs(x).max()
