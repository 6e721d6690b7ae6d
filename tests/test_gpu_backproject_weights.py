"""Single weights of A^T with tilted detectors: one view at a time, pixels far
enough apart that no voxel sees two, so every voxel of the result is one weight
h_b h_z dl against the FP64 oracle.

Bound, relative to the largest weight: a crossing's offset from a voxel is a
sum of three terms below 2, each rounded to float32 (2^-24 of a number up to 2,
twice, and of one up to 1): 2.5 * 2^-23 a coordinate, one product's 2^-24 and
the path length's four roundings, 4 * 2^-24 -- 7.5 * 2^-23 = 8.9e-7."""
import numpy as np
import pytest

import oracle as O
from paper_2103_10329_gb300 import mgct, synth
from tests.helpers import check_err, cuda, gpu_geom, oracle_scan, scan_desc, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_10329_gb300 import build
    build.build()
    O.build()


# tilts of a drift walk, and forms with and without a test of each ray's class; one
# view of 60 voxels' height takes the tilt kernel
@pytest.mark.parametrize("n,nu,tilt", [(64, 96, 0.004), (64, 90, 0.1), (61, 80, 0.25)])
def test_tilted_weights(n, nu, tilt):
    nviews = 8
    drift = synth.drift_walk(nviews, 3, sigma_px=0.4, half_diag_px=1.0)
    drift[:, 4] = tilt * np.where(np.arange(nviews) % 2, -1.0, 1.0) * np.linspace(0.4, 1.0, nviews)
    d = scan_desc(n, nu, nu, nviews, 15, levels=1, drift=drift)
    g = gpu_geom(d)
    og = O.level_geometry(oracle_scan(d), 0)
    y = np.zeros((nviews, nu, nu), dtype=np.float32)
    for k in range(nviews):
        y[k, k % 8::8, (3 * k) % 8::8] = 1.0
    for k in range(nviews):
        one = np.zeros_like(y)
        one[k] = y[k]
        ref = O.backproject(og, one.astype(np.float64))
        got = to_np(mgct.backproject(g, cuda(y[k:k + 1]), views=(k, 1, 1)))
        check_err(np.abs(got - ref) / ref.max(), 8.9e-7)
