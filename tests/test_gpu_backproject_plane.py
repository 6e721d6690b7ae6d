"""The plane-wise A^T (tilt-free geometries) at the sizes where it can go
wrong: tile edges along z (64 and 128 heights), along the planes and columns
(8), detectors coarser than the voxels (row step above 1), finer (below 0.4:
rows one by one), of fewer than five rows, and views whose rays miss most of
the volume; both entry points, against the FP64 oracle.  The bound is the
operators' own float32 bound."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2103_10329_gb300 import mgct
from tests.helpers import TOL_F32, check_err, cuda, gpu_geom, oracle_scan, rel_err, scan_desc, to_np

pytestmark = pytest.mark.gpu

# n, nu, nv, views
SIZES = [(5, 9, 7, 3), (8, 12, 4, 5), (9, 14, 30, 70), (33, 20, 25, 9), (63, 95, 61, 6), (65, 97, 140, 6),
         (129, 150, 45, 5), (17, 130, 150, 4), (96, 160, 30, 5)]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_10329_gb300 import build
    build.build()
    O.build()


@pytest.mark.parametrize("n,nu,nv,nviews", SIZES)
def test_public_and_solver(n, nu, nv, nviews):
    d = scan_desc(n, nu, nv, nviews, 77, levels=1)
    g = gpu_geom(d)
    y = np.random.default_rng(8).random((nviews, nv, nu)).astype(np.float32)
    ref = O.backproject(O.level_geometry(oracle_scan(d), 0), y.astype(np.float64))
    check_err(rel_err(to_np(mgct.backproject(g, cuda(y))), ref), TOL_F32)
    out = torch.full((n, n, n), 0.25, device="cuda")
    got = to_np(mgct.backproject(g, cuda(y), out=out, accumulate=True)) - 0.25
    check_err(np.abs(got - ref) / np.maximum(np.abs(ref), 1e-2 * np.abs(ref).max() + 0.25), TOL_F32)
    # the solver's A^T: with mu = 0 and no filter the direction is alpha A^T b
    stats = torch.zeros(4, dtype=torch.float64, device="cuda")
    step = mgct.landweber_direction(g, torch.zeros((n, n, n), device="cuda"), cuda(y), precond=False, stats=stats)
    check_err(rel_err(to_np(step) / float(stats[0]), ref), TOL_F32)


@pytest.mark.parametrize("nu", [40, 24, 100], ids=["step-0.6-0.9", "step-above-1", "step-below-0.4"])
def test_non_finite_pixel_stays_local(nu):
    """A NaN pixel reaches only voxels that its ray weights (closed supports:
    a voxel exactly one voxel away may take part with weight 0)."""
    n, nv, k = 32, 40, 6
    d = scan_desc(n, nu, nv, k, 5, levels=1)
    g = gpu_geom(d)
    y = np.zeros((k, nv, nu), dtype=np.float32)
    y[2, 17, nu // 3] = y[4, 25, nu // 2] = 1.0
    ref = O.backproject(O.level_geometry(oracle_scan(d), 0), y.astype(np.float64))
    y[y > 0] = np.nan
    got = np.isnan(to_np(mgct.backproject(g, cuda(y))))
    assert got[ref > 1e-6 * ref.max()].all()
    assert not got[ref == 0.0].any()
