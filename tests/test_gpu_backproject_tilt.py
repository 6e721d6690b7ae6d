"""A^T with tilted detectors at the sizes and angles where its kernels change
form: tile edges (32 heights, 16 voxel columns, 8 planes), detector steps
below half a voxel and strong drifts across a column's rows (row by row),
columns of both ray classes, and tilts beyond the plane-wise form's limit
(the per-voxel gather); the public call and the solver's A^T against the FP64
oracle, every voxel, with the operators' own float32 bound (relative to A^T|y|
where y has both signs)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2103_10329_gb300 import mgct, synth
from tests.helpers import TOL_F32, check_err, cuda, gpu_geom, oracle_scan, rel_err, scan_desc, to_np

pytestmark = pytest.mark.gpu

# n, nu, nv, views, tilt (radians: amplitude over the views; the sign alternates)
CASES = [(9, 14, 16, 5, 0.02), (17, 24, 24, 40, 0.01), (33, 50, 41, 24, 0.05), (40, 60, 60, 12, 0.0005),
         (24, 30, 36, 9, 0.3), (20, 72, 60, 6, 0.08), (31, 30, 22, 7, 0.12), (24, 36, 30, 8, 0.45)]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_10329_gb300 import build
    build.build()
    O.build()


def tilted(n, nu, nv, nviews, tilt, seed=61):
    drift = synth.drift_walk(nviews, seed, sigma_px=0.4, half_diag_px=1.0)
    drift[:, 4] = tilt * np.where(np.arange(nviews) % 2, -1.0, 1.0) * np.linspace(0.3, 1.0, nviews)
    return scan_desc(n, nu, nv, nviews, seed, levels=1, drift=drift)


@pytest.mark.parametrize("n,nu,nv,nviews,tilt", CASES)
def test_tilted_backprojection(n, nu, nv, nviews, tilt):
    d = tilted(n, nu, nv, nviews, tilt)
    g = gpu_geom(d)
    og = O.level_geometry(oracle_scan(d), 0)
    rng = np.random.default_rng(9)
    y = rng.random((nviews, nv, nu)).astype(np.float32)
    ref = O.backproject(og, y.astype(np.float64))
    check_err(rel_err(to_np(mgct.backproject(g, cuda(y))), ref), TOL_F32)
    stats = torch.zeros(4, dtype=torch.float64, device="cuda")
    step = mgct.landweber_direction(g, torch.zeros((n, n, n), device="cuda"), cuda(y), precond=False, stats=stats)
    check_err(rel_err(to_np(step) / float(stats[0]), ref), TOL_F32)
    s = rng.standard_normal((nviews, nv, nu)).astype(np.float32)
    ref = O.backproject(og, s.astype(np.float64))
    scale = O.backproject(og, np.abs(s).astype(np.float64))
    e = np.abs(to_np(mgct.backproject(g, cuda(s))) - ref) / np.maximum(scale, 1e-2 * scale.max())
    check_err(e, TOL_F32)


def test_tilted_osemtr_pass():
    """The two-channel form, in one pass of OS-EMTR."""
    d = tilted(20, 30, 33, 12, 0.06)
    g = gpu_geom(d)
    og = O.level_geometry(oracle_scan(d), 0)
    mu = 0.5 * synth.random_volume(20, 3).astype(np.float32)
    b = O.project(og, synth.random_volume(20, 4)).astype(np.float32)
    pi = O.project(og, np.ones((20, 20, 20)))
    ref = O.osemtr_pass(og, mu.astype(np.float64), b.astype(np.float64), n_subsets=3)
    got = to_np(mgct.osemtr_pass(g, cuda(mu), cuda(b), cuda(pi.astype(np.float32)), n_subsets=3))
    check_err(rel_err(got, ref), 1e-4)
