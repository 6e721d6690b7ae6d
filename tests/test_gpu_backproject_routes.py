"""A^T on both sides of the lines between its kernels: few views, detectors of
few rows, rows much finer and coarser than the voxels (down to 1e-5 voxel, where
a tile's middle is millions of rows away), for the public call, the solver's
A^T and OS-EMTR's two channels, with and without detector tilt; every voxel
against the FP64 oracle with the operators' float32 bound (relative to A^T|y|
where y has both signs)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2103_10329_gb300 import mgct, synth
from tests.helpers import TOL_F32, check_err, cuda, gpu_geom, oracle_scan, rel_err, scan_desc, to_np

pytestmark = pytest.mark.gpu

# n, nu, nv, views, pitch over the fan's own (row step 1.03 n / nu times that)
CASES = [
    # few views: slab kernel, then plane kernel (the solver's from 4 at 72^3)
    (40, 60, 60, 1, 1.0), (72, 108, 100, 2, 1.0), (72, 108, 100, 4, 1.0), (40, 60, 60, 3, 1.0),
    # few rows: slab kernel, plane kernel
    (66, 99, 1, 6, 1.0), (66, 99, 8, 40, 1.0),
    # fine and coarse rows: steps 0.15, 0.31, 0.33, 0.45 and 2.6 (slab kernel), 0.50 (plane kernel: row by row
    # in the near planes) and 1.7 (plane kernel, rows tested)
    (24, 36, 36, 30, 0.22), (24, 36, 16, 45, 0.45), (40, 60, 40, 20, 0.48), (66, 99, 60, 12, 0.65), (40, 40, 20, 12, 2.5),
    (40, 60, 60, 60, 0.73), (33, 50, 20, 40, 2.5),
    # plane kernel: one and two pairs of heights a lane, ragged tiles
    (63, 95, 61, 30, 1.0), (129, 150, 140, 10, 1.0), (96, 120, 70, 16, 1.0), (35, 40, 38, 40, 1.0),
    # 1e-5 voxel a row
    (4, 6, 96, 5, 1.5e-5)]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_10329_gb300 import build
    build.build()
    O.build()


def both_calls(d, y):
    """Public A^T y and the solver's, as float64 arrays."""
    g = gpu_geom(d)
    n = d["n"]
    pub = to_np(mgct.backproject(g, cuda(y)))
    stats = torch.zeros(4, dtype=torch.float64, device="cuda")
    step = mgct.landweber_direction(g, torch.zeros((n, n, n), device="cuda"), cuda(y), precond=False, stats=stats)
    return pub, to_np(step) / float(stats[0])


@pytest.mark.parametrize("n,nu,nv,nviews,scale", CASES)
def test_backprojection(n, nu, nv, nviews, scale):
    d = scan_desc(n, nu, nv, nviews, 77, levels=1, pitch=scale * synth.default_pitch(nu))
    og = O.level_geometry(oracle_scan(d), 0)
    y = np.random.default_rng(8).random((nviews, nv, nu)).astype(np.float32)
    ref = O.backproject(og, y.astype(np.float64))
    for got in both_calls(d, y):
        check_err(rel_err(got, ref), TOL_F32)
    s = np.random.default_rng(9).standard_normal((nviews, nv, nu)).astype(np.float32)
    ref = O.backproject(og, s.astype(np.float64))
    size = O.backproject(og, np.abs(s).astype(np.float64))
    out = to_np(mgct.backproject(gpu_geom(d), cuda(s)))
    check_err(np.abs(out - ref) / np.maximum(size, 1e-2 * size.max()), TOL_F32)


# gather (step below 0.5, or few views of few rows), tilt kernel
@pytest.mark.parametrize("n,nu,nv,nviews,scale,tilt", [(32, 48, 48, 8, 0.6, 0.1), (32, 48, 2, 8, 1.0, 0.05),
                                                       (32, 48, 48, 1, 1.0, 0.05), (32, 40, 48, 8, 1.0, 0.2)])
def test_tilted_backprojection(n, nu, nv, nviews, scale, tilt):
    drift = synth.drift_walk(nviews, 6, sigma_px=0.4, half_diag_px=1.0)
    drift[:, 4] = tilt * np.where(np.arange(nviews) % 2, -1.0, 1.0)
    d = scan_desc(n, nu, nv, nviews, 78, levels=1, drift=drift, pitch=scale * synth.default_pitch(nu))
    og = O.level_geometry(oracle_scan(d), 0)
    y = np.random.default_rng(8).random((nviews, nv, nu)).astype(np.float32)
    ref = O.backproject(og, y.astype(np.float64))
    for got in both_calls(d, y):
        check_err(rel_err(got, ref), TOL_F32)


# two channels: slab kernel (4 views a subset; a step of 0.34; 8 rows), plane kernel
# (15 of 24^3; 30 of 40^3), gather and tilt kernel
@pytest.mark.parametrize("n,nu,nv,nviews,subsets,scale,tilt",
                         [(20, 30, 33, 12, 3, 1.0, 0.0), (24, 36, 36, 24, 2, 0.5, 0.0), (40, 60, 8, 16, 2, 1.0, 0.0),
                          (24, 36, 30, 60, 4, 1.0, 0.0), (40, 60, 60, 60, 2, 1.0, 0.0), (24, 36, 30, 12, 3, 0.6, 0.06),
                          (24, 36, 30, 12, 3, 1.0, 0.06)])
def test_osemtr_pass(n, nu, nv, nviews, subsets, scale, tilt):
    drift = None
    if tilt:
        drift = synth.drift_walk(nviews, 6, sigma_px=0.4, half_diag_px=1.0)
        drift[:, 4] = tilt * np.where(np.arange(nviews) % 2, -1.0, 1.0)
    d = scan_desc(n, nu, nv, nviews, 61, levels=1, drift=drift, pitch=scale * synth.default_pitch(nu))
    og = O.level_geometry(oracle_scan(d), 0)
    mu = 0.5 * synth.random_volume(n, 3).astype(np.float32)
    b = O.project(og, synth.random_volume(n, 4)).astype(np.float32)
    pi = O.project(og, np.ones((n, n, n)))
    ref = O.osemtr_pass(og, mu.astype(np.float64), b.astype(np.float64), n_subsets=subsets)
    got = to_np(mgct.osemtr_pass(gpu_geom(d), cuda(mu), cuda(b), cuda(pi.astype(np.float32)), n_subsets=subsets))
    check_err(rel_err(got, ref), 1e-4)
