"""The line projector in blocks whose columns hold rays of both classes: a
plane's lines then cover the heights of two different planes, more than fit at
places, and the samples come from the volume itself.  Every row of such blocks
against the FP64 oracle, and a weighted epilogue through the same kernel (the
solver's residual and its A^T) at a ragged side; the operators' float32
bounds."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2103_10329_gb300 import mgct, synth
from tests.helpers import TOL_F32, check_err, gpu_geom, oracle_scan, rel_err, scan_desc, to_np

pytestmark = pytest.mark.gpu

# row step 0.72 (finer than the voxels); spans of up to 190 heights, 168 fit
N, NU, NV, VIEWS = 451, 640, 400, 9


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_10329_gb300 import build
    build.build()
    O.build()


@pytest.fixture(scope="module")
def scan():
    d = scan_desc(N, NU, NV, VIEWS, 31, levels=1)
    return d, gpu_geom(d), O.level_geometry(oracle_scan(d), 0)


def mixed_blocks(d):
    """(view, first column) of the 8-column blocks with rays of both classes."""
    u = (np.arange(d["nu"]) - 0.5 * (d["nu"] - 1)) * d["pitch"]
    out = []
    for k, t in enumerate(d["theta"]):
        y_major = np.abs(-4.0 * np.sin(t) + u * np.cos(t)) > np.abs(-4.0 * np.cos(t) - u * np.sin(t))
        out += [(k, u0) for u0 in range(0, d["nu"], 8) if len(set(y_major[u0:u0 + 8])) == 2]
    return out


def test_rays_of_mixed_blocks(scan):
    d, g, og = scan
    blocks = mixed_blocks(d)
    assert len(blocks) >= 3
    vol = torch.rand((N, N, N), device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    got = mgct.project(g, vol)
    rays = np.array([[k, v, u] for k, u0 in blocks for v in range(NV) for u in range(u0, min(u0 + 8, NU))])
    ref = O.project_rays(og, to_np(vol), rays)
    ri = torch.as_tensor(rays, device="cuda", dtype=torch.long)
    check_err(rel_err(to_np(got[ri[:, 0], ri[:, 1], ri[:, 2]]), ref), TOL_F32)


def test_weighted_residual(scan):
    d, g, og = scan
    mu = torch.rand((N, N, N), device="cuda", generator=torch.Generator("cuda").manual_seed(5)) * 0.5
    b = torch.rand((VIEWS, NV, NU), device="cuda", generator=torch.Generator("cuda").manual_seed(6))
    stats = torch.zeros(4, dtype=torch.float64, device="cuda")
    step = mgct.landweber_direction(g, mu, b, precond=False, stats=stats)
    p = O.project(og, to_np(mu))
    r = to_np(b) - p
    bound = 2 * TOL_F32 * (np.abs(r) * np.maximum(np.abs(p), 1e-2 * np.abs(p).max())).sum()
    assert abs(float(stats[1]) - (r ** 2).sum()) <= bound
    # voxels of the whole volume, and of the middle, where every view's rays of
    # the mixed blocks pass
    vox = synth.random_indices(40, (N, N, N), 7)
    vox = np.concatenate([vox, synth.random_indices(40, (90, 90, 90), 8) + (N - 90) // 2])
    ref = O.backproject_voxels(og, r, vox, radius=5)
    scale = O.backproject_voxels(og, np.abs(r), vox, radius=5)
    vi = torch.as_tensor(vox, device="cuda", dtype=torch.long)
    got = to_np(step[vi[:, 2], vi[:, 1], vi[:, 0]]) / float(stats[0])
    check_err(np.abs(got - ref) / np.maximum(scale, 1e-2 * scale.max()), TOL_F32)
