"""The line projector (float32 volumes from 448 voxels a side, tilt-free): a
side that fills neither its tiles of 32 nor a multiple of 4 heights, detectors
whose rows and columns fill no tile of 128 and 8, columns of both ray classes,
rows above and below the volume, and steps up to the limit beyond which the
column projector runs; sampled rays against the FP64 oracle with the operators'
float32 bound, and the residual with its norm."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2103_10329_gb300 import mgct, synth
from tests.helpers import TOL_F32, check_err, gpu_geom, oracle_scan, rel_err, scan_desc, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2103_10329_gb300 import build
    build.build()
    O.build()


# row steps at the far planes: 1.05, 1.19 (the limit is 1.2), 1.5 (column projector)
@pytest.mark.parametrize("n,nu,nv", [(450, 601, 130), (449, 528, 260), (448, 420, 65)])
def test_sampled_rays(n, nu, nv):
    nviews = 9
    d = scan_desc(n, nu, nv, nviews, 31, levels=1)
    g = gpu_geom(d)
    og = O.level_geometry(oracle_scan(d), 0)
    vol = torch.rand((n, n, n), device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    got = mgct.project(g, vol)
    rays = synth.random_indices(400, (nviews, nv, nu), 5)
    # and the detector's corners and edges of tiles
    edge = np.array([[k, v, u] for k in (0, 4, 8) for v in (0, 127 % nv, nv - 1) for u in (0, 7, nu - 1)])
    rays = np.concatenate([rays, edge])
    ref = O.project_rays(og, to_np(vol), rays)
    ri = torch.as_tensor(rays, device="cuda", dtype=torch.long)
    check_err(rel_err(to_np(got[ri[:, 0], ri[:, 1], ri[:, 2]]), ref), TOL_F32)
    # the residual and its norm
    b = torch.ones_like(got)
    s = torch.zeros(1, dtype=torch.float64, device="cuda")
    r = mgct.project(g, vol, b=b, sumsq=s)
    # r and the two roundings of b - got: 2^-24 (|got| + 2 |r|), |r| <= 1 + |got|
    assert float((r - (b - got)).abs().max()) <= 2.0 ** -24 * (2 + 3 * float(got.abs().max()))
    n2 = float((r.double() ** 2).sum())
    assert abs(float(s) - n2) <= 1e-12 * n2
    # a subset of the views is the same rays
    sub = mgct.project(g, vol, views=(2, 3, 2))
    assert torch.equal(sub, got[2:7:2])
