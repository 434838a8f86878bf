"""The tile form of the cone adjoint (plan zc = 0, 64 <= N <= 512) at the edges of its rules: ragged tiles and z
groups, two to four rows per voxel, detectors that do not cover the volume, views where both axes drive, a source
close to the volume.  Against the FP64 oracle (1e-5) and the chunk plan (1e-6, float rounding)."""
import ctypes
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_09884_gb300 import inrct, synth

pytestmark = pytest.mark.gpu

GEOMS = [
    synth.GeomSpec("cone3d", 64, 5, 90, 66, sod=200.0, sdd=300.0, span=2 * math.pi),
    synth.GeomSpec("cone3d", 65, 9, 33, 31, sod=120.0, sdd=180.0, span=2 * math.pi, angle0=0.3),        # rows and columns end inside the volume
    synth.GeomSpec("cone3d", 129, 4, 201, 333, dv=0.56, sod=1100.0, sdd=1500.0, span=2 * math.pi, angle0=math.pi / 4),  # four rows per voxel
    synth.GeomSpec("cone3d", 70, 3, 64, 77, du=0.4, dv=1.75, sod=600.0, sdd=900.0, span=2 * math.pi, angle0=0.2),  # many columns per place
    synth.GeomSpec("cone3d", 131, 2, 60, 100, du=3.0, dv=1.1, sod=140.0, sdd=400.0, span=1.0),           # pitch from 0.4: the column kernel
]


def both(g, r):
    inrct.tune_reset()
    v = inrct.backproject(g, r)
    inrct.tune_set(g, 1, 1, 8)
    c = inrct.backproject(g, r)
    inrct.tune_reset()
    return v, c


@pytest.mark.parametrize("g", GEOMS, ids=lambda g: f"{g.N}_{g.A}x{g.B}")
def test_tile_adjoint(g):
    og = O.Geometry(g.kind, g.N, g.V, g.A, g.B, g.du, g.dv, g.sod, g.sdd, g.angle0, g.span)
    r = torch.as_tensor(synth.uniform(g.m, 5).astype(np.float32), device="cuda")
    v, c = both(g, r)
    want = O.backproject(og, r.cpu().numpy().astype(np.float64))
    assert np.linalg.norm(v.cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)
    assert float((v.double() - c.double()).norm()) <= 1e-6 * float(c.double().norm())
    # a workspace without room for the padded columns takes the column kernel
    L = inrct.lib()
    gd, grd = inrct.geom_desc(g), inrct.grid_desc(3, g.N)
    nb = L.inrct_backproject_ws_bytes(ctypes.byref(gd), ctypes.byref(grd))
    ws = torch.empty(nb - 4 * 8 * g.V * g.A, dtype=torch.uint8, device="cuda")
    v2 = torch.empty_like(v)
    rc = L.backproject(ctypes.byref(gd), ctypes.byref(grd), r.data_ptr(), v2.data_ptr(), ws.data_ptr(), ws.numel(),
                       torch.cuda.current_stream().cuda_stream)
    if g is not GEOMS[-1]:  # the last one's workspace has no padding to leave out
        assert rc == 0
        assert float((v2.double() - v.double()).norm()) <= 1e-6 * float(v.double().norm())


def test_values_that_are_not_finite_reach_the_same_voxels():
    g = GEOMS[0]
    r = torch.as_tensor(synth.uniform(g.m, 6).astype(np.float32), device="cuda")
    r[[1234, 9999, 20001]] = torch.tensor([math.inf, math.nan, -math.inf], device="cuda")
    v, c = both(g, r)
    assert torch.equal(torch.isfinite(v), torch.isfinite(c))
    assert not torch.isfinite(v).all()
