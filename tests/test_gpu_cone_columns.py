"""The column form of the cone projector (plan seg = 1, N >= 128) at the edges of its rules: detector columns and
rows that fill no block, several row chunks, fine and coarse row pitches, views where both axes drive, a source
close to the volume.  Against the FP64 oracle (1e-5) and the two-segment plan (1e-6, float rounding)."""
import ctypes
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_09884_gb300 import inrct, synth

pytestmark = pytest.mark.gpu

GEOMS = [
    synth.GeomSpec("cone3d", 128, 3, 37, 32, sod=400.0, sdd=600.0, span=2 * math.pi),
    synth.GeomSpec("cone3d", 129, 4, 201, 33, dv=4.0, sod=300.0, sdd=450.0, span=2 * math.pi, angle0=math.pi / 4),
    synth.GeomSpec("cone3d", 131, 2, 190, 395, dv=0.5, sod=240.0, sdd=300.0, span=2 * math.pi, angle0=0.7),
    synth.GeomSpec("cone3d", 150, 3, 64, 130, du=3.0, dv=1.2, sod=132.0, sdd=400.0, span=2 * math.pi, angle0=0.2),
    synth.GeomSpec("cone3d", 130, 2, 60, 800, dv=0.01, sod=900.0, sdd=1800.0, span=1.0),
]


@pytest.mark.parametrize("g", GEOMS, ids=lambda g: f"{g.N}_{g.A}x{g.B}")
def test_column_projector(g):
    og = O.Geometry(g.kind, g.N, g.V, g.A, g.B, g.du, g.dv, g.sod, g.sdd, g.angle0, g.span)
    x = (synth.phantom(3, g.N, 6, 3).reshape(-1) + 0.1 * synth.uniform(g.n, 4, 0.0, 1.0)).astype(np.float32)
    y = synth.uniform(g.m, 5, 0.0, 1.0).astype(np.float32)
    xd, yd = torch.as_tensor(x, device="cuda"), torch.as_tensor(y, device="cuda")
    inrct.tune_reset()
    z, r, loss = inrct.project(g, xd, yd)
    want = O.project(og, x)
    assert np.linalg.norm(z.cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)
    assert torch.equal(r, z - yd)
    L0 = 0.5 * float(((z.double() - yd.double()) ** 2).sum())
    assert abs(loss.item() - L0) <= 1e-6 * L0  # FP32 residuals squared, FP32 sums of at most 32
    inrct.tune_set(g, 2, 1, 8)
    z2 = inrct.project(g, xd)
    inrct.tune_reset()
    assert float((z.double() - z2.double()).norm()) <= 1e-6 * float(z2.double().norm())
    # a workspace without room for the padded columns takes the row-patch form
    L = inrct.lib()
    gd, grd = inrct.geom_desc(g), inrct.grid_desc(3, g.N)
    nb = L.inrct_project_ws_bytes(ctypes.byref(gd), ctypes.byref(grd))
    pad = 4 * g.N * g.N * (-g.N % 4)
    ws = torch.empty(nb - pad, dtype=torch.uint8, device="cuda")
    z3 = torch.empty_like(z)
    rc = L.project(ctypes.byref(gd), ctypes.byref(grd), xd.data_ptr(), z3.data_ptr(), None, None, None, ws.data_ptr(), ws.numel(),
                   torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    assert float((z3.double() - z.double()).norm()) <= 1e-6 * float(z.double().norm())


def test_column_projector_first_slice():
    """All of the volume in the first slices (x = 0 and y = 0) that rays driven along x and y cross: what a warp
    interpolates right after it has cleared its shared column.  Against the two-segment plan."""
    g = synth.GeomSpec("cone3d", 160, 8, 211, 224, sod=300.0, sdd=450.0, span=2 * math.pi)
    x = torch.zeros(g.N, g.N, g.N, device="cuda")
    u = torch.as_tensor(synth.uniform(2 * g.N * g.N, 6, 0.5, 1.0).astype(np.float32), device="cuda").view(2, g.N, g.N)
    x[:, :, 0], x[:, 0, :] = u[0], u[1]
    inrct.tune_set(g, 2, 1, 8)
    want = inrct.project(g, x.view(-1))
    inrct.tune_set(g, 1, 1, 8)
    for _ in range(20):
        z = inrct.project(g, x.view(-1))
        assert float((z.double() - want.double()).norm()) <= 1e-6 * float(want.double().norm())
    inrct.tune_reset()


@pytest.mark.parametrize("g", GEOMS, ids=lambda g: f"{g.N}_{g.A}x{g.B}")
def test_column_projector_pinned(g):
    """The column form where the default takes the row patches (few columns, few rows): pinned, against the default
    and the FP64 oracle."""
    og = O.Geometry(g.kind, g.N, g.V, g.A, g.B, g.du, g.dv, g.sod, g.sdd, g.angle0, g.span)
    x = (synth.phantom(3, g.N, 6, 3).reshape(-1) + 0.1 * synth.uniform(g.n, 4, 0.0, 1.0)).astype(np.float32)
    y = synth.uniform(g.m, 5, 0.0, 1.0).astype(np.float32)
    xd, yd = torch.as_tensor(x, device="cuda"), torch.as_tensor(y, device="cuda")
    inrct.tune_reset()
    z0 = inrct.project(g, xd)
    inrct.tune_set(g, 1, 1, 8)
    z, r, loss = inrct.project(g, xd, yd)
    inrct.tune_reset()
    assert np.linalg.norm(z.cpu().numpy() - O.project(og, x)) <= 1e-5 * float(z.double().norm())
    assert float((z.double() - z0.double()).norm()) <= 1e-6 * float(z0.double().norm())
    assert torch.equal(r, z - yd)
    L0 = 0.5 * float(((z.double() - yd.double()) ** 2).sum())
    assert abs(loss.item() - L0) <= 1e-6 * L0


def test_short_detectors_take_the_row_patches():
    """By default a scan of few detector rows or few columns does not pay for the column form; one of many does take it."""
    def us(g, pin):
        x = torch.rand(g.n, device="cuda")
        inrct.tune_reset()
        if pin:
            inrct.tune_set(g, 1, 1, 8)
        best = float("inf")
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            inrct.project(g, x)
            torch.cuda._sleep(1_000_000)
            a.record()
            for _ in range(5):
                inrct.project(g, x)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        inrct.tune_reset()
        return best
    scan = lambda V, A, B: synth.GeomSpec("cone3d", 256, V, A, B, sod=640.0, sdd=960.0, span=2 * math.pi)
    for g in (scan(20, 384, 32), scan(2, 384, 384)):
        assert us(g, False) <= 0.8 * us(g, True)
    assert abs(us(scan(40, 384, 384), False) / us(scan(40, 384, 384), True) - 1) <= 0.1
