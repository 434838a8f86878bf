"""The ray tables that stay in a workspace: whatever is written to the workspace between two calls, wherever, the next
call gives the bits of a fresh one.  Every 4 KB piece of the workspace in turn, single bits, and recycled memory of
the binding's own workspaces."""
import ctypes
import math

import pytest
import torch

from paper_2604_09884_gb300 import inrct, synth

pytestmark = pytest.mark.gpu

GEOMS = [
    synth.GeomSpec("par2d", 48, 21, 69),
    synth.GeomSpec("fan2d", 64, 7, 300, sod=200.0, sdd=300.0, span=2 * math.pi),
    synth.GeomSpec("par2d", 16, 700, 1),
    synth.GeomSpec("cone3d", 33, 9, 61, 40, sod=90.0, sdd=150.0, span=2 * math.pi),
    synth.GeomSpec("cone3d", 130, 2, 150, 140, sod=300.0, sdd=450.0, span=2 * math.pi),
]


def _call(g, forward, src, ws):
    L = inrct.lib()
    gd, grd = inrct.geom_desc(g), inrct.grid_desc(g.d, g.N)
    out = torch.empty(g.m if forward else g.n, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    args = (ctypes.byref(gd), ctypes.byref(grd), src.data_ptr(), out.data_ptr())
    if forward:
        rc = L.project(*args, None, None, None, ws.data_ptr(), ws.numel(), s)
    else:
        rc = L.backproject(*args, ws.data_ptr(), ws.numel(), s)
    assert rc == 0, L.inrct_last_error().decode()
    return out


def _tables_bytes(g):  # the tables and the views come first in a workspace
    return g.V * g.A * (36 if g.kind == "cone3d" else 16) + 8 * g.V + 5 * 256


@pytest.mark.parametrize("g", GEOMS, ids=lambda g: f"{g.kind}_{g.N}_{g.V}x{g.A}")
@pytest.mark.parametrize("forward", [True, False], ids=["project", "backproject"])
def test_workspace_written_to_between_calls(g, forward):
    L = inrct.lib()
    gd, grd = inrct.geom_desc(g), inrct.grid_desc(g.d, g.N)
    nb = (L.inrct_project_ws_bytes if forward else L.inrct_backproject_ws_bytes)(ctypes.byref(gd), ctypes.byref(grd))
    src = torch.as_tensor(synth.uniform(g.n if forward else g.m, 3, 0.0, 1.0), dtype=torch.float32, device="cuda")
    want = _call(g, forward, src, torch.zeros(nb, dtype=torch.uint8, device="cuda"))
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    assert torch.equal(_call(g, forward, src, ws), want)
    for lo in range(0, min(nb, _tables_bytes(g) + 4096), 4096):
        ws[lo:lo + 4096] = 0x3f
        assert torch.equal(_call(g, forward, src, ws), want), lo
    for lo in range(5, min(nb, _tables_bytes(g)), 997):  # one bit of some entry
        ws[lo] ^= 16
        assert torch.equal(_call(g, forward, src, ws), want), lo


def test_static_scratch_without_room_for_the_checksums():
    """The allocation-free projection takes every geometry whose tables and image fit its array; where the checksums do
    not fit any more, every call builds the tables."""
    L = inrct.lib()
    limit, N, V = 16 << 20, 1200, 150

    def need(A):  # with the checksums (8 bytes per view and 32 bins, last)
        g = synth.GeomSpec("par2d", N, V, A)
        return L.inrct_project_ws_bytes(ctypes.byref(inrct.geom_desc(g)), ctypes.byref(inrct.grid_desc(2, N)))

    A = next(a for a in range(3000, 8000) if need(a) > limit)
    assert need(A) - V * -(-A // 32) * 8 + 512 <= limit
    g = synth.GeomSpec("par2d", N, V, A)
    x = torch.as_tensor(synth.uniform(g.n, 3, 0.0, 1.0), dtype=torch.float32, device="cuda")
    want = inrct.project(g, x)
    other = synth.GeomSpec("par2d", N, V, A, angle0=0.5)
    for _ in range(2):
        assert torch.equal(inrct.project_noalloc(g, x), want)
        assert not torch.equal(inrct.project_noalloc(other, x), want)


@pytest.mark.parametrize("kind", ["par2d", "fan2d"])
def test_recycled_memory_of_the_bindings_workspace(kind):
    """The allocator hands a freed workspace to the next tensor and back: a tensor of its size of which only a middle
    part is written leaves both of its ends as the call left them."""
    g = synth.GeomSpec(kind, 96, 40, 137, sod=300.0, sdd=450.0, span=2 * math.pi)
    gd, grd = inrct.geom_desc(g), inrct.grid_desc(g.d, g.N)
    src = torch.as_tensor(synth.uniform(g.m, 3, 0.0, 1.0), dtype=torch.float32, device="cuda")
    want = inrct.backproject(g, src)
    nb = inrct.lib().inrct_backproject_ws_bytes(ctypes.byref(gd), ctypes.byref(grd))
    for _ in range(3):
        t = torch.empty(nb, dtype=torch.uint8, device="cuda")
        t[4096:12288] = 0x3f
        del t
        assert torch.equal(inrct.backproject(g, src), want)
