"""The ramp filter at the edges of its tiles (bins per parity in fours, rows in twos, as many row groups per
block as fill it), against the FP64 oracle at the projector's bar of 1e-5."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_09884_gb300 import inrct, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,A", [(1, 1), (3, 2), (5, 7), (6, 8), (7, 9), (515, 33), (4096, 64), (4095, 190), (90, 729), (3, 6144)])
def test_ramp_filter_at_tile_edges(V, A):
    g = synth.GeomSpec("par2d", 64, V, A)
    og = O.Geometry(g.kind, g.N, g.V, g.A, g.B, g.du, g.dv, g.sod, g.sdd, g.angle0, g.span)
    r = synth.uniform(g.m, seed=A).astype(np.float32)
    for shift in (0, 1):  # an input that does not start on 16 bytes
        rd = torch.empty(g.m + shift, device="cuda")[shift:].copy_(torch.as_tensor(r))
        out, loss = inrct.ramp_filter(g, rd)
        want = O.ramp_filter(og, r)
        err = np.linalg.norm(out.cpu().numpy() - want) / np.linalg.norm(want)
        assert err <= 1e-5
        L0 = 0.5 * float(r.astype(np.float64) @ want)
        assert abs(loss.item() - L0) <= 1e-4 * max(abs(L0), 1e-30)


@pytest.mark.parametrize("A", [9, 12, 16, 33])
def test_ramp_loss_of_an_infinite_bin(A):
    """An infinite bin whose products with all other bins are positive or finite: the loss is +inf, not NaN from places
    past the row's end."""
    g = synth.GeomSpec("par2d", 64, 3, A)
    r = torch.full((3, A), -1.0, device="cuda")
    r[1, 2] = float("inf")
    out, loss = inrct.ramp_filter(g, r.view(-1))
    odd = (torch.arange(A) - 2) % 2 == 1
    out = out.view(3, A).cpu()
    assert (out[1][odd] == float("-inf")).all() and out[1, 2] == float("inf") and torch.isfinite(out[0]).all()
    assert loss.item() == float("inf")


@pytest.mark.parametrize("V,A", [(700, 16), (333, 100), (180, 50), (2433, 40)])
def test_ramp_filter_of_short_rows(V, A):
    """Rows side by side in small blocks: the bits of the same rows filtered one scan of 8 at a time."""
    g = synth.GeomSpec("par2d", 64, V, A)
    r = torch.as_tensor(synth.uniform(g.m, seed=A).astype(np.float32), device="cuda").view(V, A)
    out, _ = inrct.ramp_filter(g, r.view(-1))
    for lo in range(0, V - 7, 97):
        part, _ = inrct.ramp_filter(synth.GeomSpec("par2d", 64, 8, A), r[lo:lo + 8].reshape(-1))
        assert torch.equal(part.view(8, A), out.view(V, A)[lo:lo + 8])


def _device_us(fn, calls=20):
    best = float("inf")
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda._sleep(2_000_000)  # the host gets ahead
        a.record()
        for _ in range(calls):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / calls)
    return best


def test_short_rows_cost_no_more_than_long_ones():
    t = {}
    for A in (16, 256):
        g = synth.GeomSpec("par2d", 64, 180, A)
        r = torch.rand(g.m, device="cuda")
        t[A] = _device_us(lambda: inrct.ramp_filter(g, r))
    assert t[16] <= 1.5 * t[256], t
