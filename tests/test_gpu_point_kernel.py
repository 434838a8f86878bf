"""The FP32 point kernel and its weight-gradient GEMM at the edges of their tiles, against the FP64 oracle
(bars of the FP32 path: image 1e-5, gradient 1e-4 relative L2)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_09884_gb300 import inrct, synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


NETS = [
    synth.ArchSpec("siren", 2, 64, 1, omega0=30.0),              # no GEMM layer at all
    synth.ArchSpec("siren", 3, 256, 2, omega0=30.0),
    synth.ArchSpec("ffn", 2, 64, 2, n_feat=33, sigma=3.0),       # odd input width, two column tiles
    synth.ArchSpec("ffn", 3, 128, 2, n_feat=150, sigma=2.0),     # input wider than the activation buffer, ragged chunk
    synth.ArchSpec("hash", 2, 128, 2, hash_levels=5, hash_feats=1, hash_log2_T=8, hash_base=4, hash_growth=1.7),
    synth.ArchSpec("hash", 3, 64, 2, hash_levels=8, hash_feats=8, hash_log2_T=8, hash_base=2, hash_growth=1.5),
]


# points around a block's 32 and 64, and enough for 8 points per thread with a ragged last block
@pytest.mark.parametrize("k", [1, 31, 33, 64, 40001])
@pytest.mark.parametrize("spec", NETS, ids=lambda a: f"{a.kind}{a.d}d_{a.width}x{a.n_hidden}")
def test_vjp_at_tile_edges(spec, k):
    N = 211 if spec.d == 2 else 35
    n = N ** spec.d
    k = min(k, n)
    theta = synth.init_theta(spec, 2, table_scale=0.5).astype(np.float32)
    B = synth.fourier_matrix(spec.n_feat, spec.d, spec.sigma, 1).astype(np.float32) if spec.kind == "ffn" else None
    oa = O.Arch(spec.kind, spec.d, spec.width, spec.n_hidden, spec.n_feat, None if B is None else B.astype(np.float64),
                spec.omega0, **({k2: getattr(spec, k2) for k2 in ("hash_levels", "hash_feats", "hash_log2_T", "hash_base",
                                                                  "hash_growth")} if spec.kind == "hash" else {}))
    rng = np.random.default_rng(3)
    idx = np.sort(rng.choice(n, size=k, replace=False)).astype(np.int32)
    v = rng.normal(size=n).astype(np.float32)
    X = O.grid_coords(spec.d, N, idx)
    t64 = theta.astype(np.float64)
    if spec.kind != "siren":  # points whose ReLU decisions are unique in FP32
        _, _, zs, _ = O.forward(oa, t64, X, keep=True, N=N)
        ok = np.ones(k, bool)
        for z in zs[:-1]:
            ok &= (np.abs(z) >= 1e-6 * np.sqrt((z ** 2).mean())).all(axis=1)
        v[idx[~ok]] = 0.0
    h = inrct.mlp_desc(spec, inrct.FP32, B)
    dev = lambda a, t=torch.float32: torch.as_tensor(a, dtype=t, device="cuda")
    val, g = inrct.inr_virtual_loss(h, dev(theta), N, dev(idx, torch.int32), dev(v), 2.0)
    w = 2.0 * v.astype(np.float64)[idx]
    want = O.vjp(oa, t64, X, w, N=N)
    f = O.forward(oa, t64, X, N=N)
    if np.linalg.norm(want) > 0:
        assert rel(g.cpu().numpy(), want) <= 1e-4
    # FP32 values of f: 1e-5 of their size, summed with the weights
    assert abs(val.item() - float(w @ f)) <= 1e-5 * np.linalg.norm(w) * np.linalg.norm(f)
    if k == 40001 or k == n:
        img = inrct.inr_eval_grid(h, dev(theta), N).cpu().numpy()
        assert rel(img[idx], f) <= 1e-5


# few blocks (one thread sums an entry's partials) and many (32 threads): the output bias gradient is the sum of the
# weights, one per block here, exact in FP64 also where an FP32 sum of them overflows or meets infinities
@pytest.mark.parametrize("k", [1500, 40001])
@pytest.mark.parametrize("vals", [(2e38, 2e38, 2e38, 2e38), (3e38, -3e38, 3e38, 2.0), (np.inf, 1.0, 1.0, 1.0),
                                  (np.inf, -np.inf, 1.0, 1.0), (1.0, 2.0 ** -30, 2.0 ** -31, -1.0)])
def test_gradient_sums_of_any_size(vals, k):
    spec = synth.ArchSpec("siren", 2, 64, 2, omega0=30.0)
    theta = synth.init_theta(spec, 2).astype(np.float32)
    v = np.zeros(211 * 211, np.float32)
    v[[0, k // 4, k // 2, k - 1]] = np.asarray(vals, np.float32)
    dev = lambda a, t=torch.float32: torch.as_tensor(a, dtype=t, device="cuda")
    _, g = inrct.inr_virtual_loss(inrct.mlp_desc(spec, inrct.FP32, None), dev(theta), 211,
                                  dev(np.arange(k, dtype=np.int32), torch.int32), dev(v), 1.0)
    with np.errstate(invalid="ignore"):
        want = np.asarray(vals, np.float32).astype(np.float64).sum()
    assert np.array_equal(g[-1].item(), want, equal_nan=True)


# runs of equal entries in the table scatter: whole warps, none, broken by points without weight, in falling order
@pytest.mark.parametrize("order", ["dense", "reversed", "one point", "alternating weights", "shuffled"])
@pytest.mark.parametrize("spec", NETS[4:], ids=lambda a: f"{a.kind}{a.d}d_{a.width}x{a.n_hidden}")
def test_table_scatter_runs(spec, order):
    N = 64 if spec.d == 2 else 16
    k = 200
    theta = synth.init_theta(spec, 5, table_scale=0.5).astype(np.float32)
    rng = np.random.default_rng(7)
    idx = np.arange(k) + 3
    if order == "reversed":
        idx = idx[::-1].copy()
    elif order == "one point":
        idx = np.full(k, 77)
    elif order == "shuffled":
        idx = rng.permutation(N ** spec.d)[:k]
    v = rng.normal(size=N ** spec.d).astype(np.float32)
    if order == "alternating weights":
        v[::2] = 0.0
    names = ("hash_levels", "hash_feats", "hash_log2_T", "hash_base", "hash_growth")
    oa = O.Arch(spec.kind, spec.d, spec.width, spec.n_hidden, 0, None, spec.omega0, **{a: getattr(spec, a) for a in names})
    X = O.grid_coords(spec.d, N, idx)
    _, _, zs, _ = O.forward(oa, theta.astype(np.float64), X, keep=True, N=N)
    ok = np.ones(k, bool)
    for z in zs[:-1]:  # points whose ReLU decisions are unique in FP32
        ok &= (np.abs(z) >= 1e-6 * np.sqrt((z ** 2).mean())).all(axis=1)
    v[idx[~ok]] = 0.0
    dev = lambda a, t=torch.float32: torch.as_tensor(a, dtype=t, device="cuda")
    _, g = inrct.inr_virtual_loss(inrct.mlp_desc(spec, inrct.FP32, None), dev(theta), N, dev(idx, torch.int32), dev(v), 1.0)
    want = O.vjp(oa, theta.astype(np.float64), X, v.astype(np.float64)[idx], N=N)
    assert rel(g.cpu().numpy(), want) <= 1e-4


def test_step_without_room_for_shared_weights():
    """A step copies the weights once where its workspace has room, else per call: the same bits either way."""
    spec = synth.ArchSpec("siren", 2, 64, 2, omega0=30.0)
    g = synth.GeomSpec("par2d", 40, 16, 61)
    h = inrct.mlp_desc(spec, inrct.FP32, None)
    idx = torch.arange(3, 903, dtype=torch.int32, device="cuda")
    y = torch.linspace(0, 1, g.m, device="cuda")
    full = inrct.step_ws_bytes(g, h, idx.numel())
    copies = 4 * (2 * 64 + 2 * 64 * 64)  # W_1^T, W_2^T and W_2
    out = []
    for nbytes in (full, full - copies):
        th = torch.as_tensor(synth.init_theta(spec, 2).astype(np.float32), device="cuda")
        m, s = torch.zeros_like(th), torch.zeros_like(th)
        grad = torch.zeros(spec.p, dtype=torch.float64, device="cuda")
        loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        inrct.grad_step(g, h, th, y, idx, 1.0, inrct.adam(lr=1e-3, t=1), m, s, loss, grad, ws=ws)
        out.append((th, grad, loss))
    assert all(torch.equal(a, b) for a, b in zip(*out)) and out[0][1].abs().max() > 0


@pytest.mark.parametrize("k", [1, 33, 95])
def test_only_listed_points_reach_the_sums(k):
    """A network that is finite at the listed points and not at grid point 0 (a pre-activation overflows there): the
    gradient and the virtual loss of a list that fills no block are those of the list filled up with
    other finite points at no weight, and finite."""
    spec, N = synth.ArchSpec("siren", 2, 64, 2, omega0=1.0), 32
    theta = synth.init_theta(spec, 2).astype(np.float32)
    theta[[0, 1]] = 2e38  # the first unit's weights: 2e38 (x + y) overflows at the corner only
    xy = (2 * np.arange(N) + 1 - N) / N
    near = np.abs(xy[:, None] + xy[None, :]) < 1.0
    idx = np.flatnonzero(near.reshape(-1))[:: near.sum() // 96][:k].astype(np.int32)
    assert idx.size == k and 0 not in idx
    v = np.random.default_rng(3).normal(size=N * N).astype(np.float32)
    dev = lambda a, t=torch.float32: torch.as_tensor(a, dtype=t, device="cuda")
    h = inrct.mlp_desc(spec, inrct.FP32, None)
    assert not torch.isfinite(inrct.inr_eval_grid(h, dev(theta), N)[0])
    val, g = inrct.inr_virtual_loss(h, dev(theta), N, dev(idx, torch.int32), dev(v), 1.0)
    assert torch.isfinite(g).all() and torch.isfinite(val).all()
    extra = np.flatnonzero(near.reshape(-1) & ~np.isin(np.arange(N * N), idx))[: -k % 64].astype(np.int32)
    v[extra] = 0.0
    val2, g2 = inrct.inr_virtual_loss(h, dev(theta), N, dev(np.r_[idx, extra], torch.int32), dev(v), 1.0)
    assert rel(g.cpu().numpy(), g2.cpu().numpy()) <= 1e-5 and abs(val.item() - val2.item()) <= 1e-5 * abs(val2.item())


@pytest.mark.parametrize("vals", [(1.0, 2.0 ** -28, 2.0 ** -52, 2.0 ** -29), (2.0 ** 40, 1.0, 2.0 ** -12, -2.0 ** 40),
                                  (-1.0, 2.0 ** -26 + 2.0 ** -49, 2.0 ** -51, 2.0 ** -27)])
def test_gradient_sums_keep_the_bits_of_fp64(vals):
    """Partial sums whose total takes 53 bits: the output bias gradient is their FP64 sum exactly (one per block, as
    above; one thread adds them)."""
    spec, k = synth.ArchSpec("siren", 2, 64, 2, omega0=30.0), 1500
    theta = synth.init_theta(spec, 2).astype(np.float32)
    v = np.zeros(211 * 211, np.float32)
    v[[0, k // 4, k // 2, k - 1]] = np.asarray(vals, np.float32)
    dev = lambda a, t=torch.float32: torch.as_tensor(a, dtype=t, device="cuda")
    g = inrct.inr_weighted_vjp(inrct.mlp_desc(spec, inrct.FP32, None), dev(theta), 211,
                               dev(np.arange(k, dtype=np.int32), torch.int32), dev(v), 1.0)
    assert g[-1].item() == np.asarray(vals, np.float32).astype(np.float64).sum()


# one large term among small ones that a long chain of FP32 additions would lose, each below half an ulp of the sum
@pytest.mark.parametrize("W", [64, 128, 256])
@pytest.mark.parametrize("N", [16, 256])  # 4 and 8 points per thread
def test_output_sums_are_short(W, N):
    """All activations 1: f is the sum of the output weights, in at most 14 roundings of values below 2 (a tree over
    32 lanes and 8 warps), and an output weight's gradient the sum of the point weights, at most 18 (a sixteenth of
    64 points, then pairs) per block of points."""
    spec = synth.ArchSpec("ffn", 2, W, 1, n_feat=32, sigma=1.0)
    B = synth.fourier_matrix(32, 2, 1.0, 1).astype(np.float32)
    dev = lambda a, t=torch.float32: torch.as_tensor(a, dtype=t, device="cuda")
    h = inrct.mlp_desc(spec, inrct.FP32, B)
    small = np.float32(1.5 * 2.0 ** -25)
    for big in (0, 5, W - 1):
        theta = np.zeros(spec.p, np.float32)
        theta[64 * W:64 * W + W] = 1.0        # hidden biases
        theta[64 * W + W:64 * W + 2 * W] = small
        theta[64 * W + W + big] = 1.0
        f = inrct.inr_eval_grid(h, dev(theta), N).double().cpu().numpy()
        want = 1.0 + (W - 1) * float(small)
        assert np.abs(f - want).max() <= 14 * 2.0 ** -24
    k = min(N * N, 16384)
    v = np.zeros(N * N, np.float32)
    v[:64] = small
    v[3] = 1.0
    g = inrct.inr_weighted_vjp(h, dev(theta), N, dev(np.arange(k), torch.int32), dev(v), 1.0).cpu().numpy()
    assert np.abs(g[64 * W + W:] - (1.0 + 63 * float(small))).max() <= 18 * 2.0 ** -24


@pytest.mark.parametrize("W,runs", [(64, 608), (256, 38)])
@pytest.mark.parametrize("L", [3, 9])
def test_weight_gradient_sums_of_deep_networks(W, L, runs):
    """The last hidden layer's weight gradient with all activations 1 is the sum of the point weights.  One of them is
    1, the others below half an ulp of it and lost in the same FP32 run: runs of at most 1 / `runs` of the points,
    in whole slabs of 16, however many layers share the launch."""
    spec, n = synth.ArchSpec("ffn", 2, W, L, n_feat=32, sigma=1.0), 1 << 16
    B = synth.fourier_matrix(32, 2, 1.0, 1).astype(np.float32)
    dev = lambda a, t=torch.float32: torch.as_tensor(a, dtype=t, device="cuda")
    theta = np.zeros(spec.p, np.float32)
    theta[64 * W:65 * W] = 1.0
    for l in range(1, L):  # zero weights, biases 1
        theta[65 * W + l * W * (W + 1) - W:65 * W + l * W * (W + 1)] = 1.0
    theta[-W - 1:-1] = 1.0
    small = np.float32(1.5 * 2.0 ** -25)
    v = np.full(n, small, np.float32)
    v[n // 2 + 5] = 1.0
    g = inrct.inr_weighted_vjp(inrct.mlp_desc(spec, inrct.FP32, B), dev(theta), 256, dev(np.arange(n), torch.int32), dev(v), 1.0)
    dW = g[-W - 1 - W * (W + 1):-W - 1 - W].cpu().numpy()
    run = -(-(-(-n // runs)) // 16) * 16
    assert np.abs(dW - (1.0 + (n - 1) * float(small))).max() <= (run + 32) * 2.0 ** -24


@pytest.mark.parametrize("W,F", [(64, 1777), (256, 1681)])
def test_widest_input(W, F):
    """Fourier features up to the last column the path takes."""
    spec, N, k = synth.ArchSpec("ffn", 2, W, 2, n_feat=F, sigma=2.0), 40, 77
    theta = synth.init_theta(spec, 2).astype(np.float32)
    B = synth.fourier_matrix(F, 2, spec.sigma, 1).astype(np.float32)
    oa = O.Arch(spec.kind, 2, W, 2, F, B.astype(np.float64), spec.omega0)
    idx = np.sort(np.random.default_rng(3).choice(N * N, size=k, replace=False)).astype(np.int32)
    X, t64 = O.grid_coords(2, N, idx), theta.astype(np.float64)
    v = np.random.default_rng(4).normal(size=N * N).astype(np.float32)
    _, _, zs, _ = O.forward(oa, t64, X, keep=True)
    for z in zs[:-1]:  # points whose ReLU decisions are unique in FP32
        v[idx[(np.abs(z) < 1e-6 * np.sqrt((z ** 2).mean())).any(axis=1)]] = 0.0
    dev = lambda a, t=torch.float32: torch.as_tensor(a, dtype=t, device="cuda")
    h = inrct.mlp_desc(spec, inrct.FP32, B)
    g = inrct.inr_weighted_vjp(h, dev(theta), N, dev(idx, torch.int32), dev(v), 1.0).cpu().numpy()
    assert rel(g, O.vjp(oa, t64, X, v.astype(np.float64)[idx])) <= 1e-4
    assert rel(inrct.inr_eval_grid(h, dev(theta), N).cpu().numpy()[idx], O.forward(oa, t64, X)) <= 1e-5
