"""The FP32 decoder kernels at the edges of their tiles: forward tiles of 64
and 128 points, backward blocks of 32 rows dealt to the CTAs in ranges of up
to four at a time, and the per-material sums' row lists, against the FP64
oracle.  Bounds: an output is a chain of three 64- to 71-term FP32 sums, each
within 71 roundings of 2^-24 of its terms' magnitudes (4e-6), and the head's
log-space terms; a gradient adds sums over the batch: 1e-5 relative L2 for
the outputs, 1e-4 for the gradients, where a ReLU within rounding of zero may
fall either way."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import mlp
from paper_2406_17782_gb300.api import GBuffer

pytestmark = pytest.mark.gpu


def rel(a, b):
    b = np.asarray(b, np.float64)
    return np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-30)


def backward_either_way(p, cache, dy, got):
    """The oracle's (parameter gradient, input gradient).  A pre-activation
    within the rounding of its FP32 sum (a few 2^-24 of its terms' magnitudes)
    has no certain side of the ReLU, and either gives a valid gradient: the
    side is taken that `got` agrees with better."""
    grad, dx = mlp.decoder_backward(p, cache, dy)
    ins = {"a1": ("x", "W1"), "a2": ("h1", "W2"), "a3": ("h2", "W3")}
    for name, (src, w) in ins.items():
        mags = np.abs(cache[src]) @ np.abs(p[w]).T
        for r, u in np.argwhere(np.abs(cache[name]) < 4 * 2.0 ** -24 * mags):
            other = {k: v.copy() if k == name else v for k, v in cache.items()}
            other[name][r, u] = -other[name][r, u]
            g2, dx2 = mlp.decoder_backward(p, other, dy)
            if rel(got, mlp.pack(g2, mlp.DEC_SHAPES)) < rel(got, mlp.pack(grad, mlp.DEC_SHAPES)):
                cache, grad, dx = other, g2, dx2
    return grad, dx


def setup(n, n_mat, seed):
    g = W.training_queries(n, n_mat, stream=f"fp32-tiles-{n}")
    dec = W.decoder_init(seed)
    lat = W.random_latents(n_mat, seed)
    return g, dec, lat


@pytest.mark.parametrize("n,n_mat", [(1, 1), (63, 3), (64, 3), (65, 3), (129, 5), (19456, 4), (38912, 4), (38913, 9)])
def test_forward_tiles(fab, n, n_mat):
    g, dec, lat = setup(n, n_mat, 21)
    y = fab.decoder_forward(GBuffer.from_numpy(g), torch.from_numpy(lat).cuda(), torch.from_numpy(dec).cuda())
    fab.sync_status()
    idx = np.unique(np.concatenate([np.arange(min(n, 200)), np.arange(max(0, n - 200), n)]))
    sub = W.subset(g, idx)
    want = mlp.decoder_forward(mlp.unpack(dec, mlp.DEC_SHAPES), mlp.decoder_inputs(lat, sub["material"], sub))
    assert rel(y.cpu().numpy()[idx], want) < 1e-5


@pytest.mark.parametrize("n,n_mat", [(1, 1), (31, 2), (32, 2), (33, 2), (127, 3), (129, 1), (4864, 7), (4865, 1), (9733, 300)])
def test_backward_blocks(fab, n, n_mat):
    """(4864 rows are one block on each of 152 CTAs; one material makes every
    row match, so that the row lists fill up and are emptied on the way.)"""
    g, dec, lat = setup(n, n_mat, 22)
    dy = np.random.default_rng(n).standard_normal((n, 4)).astype(np.float32)
    ddec, dlat = fab.decoder_backward(GBuffer.from_numpy(g), torch.from_numpy(lat).cuda(), torch.from_numpy(dec).cuda(),
                                      torch.from_numpy(dy).cuda())
    fab.sync_status()
    p = mlp.unpack(dec, mlp.DEC_SHAPES)
    _, cache = mlp.decoder_forward(p, mlp.decoder_inputs(lat, g["material"], g), keep=True)
    want, dx = backward_either_way(p, cache, dy.astype(np.float64), ddec.cpu().numpy())
    want_lat = np.zeros((n_mat, 32))
    np.add.at(want_lat, g["material"].astype(np.int64), dx[:, :32])
    assert rel(ddec.cpu().numpy(), mlp.pack(want, mlp.DEC_SHAPES)) < 1e-4
    assert rel(dlat.cpu().numpy(), want_lat) < 1e-4


@pytest.mark.parametrize("offset", [1, 3, 4, 7])
def test_unaligned_arrays(fab, offset):
    """Materials, latents and parameters that start off a 16-byte boundary give
    the same results as aligned copies, bit for bit in the forward pass."""
    n, n_mat = 2777, 11
    g, dec, lat = setup(n + offset, n_mat, 23)
    full = GBuffer.from_numpy(g)
    view = GBuffer(*(getattr(full, k)[offset:] for k in ("u", "v", "radius", "wi", "wo", "material")))
    copy = GBuffer(*(getattr(full, k)[offset:].clone() for k in ("u", "v", "radius", "wi", "wo", "material")))

    def off(a):
        buf = torch.zeros(a.size + offset, device="cuda")
        buf[offset:] = torch.from_numpy(a).cuda().flatten()
        return buf[offset:].view(a.shape)

    dy = torch.randn((n, 4), generator=torch.Generator("cuda").manual_seed(5), device="cuda")
    args = [(copy, torch.from_numpy(lat).cuda(), torch.from_numpy(dec).cuda()), (view, off(lat), off(dec))]
    y = [fab.decoder_forward(*a) for a in args]
    d = [fab.decoder_backward(*a, dy) for a in args]
    fab.sync_status()
    assert torch.equal(y[0], y[1])
    assert torch.equal(d[0][0], d[1][0])
    assert rel(d[1][1].cpu().numpy(), d[0][1].cpu().numpy()) < 1e-5


def test_bad_material_rows_do_not_contribute(fab):
    n, n_mat = 200, 4
    g, dec, lat = setup(n, n_mat, 24)
    bad = {k: v.copy() for k, v in g.items()}
    bad["material"][[5, 70, 199]] = 1000
    dy = np.random.default_rng(1).standard_normal((n, 4)).astype(np.float32)
    keep = np.delete(np.arange(n), [5, 70, 199])
    from paper_2406_17782_gb300 import FabricError
    z, p = torch.from_numpy(lat).cuda(), torch.from_numpy(dec).cuda()
    got = fab.decoder_backward(GBuffer.from_numpy(bad), z, p, torch.from_numpy(dy).cuda())
    with pytest.raises(FabricError):
        fab.sync_status()
    want = fab.decoder_backward(GBuffer.from_numpy(W.subset(g, keep)), z, p, torch.from_numpy(dy[keep]).cuda())
    fab.sync_status()
    for a, b in zip(got, want):
        assert rel(a.cpu().numpy(), b.cpu().numpy()) < 1e-5


@pytest.mark.parametrize("offset", [0, 1])
def test_latent_rows_no_id_can_name(fab, offset):
    """Ids have 16 bits, latent tables may have more rows: those past 65 536
    get zero gradients, the others theirs, whether the ids can be read as
    16-byte words or not."""
    n, n_lat = 4001, 65540
    g, dec, _ = setup(n + offset, 8, 25)
    full = GBuffer.from_numpy(g)
    full.material[::2] = -1                       # 65 535, the last id there is
    view = GBuffer(*(getattr(full, k)[offset:] for k in ("u", "v", "radius", "wi", "wo", "material")))
    lat = torch.randn((n_lat, 32), generator=torch.Generator("cuda").manual_seed(6), device="cuda")
    dy = torch.randn((n, 4), generator=torch.Generator("cuda").manual_seed(7), device="cuda")
    _, dlat = fab.decoder_backward(view, lat, torch.from_numpy(dec).cuda(), dy)
    fab.sync_status()
    assert not dlat[65536:].any() and not dlat[8:65535].any()
    assert dlat[65535].any() and all(dlat[m].any() for m in range(8))
