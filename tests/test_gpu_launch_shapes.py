"""Every launch shape of the tensor-core decoder computes every point the
same way, so all shapes the autotuner may pick must give bit-identical
outputs: tile pipelines per CTA, CTAs per SM, and one or two warpgroups per
tile pipeline (two threads per tile row splitting the encoding and the
epilogue columns), for the single-buffer and the batched (segment table)
kernels, in every operand precision."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_2406_17782_gb300 import autotune
from paper_2406_17782_gb300.api import GBuffer

pytestmark = pytest.mark.gpu

SHAPES = autotune.DECODER_CANDIDATES


@pytest.fixture(scope="module")
def frame(fab):
    mats = W.frame_materials()
    fab.set_materials(mats)
    fab.set_params(W.decoder_init(), W.encoder_init())
    lat = torch.from_numpy(W.random_latents(len(mats))).cuda()
    # ragged: a full tile count plus a tail, several tiles per CTA at 1-4 CTAs/SM
    g = GBuffer.from_numpy(W.subset(W.frame_gbuffer(), np.arange(0, 152 * 4 * 128 * 2 + 77)))
    yield lat, g
    fab.set_launch_config(0, 0, 0, 0)


@pytest.mark.parametrize("prec", ["fp16", "bf16", "fp8"])
def test_all_launch_shapes_agree_bitwise(fab, frame, prec):
    lat, g = frame
    fab.prepare_neural(lat, prec)
    fab.set_launch_config(0, 0, 0, 0)
    want_rgb, want_c = fab.shade_neural_prepared(g, prec, comps=True)
    fab.sync_status()
    for wg, ctas, h in SHAPES:
        fab.set_launch_config(ctas, wg, 0, h)
        rgb, comps = fab.shade_neural_prepared(g, prec, comps=True)
        fab.sync_status()
        assert torch.equal(rgb, want_rgb) and torch.equal(comps, want_c), (prec, wg, ctas, h)


@pytest.mark.parametrize("h", [1, 2])
def test_batched_kernel_with_two_warpgroups_per_tile(fab, frame, h):
    lat, _ = frame
    frame_host = W.frame_gbuffer()
    segs = []
    for k, n in enumerate([5000, 1, 129, 0, 4097, 70_000]):
        host = W.subset(frame_host, np.arange(1000 * k, 1000 * k + n))
        segs.append((GBuffer.from_numpy(host), torch.full((n, 3), float("nan"), device="cuda"),
                     torch.full((n, 4), float("nan"), device="cuda")))
    fab.prepare_neural(lat, "fp16")
    fab.set_launch_config(0, 0, 0, h)
    plan = fab.plan(segs)
    plan.shade("fp16")
    fab.sync_status()
    fab.set_launch_config(0, 0, 0, 0)
    for g, rgb, comps in segs:
        if g.n == 0:
            continue
        want_rgb, want_c = fab.shade_neural_prepared(g, "fp16", comps=True)
        fab.sync_status()
        assert torch.equal(rgb, want_rgb) and torch.equal(comps, want_c)
    plan.close()


@pytest.mark.parametrize("n_mat", [1, 4, 5, 31, 32])
def test_encoder_of_records_passed_with_the_launch(fab, n_mat):
    """Few records travel with the launch, more through device memory: the
    same latents bit for bit."""
    mats = W.training_materials(8)[:64]
    fab.set_params(W.decoder_init(), W.encoder_init())
    assert torch.equal(fab.encode_params(mats[:n_mat]), fab.encode_params(mats)[:n_mat])


@pytest.mark.parametrize("prec", ["fp16", "bf16", "fp8"])
@pytest.mark.parametrize("n_mat", [1, 9, 10, 25, 26, 89])
def test_tiles_encoded_ahead(fab, n_mat, prec):
    """One thread per row encodes the next tile while a tile's products run,
    two encode each tile when it starts: the same bits at the edges of the
    tiles and of the rounds over them, and for every width of layer 1 (from
    10 materials on its operand continues in another one's columns)."""
    mats = np.resize(W.training_materials(8), n_mat)
    fab.set_materials(mats)
    fab.set_params(W.decoder_init(), W.encoder_init())
    fab.prepare_neural(torch.from_numpy(W.random_latents(n_mat)).cuda(), prec)
    wave = fab.sm_count * 4 * 128
    host = W.frame_gbuffer()
    try:
        for n in (1, 127, 129, wave - 1, wave + 1, 3 * wave + 5):
            part = W.subset(host, np.arange(n))
            part["material"] = (np.arange(n) * 7 % n_mat).astype(np.uint16)
            part["u"] = part["u"].copy()
            part["u"][::5] = np.resize(np.float32([0.0, -1e-12, 0.5, -3.25, 1e5, 0.9999999]), len(part["u"][::5]))
            g = GBuffer.from_numpy(part)
            got = []
            for h in (1, 2):
                fab.set_launch_config(0, 0, 0, h)
                got.append(fab.shade_neural_prepared(g, prec, comps=True))
                fab.sync_status()
            assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1]), n
    finally:
        fab.set_launch_config(0, 0, 0, 0)


def test_launches_of_different_shapes_back_to_back(fab, frame):
    """Each launch starts under the one before, whose CTAs are of another
    size and hold other amounts of tensor memory."""
    lat, g = frame
    fab.prepare_neural(lat, "fp16")
    want, _ = fab.shade_neural_prepared(g, "fp16")
    outs = [torch.full_like(want, float("nan")) for _ in SHAPES]
    for _ in range(20):
        for out, (wg, ctas, h) in zip(outs, SHAPES):
            fab.set_launch_config(ctas, wg, 0, h)
            fab.shade_neural_prepared(g, "fp16", out_rgb=out)
    fab.sync_status()
    fab.set_launch_config(0, 0, 0, 0)
    assert all(torch.equal(out, want) for out in outs)


@pytest.mark.parametrize("n_mat", [1, 33, 88, 89])
def test_encoder_of_records_from_device_memory(fab, n_mat):
    """Up to 89 records travel with the launch, 90 and more through device
    memory: the same latents bit for bit."""
    mats = np.resize(W.training_materials(8), 300)
    mats["twist_deg"] += np.arange(300, dtype=np.float32) / 100.0
    fab.set_params(W.decoder_init(), W.encoder_init())
    for more in (90, 300):
        assert torch.equal(fab.encode_params(mats[:n_mat]), fab.encode_params(mats[:more])[:n_mat])
