"""The work that users of this framework have it do, as cases that can be timed.

A renderer edits a material and redraws a preview, draws whole frames with
the neural decoder (one G-buffer, many ragged segments at once, or buffers in
host memory), renders supersampled ground truth and measures its error
against it; a trainer generates data with the reference kernel and trains the
two networks on it, by the library's own steps or through torch.autograd.
Inputs follow the distributions of those workloads (a 1080p frame of eight
weaves, a batched 4K draw, Table-2 training queries, batches of 65 536), drawn
on the GPU from the seed.  ``exact`` restates what each call computes in 64
bits with plain torch.
"""
from __future__ import annotations

import math
import os
import struct
import tempfile
import zlib

import numpy as np
import torch

from paper_2406_17782_gb300.api import DecoderFunction, EncoderFunction, Fabric, GBuffer

DEV = "cuda"
MATERIAL = np.dtype([("pattern", np.int32), ("twist_deg", np.float32), ("incl_deg", np.float32),
                     ("alpha", np.float32, (2,)), ("beta", np.float32, (2,)), ("kd", np.float32, (2, 3)),
                     ("ks", np.float32, (2, 3)), ("gap", np.float32), ("w_blend", np.float32)])
DEC = [(64, 71), (64, 64), (64, 64), (4, 64)]              # (out, in) of each layer
ENC = [(128, 22), (128, 128), (32, 128)]
PAPER_ENC = [(128, 22), (128, 128), (64, 128)]
LR = 3e-4                                                   # the middle of the training schedule 3e-3 .. 1e-5
PAPER_LR = 1e-4
RESUME_STEP = 20000


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # a material edit and the redraw of a 64 x 64 preview: encoder, latent fold and packing, decoder
        dict(name="edit_preview", kind="edit", n=4096, n_mat=1, prec="fp16", comps=False),
        # the frame loop: a 1920 x 1080 G-buffer of eight fabrics, operands prepared once per edit
        dict(name="frame_1080p", kind="frame", n=2073600, n_mat=8, prec="fp16", comps=False),
        # 4K view with interleaved materials and 256 ragged tiles of four views, one persistent launch
        dict(name="batched_4k", kind="plan", n=8294400, segments=256, n_mat=8, prec="bf16", comps=False),
        # the same 1080p frame from and to page-locked host memory
        dict(name="host_frame", kind="host", n=2073600, n_mat=8, prec="fp16", chunk=0),
        # the supersampled reference of the 1080p frame
        dict(name="reference_1080p", kind="reference", n=2073600, n_mat=8, nx=16, ny=16, wide=False, vis=False),
        # training data at the paper's 2048 samples a query, with the inter-yarn visibility model
        dict(name="data_visibility", kind="reference", n=8190, n_mat=256, nx=64, ny=32, wide=True, vis=True),
        # one training step in the default precision
        dict(name="train_fp32", kind="train", n=65536, n_mat=256, prec="fp32", steps=1, loss="eq11"),
        # a stretch of an epoch on the tensor cores, in one native call
        dict(name="train_bf16_epoch", kind="train", n=65536, n_mat=256, prec="bf16", steps=8, loss="rendered"),
        # a user's own training loop: both networks through torch.autograd, a ragged batch
        dict(name="autograd_step", kind="autograd", n=10007, n_mat=37),
        # 1080p frame by the paper's decoder structure, also with the four components
        dict(name="paper_frame_w128", kind="paper", n=2073600, n_mat=8, width=128, prec="fp16", comps=True),
        # one training step of the paper's structure
        dict(name="paper_train_w128", kind="paper_train", n=65536, n_mat=256, width=128, ablation="full",
             loss="rendered"),
        # error of a lit 1080p RGB frame against its ground truth
        dict(name="frame_error", kind="error", n=2073600 * 3, weighted=True),
    ]


def _log_int(rng, lo, hi):
    return int(math.floor(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["edit", "frame", "plan", "host", "reference", "reference", "train", "train", "autograd",
                       "paper", "paper_train", "error"])
    if kind == "edit":
        return dict(kind=kind, n=_log_int(rng, 1, 65536), n_mat=rng.randint(1, 32),
                    prec=rng.choice(["fp16", "bf16", "fp8"]), comps=rng.random() < 0.5)
    if kind == "frame":
        prec = rng.choice(["fp16", "fp16", "bf16", "fp8", "fp32"])
        return dict(kind=kind, n=_log_int(rng, 16384, 262144 if prec == "fp32" else 2073600), n_mat=rng.randint(1, 32),
                    prec=prec, comps=rng.random() < 0.5)
    if kind == "plan":
        return dict(kind=kind, n=_log_int(rng, 16384, 8294400), segments=rng.randint(0, 256), n_mat=rng.randint(1, 32),
                    prec=rng.choice(["fp16", "bf16", "fp8"]), comps=rng.random() < 0.5)
    if kind == "host":
        return dict(kind=kind, n=_log_int(rng, 4096, 2073600), n_mat=rng.randint(1, 32),
                    prec=rng.choice(["fp16", "bf16"]), chunk=rng.choice([0, 0, 100000]))
    if kind == "reference":
        vis = rng.random() < 0.4
        nx, ny = rng.choice([(1, 1), (2, 2), (4, 4), (5, 3), (8, 8), (16, 16), (32, 32), (64, 32)])
        most = (1 << 23 if vis else 2073600 * 256) // (nx * ny)
        return dict(kind=kind, n=_log_int(rng, max(1, min(2073600, most) // 64), min(2073600, most)),
                    n_mat=rng.randint(1, 256), nx=nx, ny=ny, wide=rng.random() < 0.5, vis=vis)
    if kind == "train":
        prec = rng.choice(["fp32", "bf16"])
        return dict(kind=kind, n=_log_int(rng, 512, 65536), n_mat=_log_int(rng, 8, 465), prec=prec,
                    steps=1 if prec == "fp32" else rng.randint(1, 8), loss=rng.choice(["eq11", "rendered"]))
    if kind == "autograd":
        return dict(kind=kind, n=_log_int(rng, 100, 65536), n_mat=rng.randint(1, 256))
    if kind == "paper":
        return dict(kind=kind, n=_log_int(rng, 4096, 2073600), n_mat=rng.randint(1, 32), width=rng.choice([64, 128]),
                    prec=rng.choice(["fp16", "bf16"]), comps=rng.random() < 0.5)
    if kind == "paper_train":
        return dict(kind=kind, n=_log_int(rng, 512, 65536), n_mat=_log_int(rng, 8, 465), width=rng.choice([64, 128]),
                    ablation=rng.choice(["full", "full", "no_oneblob", "no_fusion"]),
                    loss=rng.choice(["eq11", "rendered"]))
    return dict(kind="error", n=_log_int(rng, 1000, 1 << 24), weighted=rng.random() < 0.5)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _rng(seed):
    return np.random.default_rng([seed, 17]), torch.Generator(DEV).manual_seed(1000003 * seed + 29)


def _uniform(gen, shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, device=DEV)


def _materials(r, n, table2=False):
    """n materials over the weaves; frame-like, or every other one from the paper's Table 2."""
    m = np.zeros(n, MATERIAL)
    m["pattern"] = np.arange(n) % (12 if table2 else 8)
    m["twist_deg"] = r.uniform(0.0, 30.0, n)
    m["incl_deg"] = 30.0
    m["alpha"] = r.uniform(0.1, 0.4, (n, 2))
    m["beta"] = 1.0
    if table2:
        odd = np.arange(n) % 2 == 1
        m["twist_deg"] = np.where(odd, r.choice([-30.0, 0.0, 30.0], n), m["twist_deg"])
        m["incl_deg"] = np.where(odd, r.uniform(15.0, 45.0, n), m["incl_deg"])
        m["alpha"] = np.where(odd[:, None], r.uniform(0.1, 1.0, (n, 2)), m["alpha"])
        m["beta"] = np.where(odd[:, None], r.uniform(0.0, 2.0, (n, 2)), m["beta"])
    m["kd"] = r.uniform(0.2, 0.8, (n, 2, 3))
    m["ks"] = r.uniform(0.2, 0.8, (n, 2, 3))
    m["gap"] = 0.2
    m["w_blend"] = 0.5
    return m


def _directions(gen, n):
    z = _uniform(gen, n)
    phi = _uniform(gen, n, 0.0, 2.0 * math.pi)
    s = torch.sqrt((1.0 - z * z).clamp_min(0.0))
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], 1)


def _gbuffer(gen, n, material, wide=False):
    """Frame footprints (half side log-uniform in [1e-4, 1e-1] repeats), or half of them Table 2's (up to five)."""
    r = torch.exp(_uniform(gen, n, math.log(1e-4), math.log(1e-1)))
    if wide:
        side = torch.where(_uniform(gen, n) < 0.5, _uniform(gen, n, 1.0, 5.0), _uniform(gen, n))
        r = torch.where(_uniform(gen, n) < 0.5, r, (0.5 * side).clamp_min(1e-6))
    return GBuffer(u=_uniform(gen, n, 0.0, 50.0), v=_uniform(gen, n, 0.0, 50.0), radius=r, wi=_directions(gen, n),
                   wo=_directions(gen, n), material=material.to(torch.int16))


def _slice(g, a, b):
    return GBuffer(*(getattr(g, k)[a:b] for k in ("u", "v", "radius", "wi", "wo", "material")))


def _bands(n, n_mat):
    """Materials in vertical bands of a frame 1920 points wide."""
    x = torch.arange(n, device=DEV) % 1920
    return (x * n_mat // 1920).clamp_max(n_mat - 1)


def _any_material(gen, n, n_mat):
    return torch.randint(0, n_mat, (n,), generator=gen, device=DEV)


def _weights(r, layers, he=True):
    out = []
    for o, i in layers:
        b = math.sqrt(6.0 / i) if he else 1.0 / math.sqrt(i)
        out += [r.uniform(-b, b, o * i), r.uniform(-1.0 / math.sqrt(i), 1.0 / math.sqrt(i), o)]
    return np.concatenate(out).astype(np.float32)


def _targets(gen, n):
    """Components as the reference gives them: diffuse below about one, specular heavy-tailed, some of them zero."""
    c = torch.exp(torch.randn((n, 2), generator=gen, device=DEV) - 2.0)
    s = torch.exp(1.5 * torch.randn((n, 2), generator=gen, device=DEV) - 3.0)
    t = torch.cat([c, s], 1)
    return t * (_uniform(gen, (n, 4)) > 0.1)


def _paper_layers(width, ablation):
    if ablation == "no_fusion":
        return [(width, 93)] + [(width, width)] * 5 + [(4, width)]
    k0 = 64 + (3 if ablation == "no_oneblob" else 24)
    return [(width, k0), (width, width), (width, width + 5)] + [(width, width)] * 3 + [(4, width)]


class _Pointer:
    """A device array of the library as torch.as_tensor takes it; the tensor keeps this object, and so the context
    that owns the memory."""

    def __init__(self, fab, ptr, n):
        self.fab = fab
        self.__cuda_array_interface__ = dict(shape=(n,), typestr="<f4", data=(ptr, False), version=3, strides=None)


def _moments(r, n):
    """Adam moments in the middle of a training run."""
    s = 10.0 ** r.uniform(-4.0, -2.5, n)
    return (0.3 * s * r.standard_normal(n)).astype(np.float32), (s * s).astype(np.float32)


def _resume(fab, dec, enc, m, v):
    """Loads a checkpoint file of these parameters and moments, as a resumed run does."""
    body = b"FABCKPT1" + struct.pack("<IIIq", 1, dec.size, enc.size, RESUME_STEP)
    body += dec.tobytes() + enc.tobytes() + m.tobytes() + v.tobytes()
    fd, path = tempfile.mkstemp(suffix=".ckpt")
    with os.fdopen(fd, "wb") as f:
        f.write(body + struct.pack("<I", zlib.crc32(body)))
    fab.checkpoint_load(path)
    os.unlink(path)


def _inputs(case, seed):
    """Everything of a case that is drawn: used by prepare and by exact."""
    r, gen = _rng(seed)
    kind, n = case["kind"], case["n"]
    d = dict(case)
    if kind == "error":
        d["a"] = _uniform(gen, n)
        d["b"] = d["a"] + 0.02 * torch.randn(n, generator=gen, device=DEV)
        d["w"] = _directions(gen, n // 3 + 1) if case["weighted"] else None
        return d
    n_mat = case["n_mat"]
    training = kind in ("train", "paper_train", "autograd")
    d["mats"] = _materials(r, n_mat, table2=training or case.get("vis", False) or n_mat > 8)
    if kind in ("paper", "paper_train"):
        d["dec"] = _weights(r, _paper_layers(case["width"], case.get("ablation", "full")), he=not training)
        d["enc"] = _weights(r, PAPER_ENC, he=False)
    else:
        d["dec"] = _weights(r, DEC, he=not training)
        d["enc"] = _weights(r, ENC, he=False)
    if kind == "train":
        d["m"], d["v"] = _moments(r, d["dec"].size + d["enc"].size)
    if kind == "plan":
        # one buffer holds the view and the ragged tiles, each from a multiple of 128 points on; the case itself
        # gives the tiles' sizes, the seed what is in them
        q = np.random.default_rng([n, case["segments"]])
        sizes = [n] + [int(s) for s in np.floor(np.exp(q.uniform(math.log(256), math.log(65536), case["segments"])))]
        starts = np.concatenate([[0], np.cumsum([-(-s // 128) * 128 for s in sizes])])
        d["segs"] = [(int(a), int(a) + s) for a, s in zip(starts, sizes)]
        total = int(starts[-1])
        tile = torch.arange(n, device=DEV)
        tile = (tile // 3840 // 16) * 240 + (tile % 3840) // 16
        d["g"] = _gbuffer(gen, total, torch.cat([((tile * 0x9E3779B1) >> 7) % n_mat,
                                                 _any_material(gen, total - n, n_mat)]))
    elif training:
        total = n * case.get("steps", 1)
        d["g"] = _gbuffer(gen, total, _any_material(gen, total, n_mat), wide=True)
        d["target"] = _targets(gen, total)
    else:
        banded = kind in ("frame", "paper", "host") or (kind == "reference" and not case["wide"])
        d["g"] = _gbuffer(gen, n, _bands(n, n_mat) if banded else _any_material(gen, n, n_mat),
                          wide=case.get("wide", False))
    if kind == "autograd":
        d["feats"] = _features(d["mats"]).float()
        d["dy"] = torch.randn((n, 4), generator=gen, device=DEV) / n
    if kind in ("frame", "plan", "host"):
        d["latents"] = torch.randn((n_mat, 32), generator=gen, device=DEV)
    if kind == "paper":
        d["latents"] = torch.randn((n_mat, 64), generator=gen, device=DEV)
    return d


# --------------------------------------------------------------------------
# what is run
# --------------------------------------------------------------------------
def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    fab = d["fab"] = Fabric()
    if kind == "error":
        return d
    if kind in ("train", "paper_train"):
        fab.set_train_materials(d["mats"])
        fab.set_train_loss(case["loss"])
    if kind in ("edit", "frame", "plan", "host", "reference", "paper"):
        fab.set_materials(d["mats"])
    if kind in ("paper", "paper_train"):
        fab.paper_set_params(case["width"], d["dec"], d["enc"], case.get("ablation", "full"))
    elif kind == "train":
        fab.set_train_precision(case["prec"])
        _resume(fab, d["dec"], d["enc"], d["m"], d["v"])
        pd, pe = fab.param_tensors()
        d["theta"] = [torch.as_tensor(_Pointer(fab, p, a.size), device=DEV)
                      for p, a in ((pd, d["dec"]), (pe, d["enc"]))]
        d["losses"] = torch.zeros(case["steps"], dtype=torch.float64, device=DEV)
    elif kind in ("edit", "frame", "plan", "host"):
        fab.set_params(d["dec"], d["enc"])
    if kind in ("frame", "host", "paper"):
        d["rgb"] = torch.empty((case["n"], 3), device=DEV)
        d["comps_out"] = torch.empty((case["n"], 4), device=DEV) if case.get("comps") else None
    if kind in ("frame", "plan", "host"):
        fab.prepare_neural(d["latents"], case["prec"])
    if kind == "host":
        g = d["g"]
        d["g"] = GBuffer(*(getattr(g, k).cpu().pin_memory() for k in ("u", "v", "radius", "wi", "wo", "material")))
        d["rgb"] = torch.empty((case["n"], 3)).pin_memory()
    if kind == "paper":
        fab.paper_prepare(d["latents"], case["prec"])
    if kind == "plan":
        d["rgb"] = torch.zeros((d["g"].n, 3), device=DEV)
        d["comps_out"] = torch.zeros((d["g"].n, 4), device=DEV) if case["comps"] else None
        d["plan"] = fab.plan([(_slice(d["g"], a, b), d["rgb"][a:b], d["comps_out"][a:b] if case["comps"] else None)
                              for a, b in d["segs"]])
    if kind == "reference":
        fab.set_visibility(case["vis"])
    if kind == "autograd":
        d["p_dec"] = torch.tensor(d["dec"], device=DEV, requires_grad=True)
        d["p_enc"] = torch.tensor(d["enc"], device=DEV, requires_grad=True)
    return d


def run(s):
    kind, fab = s["kind"], s["fab"]
    if kind == "edit":
        z = fab.encode_params(s["mats"])
        rgb, comps = fab.shade_neural(s["g"], z, s["prec"], comps=s["comps"])
        return {"latents": z, "rgb": rgb, "comps": comps}
    if kind == "frame":
        rgb, comps = fab.shade_neural_prepared(s["g"], s["prec"], out_rgb=s["rgb"], out_comps=s["comps_out"])
        return {"rgb": rgb, "comps": comps}
    if kind == "plan":
        s["plan"].shade(s["prec"])
        return {"rgb": s["rgb"], "comps": s["comps_out"]}
    if kind == "host":
        rgb, _ = fab.shade_neural_host(s["g"], s["prec"], out_rgb=s["rgb"], chunk_points=s["chunk"])
        return rgb
    if kind == "reference":
        rgb, comps = fab.shade_reference(s["g"], s["nx"], s["ny"], 0xDA7A, comps=True)
        return {"rgb": rgb, "comps": comps}
    if kind == "train":
        if s["steps"] == 1:
            fab.train_step(s["g"], s["target"], LR, loss_out=s["losses"])
        else:
            fab.train_steps(s["g"], s["target"], s["n"], s["steps"], RESUME_STEP, 3 * RESUME_STEP, 3e-4, 1e-5,
                            loss_out=s["losses"])
        return {"loss": s["losses"], "dec": s["theta"][0], "enc": s["theta"][1]}
    if kind == "autograd":
        s["p_dec"].grad = s["p_enc"].grad = None
        z = EncoderFunction.apply(s["p_enc"], s["feats"], fab)
        y = DecoderFunction.apply(s["p_dec"], z, fab, s["g"])
        y.backward(s["dy"])
        return {"y": y, "dec": s["p_dec"].grad, "enc": s["p_enc"].grad}
    if kind == "paper":
        rgb, comps = fab.paper_shade_prepared(s["g"], s["prec"], out_rgb=s["rgb"], out_comps=s["comps_out"])
        return {"rgb": rgb, "comps": comps}
    if kind == "paper_train":
        loss = fab.paper_train_step(s["g"], s["target"], PAPER_LR)
        return {"loss": loss, "grad": fab.paper_gradient()}
    if s["weighted"]:
        return fab.error_stats(s["a"], s["b"], weights=s["w"].view(-1)[2:], group=3, weight_stride=3)
    return fab.error_stats(s["a"], s["b"])


def work(case):
    kind, n = case["kind"], case["n"]
    n_mat = case.get("n_mat", 0)
    flops = lambda layers: 2 * sum(o * i for o, i in layers)  # noqa: E731
    params = lambda layers: 4 * sum(o * i + o for o, i in layers)  # noqa: E731
    out = 28 if case.get("comps") else 12
    folded = [(64, 39)] + DEC[1:]
    if kind == "error":
        return dict(bytes=8 * n + (12 * (n // 3) if case["weighted"] else 0), flops=6 * n)
    if kind == "edit":
        return dict(bytes=n * (38 + out) + params(DEC) + params(ENC) + n_mat * (84 + 128),
                    flops=n * flops(folded) + n_mat * flops(ENC))
    if kind in ("frame", "host"):
        return dict(bytes=n * (38 + out), flops=n * flops(folded))
    if kind == "plan":
        n += int(case["segments"] * (65536 - 256) / math.log(256))
        return dict(bytes=n * (38 + out), flops=n * flops(folded))
    if kind == "reference":
        # about 150 operations of Eq. 1-5 a sample (frame, distribution, masking, sums)
        return dict(bytes=n * (38 + 28), flops=n * case["nx"] * case["ny"] * 150)
    if kind == "train":
        p = params(DEC) + params(ENC)
        return dict(bytes=case["steps"] * (n * 54 + 6 * p),
                    flops=case["steps"] * (3 * n * flops(DEC) + 3 * n_mat * flops(ENC)))
    if kind == "autograd":
        return dict(bytes=n * (38 + 32) + 2 * (params(DEC) + params(ENC)), flops=3 * n * flops(DEC))
    layers = _paper_layers(case["width"], case.get("ablation", "full"))
    if kind == "paper":
        return dict(bytes=n * (38 + out), flops=n * flops([(case["width"], 24)] + layers[1:]))
    p = params(layers) + params(PAPER_ENC)
    return dict(bytes=n * 54 + 7 * p, flops=3 * n * flops(layers) + 3 * n_mat * flops(PAPER_ENC))


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------
def _unflat(flat, layers):
    out, at = [], 0
    for o, i in layers:
        out += [flat[at:at + o * i].view(o, i), flat[at + o * i:at + o * i + o]]
        at += o * i + o
    return out


def _octaves(u):
    f = u - u.floor()
    out = []
    for k in range(8):
        fk = f * 2.0 ** k
        a = 2.0 * math.pi * (fk - fk.floor())
        out += [torch.sin(a), torch.cos(a)]
    return torch.stack(out, 1)


def _query(g):
    c0, c1 = 0.5 * math.log(1e-5), 0.5 * math.log(1e3)
    ell = (torch.log(g.radius.double().clamp_min(2.0 ** -20)) - c0) / c1
    return torch.cat([_octaves(g.u.double()), _octaves(g.v.double()), ell[:, None], g.wi.double(), g.wo.double()], 1)


def _index(g):
    return g.material.long() & 0xFFFF


def _decode(dec, z, g):
    w = _unflat(dec, DEC)
    h = torch.cat([z[_index(g)], _query(g)], 1)
    for k in (0, 2, 4):
        h = torch.relu(h @ w[k].T + w[k + 1])
    return h @ w[6].T + w[7]


def _features(mats):
    f = np.zeros((len(mats), 22))
    f[np.arange(len(mats)), mats["pattern"]] = 1.0
    for k, a in enumerate([mats["twist_deg"].astype(np.float64) / 30.0, mats["incl_deg"].astype(np.float64) / 45.0,
                           mats["alpha"][:, 0], mats["beta"][:, 0], mats["alpha"][:, 1], mats["beta"][:, 1]]):
        f[:, 16 + k] = a
    return torch.tensor(f, device=DEV)


def _lrelu(x):
    return torch.where(x > 0, x, 0.01 * x)


def _encode(enc, feats, layers):
    w = _unflat(enc, layers)
    h1 = _lrelu(feats @ w[0].T + w[1])
    h2 = _lrelu(h1 @ w[2].T + w[3] + h1)
    return h2 @ w[4].T + w[5]


def _onto_rgb(comps, mats, idx):
    kd = torch.tensor(mats["kd"].astype(np.float64), device=DEV)[idx]
    ks = torch.tensor(mats["ks"].astype(np.float64), device=DEV)[idx]
    c = comps[:, :, None]
    return kd[:, 0] * c[:, 0] + kd[:, 1] * c[:, 1] + ks[:, 0] * c[:, 2] + ks[:, 1] * c[:, 3]


def _shade(net, mats, g, comps):
    """Pieces of the G-buffer through `net`, the inverse of Eq. 9 and Eq. 8."""
    rgbs, cs = [], []
    for s in range(0, g.n, 1 << 18):
        p = _slice(g, s, s + (1 << 18))
        y = net(p)
        c = torch.cat([y[:, :2].clamp_min(0.0), (torch.expm1(y[:, 2:]) / 100.0).clamp_min(0.0)], 1)
        rgbs.append(_onto_rgb(c, mats, _index(p)))
        cs.append(c)
    return torch.cat(rgbs), torch.cat(cs) if comps else None


def _blob(s, periodic):
    d = s[:, None] - (torch.arange(8, device=DEV, dtype=torch.float64) + 0.5) / 8.0
    if not periodic:
        return torch.exp(-32.0 * d * d)
    d = d - d.round()
    return sum(torch.exp(-32.0 * (d + m) ** 2) for m in range(-2, 3))


def _paper_net(dec, z, g, width, ablation):
    w = _unflat(dec, _paper_layers(width, ablation))
    lin = lambda k, x: x @ w[2 * k].T + w[2 * k + 1]  # noqa: E731
    u, v = g.u.double(), g.v.double()
    u, v = u - u.floor(), v - v.floor()
    t = torch.log(g.radius.double().clamp_min(2.0 ** -20) / 1e-4) / math.log(2.5e4)
    blob = torch.stack([u, v, t], 1) if ablation == "no_oneblob" else \
        torch.cat([_blob(u, True), _blob(v, True), _blob(t, False)], 1)
    ang = torch.cat([g.wi.double(), g.wo.double()[:, :2]], 1)
    x = [z[_index(g)], blob]
    h = _lrelu(lin(1, _lrelu(lin(0, torch.cat(x + [ang] if ablation == "no_fusion" else x, 1)))))
    k1 = _lrelu(lin(2, h if ablation == "no_fusion" else torch.cat([h, ang], 1)))
    k3 = _lrelu(lin(4, _lrelu(lin(3, k1))) + k1)
    return lin(6, _lrelu(lin(5, k3)))


def _loss(y, target, wz, mode):
    if mode == "eq11":
        t = torch.cat([target[:, :2], torch.log(100.0 * target[:, 2:] + 1.0)], 1)
        lam = torch.tensor([0.1, 0.1, 0.4, 0.4], dtype=torch.float64, device=DEV)
        return (lam * ((y - t) ** 2).mean(0)).sum()
    c = torch.cat([y[:, :2], torch.expm1(y[:, 2:].clamp_max(12.0)) / 100.0], 1)
    return (((c - target) * wz.clamp_min(0.0)[:, None]) ** 2).sum() / len(y)


def _exact_train(d):
    n, steps, nd = d["n"], d["steps"], d["dec"].size
    theta = torch.tensor(np.concatenate([d["dec"], d["enc"]]), dtype=torch.float64, device=DEV)
    m, v = (torch.tensor(d[k], dtype=torch.float64, device=DEV) for k in ("m", "v"))
    feats, losses = _features(d["mats"]), []
    for k in range(steps):
        p = theta.clone().requires_grad_(True)
        g, t = _slice(d["g"], k * n, (k + 1) * n), d["target"][k * n:(k + 1) * n].double()
        loss = _loss(_decode(p[:nd], _encode(p[nd:], feats, ENC), g), t, g.wi[:, 2].double(), d["loss"])
        grad, = torch.autograd.grad(loss, p)
        lr = LR if steps == 1 else 1e-5 + (3e-4 - 1e-5) * 0.5 * (1.0 + math.cos(
            math.pi * (RESUME_STEP + k) / (3 * RESUME_STEP)))
        at = RESUME_STEP + k + 1
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
        theta = theta - lr * (m / (1 - 0.9 ** at)) / (torch.sqrt(v / (1 - 0.999 ** at)) + 1e-8)
        losses.append(loss.detach())
    return {"loss": torch.stack(losses), "dec": theta[:nd], "enc": theta[nd:]}


# the twelve weaves: rows, columns, and where the warp lies on top at row i, column j
_WEAVES = [
    (2, 2, lambda i, j: (i + j) % 2 == 0), (3, 3, lambda i, j: (i - j) % 3 < 2), (4, 4, lambda i, j: (i - j) % 4 < 3),
    (5, 5, lambda i, j: (i - 2 * j) % 5 != 0), (5, 5, lambda i, j: (i - 3 * j) % 5 == 0),
    (4, 4, lambda i, j: (i // 2 + j // 2) % 2 == 0),
    (4, 8, lambda i, j: (i - j) % 4 < 2 if j < 4 else (i + j) % 4 < 2), (4, 2, lambda i, j: (i // 2 + j) % 2 == 0),
    (5, 5, lambda i, j: (i - j) % 5 < 4), (8, 8, lambda i, j: (i - j) % 8 < 7),
    (8, 8, lambda i, j: (i - 3 * j) % 8 == 0), (10, 5, lambda i, j: (i // 2 - 3 * j) % 5 == 0)]


def _weave_tables():
    """Per weave [16 * 16] cells: warp on top, length of the float and the cell's place in it."""
    top, length, place = (np.zeros((12, 256), np.int64) for _ in range(3))
    for w, (rows, cols, on) in enumerate(_WEAVES):
        bit = np.array([[bool(on(i, j)) for j in range(cols)] for i in range(rows)])
        for i in range(rows):
            for j in range(cols):
                line, at = (bit[:, j], i) if bit[i, j] else (bit[i], j)
                k = len(line)
                back = 0
                while back + 1 < k and line[(at - back - 1) % k] == bit[i, j]:
                    back += 1
                fwd = 0
                while fwd + 1 < k and line[(at + fwd + 1) % k] == bit[i, j]:
                    fwd += 1
                whole = bool((line == bit[i, j]).all())
                top[w, 16 * i + j] = bit[i, j]
                length[w, 16 * i + j] = k if whole else back + fwd + 1
                place[w, 16 * i + j] = at if whole else back
    return [torch.tensor(a, device=DEV) for a in (top, length, place)]


def _shift(z, k):
    """Logical shift right of 64-bit words kept as int64."""
    return (z >> k) & ((1 << (64 - k)) - 1)


def _signed(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _mix(z):
    z = (z ^ _shift(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shift(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ _shift(z, 31)


def _offsets(k, xi, n, r):
    """((k + xi) (2 / n) - 1) r, each step rounded to 32 bits, then to 0.32 fixed point."""
    t = (k.float() + xi) * torch.tensor(np.float32(2.0) / np.float32(n), device=DEV)
    return torch.round((t - 1.0) * r * 4294967296.0).long()


def _exact_reference(d):
    """The stratified footprint integral of Eq. 3-5 over the same samples."""
    g, mats, nx, ny = d["g"], d["mats"], d["nx"], d["ny"]
    top, length, place = _weave_tables()
    rec = lambda k: torch.tensor(mats[k].astype(np.float64), device=DEV)  # noqa: E731
    pattern = torch.tensor(mats["pattern"].astype(np.int64), device=DEV)
    size = torch.tensor([[w[0], w[1]] for w in _WEAVES], device=DEV)
    psi, incl, alpha, beta = rec("twist_deg") * math.pi / 180, rec("incl_deg") * math.pi / 180, rec("alpha"), rec("beta")
    gap, blend = rec("gap"), rec("w_blend")
    k = torch.arange(nx * ny, device=DEV)
    out = torch.empty((g.n, 4), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 22) // (nx * ny))
    low = (1 << 32) - 1
    for s in range(0, g.n, step):
        e = min(g.n, s + step)
        m = _index(g)[s:e]
        r32 = g.radius[s:e, None]
        h = _mix(0xDA7A + torch.arange(s + 1, e + 1, device=DEV) * _signed(0x9E3779B97F4A7C15))
        h = _mix(h[:, None] + k)
        pos = []
        for c, kk, n, x in ((g.u[s:e], k % nx, nx, _shift(h, 40)), (g.v[s:e], k // nx, ny, _shift(h, 16) & 0xFFFFFF)):
            centre = torch.round((c - c.floor()) * 4294967296.0).long()
            pos.append((centre[:, None] + _offsets(kk, x.float() * 2.0 ** -24, n, r32)) & low)
        pat = pattern[m][:, None]
        wu, wv = pos[0] * size[pat, 1], pos[1] * size[pat, 0]
        cell = 16 * (wv >> 32) + (wu >> 32)
        su, sv = wu & low, wv & low
        warp = top[pat, cell] == 1
        s_top, s_along = torch.where(warp, su, sv), torch.where(warp, sv, su)
        gf = (0.5 * gap[m] * 4294967296.0).floor().long()[:, None]
        body = (s_top >= gf) & (s_top <= low - gf)
        gm = 1.0 - gap[m][:, None]
        x = torch.where(body, (2.0 * s_top.double() * 2.0 ** -32 - 1.0) / gm,
                        ((2.0 * s_along.double() * 2.0 ** -32 - 1.0) / gm).clamp(-1.0, 1.0))
        along = (place[pat, cell] + s_along.double() * 2.0 ** -32) / length[pat, cell].clamp_min(1)
        theta = torch.where(body, incl[m][:, None] * (1.0 - 2.0 * along), torch.zeros_like(x))
        is_warp = warp == body                                  # the yarn that shows
        pick = lambda t: torch.where(is_warp, t[m, 0][:, None], t[m, 1][:, None])  # noqa: E731
        hc = -pick(beta) * (math.pi / 2) * torch.sin(math.pi * x / 2)
        ha = torch.tan(theta)
        # axes: a along the yarn, c across it; vectors as (a, c, z) components
        inv = torch.rsqrt(ha * ha + hc * hc + 1.0)
        na, nc, nz = -ha * inv, -hc * inv, inv
        it = torch.rsqrt(1.0 + ha * ha)
        ta, tz = it, ha * it
        # n x t0 in world axes (x, y, z): the warp runs along y, the weft along x
        n_x, n_y = torch.where(is_warp, nc, na), torch.where(is_warp, na, nc)
        zero = torch.zeros_like(ta)
        t_x, t_y = torch.where(is_warp, zero, ta), torch.where(is_warp, ta, zero)
        cp, sp = torch.cos(psi[m])[:, None], torch.sin(psi[m])[:, None]
        p_x = cp * t_x + sp * (n_y * tz - nz * t_y)
        p_y = cp * t_y + sp * (nz * t_x - n_x * tz)
        p_z = cp * tz + sp * (n_x * t_y - n_y * t_x)
        wi, wo = g.wi[s:e].double(), g.wo[s:e].double()
        hv = wi + wo
        hv = hv / hv.norm(dim=1, keepdim=True)
        dot = lambda w, a, b, c: w[:, 0:1] * a + w[:, 1:2] * b + w[:, 2:3] * c  # noqa: E731
        ci, co = dot(wi, n_x, n_y, nz).clamp_min(0.0), dot(wo, n_x, n_y, nz).clamp_min(0.0)
        ti, to, tau = (dot(w, p_x, p_y, p_z) for w in (wi, wo, hv))
        al = pick(alpha)
        bl = blend[m][:, None]
        fd = bl * ci / (math.pi * wi[:, 2:3].clamp_min(1e-3)) + (1.0 - bl) / math.pi
        diff = fd * ci * co / nz
        q = 1.0 - tau * tau + (tau / al) ** 2
        X = torch.sqrt((1.0 - (1.0 - al * al) * ti * ti).clamp_min(0.0)) * co + \
            torch.sqrt((1.0 - (1.0 - al * al) * to * to).clamp_min(0.0)) * ci
        lit = (ci > 0) & (co > 0)
        cc = torch.where(lit, ci * co, torch.ones_like(ci))
        X = torch.where(lit, X, torch.ones_like(X))
        spec = torch.where(lit, cc * -torch.expm1(-2.0 * X / cc) / X / (math.pi * al * q * q) / 4.0 / nz, zero)
        area = (co / nz).sum(1)
        sums = torch.stack([(diff * is_warp).sum(1), (diff * ~is_warp).sum(1), (spec * is_warp).sum(1),
                            (spec * ~is_warp).sum(1)], 1)
        out[s:e] = torch.where(area[:, None] > 0, sums / torch.where(area > 0, area, torch.ones_like(area))[:, None],
                               torch.zeros_like(sums))
    return {"rgb": _onto_rgb(out, mats, _index(g)), "comps": out}


def exact(case, seed):
    kind = case["kind"]
    if case.get("prec") == "fp8" or case.get("vis"):
        # E4M3 operands are a tenth off by design; a march's decisions have no value between their two
        return None
    d = _inputs(case, seed)
    if kind == "error":
        w = d["w"][:, 2].double().repeat_interleave(3)[:d["n"]] if case["weighted"] else 1.0
        e, b = w * (d["a"].double() - d["b"].double()), w * d["b"].double()
        return torch.stack([(e * e).sum(), (b * b).sum(), e.abs().max()])
    if kind == "reference":
        return _exact_reference(d)
    if kind == "train":
        return _exact_train(d)
    f64 = lambda a: torch.tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
    dec, enc = f64(d["dec"]), f64(d["enc"])
    if kind == "autograd":
        dec.requires_grad_(True)
        enc.requires_grad_(True)
        y = _decode(dec, _encode(enc, d["feats"].double(), ENC), d["g"])
        gd, ge = torch.autograd.grad(y, (dec, enc), d["dy"].double())
        return {"y": y.detach(), "dec": gd, "enc": ge}
    if kind == "paper_train":
        p = torch.cat([dec, enc]).requires_grad_(True)
        z = _encode(p[dec.numel():], _features(d["mats"]), PAPER_ENC)
        y = _paper_net(p[:dec.numel()], z, d["g"], case["width"], case["ablation"])
        loss = _loss(y, d["target"].double(), d["g"].wi[:, 2].double(), case["loss"])
        grad, = torch.autograd.grad(loss, p)
        return {"loss": loss.detach(), "grad": grad}
    if kind == "edit":
        z = _encode(enc, _features(d["mats"]), ENC)
        rgb, comps = _shade(lambda g: _decode(dec, z, g), d["mats"], d["g"], case["comps"])
        return {"latents": z, "rgb": rgb, "comps": comps}
    if kind == "paper":
        z = d["latents"].double()
        rgb, comps = _shade(lambda g: _paper_net(dec, z, g, case["width"], "full"), d["mats"], d["g"], case["comps"])
        return {"rgb": rgb, "comps": comps}
    z = d["latents"].double()
    rgb, comps = _shade(lambda g: _decode(dec, z, g), d["mats"], d["g"], case.get("comps", False))
    if kind == "plan":
        inside = torch.zeros(d["g"].n, dtype=torch.bool, device=DEV)
        for a, b in d["segs"]:
            inside[a:b] = True
        rgb, comps = (None if x is None else x * inside[:, None] for x in (rgb, comps))
    return rgb if kind == "host" else {"rgb": rgb, "comps": comps}
