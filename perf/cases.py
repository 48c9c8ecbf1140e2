"""Performance cases: the calls that a user of this package makes, over the sizes and options they are made with.

Every case goes through the public entry points of `paper_2507_19131_b200.binding` (and `calibrate` for the
post-training flow): a single Two-Branch block, a backbone on a token map, a backbone on an image (stem and output
norms inside the call), and the min/max calibration of a backbone.  Shapes, bit widths, ratios and input distributions
are those of the workloads in `synth.py`, plus classification-sized images and ragged photograph sizes.  Weights and
feature maps are drawn on the GPU from the seed; all results are whole-tensor outputs of the call."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_19131_b200 import binding as mq
from paper_2507_19131_b200 import calibrate, synth

F32 = np.float32
MODELS = {"swin_t": synth.SWIN_T, "swin_s": synth.SWIN_S, "swin_b": synth.SWIN_B,
          "stage1_pair": dict(dims=[96], depths=[2], heads=[3])}
SITES = calibrate.SITES


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, model="", dim=0, shift=0, batch=1, height=0, width=0, image=False, w_bits=4,
             hi_bits=8, lo_bits=4, low_ratio=0.5, prune_ratio=0.0, byte_codes_min_dim=0, values="blobs", stream="own")
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one W-MSA block on a 56x56 map (64 windows), selection outputs wanted, torch's default stream
        _case("block_56x56x96", "block", dim=96, height=56, width=56, w_bits=8, values="outliers", stream="default"),
        # one SW-MSA block of a deep stage of a detector-sized image, three window classes, default stream
        _case("block_50x84x384_pruned", "block", dim=384, shift=3, height=50, width=84, prune_ratio=0.2, stream="default"),
        # classification-sized image through stem, backbone and output norms: latency and launch count
        _case("swin_t_image_224", "backbone", model="swin_t", height=224, width=224, image=True, byte_codes_min_dim=384),
        # the same size as token maps in a batch
        _case("swin_t_224_batch16", "backbone", model="swin_t", batch=16, height=56, width=56, byte_codes_min_dim=384),
        # stage-1 block pair (W-MSA, SW-MSA with mask) on heavy-tailed activations, W8, torch's default stream
        _case("stage1_pair_200x334_batch2", "backbone", model="stage1_pair", batch=2, height=200, width=334, w_bits=8,
              low_ratio=0.3, values="student_t", stream="default"),
        # the benchmark's workload: Swin-T at 800x1333 (token map behind the stem), half of the windows low-bit
        _case("swin_t_800x1333", "backbone", model="swin_t", height=200, width=334, byte_codes_min_dim=384),
        # image in, normed stage maps out, every block bit-packed (the library's default storage), a quarter low-bit
        _case("swin_t_image_800x1333", "backbone", model="swin_t", height=800, width=1333, image=True, low_ratio=0.25),
        # a small batch of ragged photographs, mostly low-bit with some windows pruned, torch's default stream
        _case("swin_t_image_427x640_batch3", "backbone", model="swin_t", batch=3, height=427, width=640, image=True,
              low_ratio=0.75, prune_ratio=0.1, stream="default"),
        # Swin-S at 1024x1024, A4 high / A2 low, a fifth of the windows pruned
        _case("swin_s_1024_batch4", "backbone", model="swin_s", batch=4, height=256, width=256, hi_bits=4, lo_bits=2,
              prune_ratio=0.2, byte_codes_min_dim=384, values="normal"),
        # Swin-B at 1536x1536, W8: the largest forward
        _case("swin_b_1536_batch2", "backbone", model="swin_b", batch=2, height=384, width=384, w_bits=8,
              byte_codes_min_dim=384),
        # post-training flow: one 800x1333 sample (host array) sets the quantizers of a Swin-T backbone
        _case("calibrate_swin_t_800x1333", "calibrate", model="swin_t", height=200, width=334),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: kind, model, sizes (log-uniform, ragged), ratios, bit widths, storage and stream at random."""
    kind = rng.choice(["block", "block", "backbone", "backbone", "backbone", "backbone", "backbone", "calibrate"])
    bits = rng.choice([(8, 4), (8, 4), (8, 4), (4, 2)])
    c = _case("", kind, w_bits=rng.choice([4, 8]), hi_bits=bits[0], lo_bits=bits[1],
              low_ratio=round(rng.uniform(0.0, 0.8), 2), prune_ratio=rng.choice([0.0, 0.0, round(rng.uniform(0.05, 0.3), 2)]),
              byte_codes_min_dim=rng.choice([0, 384]), values=rng.choice(["blobs", "normal", "student_t", "outliers"]),
              stream=rng.choice(["own", "default"]))
    del c["name"]
    aspect = math.exp(rng.uniform(-0.5, 0.5))
    if kind == "block":
        c["dim"] = rng.choice([96, 128, 192, 256, 384, 512, 768, 1024])
        c["shift"] = rng.choice([0, 3])
        # tokens of a map of that width in a backbone: 56^2 ... 400^2 tokens at 96 channels, a quarter per doubling
        side = _log_int(rng, 56, 400) / (c["dim"] / 96.0)
        c["batch"] = rng.choice([1, 1, 2, 4])
        side = max(side, 7.0)
    elif kind == "calibrate":
        c["model"] = "swin_t"
        side = _log_int(rng, 56, 240)
        aspect = math.exp(rng.uniform(-0.25, 0.25))
    else:
        c["model"] = rng.choice(["swin_t", "swin_t", "swin_t", "swin_s", "swin_b", "stage1_pair"])
        c["image"] = c["model"] != "stage1_pair" and rng.random() < 0.5
        # tokens of the whole batch: a 224x224 image ... nearly two 1536x1536 images
        tokens = _log_int(rng, 56 * 56, 1.8 * 384 * 384)
        c["batch"] = max(1, min(16, _log_int(rng, 1, 16), tokens // (56 * 56)))
        # neither side of the map beyond 384 tokens
        side = min(math.sqrt(tokens / c["batch"]), 384.0 / math.sqrt(max(aspect, 1.0 / aspect)))
    c["height"], c["width"] = max(7, int(side / math.sqrt(aspect))), max(7, int(side * math.sqrt(aspect)))
    if c["image"]:
        c["height"], c["width"] = 4 * c["height"] - rng.randrange(4), 4 * c["width"] - rng.randrange(4)
    return c


# ---- what a user's program has in hand before the call ----------------------------------------------------------------
_ctx = None
_own_stream = None


def _context():
    """One library context and one stream of its own per process, as a serving program keeps them."""
    global _ctx, _own_stream
    if _ctx is None:
        _ctx = mq.Context(0)
        _own_stream = torch.cuda.Stream()
    return _ctx


class _Draw:
    """Numbers from the seed: large arrays on the GPU, short vectors with numpy."""

    def __init__(self, seed):
        self.np = np.random.default_rng(seed)
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda")

    def linear(self, out_f, in_f, bits):
        """N(0, 0.02^2) weights quantized per output channel (max-abs / qmax)."""
        w = self.normal(out_f, in_f) * 0.02
        qmax = (1 << (bits - 1)) - 1
        scale = w.abs().amax(dim=1) / qmax
        codes = torch.clamp(torch.round(w / scale[:, None]), -qmax, qmax).to(torch.int8)
        return synth.Linear(codes.cpu().numpy(), scale.cpu().numpy(), bits)

    def block(self, dim, shift, w_bits, hi_bits, lo_bits, score_range=6.0):
        hi = synth.make_branch(self.np, dim, 4 * dim, hi_bits)
        lo = synth.make_branch(self.np, dim, 4 * dim, lo_bits, biases=[hi.b_qkv, hi.b_proj, hi.b_fc1, hi.b_fc2])
        heads = dim // 32
        relpos = (2.0 * self.np.standard_normal((169, heads), dtype=F32)).astype(F32)
        return synth.Block(dim, heads, 7, shift, 4 * dim, self.linear(3 * dim, dim, w_bits), self.linear(dim, dim, w_bits),
                           self.linear(4 * dim, dim, w_bits), self.linear(dim, 4 * dim, w_bits), relpos, hi, lo,
                           float(F32(127.0 / score_range)))

    def vec(self, n, mean):
        return (mean + 0.02 * self.np.standard_normal(n, dtype=F32)).astype(F32)

    def backbone(self, model, w_bits, hi_bits, lo_bits):
        m = MODELS[model]
        blocks, merges = [], []
        for s, (c, depth) in enumerate(zip(m["dims"], m["depths"])):
            rng_s = 6.0
            if s > 0:
                p = m["dims"][s - 1]
                rng_s = 6.0 * 0.02 * math.sqrt(4 * p)
                merges.append(synth.Merge(self.vec(4 * p, 1.0), self.vec(4 * p, 0.0), synth.make_aq(-6.0, 6.0, hi_bits),
                                          self.linear(2 * p, 4 * p, w_bits)))
            for i in range(depth):
                blocks.append(self.block(c, 0 if i % 2 == 0 else 3, w_bits, hi_bits, lo_bits, rng_s))
        return synth.Backbone(list(m["dims"]), list(m["depths"]), list(m["heads"]), blocks, merges)

    def bumps(self, batch, h, w):
        """3-8 Gaussian bumps per image in [0, 1]: foreground objects on a quiet background."""
        yy = torch.arange(h, device="cuda", dtype=torch.float32)[:, None]
        xx = torch.arange(w, device="cuda", dtype=torch.float32)[None, :]
        out = torch.zeros((batch, h, w), device="cuda")
        for b in range(batch):
            for _ in range(int(self.np.integers(3, 9))):
                cy, cx = self.np.uniform(0, h), self.np.uniform(0, w)
                sy, sx = self.np.uniform(0.03, 0.10) * h, self.np.uniform(0.03, 0.10) * w
                out[b] = torch.maximum(out[b], torch.exp(-0.5 * (((yy - cy) / sy) ** 2 + ((xx - cx) / sx) ** 2)))
        return out

    def feature_map(self, values, b, h, w, c):
        x = self.normal(b, h, w, c)
        if values == "blobs":
            return x * 0.3 * (1.0 + 3.0 * self.bumps(b, h, w))[..., None]
        if values == "student_t":
            # three degrees of freedom: N / sqrt(chi2_3 / 3)
            chi = sum(self.normal(b, h, w, c).square_() for _ in range(3))
            return x / torch.sqrt(chi / 3.0)
        if values == "outliers":
            x[..., torch.from_numpy(self.np.choice(c, size=4, replace=False)).cuda()] *= 20.0
        return x

    def image(self, b, h, w):
        """Standardised pixels: smooth bumps plus noise."""
        return self.normal(b, h, w, 3) * 0.5 + (2.0 * self.bumps(b, h, w) - 0.5)[..., None]


def prepare(case, seed):
    ctx = _context()
    d = _Draw(seed)
    st = dict(case=case, ctx=ctx, stream=_own_stream if case["stream"] == "own" else None)
    b, h, w = case["batch"], case["height"], case["width"]
    packed = case["byte_codes_min_dim"] == 0
    if case["kind"] == "block":
        dim = case["dim"]
        blk = d.block(dim, case["shift"], case["w_bits"], case["hi_bits"], case["lo_bits"])
        st["block"] = mq.DeviceBlock(ctx, blk, byte_codes=not packed and dim >= case["byte_codes_min_dim"])
        st["x"] = d.feature_map(case["values"], b, h, w, dim).contiguous()
    elif case["kind"] == "calibrate":
        st["backbone"] = d.backbone(case["model"], case["w_bits"], case["hi_bits"], case["lo_bits"])
        st["x"] = d.feature_map(case["values"], b, h, w, st["backbone"].dims[0]).cpu().numpy()
    else:
        bb = d.backbone(case["model"], case["w_bits"], case["hi_bits"], case["lo_bits"])
        embed = norms = None
        if case["image"]:
            c0 = bb.dims[0]
            embed = synth.Embed(d.vec(c0, 1.0), d.vec(c0, 0.0), d.vec(c0, 0.0), synth.make_aq(-3.0, 3.0, 8),
                                d.linear(c0, 48, 8))
            norms = [(d.vec(c, 1.0), d.vec(c, 0.0)) for c in bb.dims]
            st["x"] = d.image(b, h, w).contiguous()
        else:
            st["x"] = d.feature_map(case["values"], b, h, w, bb.dims[0]).contiguous()
        st["backbone"] = mq.DeviceBackbone(ctx, bb, b, h, w, embed=embed, norms=norms,
                                           byte_codes_min_dim=None if packed else case["byte_codes_min_dim"])
        st["low"] = [case["low_ratio"]] * st["backbone"].npairs
        st["prune"] = [case["prune_ratio"]] * st["backbone"].npairs if case["prune_ratio"] > 0 else None
    return st


def _call(st):
    case = st["case"]
    if case["kind"] == "block":
        r = mq.block_forward(st["ctx"], st["block"], st["x"], case["low_ratio"], case["prune_ratio"], selection=True)
        return dict(y=r.y, cls=r.cls, order=r.order, scores=r.scores)
    if case["kind"] == "calibrate":
        bb = calibrate.calibrate_backbone(st["ctx"], st["backbone"], st["x"])
        aqs = [getattr(br, s) for blk in bb.blocks for br in (blk.hi, blk.lo) for s in SITES] + [m.aq for m in bb.merges]
        return dict(scale=np.array([q.scale for q in aqs], F32), zero_point=np.array([q.zp for q in aqs], np.int32),
                    score_inv_scale=np.array([blk.score_inv_scale for blk in bb.blocks], F32))
    return mq.backbone_forward(st["ctx"], st["backbone"], st["x"], st["low"], st["prune"])


def run(state):
    if state["stream"] is None:
        return _call(state)
    with torch.cuda.stream(state["stream"]):
        return _call(state)


# ---- what a pass cannot do without --------------------------------------------------------------------------------------
def _block_work(dim, b, h, w, low, prune):
    """(operations, parameter bytes) of one block: integer products of the rows of all windows that are not pruned."""
    n_hi, n_lo, _ = mq.branch_counts(h, w, low, prune)
    rows = 49 * b * (n_hi + n_lo)
    return rows * (2 * 12 * dim * dim + 4 * 49 * dim), 12 * dim * dim + 4 * (2 * 9 * dim + 2 * 9 * dim + 169 * dim // 32)


def work(case):
    b, h, w = case["batch"], case["height"], case["width"]
    low, prune = case["low_ratio"], case["prune_ratio"]
    if case["kind"] == "block":
        ops, par = _block_work(case["dim"], b, h, w, low, prune)
        windows = b * (-(-h // 7)) * (-(-w // 7))
        return {"bytes": 2 * 4 * b * h * w * case["dim"] + par + windows * (1 + 4 + 8), "flops": ops}
    m = MODELS[case["model"]]
    calib = case["kind"] == "calibrate"
    ops, byt = 0, 0
    if case["image"]:
        byt += 4 * b * h * w * 3
        h, w = (h + 3) // 4, (w + 3) // 4
        ops += 2 * b * h * w * 48 * m["dims"][0]
        byt += 48 * m["dims"][0]
    else:
        byt += 4 * b * h * w * m["dims"][0]
    for s, (c, depth) in enumerate(zip(m["dims"], m["depths"])):
        if s > 0:
            p = m["dims"][s - 1]
            h, w = (h + 1) // 2, (w + 1) // 2
            ops += 2 * b * h * w * 4 * p * c
            byt += 4 * p * c + 4 * (8 * p + c)
        for _ in range(depth):
            o, par = _block_work(c, b, h, w, 0.0 if calib else low, 0.0 if calib else prune)
            ops += 2 * o if calib else o             # calibration runs every block through both branches
            byt += par
        if not calib:
            byt += 4 * b * h * w * c                 # the stage's output map
    return {"bytes": byt, "flops": ops}


def tolerance(case):
    """The forward is defined to the bit (integer products, and binary32 steps in a fixed order because every one of them
    decides codes downstream).  Calibration: binary32 extremes of sums in binary64."""
    return {"rel": 1e-6, "max": 1e-5} if case["kind"] == "calibrate" else "exact"
