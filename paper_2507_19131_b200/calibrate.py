"""Min/max calibration of the activation quantizers (the step in front of the path in the post-training flow).

MixA-Q Section 4.3: one calibration sample; the FULL feature map (all windows, not the windows a branch will later
see) initialises the step sizes of both the high- and the low-precision branch, so that the two branches share their
calibration data and differ only in bit width.

Everything is computed by the library (mixaq_calibrate_block / mixaq_calibrate_merge run the floating-point block with
min/max observers at the seven quantizer sites; mixaq_aq_from_range turns a range into a quantizer).  This module only
walks the backbone, marshals the arguments and copies the results into a parameter object the forward consumes.
It needs the CUDA library and a device, like the rest of the package.
"""
from __future__ import annotations

import copy
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from . import binding as mq
from . import synth

SITES = ("qkv_in", "q", "k", "v", "proj_in", "fc1_in", "fc2_in")


def _aq(lo: float, hi: float, bits: int) -> synth.AQ:
    scale, inv, zp = mq.aq_from_range(lo, hi, bits)
    return synth.AQ(bits, scale, inv, zp)


_upload_streams = {}


def _upload_stream(device) -> torch.cuda.Stream:
    """One upload stream per device: the caching allocator keeps memory per stream, a new stream per call would not reuse it."""
    if device not in _upload_streams:
        _upload_streams[device] = torch.cuda.Stream(device)
    return _upload_streams[device]


def calibrate_backbone(ctx: "mq.Context", bb, x0: np.ndarray):
    """Returns a deep copy of `bb` whose activation quantizers (both branches of every block, every merge) and score
    steps come from the calibration sample x0 [B,H,W,C0].  Every block is calibrated on the full feature map, once
    through each branch's own LayerNorm parameters and biases; the sample is propagated through the floating-point
    model with the high branch's."""
    dev = mq._Dev(ctx.device)
    # The copy of the result object and the upload of the next block's parameters run on helper threads while the
    # library calibrates the current block (its calls wait for the device without holding the interpreter).  Swin-T on a
    # 200 x 334 map: 10 ms of uploads beside 12 ms of kernels.
    side = _upload_stream(ctx.device)

    def upload(make, params):
        with torch.cuda.device(ctx.device), torch.cuda.stream(side):
            struct = make(dev, params)
            side.synchronize()
        return struct

    with ThreadPoolExecutor(1) as pool, ThreadPoolExecutor(1) as copier:
        copied = copier.submit(copy.deepcopy, bb)
        jobs, k = [], 0                              # parameters in the order of use: merge of a stage, its blocks
        for s, d in enumerate(bb.depths):
            if s > 0:
                jobs.append((mq.fill_merge_struct, bb.merges[s - 1]))
            jobs += [(mq.fill_block_struct, b) for b in bb.blocks[k:k + d]]
            k += d
        structs = [pool.submit(upload, *j) for j in jobs]
        x = torch.from_numpy(np.ascontiguousarray(x0, np.float32)).to(ctx.device)
        found, step = [], 0
        for s, d in enumerate(bb.depths):
            if s > 0:
                x, rng = mq.calibrate_merge(ctx, structs[step].result(), x)
                found.append(rng)
                step += 1
            for _ in range(d):
                bs = structs[step].result()
                y_next, rng_hi = mq.calibrate_block(ctx, bs, 0, x)
                _, rng_lo = mq.calibrate_block(ctx, bs, 1, x)
                found.append((rng_hi, rng_lo))
                x = y_next
                step += 1
        out = copied.result()
    it, k = iter(found), 0
    for s, d in enumerate(out.depths):
        if s > 0:
            m = out.merges[s - 1]
            m.aq = _aq(*next(it), m.aq.bits)
        for blk in out.blocks[k:k + d]:
            for br, rng in zip((blk.hi, blk.lo), next(it)):
                for site in SITES:
                    setattr(br, site, _aq(rng[site][0], rng[site][1], br.bits))
                if br is blk.hi:
                    # the int8 score codes span the block's input map
                    blk.score_inv_scale = float(np.float32(127.0 / max(1e-12, max(abs(rng["x_in"][0]), abs(rng["x_in"][1])))))
        k += d
    return out
