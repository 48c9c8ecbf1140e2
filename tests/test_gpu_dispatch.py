"""The size, width and value ranges between which the library chooses another kernel or another branch of one, at their
edges: each against the CPU oracle, bit for bit."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_19131_b200 import synth  # noqa: E402
from test_gpu_parity import F32, ctx, dev, mq, run_block_case  # noqa: E402,F401


@pytest.mark.parametrize("dim,H,W,bits", [(96, 312, 319, (8, 4)), (128, 270, 278, (4, 2)), (192, 221, 230, (8, 2)),
                                          (256, 194, 196, (8, 4))])
def test_streaming_layer_norm_just_above_its_threshold(orc, mq, ctx, dim, H, W, bits):
    """Ragged maps with a few windows more than the streaming kernel's lower limit; row counts that are no multiple of
    the rows of a warp, in both branches."""
    blk = synth.make_block(np.random.default_rng(dim), dim, dim // 32, 3, 4, *bits)
    run_block_case(orc, mq, ctx, blk, synth.input_student_t(dim, 1, H, W, dim), 0.35, taps=False)


@pytest.mark.parametrize("H,W", [(7, 7), (28, 56), (76, 20), (21, 70), (56, 56), (34, 90), (63, 49)])
def test_window_selection_by_window_count(orc, mq, ctx, H, W):
    """1 and 32 windows per image (one launch), 33, 30 and 63 to 65, with ties, in every order of two ratios."""
    blk = synth.make_block(np.random.default_rng(H), 32, 1, 3, 8, 8, 4)
    x = np.round(synth.input_student_t(W, 3, H, W, 32))
    for low, prune, rev in [(0.5, 0.0, False), (0.25, 0.25, True)]:
        run_block_case(orc, mq, ctx, blk, x, low, prune, reverse=rev, taps=False)


@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("H,W", [(21, 28), (56, 56)])
def test_window_selection_by_a_callers_large_energies(orc, mq, ctx, H, W, reverse):
    """A caller's energies up to 2^31: window scores beyond 2^32 whose lower halves are in another order."""
    rng = np.random.default_rng(H)
    blk, x = synth.make_block(rng, 32, 1, 3, 8, 8, 4), synth.input_student_t(W, 2, H, W, 32)
    energy = rng.integers(0, 2 ** 31, size=(2, H, W)).astype(np.int32)
    ref = orc.block_forward(blk, x, 0.5, 0.25, energy_map=energy, reverse=reverse)
    assert (ref.scores > 2 ** 32).all() and (np.argsort(ref.scores) != np.argsort(ref.scores.astype(np.int32))).any()
    got = mq.block_forward(ctx, mq.DeviceBlock(ctx, blk), dev(x), 0.5, 0.25, energy=dev(energy), reverse=reverse, selection=True)
    for name, want in (("scores", ref.scores), ("order", ref.order), ("cls", ref.cls), ("y", ref.y)):
        assert np.array_equal(getattr(got, name).cpu().numpy(), want), name


@pytest.mark.parametrize("dim,windows", [(32, (27, 28)), (32, (28, 28)), (64, (28, 28)), (96, (28, 28)), (1024, (1, 2))])
def test_gemm_tilings_around_their_limits(orc, mq, ctx, dim, windows):
    """Just fewer and just more than two row tiles per SM, tile widths 32 to 256, more accumulators than
    tiles, remainders in the last row tile of both branches."""
    blk = synth.make_block(np.random.default_rng(dim), dim, dim // 32, 0, 4, 8, 4, share_bias=False)
    x = synth.input_student_t(dim, 1, 7 * windows[0], 7 * windows[1] - 2, dim)
    run_block_case(orc, mq, ctx, blk, x, 0.55, taps=False)


@pytest.mark.parametrize("dim,H,W", [(96, 35, 42), (96, 21, 74), (384, 35, 41), (384, 28, 56)])
def test_gemm_epilogue_warps_around_their_limit(orc, mq, ctx, dim, H, W):
    """12 and 14 row tiles, with remainders in the last tile."""
    blk = synth.make_block(np.random.default_rng(dim + W), dim, dim // 32, 3, 8, 8, 4, share_bias=False)
    run_block_case(orc, mq, ctx, blk, synth.input_student_t(dim, 1, H, W, dim), 0.5, taps=False)


@pytest.mark.parametrize("bits,mult,low,prune", [((8, 4), 4, 0.9, 0.0), ((4, 2), 4, 0.0, 0.0), ((2, 2), 4, 0.5, 0.3), ((2, 2), 10, 0.5, 0.0),
                                                 ((2, 2), 12, 0.5, 0.0), ((4, 2), 4, 0.5, 1.0)])
def test_one_code_per_byte_inside_a_packed_workspace(orc, mq, ctx, bits, mult, low, prune):
    """Every row in one branch, hidden layers up to and beyond what the room of two-bit codes allows, all windows pruned; the
    taps of the same call stay bit-packed."""
    rng = np.random.default_rng(mult)
    blk = synth.make_block(rng, 64, 2, 3, 4, *bits, share_bias=False)
    blk.hidden = 64 * mult
    blk.fc1, blk.fc2 = synth.make_linear(rng, blk.hidden, 64, 4), synth.make_linear(rng, 64, blk.hidden, 4)
    for br in (blk.hi, blk.lo):
        br.b_fc1 = (0.02 * rng.standard_normal(blk.hidden)).astype(F32)
    x = synth.input_student_t(mult, 2, 20, 30, 64)
    for taps in (False, True):
        run_block_case(orc, mq, ctx, blk, x, low, prune, taps=taps)


@pytest.mark.parametrize("dim,sign", [(128, 1), (128, -1), (192, 1), (384, -1), (384, 0)])
def test_gemm_accumulators_beyond_the_bias_trick(orc, mq, ctx, dim, sign):
    """Weights of full magnitude: sums of 128 products of 255 x 127 stay below 2^22, from 192 on they may not, and the
    epilogues then convert them with integer instructions."""
    rng = np.random.default_rng(dim + sign)
    blk = synth.make_block(rng, dim, dim // 32, 3, 8, 8, 4)
    for lin in (blk.qkv, blk.proj, blk.fc1, blk.fc2):
        lin.codes[:] = 127 * (sign if sign else rng.choice([-1, 1], size=lin.codes.shape))
        lin.scale[:] = (lin.scale * F32(0.05)).astype(F32)
    run_block_case(orc, mq, ctx, blk, synth.input_blobs(dim, 1, 17, 23, dim, bg_std=0.5, gain=4.0), 0.4)


@pytest.mark.parametrize("dim", [96, 384])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_gemm_code_outputs_of_a_column_without_a_finite_step(orc, mq, ctx, dim, value):
    """One step of a q, a k, a v and an fc1 channel is no number or infinite, in columns whose sums stay below 2^22 (dim 96) and in
    columns whose sums may not: the codes are those of the contract (0 for what is no number)."""
    rng = np.random.default_rng(dim)
    blk = synth.make_block(rng, dim, dim // 32, 3, 8, 8, 4)
    for lin, channels in ((blk.qkv, (5, dim + 9, 2 * dim + 30)), (blk.fc1, (7, 3 * dim + 1))):
        lin.codes[list(channels)] = 127 * rng.choice([-1, 1], size=(len(channels), dim), p=[0.02, 0.98]).astype(np.int8)
        lin.scale[list(channels)] = value
    run_block_case(orc, mq, ctx, blk, synth.input_student_t(dim, 1, 17, 23, dim), 0.4)


@pytest.mark.parametrize("dim,bits,factor", [(96, (8, 4), 20.0), (32, (4, 2), 20.0), (128, (8, 2), 20.0), (128, (8, 4), 3000.0),
                                             (64, (4, 2), 3000.0)])
def test_gemm_code_outputs_far_beyond_their_range(orc, mq, ctx, dim, bits, factor):
    """Sums of which most lie beyond both ends of the codes: within the 16-bit patterns of the fast quantizers, and beyond
    them, where all codes come from the contract's own operations; rows that are no multiple of a warp's."""
    blk = synth.make_block(np.random.default_rng(dim), dim, dim // 32, 3, 4, *bits, share_bias=False)
    for lin in (blk.qkv, blk.fc1):
        lin.scale[:] = (lin.scale * F32(factor)).astype(F32)
    for taps in (False, True):
        run_block_case(orc, mq, ctx, blk, synth.input_student_t(dim, 1, 17, 23, dim), 0.4, taps=taps)


@pytest.mark.parametrize("pairs", [5, 10])
@pytest.mark.parametrize("own_stream", [False, True])
def test_block_graphs_follow_data_buffers_and_switch(orc, mq, pairs, own_stream):
    """Repeated block calls (recorded at the second, replayed from the third) see fresh data; more sets of buffers than
    calls are remembered, and the switch that turns the graphs off, change nothing."""
    blk = synth.make_block(np.random.default_rng(3), 64, 2, 3, 4, 8, 4)
    xs = [synth.input_blobs(s, 1, 15, 22, 64, bg_std=0.5, gain=4.0) for s in range(3)]
    want = [orc.block_forward(blk, x, 0.5, 0.25).y for x in xs]
    ctx = mq.Context(0)
    stream = torch.cuda.Stream() if own_stream else torch.cuda.default_stream()
    with torch.cuda.stream(stream):
        db = mq.DeviceBlock(ctx, blk)
        bufs = [(dev(xs[0]), torch.empty(xs[0].shape, device="cuda")) for _ in range(pairs)]
        for step in range(6):
            if step == 4:
                ctx.set_graph_cache(False)
            for xd, yd in bufs:
                xd.copy_(torch.from_numpy(xs[step % 3]))
                yd.zero_()
                mq.block_forward(ctx, db, xd, 0.5, 0.25, y=yd)
                stream.synchronize()
                assert np.array_equal(yd.cpu().numpy(), want[step % 3]), f"step {step}"
    ctx.close()


@pytest.mark.parametrize("own_stream", [False, True])
def test_output_norms_of_recorded_calls_after_eviction(orc, mq, own_stream):
    """Backbones with output norms (a branch of the graph) on 17 input buffers, one more than graphs are kept: the calls that
    displace a graph, those that are displaced and those that stay give the oracle's maps."""
    wl = synth.tiny_backbone(ratio=0.4, prune=0.2)
    rng = np.random.default_rng(31)
    norms = [((1.0 + 0.05 * rng.standard_normal(c)).astype(F32), (0.05 * rng.standard_normal(c)).astype(F32)) for c in wl.backbone.dims]
    xs = [wl.x, np.ascontiguousarray(wl.x[:, ::-1])]
    want = [[orc.layernorm(o, g, b) for o, (g, b) in zip(orc.backbone_forward(wl.backbone, x, wl.low_ratios, wl.prune_ratios), norms)]
            for x in xs]
    ctx = mq.Context(0)
    stream = torch.cuda.Stream() if own_stream else torch.cuda.default_stream()
    with torch.cuda.stream(stream):
        dbb = mq.DeviceBackbone(ctx, wl.backbone, wl.B, wl.H, wl.W, norms=norms)
        bufs = [dev(xs[0]) for _ in range(17)]

        def call(i, which):
            bufs[i].copy_(torch.from_numpy(xs[which]))
            for o in dbb.outs:
                o.zero_()
            got = mq.backbone_forward(ctx, dbb, bufs[i], wl.low_ratios, wl.prune_ratios)
            stream.synchronize()
            for st, (g, w) in enumerate(zip(got, want[which])):
                assert np.array_equal(g.cpu().numpy(), w), f"buffer {i}, stage {st}"
        for step in range(3):                                   # issued, recorded, replayed
            for i in range(16):
                call(i, step % 2)
        for step in range(24):                                  # 40 replays in all earn a further recording
            call(0, step % 2)
        for step in range(3):                                   # displaces the graph of buffer 1
            call(16, step % 2)
        for i in range(4):
            call(i, 1)
        assert ctx.device_status() == 0
    ctx.close()


def test_two_threads_share_a_context(orc, mq):
    """Blocks and backbones from two threads, each on a stream of its own, through issue, recording and replay."""
    import threading
    wl = synth.tiny_backbone(ratio=0.4, prune=0.2)
    blk = synth.make_block(np.random.default_rng(3), 64, 2, 3, 4, 8, 4)
    rng = np.random.default_rng(32)
    norms = [((1.0 + 0.05 * rng.standard_normal(c)).astype(F32), (0.05 * rng.standard_normal(c)).astype(F32)) for c in wl.backbone.dims]
    xb = [wl.x, np.ascontiguousarray(wl.x[:, ::-1])]
    xk = [synth.input_blobs(s, 1, 15, 22, 64, bg_std=0.5, gain=4.0) for s in range(2)]
    want_b = [[orc.layernorm(o, g, b) for o, (g, b) in zip(orc.backbone_forward(wl.backbone, x, wl.low_ratios, wl.prune_ratios), norms)]
              for x in xb]
    want_k = [orc.block_forward(blk, x, 0.5, 0.25).y for x in xk]
    ctx = mq.Context(0)
    failed = []

    def work(t):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                dbb, db = mq.DeviceBackbone(ctx, wl.backbone, wl.B, wl.H, wl.W, norms=norms), mq.DeviceBlock(ctx, blk)
                bufs = [(dev(xb[0]), dev(xk[0]), torch.empty(xk[0].shape, device="cuda")) for _ in range(3)]
                for step in range(15):
                    which = (step + t) % 2
                    x, k, y = bufs[step % 3]
                    x.copy_(torch.from_numpy(xb[which])), k.copy_(torch.from_numpy(xk[which])), y.zero_()
                    got = mq.backbone_forward(ctx, dbb, x, wl.low_ratios, wl.prune_ratios)
                    mq.block_forward(ctx, db, k, 0.5, 0.25, y=y)
                    stream.synchronize()
                    assert all(np.array_equal(g.cpu().numpy(), w) for g, w in zip(got, want_b[which])), f"thread {t}, step {step}"
                    assert np.array_equal(y.cpu().numpy(), want_k[which]), f"thread {t}, step {step}"
        except BaseException as e:                              # noqa: BLE001
            failed.append(e)
    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("w_bits,H,W,dim", [(8, 9, 15, 96), (6, 8, 16, 32), (2, 12, 11, 128)])
def test_calibration_products_by_weight_width(orc, mq, ctx, w_bits, H, W, dim):
    """Weights whose products are fused (2 to 6 bits) and are not (8), at row counts around a tile of 128."""
    blk = synth.make_block(np.random.default_rng(w_bits), dim, dim // 32, 3, w_bits, 8, 4)
    x = synth.input_blobs(5, 1, H, W, dim, bg_std=0.5, gain=3.0)
    params = mq._Dev(ctx.device)                                  # keeps the uploads alive
    bs = mq.fill_block_struct(params, blk)
    y, got = mq.calibrate_block(ctx, bs, 0, dev(x))
    want_y, want = orc.block_observe_fp(blk, "hi", x)
    assert np.array_equal(y.cpu().numpy(), want_y)
    for site, span in want.items():
        assert got[site] == span, site


@pytest.mark.parametrize("H,W", [(21, 22), (63, 71)])
def test_selection_outputs_at_odd_addresses(orc, mq, ctx, H, W):
    """Class, order and score buffers that are not aligned to their elements, with both selection routes (12 windows: one
    launch, 99: two), issued and as a recorded graph: as from aligned ones."""
    import ctypes as C
    blk = synth.make_block(np.random.default_rng(H), 32, 1, 3, 8, 8, 4)
    x = dev(synth.input_blobs(W, 1, H, W, 32, bg_std=0.5, gain=4.0))
    db = mq.DeviceBlock(ctx, blk)
    want = mq.block_forward(ctx, db, x, 0.4, 0.2, selection=True)
    n, y, ws = want.cls.numel(), torch.empty_like(x), db.workspace(1, H, W)
    raw = {name: torch.zeros(off + n * size + 64, dtype=torch.uint8, device="cuda")
           for name, off, size in (("cls", 3, 1), ("order", 2, 4), ("score", 4, 8))}
    sel = mq.Selection(raw["cls"].data_ptr() + 3, raw["order"].data_ptr() + 2, raw["score"].data_ptr() + 4, None, None, None)
    for _ in range(3):
        for t in raw.values():
            t.fill_(0xEE)
        ctx.check(mq.lib().mixaq_block_forward(ctx.h, C.byref(db.s), mq._ptr(x), mq._ptr(y), 1, H, W, C.c_float(0.4), C.c_float(0.2), None,
                                               C.byref(sel), mq._ptr(ws), C.c_size_t(ws.numel()), None, mq._stream_ptr()))
        for name, off, ref in (("cls", 3, want.cls), ("order", 2, want.order), ("score", 4, want.scores)):
            got = raw[name].cpu().numpy()
            end = off + ref.numel() * ref.element_size()
            assert got[off:end].tobytes() == ref.cpu().numpy().tobytes(), name
            assert (got[:off] == 0xEE).all() and (got[end:] == 0xEE).all(), name
        assert torch.equal(y, want.y)


def observe_merge(mq, ctx, m, x, N):
    """mixaq_calibrate_merge with any number of output channels (the binding allocates 2 * dim)."""
    B, H, W, _ = x.shape
    params, xd = mq._Dev(ctx.device), dev(x)
    ms, r = mq.fill_merge_struct(params, m), mq.RangeS()
    y = torch.empty((B, (H + 1) // 2, (W + 1) // 2, N), device="cuda")
    ws = torch.empty(mq.lib().mixaq_calibrate_merge_workspace_bytes(ctypes.byref(ms), B, H, W), dtype=torch.uint8, device="cuda")
    ctx.check(mq.lib().mixaq_calibrate_merge(ctx.h, ctypes.byref(ms), mq._ptr(xd), mq._ptr(y), B, H, W, ctypes.byref(r), mq._ptr(ws),
                                             ctypes.c_size_t(ws.numel()), mq._stream_ptr()))
    return y.cpu().numpy(), (r.lo, r.hi)


@pytest.mark.parametrize("N,dim,low,large", [(52, 32, 45, False), (31, 32, 36, True), (300, 64, 45, True), (64, 32, 31, True), (96, 32, 130, True)])
def test_calibration_products_of_rows_with_a_wide_range(orc, mq, ctx, N, dim, low, large):
    """Rows whose values span 2^-low to 1 of their largest, ragged widths.  `large`: the channel of the largest value meets
    weights of zero, so that the sums are those of the small values alone."""
    rng = np.random.default_rng(N)
    m = synth.make_merge(rng, dim, 8, 8)
    m.red = synth.make_linear(rng, N, 4 * dim, 8)
    m.ln_g = np.exp2(-rng.uniform(low - 1 if large else 0, low, 4 * dim)).astype(F32)
    m.ln_b = np.zeros(4 * dim, F32)
    if large:
        m.ln_g[5] = 1.0
        m.red.codes[:, 5] = 0
    x = synth.input_student_t(N, 1, 23, 27, dim)
    x[0, 4:9] = 0.0                                                # rows of zeros among them
    y, got_span = observe_merge(mq, ctx, m, x, N)
    want, span = orc.merge_observe_fp(m, x)
    assert got_span == span
    # each output against sum |a w| of its own: 2^-53 per term for the running sum of either side, one rounding to binary32 each
    pad = np.zeros((24, 28, dim), F32)
    pad[:23, :27] = x[0]
    ln = orc.layernorm(np.concatenate([pad[dy::2, dx::2] for dx in (0, 1) for dy in (0, 1)], axis=-1), m.ln_g, m.ln_b)
    terms = np.abs(ln.astype(np.float64)) @ np.abs(m.red.codes.astype(np.float64) * m.red.scale[:, None].astype(np.float64)).T
    bound = 2.0 ** -23 * np.abs(want) + 2.0 ** -149 + 2 * (4 * dim + 2) * 2.0 ** -53 * terms
    assert (np.abs(y.astype(np.float64) - want) <= bound).all()
    assert ctx.device_status() == 0


@pytest.mark.parametrize("shift,branch", [(0, 0), (3, 1)])
def test_calibration_products_of_a_block_with_a_wide_range_at_every_layer(orc, mq, ctx, shift, branch):
    """At the input of all four products one channel is near 1 and meets weights of zero, the others are near 2^-45; steps bring
    what they leave back to the size of the residuals.  Ragged map: pad rows take no part in the last scatter."""
    dim, small = 64, F32(2.0 ** -45)
    blk = synth.make_block(np.random.default_rng(7 + shift), dim, dim // 32, shift, 8, 8, 4, share_bias=False)
    for br in (blk.hi, blk.lo):
        for g, b in ((br.ln1_g, br.ln1_b), (br.ln2_g, br.ln2_b)):
            b[:] = 0.0
            g[:] = g * small
            g[3] = 1.0
        for b in (br.b_qkv, br.b_proj, br.b_fc1, br.b_fc2):
            b[:] = 0.0
        br.b_fc1[7] = 4.0
    for lin, channel in ((blk.qkv, 3), (blk.proj, 5), (blk.fc1, 3), (blk.fc2, 7)):
        lin.codes[:, channel] = 0
        lin.scale[:] = (lin.scale / small).astype(F32)
    for lin, big in ((blk.qkv, 2 * dim + 5), (blk.fc1, 7)):       # and small again: the v channels but one, the hidden ones but one
        rows = np.arange(lin.scale.size)
        lin.scale[(rows != big) & (rows >= (2 * dim if lin is blk.qkv else 0))] *= small
    x = synth.input_blobs(5, 2, 12, 17, dim, bg_std=0.5, gain=3.0)
    params = mq._Dev(ctx.device)
    y, got = mq.calibrate_block(ctx, mq.fill_block_struct(params, blk), branch, dev(x))
    want_y, want = orc.block_observe_fp(blk, ("hi", "lo")[branch], x)
    # a binary32 rounding (6e-8) may fall the other way in each of the products; the layers behind it amplify it by less than 100
    assert np.abs(y.cpu().numpy() - want_y).max() <= 6e-6 * np.abs(want_y - x).max() + 2.0 ** -22 * np.abs(want_y).max()
    for site, (lo, hi) in want.items():
        assert max(abs(got[site][0] - lo), abs(got[site][1] - hi)) <= 6e-6 * (hi - lo), site
    assert ctx.device_status() == 0


def test_calibration_products_longer_than_an_int32_sum(orc, mq, ctx):
    """fc2 over 32 896 hidden channels is drained from the accumulators in two parts."""
    rng = np.random.default_rng(8)
    blk = synth.make_block(rng, 32, 1, 0, 8, 8, 4)
    blk.hidden = 32768 + 128
    blk.fc1, blk.fc2 = synth.make_linear(rng, blk.hidden, 32, 8), synth.make_linear(rng, 32, blk.hidden, 8)
    for br in (blk.hi, blk.lo):
        br.b_fc1 = (0.02 * rng.standard_normal(blk.hidden)).astype(F32)
    x = synth.input_blobs(5, 1, 7, 7, 32, bg_std=0.5, gain=3.0)
    params = mq._Dev(ctx.device)
    y, got = mq.calibrate_block(ctx, mq.fill_block_struct(params, blk), 0, dev(x))
    want_y, want = orc.block_observe_fp(blk, "hi", x)
    assert np.array_equal(y.cpu().numpy(), want_y)
    assert all(got[site] == span for site, span in want.items())


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_calibration_products_of_rows_that_are_not_finite(orc, mq, ctx, value):
    """A token that is not finite reaches the rows of its window as the plain sums have it, and no others."""
    blk = synth.make_block(np.random.default_rng(4), 64, 2, 0, 4, 8, 4)
    x = synth.input_blobs(5, 1, 14, 21, 64, bg_std=0.5, gain=3.0)
    x[0, 3, 4, 5] = value
    params = mq._Dev(ctx.device)
    y, _ = mq.calibrate_block(ctx, mq.fill_block_struct(params, blk), 0, dev(x))
    want_y, _ = orc.block_observe_fp(blk, "hi", x)
    assert np.isnan(want_y).any() and np.array_equal(np.isnan(y.cpu().numpy()), np.isnan(want_y))
    finite = ~np.isnan(want_y)
    assert np.array_equal(y.cpu().numpy()[finite], want_y[finite])
