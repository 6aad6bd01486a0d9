"""The edges of the kernels' tiles: sizes one below, at and one above what a tile, a panel, a cluster or a launch holds."""
import numpy as np
import pytest
import torch

import dc_workloads as wl
from oracle import dc_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dc():
    import paper_2609_35115_b200 as dc
    dc.load_library()
    return dc


def _util():
    from tests import gpu_util
    return gpu_util


def _batch_equals_single(dc, cfg, n, chunks=3, max_batch=None, ragged=True, options=0):
    """Every stream of n batched calls gives the bytes of its own calls; returns a stream's input and output."""
    w = wl.make_workload(cfg)
    m = dc.Model(cfg, w.weights, max_batch=max_batch or n, options=options)
    streams = [m.open_stream() for _ in range(n)]
    gen = torch.Generator(device="cuda").manual_seed(n)
    feats, outs = [], []
    for c in range(chunks):
        T = [cfg.f_chunk if not ragged or c == 0 else 1 + (7 * i + 5 * c) % cfg.f_chunk for i in range(n)]
        feats.append([torch.randn(t, cfg.in_dim, generator=gen, device="cuda") for t in T])
        outs.append([torch.zeros(t, cfg.out_per_frame, device="cuda") for t in T])
        dc.decode_batch(m, streams, feats[-1], outs[-1])
    torch.cuda.synchronize()
    for i, s in enumerate(streams):
        s.reset()
        for c in range(chunks):
            assert torch.equal(s.decode_chunk(feats[c][i]).flatten(), outs[c][i].flatten()), (n, i, c)
    assert m.counters()[4] == 0
    for s in streams:
        s.close()
    m.destroy()
    x = torch.cat([f[-1] for f in feats]).cpu().numpy()
    bounds = np.cumsum([0] + [f[-1].shape[0] for f in feats]).tolist()
    return w.weights, x, bounds, torch.cat([o[-1].flatten() for o in outs]).cpu().numpy()


# channels: one panel of 64 and more, remainders of 4; frames around the 128-row tile; dilations that share a panel (<= 4) and not
@pytest.mark.parametrize("hidden,dilations,T", [(4, (1, 4), 127), (64, (4, 5), 128), (68, (2, 1), 129), (60, (9, 1), 1), (132, (1, 64), 257)])
def test_tap_convolution_tiles(dc, hidden, dilations, T):
    gu = _util()
    cfg = wl.CONFIGS["cfg1"].replace(name="tiles", hidden=hidden, dilations=dilations, f_chunk=T, n_chunks=3, seed=31, bias_std=0.3)
    bounds = [0, T, T + 1, 2 * T + 1]
    w = wl.make_workload(cfg, boundaries=[bounds])
    m = dc.Model(cfg, w.weights)
    got = gu.run_gpu_stream(m, w.streams[0].feats, bounds)
    assert gu.rel_err(got, orc.run_offline(cfg, w.weights, w.streams[0].feats, bounds)) <= 1e-4
    m.destroy()


# the head's runs of 61 frames and 64 channels, and the batches whose short first layers share tiles (up to 56 frames): even and odd
@pytest.mark.parametrize("mel,channels,f_chunk,n", [(8, (264, 128, 4), 56, 33), (8, (264, 128, 68), 57, 33), (80, (512, 64, 64), 56, 20), (80, (256, 128, 132), 1, 50),
                                                    (8, (128, 256, 8), 61, 2), (8, (16, 8, 8), 5, 64)])
def test_vocoder_batch_tiles(dc, mel, channels, f_chunk, n):
    gu = _util()
    cfg = wl.tiny_vocoder(mel_dim=mel, up_channels=channels, f_chunk=f_chunk, n_chunks=3, seed=32)
    weights, x, bounds, got = _batch_equals_single(dc, cfg, n)
    assert gu.rel_err(got, orc.run_offline(cfg, weights, x, bounds).reshape(-1)) <= 1e-4


# tiles of 64 frames: alone (32 columns each) and in batches; the first layer of the first case takes 64 columns with one panel of input channels, that of the last
# 64 columns with two panels (at 148 SMs); the last frames of a tile, a second and a third tile of one frame; the bytes of single calls, which take other tiles
@pytest.mark.parametrize("mel,channels,f_chunk,n", [(8, (512, 64, 64), 56, 12), (80, (512, 256, 64), 50, 3), (80, (256, 128, 132), 33, 2), (80, (512, 128, 64), 65, 5),
                                                    (80, (512, 128, 64), 129, 5)])
def test_vocoder_small_tiles(dc, mel, channels, f_chunk, n):
    gu = _util()
    cfg = wl.tiny_vocoder(mel_dim=mel, up_channels=channels, f_chunk=f_chunk, n_chunks=3, seed=42)
    weights, x, bounds, got = _batch_equals_single(dc, cfg, n)
    assert gu.rel_err(got, orc.run_offline(cfg, weights, x, bounds).reshape(-1)) <= 1e-4


# batches on both sides of one and two slots per cluster and of the kernels of their own; every cluster size; keys with a gap between
# prompt and history, one block and several
@pytest.mark.parametrize("hidden,heads,n,kw", [
    (512, 8, 7, {}), (512, 8, 8, {}), (512, 16, 15, {}), (256, 4, 3, dict(f_prompt=13, kv_cap=150)), (128, 4, 2, dict(cfg_scale=0.7)),
    (64, 1, 5, dict(kv_cap=300, f_lookahead=6)), (192, 3, 3, dict(f_prompt=130)), (64, 2, 64, dict(f_prompt=9, f_chunk=56))])
def test_flow_cluster_edges(dc, hidden, heads, n, kw):
    gu = _util()
    cfg = wl.tiny_flow(hidden=hidden, n_heads=heads, head_dim=hidden // heads, n_steps=2, seed=33, **kw)
    weights, x, bounds, got = _batch_equals_single(dc, cfg, n, max_batch=2 * n)
    if not cfg.f_lookahead:      # (a call's look-ahead frames are presented again by the next one: other tests compare those)
        assert gu.rel_err(got.reshape(-1, cfg.out_per_frame), orc.run_offline(cfg, weights, x, bounds)) <= 2e-2


def test_single_panel_sums_keep_fp32_precision(dc):
    """Ten layers of 64 channels (one panel each): the taps' sums are added rounded to nearest.  Sums of the FP32 pipe end at 1.8e-6 to 2.1e-6 of
    the output's norm over six seeds, one truncating accumulator for all taps at 3.5e-6 to 5.0e-6; the bound lies between.  Four streams
    fill the 64-column tiles, one the 32-column ones: the same bytes."""
    gu = _util()
    cfg = wl.CONFIGS["cfg4"].replace(name="single_panel", mel_dim=64, up_channels=(64, 64, 64, 64), n_streams=4, n_chunks=2)
    bounds = [0, cfg.f_chunk, 2 * cfg.f_chunk]
    w = wl.make_workload(cfg, boundaries=[bounds] * 4)
    m = dc.Model(cfg, w.weights, max_batch=4)
    streams = [m.open_stream() for _ in range(4)]
    feats = torch.stack([torch.from_numpy(s.feats) for s in w.streams]).cuda()
    outs = [torch.zeros(4, cfg.f_chunk, cfg.out_per_frame, device="cuda") for _ in range(2)]
    for c in range(2):
        dc.decode_batch(m, streams, feats[:, bounds[c]:bounds[c + 1]].contiguous(), outs[c])
    got = torch.cat(outs, dim=1).reshape(4, -1).cpu().numpy()
    ref = np.stack([orc.run_offline(cfg, w.weights, s.feats, bounds).reshape(-1) for s in w.streams]).astype(np.float64)
    err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.mean() <= 3e-6, err
    assert np.array_equal(gu.run_gpu_stream(m, w.streams[0].feats, bounds).reshape(-1), got[0])
    for s in streams:
        s.close()
    m.destroy()


# full batches of an odd number of slots, two per cluster: the last cluster's second slot does not exist, in no buffer
@pytest.mark.parametrize("hidden,n", [(512, 9), (512, 13), (256, 17), (128, 35)])
def test_flow_cluster_odd_full_batch(dc, hidden, n):
    gu = _util()
    cfg = wl.tiny_flow(hidden=hidden, n_heads=hidden // 64, head_dim=64, mel_dim=80, n_steps=2, seed=34)
    weights, x, bounds, got = _batch_equals_single(dc, cfg, n)
    assert gu.rel_err(got.reshape(-1, cfg.out_per_frame), orc.run_offline(cfg, weights, x, bounds)) <= 2e-2


# one slot per cluster has products of 64 rows, sixteen of a quarter of tensor memory each (eight of them left context): chunks that end at, in front of and
# behind a quarter's last row; the bytes of two slots per cluster
@pytest.mark.parametrize("hidden,rounded", [(64, False), (128, True), (512, False)])
def test_flow_cluster_one_slot_rows(dc, hidden, rounded):
    cfg = wl.tiny_flow(hidden=hidden, n_heads=hidden // 32, head_dim=32, mel_dim=80, n_steps=2, f_chunk=56, seed=41)
    w = wl.make_workload(cfg)
    n = {64: 80, 128: 40, 512: 9}[hidden]      # more than the resident clusters
    m = dc.Model(cfg, w.weights, max_batch=n, options=dc.OPT_ROUNDED_NORM if rounded else 0)
    one, many = m.open_stream(), [m.open_stream() for _ in range(n)]
    gen = torch.Generator(device="cuda").manual_seed(hidden)
    for T in (56, 1, 7, 8, 9, 23, 24, 25, 39, 40, 41, 55):
        x = torch.randn(T, cfg.in_dim, generator=gen, device="cuda")
        outs = [torch.zeros(T, cfg.mel_dim, device="cuda") for _ in range(n)]
        dc.decode_batch(m, many, [x] * n, outs)
        got = one.decode_chunk(x)
        assert got.isfinite().all() and all(torch.equal(got, o) for o in outs), T
    assert m.counters()[4] == 0
    for s in [one] + many:
        s.close()
    m.destroy()


# the rounded norm rewrites the panel of one slot or of two: full batches of an odd and an even number, guided passes; the bytes of single calls and of the
# kernels of their own (the option keeps them apart)
@pytest.mark.parametrize("n,kw", [(7, {}), (9, {}), (14, {}), (1, dict(cfg_scale=0.7)), (3, dict(cfg_scale=0.7))])
def test_flow_cluster_rounded_norm(dc, n, kw):
    gu = _util()
    cfg = wl.tiny_flow(hidden=512, n_heads=8, head_dim=64, mel_dim=80, n_steps=2, seed=40, **kw)
    weights, x, bounds, got = _batch_equals_single(dc, cfg, n, options=dc.OPT_ROUNDED_NORM)
    assert gu.rel_err(got.reshape(-1, cfg.out_per_frame), orc.run_offline(cfg, weights, x, bounds)) <= 2e-2
    assert np.array_equal(got, _batch_equals_single(dc, cfg, n, options=dc.OPT_ROUNDED_NORM | dc.OPT_CTA_PAIRS)[3])


# large scores: a later key block's maximum exceeds the reference by more than 2^8 and the accumulated output is rescaled (counted in the oracle's scores, wherever
# the blocks begin).  One and two slots per cluster and kernels of their own: each has its own rows in tensor memory, and all give the same bytes.
# The bound: scores of 14 binary orders turn last bits of a product into percents of a weight.  The oracle differs from itself by 3.2e-2 of RMS with scores in fp32,
# by 3.8e-2 with its weights rounded against another reference, by 3.4e-2 with two accumulators rescaled as on the device; twice the largest.  Without the rescaling
# of the row sums it differs by 0.64, without that of the accumulated output by 2.1, with half of the columns rescaled twice by 1.9.
@pytest.mark.parametrize("heads", [8, 16])
def test_attention_rescale_in_every_form(dc, heads, monkeypatch):
    cfg = wl.tiny_flow(hidden=512, n_heads=heads, head_dim=512 // heads, mel_dim=80, n_steps=2, kv_cap=500, f_chunk=50, seed=44)
    w, at = wl.make_workload(cfg).weights.copy(), 0
    for name, shape, _ in wl.blob_layout(cfg):
        n = int(np.prod(shape))
        if "q" in name.lower() and len(shape) == 2:
            w[at:at + n] *= 10.0          # scores of 14 binary orders, the largest of 128 some 30 above their mean
        at += n
    m = dc.Model(cfg, w, max_batch=20)
    streams = [m.open_stream() for _ in range(20)]
    gen = torch.Generator(device="cuda").manual_seed(44)
    x = [torch.randn(cfg.f_chunk, cfg.in_dim, generator=gen, device="cuda") for _ in range(12)]
    outs = {}
    for n in (1, 9, 20):
        for s in streams:
            s.reset()
        for c in x:
            out = torch.zeros(n, cfg.f_chunk, cfg.mel_dim, device="cuda")
            dc.decode_batch(m, streams[:n], c.expand(n, -1, -1).contiguous(), out)
        outs[n] = out
    assert m.counters()[4] == 0 and outs[1].isfinite().all()
    for n in (9, 20):
        assert torch.equal(outs[n], outs[1].expand(n, -1, -1)), n
    rescaled, attend = [], orc._attend

    def counting(cfg, q, k, v, rb):
        dh = cfg.head_dim
        for e in range(cfg.n_heads if k.shape[0] > 300 else 0):
            s = (q[:, e * dh:(e + 1) * dh] @ k[:, e * dh:(e + 1) * dh].T) * (np.log2(np.e) / np.sqrt(dh))
            count = []
            for phi in range(8):          # the first block holds 128 - phi keys; block b follows block b - 2 into its accumulator
                top = [s[:, max(0, 128 * i - phi):128 * (i + 1) - phi].max(axis=1) for i in range((k.shape[0] + phi + 127) // 128)]
                count.append(sum(int((top[i] > top[i - 2] + 8.0).sum()) for i in range(2, min(4, len(top)))))
            rescaled.append(min(count))
        return attend(cfg, q, k, v, rb)

    monkeypatch.setattr(orc, "_attend", counting)
    ref = orc.run_stream(cfg, w, torch.cat(x).cpu().numpy(), list(range(0, 12 * cfg.f_chunk + 1, cfg.f_chunk)))
    assert sum(rescaled) >= 100
    assert _util().rel_err(outs[1][0].cpu().numpy(), ref[-cfg.f_chunk:]) <= 8e-2
    for s in streams:
        s.close()
    m.destroy()


# one reduction block per conv product (hidden 64): 32- and 64-column tiles, whose epilogue exchanges more rows than one pipeline stage holds
@pytest.mark.parametrize("n", [76, 150])
def test_conv_exchange_of_one_reduction_block(dc, n):
    gu = _util()
    cfg = wl.tiny_flow(n_steps=2, seed=35)
    weights, x, bounds, got = _batch_equals_single(dc, cfg, n, options=dc.OPT_CTA_PAIRS)    # (the option keeps the kernels apart)
    assert gu.rel_err(got.reshape(-1, cfg.out_per_frame), orc.run_offline(cfg, weights, x, bounds)) <= 2e-2


# the row exchanges of the cluster step's epilogues lie where the next stage's activations land: one and two slots per cluster, guided passes
@pytest.mark.parametrize("n,kw", [(1, {}), (9, {}), (2, dict(cfg_scale=0.7))])
def test_flow_cluster_exchange_repeats(dc, n, kw):
    cfg = wl.tiny_flow(hidden=512, n_heads=8, head_dim=64, mel_dim=80, n_steps=8, f_chunk=50, seed=36, **kw)
    w = wl.make_workload(cfg)
    m = dc.Model(cfg, w.weights, max_batch=2 * n)
    streams = [m.open_stream() for _ in range(n)]
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn(n, cfg.f_chunk, cfg.in_dim, generator=gen, device="cuda")
    outs = torch.zeros(40, n, cfg.f_chunk, cfg.mel_dim, device="cuda")
    for out in outs:
        for s in streams:
            s.reset()
        dc.decode_batch(m, streams, x, out)
    assert m.counters()[4] == 0
    assert torch.equal(outs, outs[:1].expand_as(outs))
    for s in streams:
        s.close()
    m.destroy()


# a stream that has held NaN is reset: its new session's history does not fill the gap behind the prompt rows yet.  One kernel per chunk and
# kernels of their own, both head widths, wavefront
@pytest.mark.parametrize("kw", [dict(hidden=128, head_dim=64), dict(hidden=128, head_dim=32), dict(hidden=192, head_dim=64), dict(hidden=192, head_dim=32)])
@pytest.mark.parametrize("f_prompt", [13, 17])
def test_reset_leaves_nothing_of_the_session_before(dc, kw, f_prompt):
    cfg = wl.tiny_flow(f_prompt=f_prompt, n_heads=kw["hidden"] // kw["head_dim"], n_steps=2, seed=37, **kw)
    w = wl.make_workload(cfg)
    m = dc.Model(cfg, w.weights, max_batch=cfg.n_steps)
    gen = torch.Generator(device="cuda").manual_seed(f_prompt)
    x = torch.randn(f_prompt + 21, cfg.in_dim, generator=gen, device="cuda")
    cuts = list(range(0, f_prompt, cfg.f_chunk)) + [f_prompt, f_prompt + 1, f_prompt + 2, f_prompt + 11, f_prompt + 21]
    fresh, used = m.open_stream(), m.open_stream()
    for _ in range(8):
        assert used.decode_chunk(torch.full((cfg.f_chunk, cfg.in_dim), float("nan"), device="cuda")).isnan().all()
    used.reset()
    for a, b in zip(cuts, cuts[1:]):
        got = used.decode_chunk(x[a:b].contiguous())
        assert torch.equal(got, fresh.decode_chunk(x[a:b].contiguous())) and got.isfinite().all(), (a, b)
    for s in (fresh, used):
        s.reset()
    used.decode_wavefront(torch.full((8 * cfg.f_chunk, cfg.in_dim), float("nan"), device="cuda"))
    used.reset()
    assert torch.equal(used.decode_wavefront(x), fresh.decode_wavefront(x))
    for s in (fresh, used):
        s.close()
    m.destroy()


def test_ring_of_more_than_2_to_32_elements(dc):
    """A vocoder ring of 2^20 rows of 4,100 channels (34 GB): element offsets beyond 32 bits.  The same frames in short chunks, whose rings are small, give
    the same bytes."""
    cfg = wl.tiny_vocoder(mel_dim=4, up_strides=(16, 16, 1), up_channels=(4, 4, 4100, 4), res_dilations=(), f_chunk=4096, seed=38)
    w = wl.make_workload(cfg.replace(n_chunks=1))
    x = torch.from_numpy(w.streams[0].feats).cuda()
    big, small = dc.Model(cfg, w.weights), dc.Model(cfg.replace(f_chunk=64), w.weights)
    a, b = big.open_stream(), small.open_stream()
    got = a.decode_chunk(x).flatten()
    want = torch.cat([b.decode_chunk(x[t:t + 64].contiguous()).flatten() for t in range(0, 4096, 64)])
    assert torch.equal(got, want) and got.isfinite().all()
    for s, m in ((a, big), (b, small)):
        s.close()
        m.destroy()


# one kernel of clusters (1, 14 streams), kernels of their own (15): a profiled call launches what the same call launches otherwise
@pytest.mark.parametrize("n,cluster", [(1, 1), (14, 1), (15, 0)])
def test_profile_brackets_the_launches_of_a_call(dc, n, cluster):
    cfg = wl.CONFIGS["cfg3"].replace(n_steps=2)
    m = dc.Model(cfg, wl.make_weights(cfg, np.random.default_rng(39)), max_batch=n, options=dc.OPT_NO_GRAPH)
    streams = [m.open_stream() for _ in range(n)]
    x, out = torch.randn(n, cfg.f_chunk, cfg.in_dim, device="cuda"), torch.zeros(n, cfg.f_chunk, cfg.mel_dim, device="cuda")
    before = m.counters()[5]
    dc.decode_batch(m, streams, x, out)
    launched = m.counters()[5] - before
    m.profile_begin()
    dc.decode_batch(m, streams, x, out)
    ms, count = m.profile_end()
    assert sum(count.values()) == launched and count["flow_cluster"] == cluster
    assert all(ms[k] > 0 for k in count if count[k])
    for s in streams:
        s.close()
    m.destroy()


# two slots per cluster (fourteen streams, seven guided ones) and one, from the empty window to the full one, one to five key blocks, beside copies that
# hold up the loads of carried rows: the same bytes every time.  (A wait of the K/V ring that passed early showed in 2 of 8,700 such rounds, and only in an attention
# with a shorter softmax: the walk of the ring on the host is what tests the wait.)
@pytest.mark.parametrize("net,n", [("cfg3", 14), ("cfg3_guided", 7), ("cfg3", 1)])
def test_cluster_step_repeats_beside_copies(dc, net, n):
    cfg = {**wl.CONFIGS, **wl.EXTRA_CONFIGS}[net]
    m = dc.Model(cfg, wl.make_weights(cfg, np.random.default_rng(1)), max_batch=n)
    streams = [m.open_stream() for _ in range(n)]
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = [torch.randn(n, cfg.f_chunk, cfg.in_dim, generator=gen, device="cuda") for _ in range(12)]
    out = torch.zeros(12, n, cfg.f_chunk, cfg.out_per_frame, device="cuda")
    side, a, b = torch.cuda.Stream(), torch.zeros(1 << 26, device="cuda"), torch.zeros(1 << 26, device="cuda")
    first, bad = None, torch.zeros((), device="cuda", dtype=torch.int64)
    for r in range(200):
        with torch.cuda.stream(side):
            for _ in range(4):
                b[: 1 << (19 + r % 8)].copy_(a[: 1 << (19 + r % 8)])
        for s in streams:
            s.reset()
        for c in range(12):
            dc.decode_batch(m, streams, x[c], out[c])
        if first is None:
            first = out.clone()
        bad += (out != first).any()
    assert int(bad) == 0 and first.isfinite().all() and m.counters()[4] == 0
    for s in streams:
        s.close()
    m.destroy()
