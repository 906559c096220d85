"""Edges of the paths that a size decides: row tiles and K splits of the tensor-core projection, the shrink over rows that
pick their adapters one by one, tensor-core attention (trees, many streams, causal passes of one and two row blocks), and the
variants of the kernel-per-projection decode path -- each against the CPU oracle."""
import numpy as np
import pytest

import gen
from oracle import ref
from tests.helpers import check_argmax, compare
from tests.test_gpu_kernels import dev, mb, run_attention, run_linear  # noqa: F401  (mb: fixture)
from tests.test_gpu_model import GpuModel, compare_kv, make_pair  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# ------------------------------------------------------------------ projections of many rows
@pytest.mark.parametrize("M", [9, 32, 33, 64, 65, 96, 97, 128, 129, 192, 193, 256, 257, 385])
def test_projection_row_tiles(mb, M):
    """Row counts at the edges of the row tiles, a ragged last column tile (N = 8 x 128 + 16), adapters and base rows."""
    got, want = run_linear(mb, 512, 1040, 128, M, 8, 16, seed=M)
    compare(got, want, f"row tiles M{M}")


@pytest.mark.parametrize("K,N,G,M", [
    (256, 16, 64, 9),            # one column tile of 16, the smallest K that is split
    (4096, 256, 128, 40),        # few columns: the widest split of K
    (14336, 128, 128, 250),      # the longest K in two row blocks
    (320, 4096, 64, 700),        # K of an odd number of steps, more tiles than CTAs: each stays for further ones
    (192, 9600, 64, 180),        # the same with fewer steps than weight stages
    (192, 9600, 64, 90),
    (64, 15376, 64, 280),        # the 96-row tile, again more tiles than CTAs
    (2048, 3072, 128, 96), (2048, 3072, 128, 192),   # clusters of four would not all fit at once: split in two
])
def test_projection_splits_and_persistent_tiles(mb, K, N, G, M):
    for n_ad, rank in ((0, 0), (3, 8)):
        got, want = run_linear(mb, K, N, G, M, n_ad, rank, seed=K + N + M + n_ad)
        compare(got, want, f"projection K{K} N{N} M{M} adapters {n_ad}")


@pytest.mark.parametrize("K,N,M", [(192, 1040, 40), (320, 1040, 64), (64, 16, 128), (2048, 272, 65), (832, 1040, 128), (4096, 400, 100)])
def test_projection_of_few_columns(mb, K, N, M):
    """Fewer steps than pairs of unpacking groups, K splits down to a pair of rows a warp."""
    got, want = run_linear(mb, K, N, 64, M, 0, 0, seed=K + N + M)
    compare(got, want, f"few columns K{K} N{N} M{M}")


@pytest.mark.parametrize("K,N,M,plan", [
    (320, 4112, 200, (64, 1, 4)), (832, 4112, 250, (64, 1, 4)), (1088, 4112, 65, (64, 2, 4)), (2048, 2064, 33, (64, 4, 4)),
    (2048, 528, 200, (64, 4, 4)), (8192, 528, 100, (64, 8, 4)), (8192, 272, 250, (64, 8, 4)), (2048, 4112, 200, (128, 2, 4)),
    (3136, 4112, 100, (128, 4, 4)), (8192, 528, 250, (128, 8, 4)),
])
def test_projection_with_four_unpacking_groups(mb, K, N, M, plan):
    """Tiles of 64 and 128 rows whose grid leaves every CTA an SM (the projection ahead of an expand of its own): steps that the groups
    share unevenly, K splits down to a pair of rows a warp."""
    assert mb.mlora_debug_gemm_plan(M, K, N, 0) == plan
    got, want = run_linear(mb, K, N, 64, M, 70, 16, seed=K + N + M)
    compare(got, want, f"four groups K{K} N{N} M{M}")


@pytest.mark.parametrize("P", [100, 200])
def test_prefill_with_four_unpacking_groups(GpuModel, P):
    """The other epilogues with four groups: q,k,v, o, gate/up and down of one layer of 2048."""
    from paper_2604_18655_b200 import binding as mb
    cfg = gen.ModelCfg("four", 1, 2048, 32, 8, 64, 5632, 0, 128, 4, gen.configs.ALL7, 1, 1, P)
    shapes = ((2048, 3072), (2048, 2048), (2048, 11264), (5632, 2048))
    assert sum(mb.mlora_debug_gemm_plan(P, K, N, 0)[2] == 4 for K, N in shapes) == 4
    _, orc, gm = make_pair(GpuModel, cfg, max_suffix=2)
    x = gen.make_hidden(cfg, P, 0, 0)
    compare(gm.prefill_h(x), orc.prefill_shared(hidden=x), f"prefill of {P}")
    _, pk, pv = gm.export_kv(0, -1, 0, P)
    compare(pk, orc.prefix_k[0], "prefix K")
    compare(pv, orc.prefix_v[0], "prefix V")
    gm.close()


@pytest.mark.parametrize("M,n_ad,rank,K", [(9, 1, 1, 256), (17, 40, 12, 1024), (300, 2, 64, 8192), (64, 64, 16, 2112)])
def test_shrink_of_rows_with_their_own_adapters(mb, M, n_ad, rank, K):
    """Adapters without a row, with one, with more than the 16 of a group; ranks off the tile of eight; K shares beyond what
    the registers hold and a K that the warps share unevenly."""
    got, want = run_linear(mb, K, 256, 64, M, n_ad, rank, seed=M + rank)
    compare(got, want, f"gather shrink M{M} adapters {n_ad} rank {rank} K{K}")


@pytest.mark.parametrize("M,n_ad,rank,K,N", [
    (9, 64, 64, 256, 208),        # 4096 columns of (adapter, rank index), few of them in use
    (32, 65, 64, 512, 1040),      # more than that
    (250, 300, 20, 320, 144),     # more adapters than rows, a rank off the multiples of 8
    (129, 128, 64, 192, 4112),
    (700, 90, 24, 320, 9600),     # about eight rows an adapter: groups of sixteen rows, and more
    (4096, 5000, 9, 64, 16),      # the most rows, the narrowest output
    (40, 7, 130, 256, 64),        # a rank above 64
    (64, 40, 16, 14336, 128),     # the widest split of K
    (300, 64, 64, 1088, 528),     # T adapter by adapter ahead of the separate expand
    (600, 70, 70, 64, 48),
    (64, 70, 16, 49216, 16),      # rows too long for the row-wise shrink
])
def test_projection_with_many_adapters(mb, M, n_ad, rank, K, N):
    """Calls whose rows pick from many adapters: the expand is a kernel of its own over the ones that occur.  The workspace is the
    smallest that the call takes; rows without an adapter, adapters without matrices."""
    rng = np.random.default_rng(M + n_ad)
    qb, sc = gen.quantize_int4(rng.standard_normal((K, N)).astype(np.float32) * 0.02, 64)
    x = rng.standard_normal((M, K)).astype(np.float16)
    A = (rng.standard_normal((n_ad, rank, K)) / rank).astype(np.float16)
    B = (rng.standard_normal((n_ad, rank, N)) * 0.05).astype(np.float16)
    scale = (16.0 / rank * (1 + 0.25 * (np.arange(n_ad) % 8))).astype(np.float32)
    rows = rng.integers(-1, n_ad, size=M).astype(np.int32)
    rows[0], rows[1], rows[-1] = n_ad, -7, rows[M // 2]
    dA, dB = dev(A), dev(B)
    pa, pb = [torch.tensor([t[i].data_ptr() for i in range(n_ad)], dtype=torch.int64, device="cuda") for t in (dA, dB)]
    none = int(rows[2]) if rows[2] >= 0 else 0
    pa[none] = 0                                       # an adapter without matrices
    pb[none] = 0
    w = mb.mlora_weight_create(dev(qb), dev(sc), K, N, 64)
    need = mb.mlora_linear_workspace_bytes(w, M, rank) - 7 * M * N * 4
    ws = torch.full((need + 4096,), 255, dtype=torch.uint8, device="cuda")      # (what lies behind must stay as it is)
    ws[:16640] = 0
    y = torch.empty(M, N, dtype=torch.float32, device="cuda")
    for _ in range(2):
        mb.mlora_linear(w, dev(x), y, ws[:need], dev(rows), pa, pb, dev(scale), rank)
    torch.cuda.synchronize()
    rows = np.where((rows >= n_ad) | (rows == none), -1, np.maximum(rows, -1))
    f = np.float64
    want = ref.linear_lora(x.astype(f), ref.dequant(qb, sc, 64).astype(f), rows, list(A.astype(f)), list(B.astype(f)), scale.astype(f))
    mb.mlora_weight_destroy(w)
    compare(y.cpu().numpy(), want, f"M{M} adapters {n_ad}x{rank} K{K} N{N}")
    assert bool((ws[need:] == 255).all())


@pytest.mark.parametrize("rows", [(8, 3, 8, 1), (40, 200, 9, 40), (64, 12, 300, 64), (8, 40, 5, 200)])
def test_calls_that_follow_one_another_on_one_workspace(mb, rows):
    """Calls chained by programmatic launches, nothing waited for in between: other rows, other adapters (few, many, none) and
    other inputs each time on one workspace, every call's result in fp16 the input of the next but one."""
    K = 512
    rng = np.random.default_rng(sum(rows))
    stream = torch.cuda.Stream()
    sets = [None]
    for n_ad, rank in ((4, 16), (70, 64)):
        A = (rng.standard_normal((n_ad, rank, K)) / rank).astype(np.float16)
        B = (rng.standard_normal((n_ad, rank, K)) * 0.05).astype(np.float16)
        dA, dB = dev(A), dev(B)
        ptr = [torch.tensor([t[i].data_ptr() for i in range(n_ad)], dtype=torch.int64, device="cuda") for t in (dA, dB)]
        sets.append((A, B, rank, (dA, dB), ptr, torch.full((n_ad,), 16.0 / rank, device="cuda")))
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        ws, Wd = [], []
        for i in range(2):
            qb, sc = gen.quantize_int4(rng.standard_normal((K, K)).astype(np.float32) * 0.04, 64)
            ws.append(mb.mlora_weight_create(dev(qb), dev(sc), K, K, 64))
            Wd.append(ref.dequant(qb, sc, 64).astype(np.float64))
        work = torch.zeros(max(mb.mlora_linear_workspace_bytes(ws[0], m, 64) for m in rows), dtype=torch.uint8, device="cuda")
        plan, src = [], [dev(rng.standard_normal((max(rows), K)).astype(np.float16)) for _ in range(2)]
        for i in range(10):
            M, st = rows[i % 4], sets[(i + 1) % 3]
            idx = rng.integers(-1, len(st[0]), size=M).astype(np.int32) if st else None
            plan.append((M, st, idx, dev(idx) if st else None, torch.empty(M, K, device="cuda"), torch.empty(max(rows), K, dtype=torch.float16, device="cuda")))
        stream.synchronize()
        ins = []
        for i, (M, st, idx, d_idx, y, h) in enumerate(plan):
            x = src[i] if i < 2 else plan[i - 2][5]
            ins.append(x)
            mb.mlora_linear(ws[i % 2], x[:M], y, work, *((d_idx, *st[4], st[5], st[2]) if st else ()))
            for j in (i - 1, i) if i % 2 else ():          # (two calls straight behind one another)
                plan[j][5].copy_(src[j % 2])
                plan[j][5][:plan[j][0]].copy_(plan[j][4])
        stream.synchronize()
        for i, (M, st, idx, _, y, _) in enumerate(plan):
            x = ins[i][:M].double().cpu().numpy()
            lora = (idx, list(st[0].astype(np.float64)), list(st[1].astype(np.float64)), st[5].double().cpu().numpy()) if st else ()
            compare(y.cpu().numpy(), ref.linear_lora(x, Wd[i % 2], *lora), f"call {i}, {M} rows")
        mb.mlora_linear_status(ws[0], work)
        for w in ws:
            mb.mlora_weight_destroy(w)


def test_quantised_calls_that_follow_one_another(mb):
    """Quantiser and INT8 projection in a chain over the same buffers, nothing waited for in between."""
    K, N, stream = 512, 256, torch.cuda.Stream()
    rng = np.random.default_rng(4)
    qb, sc = gen.quantize_int4_per_channel(rng.standard_normal((K, N)).astype(np.float32) * 0.02)
    xs = [rng.standard_normal((M, K)).astype(np.float16) for M in (8, 64, 1, 17, 8)]
    dq, ds, dx, ys = dev(qb), dev(sc), [dev(x) for x in xs], [torch.empty(len(x), N, device="cuda") for x in xs]
    qx = torch.empty(64, K, dtype=torch.int8, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for x, y in zip(dx, ys):
            mb.mlora_quantize_act_int8(x, 0.03, qx[:len(x)])
            mb.mlora_linear_w4a8(dq, ds, qx[:len(x)], 0.03, y)
        stream.synchronize()
    for x, y in zip(xs, ys):
        want = ref.linear_w4a8(ref.quantize_act_int8(x, 0.03), 0.03, qb, sc)
        assert np.array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("count", [1, 7, 8, 9, 1023, 1025])
def test_quantiser_tails(mb, count):
    x = np.random.default_rng(count).standard_normal((1, count)).astype(np.float16)
    for off in (0, 1):           # (an input that starts between 16-byte boundaries)
        buf = torch.zeros(count + 8, dtype=torch.float16, device="cuda")
        buf[off:off + count] = dev(x[0])
        out = torch.zeros(count, dtype=torch.int8, device="cuda")
        mb.mlora_quantize_act_int8(buf[off:off + count].view(1, count), 0.02, out.view(1, count))
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().reshape(1, -1), ref.quantize_act_int8(x, 0.02))


@pytest.mark.parametrize("n,T,rank", [(40, 30, 20), (70, 6, 12), (9, 64, 64), (300, 1, 9), (130, 3, 64)])
def test_adapters_of_passes_with_more_streams_than_a_row_tile_has(GpuModel, n, T, rank):
    """The adapters' T has columns for the streams that one row tile can touch; further streams use them again."""
    cfg = gen.ModelCfg("streams", 1, 128, 4, 2, 64, 192, 304, 64, rank, gen.configs.ALL7, 5, n, 33, b_std=0.05)
    _, orc, gm = make_pair(GpuModel, cfg, max_suffix=T, max_tree=T)
    ids = gen.make_prompt_ids(cfg, 0)
    compare(gm.prefill(ids), orc.prefill_shared(ids, n_streams=n), "prefill logits")
    ad = [(s * 7) % 6 - 1 for s in range(n)]
    par = np.stack([np.array([-1] + [(i - 1) // 2 for i in range(1, T)], dtype=np.int32)] * n)
    tree = np.random.default_rng(n).integers(0, cfg.vocab, size=(n, T), dtype=np.int32)
    compare(gm.verify(ad, tree, par)["logits"], orc.verify_tree(ad, par, tree)["logits"], f"{n} streams of {T} rows, rank {rank}")
    gm.close()


def test_adapter_scratch_of_many_streams_stays_proportional():
    """A context for 256 streams of 64-node trees at rank 64 (one small layer) fits in half of what the adapters' T alone took
    with a column for every (stream, rank index)."""
    from paper_2604_18655_b200 import binding as mb
    cfg = gen.ModelCfg("scratch", 1, 64, 1, 1, 64, 64, 0, 64, 64, gen.configs.ALL7, 1, 256, 64)
    m = gen.make_model(cfg, 0)
    to = lambda ts: [dev(t) for t in ts]
    w, s, ga, gf = to(m.qweight), to(m.scales), to(m.rms_attn), to(m.rms_ffn)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = mb.mlora_create(cfg, w, s, ga, gf, None, None, max_adapters=1, max_streams=256, max_prefix=64, max_suffix=64, max_tree=64)
    used = before - torch.cuda.mem_get_info()[0]
    mb.mlora_destroy(ctx)
    assert used < 256 * 64 * 6 * 256 * 64 * 2 // 2, used


# ------------------------------------------------------------------ attention
@pytest.mark.parametrize("n,T,Hq,Hkv,hd,P,suf,branch", [
    (2, 9, 6, 2, 64, 129, [0, 1], (2, 3)),            # groups of three heads: 126 of a block's 128 rows
    (3, 33, 5, 1, 128, 128, [127, 128, 5], (4, 4, 3)),   # own segments over a tile's end, two blocks of rows a stream
    (1, 64, 8, 8, 64, 1, [0], (4, 4, 3)),             # one head a group, the largest tree, a prefix of one key
    (2, 16, 16, 2, 128, 0, [3, 250], (4, 3)),         # no prefix
    (1, 16, 8, 2, 64, 100, [1500], (4, 3)),           # own segments in chunks: thirteen of them,
    (3, 30, 24, 8, 128, 300, [900, 0, 380], (4, 3, 2)),   # two, of which a short segment has one; the tree across a chunk's end,
    (16, 1, 8, 8, 64, 70, [700, 3, 127, 128, 129, 255, 256, 257, 383, 384, 385, 0, 511, 512, 513, 640], ()),
    (40, 1, 32, 8, 128, 0, [400] * 39 + [1023], ()),      # one (more own segments than CTAs wanted)
])
def test_tree_attention_edges(mb, n, T, Hq, Hkv, hd, P, suf, branch):
    got, want = run_attention(mb, n, T, Hq, Hkv, hd, P, suf, branch, seed=n + T + P)
    compare(got, want, f"tree attention n{n} T{T} {Hq}q/{Hkv}kv hd{hd} P{P}")


@pytest.mark.parametrize("n,T,Hq,Hkv,hd,P,suf,branch,out_off", [
    (5, 13, 12, 4, 64, 200, [0, 1, 60, 130, 7], (3, 3), 0),       # rows of a kv head that fill no whole block
    (3, 30, 32, 8, 64, 512, [0, 640, 9], (4, 4, 2), 0),           # own segments in chunks, one stream without keys in most of them
    (2, 40, 24, 8, 128, 1000, [300, 2], (4, 4, 2), 0),
    (9, 16, 8, 1, 128, 0, [5] * 9, (4, 2, 2), 0),                 # no prefix: one chunk a row
    (2, 40, 24, 8, 64, 3000, [900, 2], (4, 4, 2), 0),             # more chunks than the kernel for few takes
    (3, 30, 32, 8, 64, 512, [0, 40, 9], (4, 4, 2), 2),            # an output that does not start on 8 bytes
])
def test_merge_of_many_rows(mb, n, T, Hq, Hkv, hd, P, suf, branch, out_off):
    got, want = run_attention(mb, n, T, Hq, Hkv, hd, P, suf, branch, seed=n + T + P, out_off=out_off)
    compare(got, want, f"merge n{n} T{T} {Hq}q/{Hkv}kv hd{hd} P{P} out + {out_off}")


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("n,T,P,suf,branch", [(3, 1, 2100, [0, 40, 90], ()), (2, 16, 130, [3, 64], (4, 2, 2))])
@pytest.mark.parametrize("out_off,ws_off", [(1, 8), (2, 0), (3, 4)])
def test_merged_attention_into_buffers_of_any_start(mb, hd, n, T, P, suf, branch, out_off, ws_off):
    """The partial-result paths (streaming + merge, tensor cores + merge) into an output that starts on any half and with
    scratch that starts on any word."""
    got, want = run_attention(mb, n, T, 8, 2, hd, P, suf, branch, seed=hd + T + out_off, out_off=out_off, ws_off=ws_off)
    compare(got, want, f"attention out + {out_off} halves, scratch + {ws_off} bytes")


@pytest.mark.parametrize("hd,n_q,n_kv,P", [(64, 32, 8, 640), (128, 24, 8, 1025), (128, 16, 8, 2100), (64, 6, 2, 257)])
def test_causal_passes_of_one_and_two_row_blocks(GpuModel, hd, n_q, n_kv, P):
    """Two row blocks a CTA from about 600 positions on; the second layer's K/V show every row of the first one's output.
    2100 positions: a second pass of 52 rows over the first one's keys."""
    cfg = gen.ModelCfg("causal", 2, 256, n_q, n_kv, hd, 320, 0, 64, 8, 15, 1, 1, P)
    _, orc, gm = make_pair(GpuModel, cfg, max_suffix=8)
    prompt = gen.make_hidden(cfg, P, 0, 0)
    want = orc.prefill_shared(hidden=prompt)
    compare(gm.prefill_h(prompt), want, "last hidden")
    for l in range(2):
        _, pk, pv = gm.export_kv(l, -1, 0, P)
        compare(pk, orc.prefix_k[l], f"prefix K of layer {l}")
        compare(pv, orc.prefix_v[l], f"prefix V of layer {l}")
    gm.close()


def test_passes_with_more_query_heads_a_group_than_a_block_has_rows(GpuModel):
    """129 query heads on one KV head: prefill, a tree pass and a decode step of nine streams keep the tensor-core projections
    and take the general attention kernel."""
    cfg = gen.ModelCfg("mqa", 2, 128, 129, 1, 64, 192, 304, 64, 4, gen.configs.ALL7, 2, 9, 40)
    _, orc, gm = make_pair(GpuModel, cfg, max_suffix=40, max_tree=6)
    ids = gen.make_prompt_ids(cfg, 0)
    compare(gm.prefill(ids), orc.prefill_shared(ids, n_streams=9), "prefill logits")
    ad = [0, 1, -1] * 3
    parent = np.array([-1, 0, 0, 1, 1, 2], dtype=np.int32)
    tree = np.random.default_rng(3).integers(0, cfg.vocab, size=(9, 6), dtype=np.int32)
    par = np.stack([parent] * 9)
    got = gm.verify(ad, tree, par)
    want = orc.verify_tree(ad, par, tree, follow_argmax=np.argmax(got["logits"], axis=1).reshape(9, 6))
    compare(got["logits"], want["logits"], "verify logits")
    toks = np.arange(3, 12, dtype=np.int32)
    _, logits = gm.decode(ad, toks)
    compare(logits, orc.decode_step(ad, tokens=toks)["logits"], "decode logits")
    gm.close()


@pytest.mark.parametrize("rms,channel,gain,decode_path", [
    (3000., None, 8., 1),       # rows whose x * gain leaves fp16 everywhere, and whose squares add up to more than 2^31
    (40., 60000., 1.5, 1),      # one massive channel
    (45., None, 1., 0), (47., None, 1., 0),     # on either side of where rows start to be scaled (a sum of 2^20 over 512 features)
])
def test_large_residual_rows(GpuModel, rms, channel, gain, decode_path):
    """A pass's residual rows travel as x * gain without their 1/rms: rows far beyond what fp16 holds give what normalised rows
    give, in prefill (one row's logits), tree passes and decode steps of nine streams.  (Decode steps of few streams on the
    path that normalises its rows first: the other one's bound is documented.)"""
    from paper_2604_18655_b200 import binding as mb
    cfg = gen.ModelCfg("large", 3, 512, 4, 2, 64, 192, 304, 64, 4, gen.configs.ALL7, 3, 9, 40, b_std=0.05)
    m = gen.make_model(cfg, 0)
    m.embed = (m.embed.astype(np.float32) * (rms / cfg.w_std)).astype(np.float16)
    if channel:
        m.embed[:, 5] = channel
    for g in m.rms_attn + m.rms_ffn + [m.rms_final]:
        g *= np.float16(gain)
    orc, gm = ref.OracleModel.from_synth(m), GpuModel(m, max_suffix=40, max_tree=6)
    mb.mlora_debug_set(gm.ctx, 6, decode_path)
    for a in range(3):
        A, B = gen.make_adapter(cfg, a, 0)
        orc.set_adapter(a, A, B, cfg.alpha)
        gm.set_adapter(a, A, B, cfg.alpha)
    ids = gen.make_prompt_ids(cfg, 0)
    compare(gm.prefill(ids), orc.prefill_shared(ids, n_streams=9), "prefill logits")
    for l in range(3):
        _, pk, pv = gm.export_kv(l, -1, 0, cfg.prompt_len)
        compare(pk, orc.prefix_k[l], f"prefix K of layer {l}")
        compare(pv, orc.prefix_v[l], f"prefix V of layer {l}")
    ad = [0, 1, -1, 2, 0, 1, 2, -1, 0]
    par = np.stack([np.array([-1, 0, 0, 1, 1, 2], dtype=np.int32)] * 9)
    tree = np.random.default_rng(3).integers(0, cfg.vocab, size=(9, 6), dtype=np.int32)
    got = gm.verify(ad, tree, par)
    want = orc.verify_tree(ad, par, tree, follow_argmax=np.argmax(got["logits"], axis=1).reshape(9, 6))
    compare(got["logits"], want["logits"], "verify logits")
    toks = np.arange(3, 12, dtype=np.int32)
    _, logits = gm.decode(ad, toks)
    compare(logits, orc.decode_step(ad, tokens=toks)["logits"], "decode logits, nine streams")
    nxt, logits = gm.decode(ad[:5], toks[:5])
    compare(logits, orc.decode_step(ad[:5], tokens=toks[:5])["logits"], "decode logits, five streams")
    only, _ = gm.decode(ad[:5], toks[:5], want_logits=False)
    check_argmax(only, orc.decode_step(ad[:5], tokens=toks[:5])["logits"], "greedy tokens")
    gm.close()


# ------------------------------------------------------------------ decode
@pytest.mark.parametrize("d_model,d_ffn,hd,n_q,n_kv,vocab,rank,n,P", [
    (3072, 4096, 128, 24, 8, 9600, 32, 8, 70),     # single-wave variants, pointer table, lm_head of K = 3072
    (4096, 1024, 128, 8, 2, 9600, 20, 3, 40),      # a rank off the multiples of 16, lm_head of K = 4096
    (512, 8192, 64, 8, 8, 304, 16, 5, 33),         # down projection of K = 8192 with few columns
    (512, 1408, 64, 8, 4, 304, 64, 8, 2101),       # streaming attention + merge with the o projection's shrink, rank 64
    (256, 512, 128, 4, 1, 304, 8, 2, 2048),
    (128, 14336, 64, 2, 1, 304, 8, 3, 9),          # gate/up in more than four CTAs an SM: the dense variant again
])
def test_decode_variants(GpuModel, d_model, d_ffn, hd, n_q, n_kv, vocab, rank, n, P):
    cfg = gen.ModelCfg("decode", 2, d_model, n_q, n_kv, hd, d_ffn, vocab, 64, rank, gen.configs.ALL7, 3, n, P)
    _, orc, gm = make_pair(GpuModel, cfg, max_suffix=8)
    ids = gen.make_prompt_ids(cfg, 0)
    compare(gm.prefill(ids), orc.prefill_shared(ids, n_streams=n), "prefill logits")
    ad = [(s % 4) - 1 for s in range(n)]
    toks = np.arange(3, 3 + n, dtype=np.int32)
    for step in range(2):
        nxt, logits = gm.decode(ad, toks)
        r = orc.decode_step(ad, tokens=toks)
        compare(logits, r["logits"], f"decode logits, step {step}")
        check_argmax(nxt, r["logits"], f"step {step}")
        toks = nxt
    compare_kv(gm, orc, cfg, n)
    gm.close()
