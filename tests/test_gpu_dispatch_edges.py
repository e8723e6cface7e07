"""Edges of the kernels and of the rules that choose between them: cluster sizes of the one-launch decode and of the ladder
decode, strides of the value quantisers, query tiles of the calibration weights, degenerate matrices of the eigen solver."""
import numpy as np
import pytest
import torch

from oracle import okq_calib_oracle as CO
from paper_2609_11582_b200 import binding as B
from paper_2609_11582_b200 import workloads as WL
from tests import harness as Hn
from tests.test_gpu_ladder import LadderCase

pytestmark = pytest.mark.gpu
D, W = 128, 32


# (sequences, KV heads), units around the steps of the rule: a cluster of 16; the most clusters of 8 and of 4 that run at once
# (15, 33); clusters of 2 up to the most of them (74); single blocks in one wave (75, 76, 148) and in two (149); the split-K pair
# (448 units would be a fourth wave); tokens: fewer windows than warps, one window, no window at all, a full and an empty raw tail
@pytest.mark.parametrize("batch,heads", [(1, 1), (2, 4), (15, 1), (33, 1), (17, 2), (74, 1), (75, 1), (76, 1), (37, 4), (149, 1), (112, 4)])
@pytest.mark.parametrize("n", [31, 32, 32 * 13 + 31])
def test_one_launch_decode_at_its_edges(batch, heads, n):
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=batch, n_kv_heads=heads, n_q_heads=7 * heads, prefix_text=40, video_chunk=70, audio_chunk=21)
    c = Hn.Case(w, n_tokens=n, meta_format=B.META_MXFP4 if batch % 2 else B.META_FP16)
    # the CUDA-core kernels are within 1e-6 of the definition, so the bound is the tensor-core path's own
    got = c.gpu_decode(0)[0]
    assert c.split_k == (batch * heads == 448 and n >= W)
    Hn.assert_attention_close(got, c.gpu_decode(0, simt=True)[0])


# four windows stay with the first block of a cluster, five are dealt out (a cluster of 16 deals from the first on)
@pytest.mark.parametrize("batch,heads,cluster", [(7, 1, 16), (15, 1, 8), (4, 4, 6), (33, 1, 4), (74, 1, 2), (148, 1, 1)])
@pytest.mark.parametrize("n", [32 * 4 + 3, 32 * 5])
def test_one_launch_decode_of_a_few_windows(batch, heads, cluster, n):
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=batch, n_kv_heads=heads, n_q_heads=7 * heads, prefix_text=40, video_chunk=70, audio_chunk=21)
    c = Hn.Case(w, n_tokens=n, meta_format=B.META_MXFP4 if batch % 2 else B.META_FP16)
    assert B.decode_plan(c.cache.c, 1, 0, B.decode_workspace_bytes(c.cache, 1)) == cluster
    Hn.assert_attention_close(c.gpu_decode(0)[0], c.gpu_decode(0, simt=True)[0])


# 16 to 22 units: clusters of six, of which four blocks merge.  No window, one, fewer than the 72 warps, one more, several per warp
@pytest.mark.parametrize("schedule", [B.SCHEDULE_WINDOW, B.SCHEDULE_CAPTION])
@pytest.mark.parametrize("batch,heads,n", [(16, 1, 31), (5, 4, 32), (11, 2, 32 * 13 + 31), (4, 4, 32 * 73), (9, 2, 32 * 200 + 5)])
def test_one_launch_decode_in_clusters_of_six(schedule, batch, heads, n):
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=batch, n_kv_heads=heads, n_q_heads=7 * heads, prefix_text=40, video_chunk=70, audio_chunk=21)
    dev = torch.device("cuda")
    cache = B.Cache(1, batch, heads, 7 * heads, max(8, (n + W - 1) // W) * W, device=dev, schedule=schedule,
                    meta_format=B.META_MXFP4 if batch % 2 else B.META_FP16)
    k, v = WL.gen_kv(w, 0, n_tokens=n)
    signs, R = WL.gen_signs(w, 0).to(dev), WL.gen_rotations(w, 0)[None].contiguous().to(dev)
    mod = WL.modality_layout(w, n).unsqueeze(0).repeat(batch, 1).contiguous().to(dev)
    B.quantize_keys(cache, 0, k.to(dev), signs)
    B.quantize_values(cache, 0, v.to(dev), mod, R)
    q = WL.gen_queries(w, 0).to(dev)
    outs = []
    for splits in (0, 2):   # against the split-K pair
        out = torch.full((1, batch, 7 * heads, D), float("nan"), device=dev)
        ws = Hn.decode_workspace(cache, 1, splits)
        assert (B.decode_plan(cache.c, 1, splits, ws.numel()) == 6) == (splits == 0)
        B.decode_attention(cache, 0, 1, q, signs, R, ws, out, num_splits=splits)
        outs.append(out.cpu().numpy().astype(np.float64))
    Hn.assert_attention_close(outs[0], outs[1])


@pytest.mark.parametrize("meta", [B.META_FP16, B.META_MXFP4])
@pytest.mark.parametrize("n", [100, 128, 128 + 159, 1024 + 127])
@pytest.mark.parametrize("batch", [2, 40])   # clusters of 8, single blocks
def test_one_launch_decode_captioning_schedule(meta, n, batch):
    """Up to four packed windows and 127 raw keys among the raw values; against the split-K pair."""
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=batch)
    dev = torch.device("cuda")
    cache = B.Cache(1, batch, w.n_kv_heads, w.n_q_heads, 1280, device=dev, meta_format=meta, schedule=B.SCHEDULE_CAPTION)
    k, v = WL.gen_kv(w, 0, n_tokens=n)
    signs, R = WL.gen_signs(w, 0).to(dev), WL.gen_rotations(w, 0)[None].contiguous().to(dev)
    mod = WL.modality_layout(w, n).unsqueeze(0).repeat(batch, 1).contiguous().to(dev)
    B.quantize_keys(cache, 0, k.to(dev), signs)
    B.quantize_values(cache, 0, v.to(dev), mod, R)
    q = WL.gen_queries(w, 0).to(dev)
    outs = []
    for splits in (0, 2):
        ws = Hn.decode_workspace(cache, 1, splits)
        out = torch.full((1, batch, w.n_q_heads, D), float("nan"), device=dev)
        B.decode_attention(cache, 0, 1, q, signs, R, ws, out, num_splits=splits)
        assert Hn.ran_split_k(ws) == (splits > 0 and n >= 128 + W)
        outs.append(out.cpu().numpy().astype(np.float64))
    Hn.assert_attention_close(outs[0], outs[1])


# blocks of four sequences (152 of them), the last one partly filled; no packed window, one, several; a full raw tail.
# The matrices may be of any size: the combine kernel's product takes them as they are.
@pytest.mark.parametrize("schedule", [B.SCHEDULE_WINDOW, B.SCHEDULE_CAPTION])
@pytest.mark.parametrize("batch,group,n,size", [(5, 5, 31, 1.0), (6, 8, 32 * 9 + 31, 1.0), (7, 1, 32 * 12, 1e20), (8, 7, 32 * 9 + 1, 1e-20)])
def test_combine_blocks_of_several_sequences(schedule, batch, group, n, size):
    layers, heads, dev = 38, 2, torch.device("cuda")
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=batch, n_kv_heads=heads, n_q_heads=heads * group, prefix_text=40, video_chunk=70, audio_chunk=21)
    cache = B.Cache(layers, batch, heads, heads * group, 32 * 14, device=dev, schedule=schedule)
    k, v = WL.gen_kv(w, 0, n_tokens=n)
    mod = WL.modality_layout(w, n).unsqueeze(0).repeat(batch, 1).contiguous().to(dev)
    signs = torch.stack([WL.gen_signs(w, l) for l in range(layers)]).to(dev)
    R = torch.stack([WL.gen_rotations(w, l) for l in range(layers)])[:, None].contiguous().to(dev)
    for l in range(layers):
        B.quantize_keys(cache, l, k.to(dev).roll(l, dims=2), signs[l])
        B.quantize_values(cache, l, v.to(dev).roll(l, dims=2), mod, R[l])
    q = torch.stack([WL.gen_queries(w, l) for l in range(layers)]).to(dev)
    ref = torch.full((layers, batch, heads * group, D), float("nan"), device=dev)

    def call(ws):
        out = torch.full_like(ref, float("nan"))
        B.decode_attention(cache, 0, layers, q, signs, size * R, ws, out)
        torch.cuda.synchronize()
        return out

    ws = Hn.decode_workspace(cache, layers, 0, call)   # no room for the one-launch kernel's pieces
    assert B.decode_plan(cache.c, layers, 0, ws.numel()) == B.PLAN_PAIR_FOUR
    out = call(ws)
    one = Hn.decode_workspace(cache, 1)
    for l in range(layers):   # the one-launch kernel, whose product is on CUDA cores
        B.decode_attention(cache, l, 1, q[l], signs[l], size * R[l], one, ref[l])
    outs = [x.cpu().numpy().astype(np.float64) for x in (out, ref)]
    top = np.abs(outs[1]).max()
    Hn.assert_attention_close(outs[0] / top, outs[1] / top)


# The combine kernel's product with R_m^T by itself: from the outputs with identity matrices and with none (the raw tail alone) follow the
# rotated sums, and from those in 64 bits the outputs for any other matrices.  Bound: four units in the last place of fp32, norm over
# norm; a chain of rounded fp32 multiply-adds has 2.1e-7 of it, a lost third bf16 term would be 2^-17.
@pytest.mark.parametrize("schedule,batch,group,layers,mod_id", [(B.SCHEDULE_WINDOW, 6, 7, 38, 0), (B.SCHEDULE_WINDOW, 3, 8, 56, 1),
                                                               (B.SCHEDULE_CAPTION, 6, 7, 38, 2)])
def test_combine_product_in_blocks_of_several_sequences(schedule, batch, group, layers, mod_id):
    heads, n, dev = 2, 32 * 12 + 17, torch.device("cuda")
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=batch, n_kv_heads=heads, n_q_heads=heads * group)
    cache = B.Cache(layers, batch, heads, heads * group, 32 * 14, device=dev, schedule=schedule)
    k, v = (x.to(dev) for x in WL.gen_kv(w, 0, n_tokens=n))
    mod = torch.full((batch, n), mod_id, dtype=torch.uint8, device=dev)
    signs = torch.stack([WL.gen_signs(w, l) for l in range(layers)]).to(dev)
    R = torch.stack([WL.gen_rotations(w, l) for l in range(layers)])[:, None].contiguous().to(dev)
    for l in range(layers):
        B.quantize_keys(cache, l, k.roll(l, dims=2), signs[l])
        B.quantize_values(cache, l, v.roll(l, dims=2), mod, R[l])
    q = torch.stack([WL.gen_queries(w, l) for l in range(layers)]).to(dev)

    def call(ws, mats=R):
        out = torch.full((layers, batch, heads * group, D), float("nan"), device=dev)
        B.decode_attention(cache, 0, layers, q, signs, mats, ws, out)
        torch.cuda.synchronize()
        return out.double()

    ws = Hn.decode_workspace(cache, layers, 0, call)   # no room for the one-launch kernel's pieces
    raw = call(ws, torch.zeros_like(R))
    sums = call(ws, torch.eye(D, device=dev).expand_as(R).contiguous()) - raw
    assert B.decode_plan(cache.c, layers, 0, ws.numel()) == B.PLAN_PAIR_FOUR and Hn.ran_split_k(ws)
    ref = torch.einsum("lbhr,lrc->lbhc", sums, R[:, 0, mod_id].double())
    assert (call(ws) - raw - ref).norm() <= 2.0 ** -22 * ref.norm()


# clusters of 1, 2, 4 and 8 blocks (by units and windows); one window; more warps than windows
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("batch,n", [(1, 32), (1, 32 * 9), (12, 32 * 20), (38, 32 * 3)])
def test_ladder_cache_and_decode_over_cluster_sizes(bits, batch, n):
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=batch, prefix_text=5, video_chunk=45, audio_chunk=19)
    c = LadderCase(w, bits, n)
    got = c.gpu_attention()
    # fp32 sums of scores of size up to 2^5 (log2 domain) over 8 tensor-core steps, truncated: 2^5 * 8 * 2^-24 = 1.5e-5 per
    # numerator at the very worst; sums over tokens average it.  The worst (sequence, head) vector may be short: ten times that.
    rel, worst, mx = Hn.attention_errors(got, c.oracle_attention())
    assert rel < 1.5e-5 and worst < 1.5e-4, (rel, worst, mx)
    if batch == 1:
        c.check_cache()


@pytest.mark.parametrize("bulk", [False, True])
def test_value_quantiser_strides(bulk):
    """Heads inside tokens and a broadcast (zero-stride) head: the same records as from a contiguous copy; the default entry
    point takes what a tensor map cannot describe, the bulk one reports it."""
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=2)
    n, dev = 32 * 5 + 7, torch.device("cuda")
    _, v = WL.gen_kv(w, 0, n_tokens=n)
    v = v.to(dev)
    R = WL.gen_rotations(w, 0)[None].contiguous().to(dev)
    mod = WL.modality_layout(w, n).unsqueeze(0).repeat(2, 1).contiguous().to(dev)

    def records(x):
        cache = B.Cache(1, 2, w.n_kv_heads, w.n_q_heads, 192, device=dev)
        B.quantize_values(cache, 0, x, mod, R, bulk=bulk)
        return cache.records.clone(), cache.v_tail.clone(), cache.modality.clone(), cache.seq_len.clone()

    inner = v.transpose(1, 2).contiguous().transpose(1, 2)
    assert all(torch.equal(a, b) for a, b in zip(records(inner), records(v)))
    shared = v[:, :1].expand(2, w.n_kv_heads, n, D)
    if bulk:
        with pytest.raises(B.OkqError) as e:
            records(shared)
        assert e.value.status == B.ERR_UNSUPPORTED
    else:
        assert all(torch.equal(a, b) for a, b in zip(records(shared), records(shared.contiguous())))


@pytest.mark.parametrize("bits", [2, 3, 4])
def test_ladder_values_with_a_broadcast_head(bits):
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=1)
    _, v = WL.gen_kv(w, 0, n_tokens=96)
    R = WL.gen_rotations(w, 0)[None].contiguous().cuda()
    mod = WL.modality_layout(w, 96).unsqueeze(0).contiguous().cuda()
    shared = v.cuda()[:, :1].expand(1, w.n_kv_heads, 96, D)
    caches = [B.LadderCache(1, w.n_kv_heads, w.n_q_heads, 96, bits) for _ in range(2)]
    for c, x in zip(caches, (shared, shared.contiguous())):
        B.ladder_quantize_values(c, x, mod, R)
    assert torch.equal(caches[0].v_codes, caches[1].v_codes) and torch.equal(caches[0].v_norm, caches[1].v_norm)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 193])
@pytest.mark.parametrize("scale", [D ** -0.5, 0.0, -0.05])
def test_calibration_weights_at_tile_edges(n, scale):
    """One more and one fewer than the 128-query and 64-key tiles; a zero and a negative softmax scale."""
    g = torch.Generator().manual_seed(n)
    q = torch.randn(3, n, D, generator=g).half()
    k = torch.randn(n, D, generator=g).half()
    w = B.calib_attention_weights(q.cuda(), k.cuda(), B.calib_workspace(3, n), sm_scale=scale).cpu().double().numpy()
    s = q.double() @ k.double().T * scale
    s = s.masked_fill(torch.ones(n, n).triu(1).bool(), -float("inf"))
    ref = s.softmax(-1).square().sum((0, 1)).numpy()
    # fp32 scores of size up to 2^3: 2^3 * 2^-21 in the exponent, twice for the square
    assert np.abs(w - ref).max() <= 1e-5 * ref.max()


def _matrices():
    g = torch.Generator().manual_seed(3)
    q = torch.linalg.qr(torch.randn(D, D, generator=g, dtype=torch.float64))[0]
    yield "zero", torch.zeros(D, D)
    yield "identity", torch.eye(D)
    yield "rank one", torch.ones(D, D)
    yield "repeated", (q * torch.tensor([5.0] * 40 + [1.0] * 48 + [0.0] * 40, dtype=torch.float64)) @ q.T
    yield "indefinite", (q * torch.linspace(-3, 3, D, dtype=torch.float64)) @ q.T
    yield "zero diagonal", torch.ones(D, D) - torch.eye(D)
    yield "tiny", 1e-30 * ((q * torch.linspace(0, 1, D, dtype=torch.float64)) @ q.T)


@pytest.mark.parametrize("name,C", list(_matrices()), ids=[n for n, _ in _matrices()])
def test_eigen_solver_on_degenerate_matrices(name, C):
    C = (0.5 * (C + C.T)).float().contiguous()
    signs = WL.gen_signs(WL.WORKLOADS["layer7b"], 0)
    R, lam, sweeps = B.calib_rotation(C.cuda(), signs.cuda(), B.calib_workspace(1, 1))
    R, lam = R.cpu().double().numpy(), lam.cpu().double().numpy()
    Cd = C.double().numpy()
    top = max(np.abs(Cd).sum(1).max(), 1e-300)
    assert 0 <= int(sweeps.item()) < 30
    # fp32 outputs of an fp64 solution: 128 products of 2^-24 each
    assert np.abs(R @ R.T - np.eye(D)).max() < 1e-5
    assert (np.diff(lam) <= 0).all()
    assert np.abs(lam - np.sort(np.linalg.eigvalsh(Cd))[::-1]).max() <= 1e-6 * top
    H = CO.hadamard_matrix(signs.numpy())
    assert np.abs(R @ Cd @ R.T - (H * lam) @ H.T).max() <= 1e-5 * top


@pytest.mark.parametrize("bits", [0, 2, 3, 4])
@pytest.mark.parametrize("row,value", [(1e-6, 1.0), (30.0, 1.0), (1e3, 1.0), (1e6, 1.0), (1.0, 4000.0), (1.0, 12000.0)])
def test_value_codes_for_any_matrix(bits, row, value):
    """Matrices with rows shorter and longer than 1, entries beyond fp16, values whose norm fp16 holds just and not at all: the
    codes of the exact chain (which a broadcast head gets), from the hot path's quantiser (0) and the ladder's."""
    n = 32 * 64 + (7 if bits == 0 else 0)
    w = WL.scaled(WL.WORKLOADS["layer7b"], batch=1, n_kv_heads=2, n_q_heads=14)
    g = torch.Generator().manual_seed(5)
    shared = (value * torch.randn(1, 1, n, D, generator=g)).clamp(-65504, 65504).half().cuda().expand(1, 2, n, D)
    R = row * WL.gen_rotations(w, 0)[None].contiguous().cuda()
    mod = WL.modality_layout(w, n).unsqueeze(0).contiguous().cuda()

    def quantised(v):
        if bits:
            c = B.LadderCache(1, 2, 14, n, bits)
            B.ladder_quantize_values(c, v, mod, R)
            return c.v_codes, c.v_norm
        c = B.Cache(1, 1, 2, 14, n + 25)
        B.quantize_values(c, 0, v, mod, R)
        return c.records, c.v_tail

    assert all(torch.equal(a, b) for a, b in zip(quantised(shared), quantised(shared.contiguous())))
