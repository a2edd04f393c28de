"""Cache policy around the codec (Section 3.3 / Section 4.1: attention sinks and a recent-token buffer in
16 bits, a 4-bit first layer, chunks compressed when the buffer overflows) and the attention over
[compressed | sinks | recent] (aquakv_decode_attn_buffered).

The attention arithmetic is checked teacher-forced, like the other attention tests: the oracle attends
over the SAME rows the kernel attended over (the decoded compressed rows it returns, then the
uncompressed rows), bar 2e-3 of the head's largest output or a one-ulp flip of the 16-bit output.  The
policy itself is plumbing: the cache it builds must equal encoding the same chunks directly."""
import dataclasses
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2501_19392_b200 import synth
from parity import gpu_bits

pytestmark = pytest.mark.gpu
DEV = "cuda"


def make(shape, n):
    from paper_2501_19392_b200 import api
    grid = synth.lloyd_grid(n, seed=7, n_samples=1 << 14, iters=25)
    return api.Codec(shape.d_kv, shape.had_block, shape.scale_group, grid, shape.dtype,
                     synth.hadamard_signs(shape.d_kv, 11), synth.hadamard_signs(shape.d_kv, 12))


def attn_check(out, q, rows_k, rows_v, shape, scale):
    """out [1, n_q, hd] against the oracle's attention over the given 16-bit rows (numpy bits [n, d])."""
    n = rows_k.shape[0]
    ref, _ = oracle.attention(shape.dtype, 1, n, shape.n_q_heads, shape.n_kv_heads, shape.head_dim, scale,
                              synth.to_bits(q.cpu()), rows_k, rows_v)
    o = out.to(torch.float64).cpu().numpy()
    ref_bits = synth.to_bits(torch.from_numpy(ref).to(out.dtype)).astype(np.int64)
    adjacent = np.abs(gpu_bits(out).astype(np.int64) - ref_bits) <= 1
    denom = np.abs(ref).max(axis=-1, keepdims=True)
    assert np.all((np.abs(o - ref) <= 2e-3 * denom) | adjacent)


@pytest.mark.parametrize("ctx,n16,with_pred", [(300, 132, True), (0, 77, False), (1000, 1500, True), (256, 0, True),
                                               (384, 4, False)])
def test_buffered_attention_is_attention_over_the_concatenation(ctx, n16, with_pred):
    from paper_2501_19392_b200 import api
    shape = dataclasses.replace(synth.CONFIGS[5], n_tokens=max(ctx, 1), n_layers=2, batch=1)
    codec = make(shape, 16)
    d, dt = shape.d_kv, shape.dtype
    scale = 1.0 / math.sqrt(shape.head_dim)
    q = synth.random_16bit((1, shape.n_q_heads, shape.head_dim), dt, 1, device=DEV)
    K16 = synth.random_16bit((1, max(n16, 1), d), dt, 2, device=DEV)[:, :n16] if n16 else None
    V16 = synth.random_16bit((1, max(n16, 1), d), dt, 3, device=DEV)[:, :n16] if n16 else None
    if ctx:
        rc = synth.random_cache(dataclasses.replace(shape, n_tokens=ctx), seed=4, device=DEV, n_layers=1)
        ad = synth.random_adapters(shape, seed=5, device=DEV)
        Kp = synth.random_16bit((ctx, d), dt, 6, device=DEV) if with_pred else None
        Vp = synth.random_16bit((ctx, d), dt, 7, device=DEV) if with_pred else None
        Kh = torch.empty((ctx, d), dtype=codec.torch_dtype, device=DEV)
        Vh = torch.empty_like(Kh)
        out, lse = codec.decode_attn_buffered(q, rc.Kcodes[0], rc.Kscales[0], rc.Vcodes[0], rc.Vscales[0], ctx,
                                              shape.n_kv_heads, scale, K16, V16, Kp, Vp,
                                              ad.Wk[1] if with_pred else None, ad.Wv[1] if with_pred else None,
                                              Khat=Kh, Vhat=Vh, want_lse=True)
        rows_k = np.concatenate([gpu_bits(Kh)] + ([gpu_bits(K16[0])] if n16 else []), axis=0)
        rows_v = np.concatenate([gpu_bits(Vh)] + ([gpu_bits(V16[0])] if n16 else []), axis=0)
        if n16 == 0:      # identical to the plain entry point
            out2, _ = codec.decode_attn(q, rc.Kcodes[0], rc.Kscales[0], rc.Vcodes[0], rc.Vscales[0], ctx,
                                        shape.n_kv_heads, scale, Kp, Vp, ad.Wk[1] if with_pred else None,
                                        ad.Wv[1] if with_pred else None)
            assert torch.equal(out, out2)
    else:
        empty_c = torch.empty((0, codec.code_bytes), dtype=torch.uint8, device=DEV)
        empty_s = torch.empty((0, codec.n_groups), dtype=torch.float16, device=DEV)
        out, lse = codec.decode_attn_buffered(q, empty_c, empty_s, empty_c, empty_s, 0, shape.n_kv_heads, scale,
                                              K16, V16, want_lse=True)
        rows_k, rows_v = gpu_bits(K16[0]), gpu_bits(V16[0])
    torch.cuda.synchronize()
    assert codec.poll_status() == 0
    attn_check(out, q, rows_k, rows_v, shape, scale)
    ref, ref_lse = oracle.attention(dt, 1, rows_k.shape[0], shape.n_q_heads, shape.n_kv_heads, shape.head_dim, scale,
                                    synth.to_bits(q.cpu()), rows_k, rows_v)
    assert np.abs(lse.cpu().numpy() - ref_lse).max() <= 1e-4


def test_policy_keeps_sinks_and_recent_tokens_and_compresses_the_rest():
    from paper_2501_19392_b200 import api, policy
    B, L, total = 2, 3, 4 + 128 + 128 + 45          # sinks + one flushed chunk + a partly filled buffer
    shape = dataclasses.replace(synth.CONFIGS[5], n_tokens=B * total, n_layers=L, batch=B)
    codec, codec0 = make(shape, 16), make(shape, 256)          # 2-bit layers, 4-bit first layer
    d, dt = shape.d_kv, shape.dtype
    kv = synth.kv_chain(shape, seed=21, device=DEV)
    ad = synth.random_adapters(shape, seed=22, device=DEV)
    K = [k.view(B, total, d) for k in kv.K]
    V = [v.view(B, total, d) for v in kv.V]
    cache = policy.BufferedKVCache(codec, ad, L, B, max_tokens=512, device=DEV, first_layer_codec=codec0)
    # a prefill of 200 tokens, then single-token steps
    cache.append([k[:, :200] for k in K], [v[:, :200] for v in V])
    assert (cache.ctx, cache.fill, cache.n_sinks_held) == (0, 196, 4)
    for t in range(200, total):
        cache.append([k[:, t:t + 1] for k in K], [v[:, t:t + 1] for v in V])
    assert (cache.ctx, cache.n_uncompressed) == (128, 4 + 128 + 45)
    torch.cuda.synchronize()
    assert codec.poll_status() == 0 and codec0.poll_status() == 0
    for b in range(B):
        for l in range(L):
            # uncompressed rows: the sinks, then tokens 132 .. total-1 in order
            exp = torch.cat([K[l][b, :4], K[l][b, 132:total]], dim=0)
            assert torch.equal(cache.K16[l][b, :cache.n_uncompressed], exp)
        # the compressed chunk is tokens 4 .. 131 encoded through the layers, first layer at 4 bits
        Kc0, Ks0, Vc0, Vs0, Kh, Vh = codec0.encode(K[0][b, 4:132].contiguous(), V[0][b, 4:132].contiguous())
        assert torch.equal(cache.Kcodes[0][b, :128], Kc0) and torch.equal(cache.Vscales[0][b, :128], Vs0)
        assert cache.Kcodes[0].shape[2] == 2 * cache.Kcodes[1].shape[2]
        for l in range(1, L):
            Kc, Ks, Vc, Vs, Kh, Vh = codec.encode(K[l][b, 4:132].contiguous(), V[l][b, 4:132].contiguous(), Kh, Vh,
                                                  ad.Wk[l], ad.Wv[l])
            assert torch.equal(cache.Kcodes[l][b, :128], Kc) and torch.equal(cache.Vcodes[l][b, :128], Vc)
            assert torch.equal(cache.Kscales[l][b, :128], Ks) and torch.equal(cache.Vscales[l][b, :128], Vs)
    # attention of every layer over [compressed | sinks | recent], teacher-forced on the decoded rows
    scale = 1.0 / math.sqrt(shape.head_dim)
    q = [synth.random_16bit((B, shape.n_q_heads, shape.head_dim), dt, 30 + l, device=DEV) for l in range(L)]
    outs = cache.attend(q, shape.n_kv_heads, scale)
    torch.cuda.synchronize()
    assert codec.poll_status() == 0 and codec0.poll_status() == 0
    for b in range(B):
        Kh = Vh = None
        for l in range(L):
            cdc = codec0 if l == 0 else codec
            args = (cache.Kcodes[l][b, :128], cache.Kscales[l][b, :128], cache.Vcodes[l][b, :128], cache.Vscales[l][b, :128])
            Kh, Vh = cdc.decode(*args, Kh, Vh, ad.Wk[l] if l else None, ad.Wv[l] if l else None)
            n16 = cache.n_uncompressed
            rows_k = np.concatenate([gpu_bits(Kh), gpu_bits(cache.K16[l][b, :n16])], axis=0)
            rows_v = np.concatenate([gpu_bits(Vh), gpu_bits(cache.V16[l][b, :n16])], axis=0)
            attn_check(outs[l][b:b + 1], q[l][b:b + 1], rows_k, rows_v, shape, scale)
    # the same with the cached keys taken as pre-RoPE keys of tokens 0 .. total-1 (Section 3.3): sinks at
    # 0 .. 3, compressed tokens at 4 .. 131, recent rows at 132 ..
    from oracle import rope as orope
    base = 500000.0
    table = codec.rope_table(shape.head_dim, base, total, DEV)
    outs_r = cache.attend(q, shape.n_kv_heads, scale, rope_table=table)
    torch.cuda.synchronize()
    assert codec.poll_status() == 0 and codec0.poll_status() == 0
    positions = np.concatenate([4 + np.arange(128), np.arange(4), np.arange(132, total)])
    for b in range(B):
        Kh = Vh = None
        for l in range(L):
            cdc = codec0 if l == 0 else codec
            args = (cache.Kcodes[l][b, :128], cache.Kscales[l][b, :128], cache.Vcodes[l][b, :128], cache.Vscales[l][b, :128])
            Kh, Vh = cdc.decode(*args, Kh, Vh, ad.Wk[l] if l else None, ad.Wv[l] if l else None)
            n16 = cache.n_uncompressed
            rows_k = np.concatenate([gpu_bits(Kh), gpu_bits(cache.K16[l][b, :n16])], axis=0)
            rows_v = np.concatenate([gpu_bits(Vh), gpu_bits(cache.V16[l][b, :n16])], axis=0)
            ref, _ = orope.attention_rope(dt, 1, rows_k.shape[0], shape.n_q_heads, shape.n_kv_heads, shape.head_dim,
                                          scale, synth.to_bits(q[l][b:b + 1].cpu()), rows_k, rows_v, positions, base)
            o = outs_r[l][b:b + 1]
            ref_bits = synth.to_bits(torch.from_numpy(ref).to(o.dtype)).astype(np.int64)
            adjacent = np.abs(gpu_bits(o).astype(np.int64) - ref_bits) <= 1
            assert np.all((np.abs(o.to(torch.float64).cpu().numpy() - ref) <= 2e-3 * np.abs(ref).max(axis=-1, keepdims=True))
                          | adjacent)
            assert not torch.equal(o, outs[l][b:b + 1])


@pytest.mark.parametrize("cfg,batch,ctx,n16,rope", [
    (5, 3, 1, 5, True),          # one token per sequence
    (5, 2, 1025, 9, False),      # one token past an attention block; the uncompressed rows fill their room
    (7, 4, 130, 3, True),        # d_kv 512
    (6, 5, 0, 4, True),          # nothing compressed
])
def test_uncompressed_rows_with_room_to_grow(cfg, batch, ctx, n16, rope):
    """decode_attn_cache on a batch whose caches and uncompressed rows have room to grow against decode_attn_buffered /
    decode_attn_rope of each sequence by itself: the arithmetic is the same, so the results agree bit for bit."""
    room, room16 = 1400, 9
    shape = dataclasses.replace(synth.CONFIGS[cfg], n_tokens=batch * room, n_layers=2, batch=batch)
    codec = make(shape, 16)
    d, dt, scale, hd = shape.d_kv, shape.dtype, 1.0 / math.sqrt(shape.head_dim), shape.head_dim
    rnd = lambda s, *sh: synth.random_16bit(sh, dt, s, device=DEV)
    K16, V16, q = rnd(1, batch, room16, d), rnd(2, batch, room16, d), rnd(3, batch, shape.n_q_heads, hd)
    prev = [rnd(5, batch * ctx, d), rnd(6, batch * ctx, d)] if ctx else [None, None]
    ad = synth.random_adapters(shape, seed=7, device=DEV)
    W = [ad.Wk[1], ad.Wv[1]] if ctx else [None, None]
    rc = synth.random_cache(shape, seed=8, device=DEV, n_layers=1)
    full = [x[0].view(batch, room, -1) for x in (rc.Kcodes, rc.Kscales, rc.Vcodes, rc.Vscales)]
    cache = [torch.empty((batch * ctx, x.shape[2]), dtype=x.dtype, device=DEV) for x in full]
    if ctx:
        codec.copy_cache(full, cache, batch, ctx, room, ctx)
        back = [torch.zeros_like(x) for x in full]
        codec.copy_cache(cache, back, batch, ctx, ctx, room)
        for x, y, z in zip(full, cache, back):
            assert torch.equal(x[:, :ctx].reshape(batch * ctx, x.shape[2]), y)
            assert torch.equal(x[:, :ctx], z[:, :ctx]) and not z[:, ctx:].any()
    table = codec.rope_table(hd, 5e5, ctx + n16 + 4, DEV) if rope else None
    pos16 = torch.arange(n16, dtype=torch.int32, device=DEV) if rope else None
    out = codec.decode_attn_cache(q, *cache, ctx, shape.n_kv_heads, scale, K16, V16, n16, table, 2, pos16, *prev, *W)
    torch.cuda.synchronize()
    assert codec.poll_status() == 0
    for b in range(batch):
        p = [x[b * ctx:(b + 1) * ctx] if x is not None else None for x in prev]
        args = (q[b:b + 1], *[c[b * ctx:(b + 1) * ctx] for c in cache], ctx, shape.n_kv_heads, scale)
        rows = (K16[b:b + 1, :n16], V16[b:b + 1, :n16])
        if rope:
            ref, _ = codec.decode_attn_rope(*args, table, 2, *rows, pos16, *p, *W)
        else:
            ref, _ = codec.decode_attn_buffered(*args, *rows, *p, *W)
        assert torch.equal(ref, out[b:b + 1])


def test_copy_rows_moves_strided_blocks_of_many_tensors():
    shape = dataclasses.replace(synth.CONFIGS[7], n_tokens=1)
    codec = make(shape, 16)
    g = torch.Generator(device=DEV).manual_seed(3)
    src = [torch.randn((3, 11, shape.d_kv), generator=g, device=DEV).to(codec.torch_dtype) for _ in range(70)]   # more than one launch holds
    dst = [torch.zeros_like(x) for x in src]
    codec.copy_rows((x[:, 2:7], y[:, 5:10]) for x, y in zip(src, dst))
    torch.cuda.synchronize()
    for x, y in zip(src, dst):
        assert torch.equal(y[:, 5:10], x[:, 2:7]) and not y[:, :5].any() and not y[:, 10:].any()


def filled_cache(B, ctx, fill, L=2, cfg=5, seed=40):
    """A cache policy object in the middle of a conversation, with random contents, and queries for it."""
    from paper_2501_19392_b200 import policy
    shape = dataclasses.replace(synth.CONFIGS[cfg], n_tokens=B * (ctx + 256), n_layers=L, batch=B)
    codec, codec0 = make(shape, 16), make(shape, 256)
    ad = synth.random_adapters(shape, seed=seed, device=DEV)
    cache = policy.BufferedKVCache(codec, ad, L, B, max_tokens=ctx + 256, device=DEV, first_layer_codec=codec0)
    for l in range(L):
        rc = synth.random_cache(dataclasses.replace(shape, n_layers=1, grid_size=256 if l == 0 else 16), seed=seed + 1 + l,
                                device=DEV, n_layers=1)
        for mine, theirs in ((cache.Kcodes, rc.Kcodes), (cache.Vcodes, rc.Vcodes), (cache.Kscales, rc.Kscales), (cache.Vscales, rc.Vscales)):
            mine[l].copy_(theirs[0].view(mine[l].shape))
        cache.K16[l].copy_(synth.random_16bit(tuple(cache.K16[l].shape), shape.dtype, seed + 10 + l, device=DEV))
        cache.V16[l].copy_(synth.random_16bit(tuple(cache.V16[l].shape), shape.dtype, seed + 20 + l, device=DEV))
    cache.ctx, cache.fill, cache.n_sinks_held = ctx, fill, cache.n_sink
    q = [synth.random_16bit((B, shape.n_q_heads, shape.head_dim), shape.dtype, seed + 30 + l, device=DEV) for l in range(L)]
    return cache, shape, q


@pytest.mark.parametrize("rope", [False, True])
def test_queries_that_do_not_follow_one_another(rope):
    """The last position of [batch, positions, heads, head_dim] queries: dense within a sequence, apart between sequences."""
    cache, shape, q = filled_cache(3, 200, 40)
    table = cache.codec.rope_table(shape.head_dim, 5e5, 400, DEV) if rope else None
    scale = 1.0 / math.sqrt(shape.head_dim)
    ref = cache.attend(q, shape.n_kv_heads, scale, rope_table=table)
    apart = []
    for x in q:
        big = torch.full((x.shape[0], 5, *x.shape[1:]), 7.0, dtype=x.dtype, device=DEV)
        big[:, -1] = x
        apart.append(big[:, -1])
    assert not apart[0].is_contiguous()
    for r, o in zip(ref, cache.attend(apart, shape.n_kv_heads, scale, rope_table=table)):
        assert torch.equal(r, o)


@pytest.mark.parametrize("rope", [False, True])
def test_sequences_served_in_several_groups(rope, monkeypatch):
    """Five sequences in one group, in groups of two, two and one, and one by one (a context longer than a group): the same
    results bit for bit."""
    from paper_2501_19392_b200 import policy
    ctx, outs = 300, []
    for tokens in (policy.GROUP_TOKENS, 2 * ctx, 2 * ctx + ctx // 2, ctx - 1):
        monkeypatch.setattr(policy, "GROUP_TOKENS", tokens)
        cache, shape, q = filled_cache(5, ctx, 40, L=3)        # its own scratch, sized for these groups
        table = cache.codec.rope_table(shape.head_dim, 5e5, 500, DEV) if rope else None
        outs.append(cache.attend(q, shape.n_kv_heads, 1.0 / math.sqrt(shape.head_dim), rope_table=table))
        torch.cuda.synchronize()
        assert cache.codec.poll_status() == 0 and cache.codec0.poll_status() == 0
    for other in outs[1:]:
        for a, b in zip(outs[0], other):
            assert torch.equal(a, b)


@pytest.mark.parametrize("queries", [2, 4])
def test_queries_of_fewer_or_more_sequences_than_the_cache_holds(queries, monkeypatch):
    """Queries of the first sequences are served, whatever the groups, and surplus ones are not looked at."""
    from paper_2501_19392_b200 import policy
    cache, shape, q = filled_cache(3, 200, 40)
    scale = 1.0 / math.sqrt(shape.head_dim)
    ref = cache.attend(q, shape.n_kv_heads, scale)
    other = [torch.cat([x, x])[:queries] for x in q]
    for tokens in (policy.GROUP_TOKENS, 2 * 200, 1):
        monkeypatch.setattr(policy, "GROUP_TOKENS", tokens)
        for r, o in zip(ref, cache.attend(other, shape.n_kv_heads, scale)):
            n = min(3, queries)
            assert o.shape[0] == queries and torch.equal(r[:n], o[:n])
    assert cache.codec.poll_status() == 0
