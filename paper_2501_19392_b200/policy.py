"""Cache policy around the codec (Section 3.3; Section 4.1 "Evaluation setup": the first four
tokens, the attention sinks, and a buffer of the 128 newest tokens are left uncompressed, and the first layer
gets 4 bits per value): the first `n_sink` tokens and the most recent tokens stay in
16 bits, older tokens are compressed in chunks of `chunk` tokens whenever the recent buffer holds
`recent + chunk` of them, and every query attends to [compressed | sinks | recent] in one call.

Host policy only: bookkeeping of which rows are where.  Compression is aquakv_encode on the flushed
chunks (layer by layer, the chunks' own reconstructions feeding the next layer), row movement is aquakv_copy_rows and
aquakv_copy_cache (all sequences, and all layers where that is possible, in one launch), attention is
aquakv_decode_attn_cache.  Sequences of a batch advance in lockstep (the same number of tokens each) and are served
together: a call for one sequence of a few thousand tokens leaves most of the chip idle.  Keys are cached as given; with a rotary table (`attend(..., rope_table=...)`, Section 3.3
"Positional embeddings": keys are compressed before RoPE) they are taken as pre-RoPE keys of tokens 0, 1, ...
and rotated by their positions when attended to: sinks at 0 .. n_sink-1, compressed
token t at n_sink + t, the recent rows after them.
"""
from __future__ import annotations

from typing import List, Optional

import torch

from . import api, chain


# Tokens that one attention pass decodes at a time (more only for a single longer sequence): enough to fill the chip for
# 28 waves of the layer kernel, and the decoded rows of a layer and its predecessor take 1 GB at d_kv = 1024.
GROUP_TOKENS = 131072


class BufferedKVCache:
    def __init__(self, codec: api.Codec, adapters, n_layers: int, batch: int, max_tokens: int, device,
                 n_sink: int = 4, recent: int = 128, chunk: int = 128, first_layer_codec: Optional[api.Codec] = None):
        """first_layer_codec: a codec with a finer grid for layer 0 (the paper's 4-bit first layer); layer 0 has
        no predictor, so only its code size differs."""
        self.codec, self.codec0 = codec, first_layer_codec or codec
        self.ad, self.L, self.B, self.dev = adapters, n_layers, batch, device
        self.n_sink, self.recent, self.chunk = n_sink, recent, chunk
        self.cap = recent + chunk                      # rows of the recent buffer
        self.max_ctx = max_tokens
        d, dt = codec.d, codec.torch_dtype
        mk = lambda *shape, dtype=dt: torch.zeros(shape, dtype=dtype, device=device)
        # uncompressed rows per layer and sequence: [sinks | recent buffer], valid rows are a prefix
        self.K16 = [mk(batch, n_sink + self.cap, d) for _ in range(n_layers)]
        self.V16 = [mk(batch, n_sink + self.cap, d) for _ in range(n_layers)]
        cb = lambda l: (self.codec0 if l == 0 else codec).code_bytes
        self.Kcodes = [mk(batch, max_tokens, cb(l), dtype=torch.uint8) for l in range(n_layers)]
        self.Vcodes = [mk(batch, max_tokens, cb(l), dtype=torch.uint8) for l in range(n_layers)]
        self.Kscales = [mk(batch, max_tokens, codec.n_groups, dtype=torch.float16) for _ in range(n_layers)]
        self.Vscales = [mk(batch, max_tokens, codec.n_groups, dtype=torch.float16) for _ in range(n_layers)]
        self.n_sinks_held = 0       # sink rows filled so far
        self.fill = 0               # valid rows of the recent buffer
        self.ctx = 0                # compressed tokens per sequence
        self._bufs = chain.PingPong(codec, batch * chunk, device)
        self._stage = [mk(batch, chunk, d) for _ in range(2)]                  # a layer's chunk of keys / values
        self._stage_cache = self._compact_cache(batch * chunk)                 # and what it is compressed to
        self._dec = None            # ping-pong buffers of the attention pass and a layer's packed cache, sized on demand
        self._dec_cache = None

    def _compact_cache(self, rows: int):
        cb = max(self.codec.code_bytes, self.codec0.code_bytes)
        mk = lambda w, dt: torch.empty(rows * w, dtype=dt, device=self.dev)
        return [mk(cb, torch.uint8), mk(self.codec.n_groups, torch.float16), mk(cb, torch.uint8), mk(self.codec.n_groups, torch.float16)]

    # -- appending ------------------------------------------------------------------------------
    def append(self, K: List[torch.Tensor], V: List[torch.Tensor]) -> None:
        """K[l], V[l]: [batch, n_new, d_kv] 16-bit, the new tokens' keys / values of every layer."""
        n_new = K[0].shape[1]
        t = 0
        while t < n_new:
            if self.n_sinks_held < self.n_sink:
                n = min(self.n_sink - self.n_sinks_held, n_new - t)
                self._store(K, V, t, n, self.n_sinks_held)
                self.n_sinks_held += n
            else:
                n = min(self.cap - self.fill, n_new - t)
                self._store(K, V, t, n, self.n_sink + self.fill)
                self.fill += n
                if self.fill == self.cap:
                    self._flush()
            t += n

    def _store(self, K, V, t, n, row):
        pairs = []
        for x, y in ((K, self.K16), (V, self.V16)):
            for l in range(self.L):
                new = x[l]
                if len(new) != self.B:
                    if len(new) < self.B:
                        raise IndexError("append: new tokens of fewer than %d sequences" % self.B)
                    new = new[:self.B]
                pairs.append((new[:, t:t + n], y[l][:, row:row + n]))
        self.codec.copy_rows(pairs)

    def _flush(self):
        """Compresses the oldest `chunk` rows of the recent buffer (all layers) and closes the gap."""
        assert self.ctx + self.chunk <= self.max_ctx, "compressed cache is full"
        s0, c, r = self.n_sink, self.chunk, self.recent
        self._encode_chunk(s0, c)
        # the remaining `recent` rows move to the front of the buffer, piece by piece: a piece's destination is what the
        # piece before it has left
        for o in range(0, r, c):
            n = min(c, r - o)
            self.codec.copy_rows((x[l][:, s0 + c + o:s0 + c + o + n], x[l][:, s0 + o:s0 + o + n])
                                 for x in (self.K16, self.V16) for l in range(self.L))
        self.fill -= c
        self.ctx += c

    def _encode_chunk(self, s0, c):
        """Algorithm 2 over the layers for one chunk of every sequence; layer 0 through the first-layer codec."""
        bufs, ad, n, dst = self._bufs, self.ad, self.B * c, self._stage_cache
        K, V = self._stage
        for l in range(self.L):
            cur, prv, has = l % 2, (l + 1) % 2, l > 0
            cdc = self.codec if has else self.codec0
            cdc.copy_rows([(self.K16[l][:, s0:s0 + c], K), (self.V16[l][:, s0:s0 + c], V)])
            cdc.encode(K.view(n, -1), V.view(n, -1), bufs.K[prv] if has else None, bufs.V[prv] if has else None,
                       ad.Wk[l] if has else None, ad.Wv[l] if has else None, ad.bk[l] if has else None,
                       ad.bv[l] if has else None, *dst, bufs.K[cur], bufs.V[cur])
            sl = slice(self.ctx, self.ctx + c)
            cdc.copy_cache(dst, [x[l][:, sl] for x in (self.Kcodes, self.Kscales, self.Vcodes, self.Vscales)], self.B, c, c,
                           self.max_ctx)

    # -- attention ------------------------------------------------------------------------------
    @property
    def n_uncompressed(self) -> int:
        return self.n_sinks_held + self.fill

    def attend(self, q: List[torch.Tensor], n_kv_heads: int, softmax_scale: float,
               rope_table: Optional[torch.Tensor] = None) -> List[torch.Tensor]:
        """The decode-and-attend loop of Algorithm 4 for every layer: q[l] [batch, n_q_heads, head_dim] -> outputs of the same shape.
        The decoded compressed rows of layer l feed layer l + 1's predictors and are dropped afterwards.
        rope_table (Codec.rope_table): the cached keys are pre-RoPE and are rotated by their positions; q[l] must
        be rotated by the caller."""
        q = [x.contiguous() for x in q]         # several sequences are one call, and a call's queries follow one another
        out = [torch.empty_like(x) for x in q]
        B = min(self.B, len(q[0]))              # queries of the first sequences only are served
        n16 = self.n_uncompressed
        pos16 = None
        if rope_table is not None and n16:
            first_recent = self.n_sinks_held + self.ctx
            pos16 = torch.cat([torch.arange(self.n_sinks_held, dtype=torch.int32, device=self.dev),
                               torch.arange(first_recent, first_recent + self.fill, dtype=torch.int32, device=self.dev)])
        group = max(1, min(B, GROUP_TOKENS // max(self.ctx, 1)))      # sequences decoded together
        if self.ctx > 0 and (self._dec is None or self._dec.K[0].shape[0] < group * self.ctx):
            rows = max(self.max_ctx, min(self.B * self.max_ctx, GROUP_TOKENS))      # enough for every later context
            self._dec = self._dec_cache = None                                      # the old buffers make room first
            self._dec, self._dec_cache = chain.PingPong(self.codec, rows, self.dev), self._compact_cache(rows)
        for b in range(0, B, group):
            bs = slice(b, min(b + group, B))
            of = lambda x: x if len(x) == group == B else x[bs]        # a tensor's part for these sequences
            n = (bs.stop - b) * self.ctx
            for l in range(self.L):
                cur, prv = l % 2, (l + 1) % 2
                has, dec = l > 0 and n > 0, self._dec if n > 0 else None
                cdc = self.codec0 if l == 0 else self.codec
                cache = [of(x[l]) for x in (self.Kcodes, self.Kscales, self.Vcodes, self.Vscales)]
                if bs.stop - b > 1 and n > 0:       # one sequence's rows are compact as they are
                    cdc.copy_cache(cache, self._dec_cache, bs.stop - b, self.ctx, self.max_ctx, self.ctx)
                    cache = self._dec_cache
                cdc.decode_attn_cache(
                    of(q[l]), *cache, self.ctx, n_kv_heads, softmax_scale, of(self.K16[l]) if n16 else None,
                    of(self.V16[l]) if n16 else None, n16, rope_table, self.n_sinks_held, pos16,
                    dec.K[prv][:n] if has else None, dec.V[prv][:n] if has else None, self.ad.Wk[l] if has else None,
                    self.ad.Wv[l] if has else None, self.ad.bk[l] if has else None, self.ad.bv[l] if has else None,
                    out=of(out[l]), Khat=dec.K[cur][:n] if dec else None, Vhat=dec.V[cur][:n] if dec else None)
        return out
