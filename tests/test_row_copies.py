"""What the binding hands to the batched row copies and to the attention over a batch's cache, without a GPU: the library call is
replaced by one that writes down its arguments.  The C entry points get no shapes, so a batch, a row count or a stride that
does not fit has to be refused here (the kernels would read or write past the end of a tensor)."""
import types

import pytest
import torch

from paper_2501_19392_b200 import api, policy

D = 256


@pytest.fixture
def calls(monkeypatch):
    made = []

    def record(name):
        def call(*args):
            made.append((name, args))
            return 0
        return call

    fake = types.SimpleNamespace(**{n: record(n) for n in ("aquakv_copy_rows", "aquakv_decode_attn_cache", "aquakv_destroy")})
    fake.aquakv_decode_attn_buffered_workspace_bytes = fake.aquakv_decode_attn_rope_workspace_bytes = lambda *a: 1024
    monkeypatch.setattr(api, "lib", fake)
    monkeypatch.setattr(api, "_stream", lambda: 0)
    return made


def make_codec():
    c = api.Codec.__new__(api.Codec)
    c.h, c.d, c.code_bytes, c.n_groups, c.torch_dtype, c._ws = None, D, D // 4, 1, torch.bfloat16, None
    return c


def rows(*shape):
    return torch.zeros((*shape, D), dtype=torch.bfloat16)


def make_cache(B=2, L=2):
    return policy.BufferedKVCache(make_codec(), None, L, B, 512, "cpu")


def test_new_tokens_of_more_sequences_than_the_cache_holds(calls):
    cache = make_cache(B=2)
    cache.append([rows(3, 1) for _ in range(2)], [rows(3, 1) for _ in range(2)])
    (name, args), = calls
    assert name == "aquakv_copy_rows" and args[1] == 4 and args[3:5] == (2, 1)      # four tensors, two sequences, one row


@pytest.mark.parametrize("shapes", [
    [(1, 1), (1, 1)],          # a sequence is missing
    [(2, 1), (1, 1)],          # ... of the second layer
])
def test_new_tokens_of_fewer_sequences(calls, shapes):
    cache = make_cache(B=2)
    with pytest.raises(IndexError):
        cache.append([rows(*s) for s in shapes], [rows(*s) for s in shapes])
    assert not calls and cache.n_sinks_held == 0


def test_new_tokens_of_unequal_count(calls):
    with pytest.raises(ValueError):
        make_cache(B=2).append([rows(2, 3), rows(2, 2)], [rows(2, 3), rows(2, 3)])
    assert not calls


@pytest.mark.parametrize("src,dst", [
    (rows(3, 4), rows(2, 4)),
    (rows(2, 4), rows(2, 3)),
    (rows(2, 4)[..., :128], rows(2, 4)[..., :128]),                                  # narrower than a row
    (rows(2, 4), rows(2, 4).float()),
    (torch.zeros((2, D, 4), dtype=torch.bfloat16).transpose(1, 2), rows(2, 4)),       # values of a row are not neighbours
])
def test_copies_that_do_not_fit(calls, src, dst):
    good = (rows(2, 4), rows(2, 4))
    for pairs in ([(src, dst)], [good, (src, dst)]):
        with pytest.raises(ValueError):
            make_codec().copy_rows(pairs)
    assert not calls


def test_copies_that_fit(calls):
    c = make_codec()
    c.copy_rows([])
    c.copy_rows([(rows(2, 9)[:, 1:5], rows(2, 7)[:, :4]), (rows(1, 4).expand(2, 4, D), rows(2, 4))])
    a = calls[1][1][2]
    assert (a[0].ld_src, a[0].pitch_src, a[0].pitch_dst) == (D, 9 * D, 7 * D) and a[1].pitch_src == 0
    one = torch.zeros((5, 1, D + 3), dtype=torch.bfloat16).transpose(0, 1)[..., :D]     # one sequence: its pitch is never used
    c.copy_rows([(one, rows(1, 5))])
    assert calls[2][1][2][0].pitch_src == 0


def attn(q, K16, V16, n16):
    return make_codec().decode_attn_cache(q, None, None, None, None, 0, 2, 0.1, K16, V16, n16)


Q = torch.zeros((2, 4, 128), dtype=torch.bfloat16)


@pytest.mark.parametrize("q,K16,V16,n16", [
    (torch.zeros((2, 8, 128), dtype=torch.bfloat16)[:, :4], rows(2, 9), rows(2, 9), 5),                       # queries apart
    (Q, rows(2, 9), rows(2, 10)[:, :9], 5),                                                                  # values pitched otherwise
    (Q, torch.as_strided(rows(40), (2, 9, D), (9 * D + 8, D, 1)), torch.as_strided(rows(40), (2, 9, D), (9 * D + 8, D, 1)), 5),
    (Q, rows(2, 9), rows(2, 9), 10),                                                                         # more rows than there are
    (Q, rows(1, 9), rows(1, 9), 5),                                                                          # a sequence is missing
    (Q, rows(2, 9), None, 5),
])
def test_uncompressed_rows_that_do_not_fit(calls, q, K16, V16, n16):
    with pytest.raises(ValueError):
        attn(q, K16, V16, n16)
    assert not calls


def test_uncompressed_rows_that_fit(calls):
    attn(Q, rows(2, 9), rows(2, 9), 5)
    attn(Q, rows(2, 9)[..., :], rows(2, 9), 0)
    attn(Q, None, None, 0)
    wide = torch.zeros((2, 9, 2 * D), dtype=torch.bfloat16)[..., :D]
    attn(Q, wide, wide, 9)
    assert [a[1][21:24] for a in calls] == [(5, D, 9), (0, D, 9), (0, D, 0), (9, 2 * D, 9)]
