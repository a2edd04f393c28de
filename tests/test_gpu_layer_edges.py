"""One predicted layer through the layer kernel against the single-phase entry points at the edges of its waves: the widths of
the GEMM's tiles in a short last wave, one warp per row for d_kv <= 512, one poller and one report per CTA.

The two paths share no kernel but form the same sums in the same order (fp32 accumulation over the input features, ascending)
and the same roundings in the rows, so everything has to agree bit for bit."""
import numpy as np
import pytest
import torch

from paper_2501_19392_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
# d_kv 1024 on 148 SMs: 36 token blocks of 128 a wave; up to 8 blocks in the last one take tiles of 64 features, up to 18 of
# 128, more of 256.  d_kv 512: 74 blocks, 18 and 37; d_kv 256: 148 blocks, 37 and 74 (of 148 token-block slots).
CASES = [(1024, 1024, t) for t in (1, 129, 1024, 1025, 2304, 2305, 4608, 4609, 5633)] + [
    (512, 512, t) for t in (1, 300, 2304, 2305, 4736, 9472, 9473)] + [(512, 64, t) for t in (257, 2305, 9600)] + [
    (512, 128, 700), (1024, 64, 1300), (256, 256, 130), (256, 64, 4737), (256, 256, 18945)]


GRIDS = [(16, synth.BF16), (64, synth.F16), (256, synth.BF16)]


@pytest.mark.parametrize("d,h,T,n,dtype", [c + g for g in GRIDS for c in CASES if g[0] == 16 or c[2] <= 5000])     # the large calls with one grid only
def test_layer_calls_equal_the_phases(d, h, T, n, dtype):
    from paper_2501_19392_b200 import api
    grid = synth.lloyd_grid(n, seed=7, n_samples=1 << 13, iters=8)
    codec = api.Codec(d, h, h, grid, dtype, synth.hadamard_signs(d, 11), synth.hadamard_signs(d, 12))
    row = lambda seed: synth.random_16bit((T, d), dtype, seed, device=DEV)
    K, V, Kp, Vp = (row(s) for s in (1, 2, 3, 4))
    Wk = (synth.random_16bit((d, d), dtype, 5, device=DEV).float() / d ** 0.5).to(K.dtype)
    Wv = (synth.random_16bit((d, 2 * d), dtype, 6, device=DEV).float() / (2 * d) ** 0.5).to(K.dtype)
    bk, bv = (torch.linspace(-0.2, 0.3, d, device=DEV) for _ in range(2))
    got = codec.encode(K, V, Kp, Vp, Wk, Wv, bk, bv)
    ck, sk, kh = codec.encode_phase(api.ROLE_KEY, K, Kp, None, Wk, bk)
    cv, sv, vh = codec.encode_phase(api.ROLE_VALUE, V, Vp, kh, Wv, bv)
    for a, b in zip(got, (ck, sk, cv, sv, kh, vh)):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    back = codec.decode(ck, sk, cv, sv, Kp, Vp, Wk, Wv, bk, bv)
    assert torch.equal(back[0], kh) and torch.equal(back[1], vh)
    assert codec.poll_status() == 0


@pytest.mark.parametrize("d,h,T", [(1024, 1024, 42000), (1024, 64, 30000), (512, 512, 60000), (512, 64, 60000), (256, 256, 90000)])
def test_repeated_calls_of_many_waves_equal_the_phases(d, h, T):
    """The prediction ring is reused every three jobs, its lines read and discarded by the row warps, then written by the
    TMA stores of other CTAs: a store that a late discard or read overtakes would show as wrong rows now and then."""
    from paper_2501_19392_b200 import api
    grid = synth.lloyd_grid(16, seed=7, n_samples=1 << 13, iters=8)
    codec = api.Codec(d, h, h, grid, synth.BF16, synth.hadamard_signs(d, 11), synth.hadamard_signs(d, 12))
    K, V, Kp, Vp = (synth.random_16bit((T, d), synth.BF16, s, device=DEV) for s in (1, 2, 3, 4))
    Wk = (synth.random_16bit((d, d), synth.BF16, 5, device=DEV).float() / d ** 0.5).to(K.dtype)
    Wv = (synth.random_16bit((d, 2 * d), synth.BF16, 6, device=DEV).float() / (2 * d) ** 0.5).to(K.dtype)
    ck, sk, kh = codec.encode_phase(api.ROLE_KEY, K, Kp, None, Wk)
    cv, sv, vh = codec.encode_phase(api.ROLE_VALUE, V, Vp, kh, Wv)
    for _ in range(8):
        for a, b in zip(codec.encode(K, V, Kp, Vp, Wk, Wv), (ck, sk, cv, sv, kh, vh)):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
        back = codec.decode(ck, sk, cv, sv, Kp, Vp, Wk, Wv)
        assert torch.equal(back[0], kh) and torch.equal(back[1], vh)
    assert codec.poll_status() == 0


def make_codec(d, h, n, dtype=synth.BF16):
    from paper_2501_19392_b200 import api
    grid = synth.lloyd_grid(n, seed=7, n_samples=1 << 13, iters=8)
    return api.Codec(d, h, h, grid, dtype, synth.hadamard_signs(d, 11), synth.hadamard_signs(d, 12))


def extreme_rows(d, h, T, dtype):
    """Rows around the border of the search table and beyond it (k of a block's h rotated values are +-sqrt(h / k), the
    others zero: 4.5 to 32 standard deviations), rows that are not finite, zeros, and ordinary ones."""
    rng = np.random.default_rng(d + h)
    H = np.array([[1.0]])
    while H.shape[0] < h:
        H = np.block([[H, H], [H, -H]])
    x = rng.standard_normal((T, d))
    ks = [k for k in (1, 1, 2, 3, 5, 12, 20, 40, 47, 49, 52, 64, 100, 200) if k <= h // 2]
    for r in range(0, T, 3):
        k = ks[(r // 3) % len(ks)]
        y = np.zeros((d // h, h))
        for b in range(d // h):
            y[b, rng.choice(h, size=k, replace=False)] = rng.choice([-1.0, 1.0], size=k) * np.sqrt(h / k)
        x[r] = (y @ H / np.sqrt(h)).reshape(d) * synth.hadamard_signs(d, 11)
    x[1] = 0.0
    for r, v in ((4, np.nan), (7, np.inf), (10, -np.inf), (T - 1, np.nan)):
        x[r, (5 * r) % d] = v
    return torch.from_numpy(x).to(synth.torch_dtype(dtype)).to(DEV)


@pytest.mark.parametrize("d,h,n,dtype", [(256, 256, 16, synth.BF16), (256, 64, 64, synth.F16), (512, 512, 16, synth.F16), (512, 512, 256, synth.BF16),
                                         (512, 64, 64, synth.BF16), (1024, 1024, 64, synth.BF16), (1024, 64, 16, synth.F16)])
def test_extreme_rows_with_a_prediction_of_zero_equal_those_without_predictor(d, h, n, dtype):
    """The layer kernel's row routines against the stand-alone ones: a predictor of zeros changes no bit of a row."""
    T = 500
    codec = make_codec(d, h, n, dtype)
    K, V = extreme_rows(d, h, T, dtype), extreme_rows(d, h, T, dtype).flip(0).contiguous()
    prev = synth.random_16bit((T, d), dtype, 3, device=DEV)
    Wk, Wv = torch.zeros((d, d), dtype=K.dtype, device=DEV), torch.zeros((d, 2 * d), dtype=K.dtype, device=DEV)
    want, got = codec.encode(K, V), codec.encode(K, V, prev, prev, Wk, Wv)
    back, plain = codec.decode(*want[:4], prev, prev, Wk, Wv), codec.decode(*want[:4])
    assert codec.poll_status() == 0
    rows = want[4].isfinite().all(1)                     # a value's prediction multiplies its reconstructed key: 0 x infinity
    assert rows.sum() >= T - 4
    same = lambda a, b: torch.equal(a.isnan(), b.isnan()) and torch.equal(a.nan_to_num(), b.nan_to_num())
    for i in (0, 1):
        assert torch.equal(got[i], want[i]) and torch.equal(got[2 + i][rows], want[2 + i][rows])
    for g, w in ((got[4:], want[4:]), (back, plain)):
        assert same(g[0], w[0]) and same(g[1][rows], w[1][rows])


@pytest.mark.parametrize("d,h,T", [(256, 256, 81000), (256, 64, 700), (512, 512, 42000), (512, 512, 90), (512, 64, 42000), (1024, 1024, 21000), (1024, 128, 21000)])
def test_strided_rows_and_calls_without_reconstructions(d, h, T):
    """Inputs and outputs with other strides than d_kv, nothing beside the rows written; without reconstructions (the keys then
    live in a ring of three waves) the same codes."""
    codec = make_codec(d, h, 16)
    wide = lambda w, s: synth.random_16bit((T, d + w), synth.BF16, s, device=DEV)[:, :d]
    K, V = wide(64, 1), wide(64, 2)
    Kp, Vp = wide(8, 3), wide(8, 4)
    Wk = (synth.random_16bit((d, d), synth.BF16, 5, device=DEV).float() / d ** 0.5).to(K.dtype)
    Wv = (synth.random_16bit((d, 2 * d), synth.BF16, 6, device=DEV).float() / (2 * d) ** 0.5).to(K.dtype)
    want = codec.encode(*(x.contiguous() for x in (K, V, Kp, Vp)), Wk, Wv)
    out = [torch.full((T, d + 24), 3.0, dtype=K.dtype, device=DEV) for _ in range(4)]
    got = codec.encode(K, V, Kp, Vp, Wk, Wv, Khat=out[0][:, :d], Vhat=out[1][:, :d])
    bare = codec.encode(K, V, Kp, Vp, Wk, Wv, want_hat=False)
    for i in range(4):
        assert torch.equal(got[i], want[i]) and torch.equal(bare[i], want[i])
    codec.decode(*want[:4], Kp, Vp, Wk, Wv, Khat=out[2][:, :d], Vhat=out[3][:, :d])
    assert codec.poll_status() == 0
    for i, o in enumerate(out):
        assert torch.equal(o[:, :d], want[4 + i % 2]) and (o[:, d:] == 3.0).all()


@pytest.mark.parametrize("T", [14000, 18432, 23100])
def test_several_layers_of_many_waves_in_one_launch_equal_layer_by_layer(T):
    """Four to six waves: the last layer reports its value rows with the next key rows, the layers before it by themselves."""
    from paper_2501_19392_b200 import chain
    d, L = 1024, 3
    codec = make_codec(d, d, 16)
    row = lambda s: synth.random_16bit((T, d), synth.BF16, s, device=DEV)
    K, V = [row(10 + l) for l in range(L)], [row(20 + l) for l in range(L)]
    W = lambda n, s: (synth.random_16bit((d, n), synth.BF16, s, device=DEV).float() / n ** 0.5).bfloat16()
    Wk, Wv = [None] + [W(d, 30 + l) for l in range(1, L)], [None] + [W(2 * d, 40 + l) for l in range(1, L)]
    ref, hats = chain.CompressedCache.empty(codec, L, T, DEV), []
    for l in range(L):
        prev = hats[-1] if l else (None, None)
        hats.append(codec.encode(K[l], V[l], *prev, Wk[l], Wv[l], None, None, ref.Kcodes[l], ref.Kscales[l], ref.Vcodes[l], ref.Vscales[l])[4:])
    for _ in range(3):
        got = chain.CompressedCache.empty(codec, L, T, DEV)
        Kh, Vh = ([torch.empty_like(K[0]) for _ in range(L)] for _ in range(2))
        codec.encode_chain(K, V, Wk, Wv, got.Kcodes, got.Kscales, got.Vcodes, got.Vscales, Khat=Kh, Vhat=Vh)
        Kb, Vb = ([torch.empty_like(K[0]) for _ in range(L)] for _ in range(2))
        codec.decode_chain(ref.Kcodes, ref.Kscales, ref.Vcodes, ref.Vscales, Wk, Wv, Khat=Kb, Vhat=Vb)
        assert codec.poll_status() == 0
        for l in range(L):
            for a, b in ((got.Kcodes, ref.Kcodes), (got.Kscales, ref.Kscales), (got.Vcodes, ref.Vcodes), (got.Vscales, ref.Vscales)):
                assert torch.equal(a[l], b[l]), l
            for a, b in ((Kh[l], hats[l][0]), (Vh[l], hats[l][1]), (Kb[l], hats[l][0]), (Vb[l], hats[l][1])):
                assert torch.equal(a, b), l
