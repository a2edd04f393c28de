"""One predicted layer through the layer kernel against the single-phase entry points at the edges of its waves: the widths of
the GEMM's tiles in a short last wave, one warp per row for d_kv <= 512, one poller and one report per CTA.

The two paths share no kernel but form the same sums in the same order (fp32 accumulation over the input features, ascending)
and the same roundings in the rows, so everything has to agree bit for bit."""
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


@pytest.mark.parametrize("d,h,T", CASES)
@pytest.mark.parametrize("n,dtype", [(16, synth.BF16), (64, synth.F16), (256, synth.BF16)])
def test_layer_calls_equal_the_phases(d, h, T, n, dtype):
    from paper_2501_19392_b200 import api
    if n != 16 and T > 5000:
        pytest.skip("the large calls with one grid only")
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
