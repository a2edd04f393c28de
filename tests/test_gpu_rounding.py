"""The row kernels' results bit for bit, from the order in which they round: the rotation's butterflies in single precision stage
by stage, the normalisation, the search and the reconstruction, restated here with one torch operation per rounding.

A packed cache outlives the build that wrote it, and a chain of layers passes every moved last bit on to codes of the layers
that follow, so the order is part of what the library promises and not only the accuracy, which the oracle
tests check.  The prediction is the library's own (aquakv_predict)."""
import numpy as np
import pytest
import torch

from paper_2501_19392_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
T = 300


def make(d, h, g, dtype, grid=None, levels=0):
    from paper_2501_19392_b200 import api
    return api.Codec(d, h, g, grid, dtype, synth.hadamard_signs(d, 11), synth.hadamard_signs(d, 12), levels=levels)


def signs(d, role):
    return torch.from_numpy(synth.hadamard_signs(d, 11 + role)).to(DEV, torch.float32)


def butterflies(x, bits):
    """Unnormalised Hadamard butterflies over the given index bits, in that order, each rounded to fp32."""
    for b in bits:
        n, d = x.shape
        v = x.view(n, d >> (b + 1), 2, 1 << b)
        x = torch.stack([v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]], dim=2).reshape(n, d)
    return x


def fma(a, b, c):
    """One rounding to fp32: the product of two fp32 values is exact in double (and so, but for one case in 2^29, the sum)."""
    return (a.double() * b.double() + c.double()).float()


def unpack(codes, bits):
    b = (codes.to(torch.int32)[:, :, None] >> torch.arange(8, device=DEV)) & 1
    return (b.view(codes.shape[0], -1, bits) << torch.arange(bits, device=DEV)).sum(-1)


def rows(codec, d, dtype, seed):
    shape = (T, d)
    X = synth.random_16bit(shape, dtype, seed, device=DEV)
    prev = synth.random_16bit(shape, dtype, seed + 1, device=DEV)
    W = (synth.random_16bit((d, d), dtype, seed + 2, device=DEV).float() / d ** 0.5).to(X.dtype)
    P = codec.predict(prev, None, W)
    return X, prev, W, P


def both_ways(codec, X, prev, W, role):
    codes, scales, hat = codec.encode_phase(role, X, prev, None, W)
    assert torch.equal(codec.decode_phase(role, codes, scales, prev, None, W), hat)
    return codes, scales, hat


@pytest.mark.parametrize("n,dtype", [(16, synth.BF16), (64, synth.F16), (256, synth.F16)])
def test_rows_of_one_warp(n, dtype):
    d = 1024
    grid = synth.lloyd_grid(n, seed=7, n_samples=1 << 14, iters=20)
    codec = make(d, d, d, dtype, grid)
    for role in (0, 1):
        X, prev, W, P = rows(codec, d, dtype, 5 + 10 * role)
        codes, scales, hat = both_ways(codec, X, prev, W, role)
        sg, s = signs(d, role), scales.float()
        y = butterflies((X.float() - P) * sg, (0, 1, 2, 8, 9, 3, 4, 5, 6, 7)) * ((1.0 / s) * (1.0 / 32.0))
        g = torch.from_numpy(grid).to(DEV)
        dx = y.view(T, -1, 2)[:, :, None, :] - g
        sq = dx * dx
        q = (sq[..., 0] + sq[..., 1]).argmin(-1)
        assert torch.equal(unpack(codes, n.bit_length() - 1), q)
        x = butterflies(g[q].reshape(T, d), (7, 3, 4, 5, 6, 1, 2, 8, 9, 0)) * (s * (1.0 / 32.0))
        assert torch.equal(hat, (P + x * sg).to(hat.dtype))


def test_the_layer_kernel_rounds_like_the_row_kernels():
    """Keys of the fused encode and decode (whose prediction stays inside the kernel) equal the phase calls' bit for bit."""
    d, dtype = 1024, synth.BF16
    codec = make(d, d, d, dtype, synth.lloyd_grid(16, seed=7, n_samples=1 << 14, iters=20))
    X, prev, W, _ = rows(codec, d, dtype, 40)
    Wv = torch.cat([W, W], dim=1).contiguous()
    codes, scales, hat = both_ways(codec, X, prev, W, 0)
    out = codec.encode(X, X, prev, prev, W, Wv)
    assert torch.equal(out[0], codes) and torch.equal(out[1], scales) and torch.equal(out[4], hat)
    Kh, Vh = codec.decode(*out[:4], prev, prev, W, Wv)
    assert torch.equal(Kh, hat) and torch.equal(Vh, out[5])


def rsqrt(h):
    return torch.rsqrt(torch.tensor(float(h), device=DEV))


@pytest.mark.parametrize("d,h,g,levels,dtype", [(512, 512, 128, 8, synth.F16), (1024, 128, 1024, 16, synth.BF16), (256, 64, 32, 4, synth.F16)])
def test_uniform_levels_after_a_rotation(d, h, g, levels, dtype):
    codec = make(d, h, g, dtype, None, levels)
    order, half = range(h.bit_length() - 1), levels // 2
    for role in (0, 1):
        X, prev, W, P = rows(codec, d, dtype, 60 + 10 * role)
        codes, scales, hat = both_ways(codec, X, prev, W, role)
        sg, rs = signs(d, role), rsqrt(h)
        v = butterflies((X.float() - P) * sg, order) * rs
        assert torch.equal((v.view(T, d // g, g).abs().amax(-1) * (1.0 / half)).half(), scales)
        sf = scales.float().repeat_interleave(g, dim=1)
        level = torch.clamp(torch.ceil(v.double() / sf.double() - 0.5), -half, half - 1).float()
        assert torch.equal(unpack(codes, levels.bit_length() - 1), level.to(torch.int64) + half)
        assert torch.equal(hat, (butterflies(level * sf, order) * rs * sg + P).to(hat.dtype))


def nearest4(y, g):
    """Index of the point whose half squared distance (less the tuple's own) is the smallest, the first of equal ones."""
    half = torch.zeros(g.shape[0], device=DEV)
    for k in range(4):
        half = fma(g[:, k], g[:, k], half)
    s = (0.5 * half).expand(y.shape[0], -1)
    for k in range(4):
        s = fma(-y[:, k:k + 1], g[:, k], s)
    return s.argmin(-1)


@pytest.mark.parametrize("d,h,dtype", [(512, 512, synth.F16), (1024, 128, synth.BF16), (256, 64, synth.BF16)])
def test_four_dimensional_grid(d, h, dtype):
    grid = synth.lloyd_grid(256, seed=7, n_samples=1 << 14, iters=20, dim=4)
    codec, g = make(d, h, d, dtype, grid), torch.from_numpy(grid).to(DEV)
    order = range(h.bit_length() - 1)
    for role in (0, 1):
        X, prev, W, P = rows(codec, d, dtype, 80 + 10 * role)
        codes, scales, hat = both_ways(codec, X, prev, W, role)
        sg, rs, r = signs(d, role), rsqrt(h), X.float() - P
        # the scale: eight values a lane, the 32 lanes of a chunk by halving distances, the chunks in order
        part, total = torch.zeros((T, d // 256, 32), device=DEV), torch.zeros(T, device=DEV)
        for i in range(8):
            v = r.view(T, d // 256, 32, 8)[..., i]
            part = fma(v, v, part)
        for off in (1, 2, 4, 8, 16):
            part = part + part[..., torch.arange(32, device=DEV) ^ off]
        for c in range(d // 256):
            total = total + part[:, c, 0]
        assert torch.equal((total * (1.0 / d)).sqrt().half()[:, None], scales)
        sf = scales.float()
        y = butterflies(r * (1.0 / sf) * sg, order) * rs
        q = torch.cat([nearest4(t, g) for t in y.view(-1, 4).split(4096)]).view(T, -1)
        assert torch.equal(codes.long(), q)
        assert torch.equal(hat, fma(butterflies(g[q].reshape(T, d), order) * rs * sg, sf, P).to(hat.dtype))


def test_four_dimensional_ties_are_decided_by_the_roundings():
    """Rows of +-1 have scale 1 and rotate to multiples of 1/4; half of the points are the others mirrored in the plane
    y_k = 1/4, so that many tuples are equally far from two points and the order of the roundings chooses."""
    d, h = 256, 64
    rng = np.random.default_rng(3)
    g = rng.standard_normal((128, 4)).astype(np.float32)
    m = g.copy()
    k = np.arange(128)
    m[k, k % 4] = np.float32(0.5) - g[k, k % 4]
    grid = np.concatenate([g, m])[rng.permutation(256)]
    codec = make(d, h, d, synth.BF16, grid)
    X = torch.from_numpy(rng.choice([-1.0, 1.0], size=(T, d))).to(DEV, torch.bfloat16)
    codes, scales, _ = codec.encode_phase(0, X)
    assert bool((scales == 1.0).all())
    y = butterflies(X.float() * signs(d, 0), range(6)) * 0.125
    q = torch.cat([nearest4(t, torch.from_numpy(grid).to(DEV)) for t in y.view(-1, 4).split(4096)]).view(T, -1)
    assert torch.equal(codes.long(), q)


def test_four_dimensional_lists_keep_what_rounding_can_choose():
    """Points far from the tuples, in pairs that differ by a few units in the last place: single precision cannot tell
    which of a pair is nearer, so both have to be among a cell's candidates for the search to equal the exhaustive one."""
    d, h = 256, 64
    rng = np.random.default_rng(4)
    g = rng.standard_normal((128, 4))
    g = (100.0 * g / np.linalg.norm(g, axis=1, keepdims=True)).astype(np.float32)
    m = g.copy()
    k = np.arange(128)
    m[k, k % 4] += (10.0 ** rng.uniform(-5, -3, 128)).astype(np.float32) * rng.choice([-1.0, 1.0], 128).astype(np.float32)
    grid = np.concatenate([g, m])[rng.permutation(256)]
    codec = make(d, h, d, synth.BF16, grid)
    X = synth.random_16bit((T, d), synth.BF16, 6, device=DEV)
    codes, scales, _ = codec.encode_phase(0, X)
    r = X.float()
    y = butterflies(r * (1.0 / scales.float()) * signs(d, 0), range(6)) * 0.125
    q = torch.cat([nearest4(t, torch.from_numpy(grid).to(DEV)) for t in y.view(-1, 4).split(4096)]).view(T, -1)
    assert torch.equal(codes.long(), q)
