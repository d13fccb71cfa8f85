"""Numerics that weights of the usual scale do not show, on one layer against a float64 restatement
of the same bf16 operands: full encodes of small encoders (dim up to 384, at most 256 tokens per
view) keep the softmax's probabilities and GELU's tanh in fp32; large and infinite scores."""
import numpy as np
import pytest

from paper_2607_12287_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2607_12287_gb300 as p
    p.load()
    return p


def _bf16(x):
    return synth.bf16_bits_to_f32(synth.f32_to_bf16_bits(np.asarray(x, np.float32))).astype(np.float64)


def _ln(x):
    c = x - x.mean(-1, keepdims=True)
    return c / np.sqrt((c * c).mean(-1, keepdims=True) + 1e-6)


def _encode(pkg, grid, dim, heads, mlp, **tensors):
    """One layer on one view whose patches embed to zero, so that the residual stream starts as `pos`:
    the tokens, and the layer's keys and values."""
    import torch
    shape = synth.EncoderShape(grid[0], grid[1], 1, dim, 1, heads, mlp, synth.GELU_TANH)
    flat = np.zeros(synth.weight_count(shape), np.uint16)
    w = synth.split_weights(shape, flat)
    for name, t in w.items():
        if name.endswith("_g"):
            t[...] = synth.f32_to_bf16_bits(np.float32([1.0]))[0]
        for key, value in tensors.items():
            if name.split(".")[-1] == key:
                t[...] = synth.f32_to_bf16_bits(np.asarray(value, np.float32).reshape(-1)).reshape(t.shape)
    enc = pkg.IncrementalViT(shape, flat, 1, 1)
    out = enc.encode_full(torch.zeros(1, grid[0], grid[1], 3, dtype=torch.uint8, device="cuda"))
    got = [t.float().cpu().numpy().astype(np.float64)[0] for t in (out, enc.cache("K", 0), enc.cache("V", 0))]
    assert enc.device_status() == 0
    enc.close()
    return got


@pytest.mark.parametrize("path", ["kernels", "persistent"])
@pytest.mark.parametrize("grid,dim,heads", [((14, 14), 192, 3), ((16, 16), 256, 8), ((12, 17), 320, 4), ((7, 10), 192, 2),
                                            ((16, 16), 384, 3), ((1, 6), 64, 4)],
                         ids=["dh64", "dh32", "dh80", "dh96", "dh128", "dh16"])
def test_probabilities_in_fp32(pkg, monkeypatch, path, grid, dim, heads):
    """Tokens come in pairs with opposite values and keys that are nearly the same, so that O is a sum of
    differences of probabilities, 1 % of them: rounding those to bf16 leaves an error of 2 to 4 % of it, the
    roundings of O and of the tokens to bf16 one of 2^-9."""
    monkeypatch.setenv("IVIT_PATH", path)
    rng = np.random.default_rng(dim)
    n, dh, half = grid[0] * grid[1], dim // heads, dim // 2
    even = rng.standard_normal((n // 2, half))
    odd = rng.standard_normal((n // 2, half // 2))
    odd = np.concatenate([odd, -odd], 1)  # (sums to zero: the pair has one mean and variance)
    pos = np.empty((n, dim))
    pos[0::2] = np.concatenate([even, odd], 1)
    pos[1::2] = np.concatenate([even, -odd], 1)
    pos = _bf16(pos)
    w_qkv = np.zeros((3 * dim, dim))
    w_qkv[:2 * dim, :half] = rng.standard_normal((2 * dim, half)) / np.sqrt(half)
    w_qkv[dim:2 * dim, half:] = 0.005 * rng.standard_normal((dim, half)) / np.sqrt(half)
    w_qkv[2 * dim:, half:] = rng.standard_normal((dim, half)) / np.sqrt(half)
    w_qkv = _bf16(w_qkv)
    gain = 2.0 ** 12
    out, k, v = _encode(pkg, grid, dim, heads, 64, pos=pos, W_qkv=w_qkv, W_o=gain * np.eye(dim))
    q = _bf16(_bf16(_ln(pos)) @ w_qkv[:dim].T).reshape(n, heads, dh)
    k, v = k.reshape(n, heads, dh), v.reshape(n, heads, dh)
    s = np.einsum("qhd,khd->hqk", q, k) / np.sqrt(dh)
    p = np.exp(s - s.max(-1, keepdims=True))
    o = np.einsum("hqk,khd->qhd", p / p.sum(-1, keepdims=True), v).reshape(n, dim)
    want = _ln(pos + gain * o)
    err = np.linalg.norm(out - want) / np.linalg.norm(want)
    assert err < 0.01, err


@pytest.mark.parametrize("path", ["kernels", "persistent"])
@pytest.mark.parametrize("grid,dim", [((14, 14), 384), ((4, 5), 384)], ids=["n196", "n20"])
def test_gelu_tanh_in_fp32(pkg, monkeypatch, path, grid, dim):
    """The MLP is h = GELU(LN(x)) added to x with a large gain, so that a hidden value rounded to another
    bf16 shows in the tokens: the hardware's tanh (2^-11) moves 0.7 % of them, fp32's one in 10^5."""
    monkeypatch.setenv("IVIT_PATH", path)
    rng = np.random.default_rng(dim)
    n = grid[0] * grid[1]
    pos = _bf16(rng.uniform(-1, 1, (n, dim)))
    gain = 2.0 ** 12
    out, _, _ = _encode(pkg, grid, dim, dim // 64, dim, pos=pos, W_1=np.eye(dim), W_2=gain * np.eye(dim))
    y = _bf16(_ln(pos))
    h = _bf16(0.5 * y * (1 + np.tanh(np.sqrt(2 / np.pi) * (y + 0.044715 * y ** 3))))
    want = _bf16(_ln(pos + gain * h))
    moved = np.mean(out != want)
    assert moved < 0.001, moved


@pytest.mark.parametrize("kernel", ["tc", "rows", "exact"])
@pytest.mark.parametrize("dim,heads", [(192, 3), (576, 8), (256, 2), (320, 10)], ids=["dh64", "dh72", "dh128", "dh32"])
def test_scores_of_minus_infinity(pkg, monkeypatch, dim, heads, kernel):
    """The first 140 keys' scores overflow to -inf, a whole key block and several warps' shares of the keys:
    they take no part, as in a softmax over all keys."""
    if kernel == "exact" and dim > 384:
        pytest.skip("full encodes of small encoders only")
    if kernel != "exact":
        monkeypatch.setenv("IVIT_ATTN", kernel)
    grid = (14, 14) if kernel == "exact" else (16, 17)
    rng = np.random.default_rng(dim)
    n, dh, masked = grid[0] * grid[1], dim // heads, 140
    half = rng.choice([-1.0, 1.0], (n, dim // 2 - 1)) * rng.choice([0.5, 1.0, 2.0], (n, dim // 2 - 1))
    pos = np.concatenate([np.zeros((n, 1)), half, np.zeros((n, 1)), -half], 1)  # (rows sum to zero exactly)
    pos[:masked, 0], pos[:masked, dim // 2] = -2.0, 2.0
    w_qkv, b_qkv = np.zeros((3 * dim, dim)), np.zeros(3 * dim)
    b_qkv[:dim] = 1e15                                                # q k = -1e40 for the masked keys,
    w_qkv[dim:2 * dim] = 1e-15 * rng.standard_normal((dim, dim)) / np.sqrt(dim)  # of order one for the others
    w_qkv[dim:2 * dim, 0] = 1e25
    w_qkv[2 * dim:] = rng.standard_normal((dim, dim)) / np.sqrt(dim)
    out, k, v = _encode(pkg, grid, dim, heads, 64, pos=pos, W_qkv=w_qkv, b_qkv=b_qkv, W_o=2.0 ** 6 * np.eye(dim))
    q = _bf16(b_qkv[:dim]).reshape(1, heads, dh)
    s = np.einsum("qhd,khd->hqk", q, k.reshape(n, heads, dh)[masked:]) / np.sqrt(dh)
    p = np.exp(s - s.max(-1, keepdims=True))
    o = np.einsum("hqk,khd->qhd", p / p.sum(-1, keepdims=True), v.reshape(n, heads, dh)[masked:]).reshape(1, dim)
    want = _ln(pos + 2.0 ** 6 * o)
    assert np.isfinite(out).all()
    err = np.linalg.norm(out - want) / np.linalg.norm(want)
    assert err < 0.01, err  # roundings of P, O and the tokens to bf16, 2^-9 each


@pytest.mark.parametrize("kernel", ["tc", "rows"])
@pytest.mark.parametrize("dim,heads", [(64, 4), (64, 2), (192, 4), (64, 1), (320, 4), (192, 2), (448, 4), (128, 1)],
                         ids=lambda x: str(x))
def test_scores_that_grow_from_block_to_block(pkg, monkeypatch, dim, heads, kernel):
    """Scores of standard deviation 12: the running maximum moves by more than 2^8 in many rows, so that sums
    and outputs of earlier key blocks are rescaled, in every padded head width."""
    monkeypatch.setenv("IVIT_ATTN", kernel)
    rng = np.random.default_rng(dim + heads)
    grid, n, dh = (20, 20), 400, dim // heads
    pos = _bf16(rng.standard_normal((n, dim)))
    w_qkv = _bf16(rng.standard_normal((3 * dim, dim)) * np.sqrt(12.0 / dim))
    out, k, v = _encode(pkg, grid, dim, heads, 64, pos=pos, W_qkv=w_qkv, W_o=2.0 ** 6 * np.eye(dim))
    q = _bf16(_bf16(_ln(pos)) @ w_qkv[:dim].T).reshape(n, heads, dh)
    s = np.einsum("qhd,khd->hqk", q, k.reshape(n, heads, dh)) / np.sqrt(dh)
    for kb in (64, 96, 128, 256):  # (the tensor-core kernel's key blocks, and one step of the few-query kernel)
        blocks = np.stack([s[..., i:i + kb].max(-1) for i in range(0, n, kb)], -1) * np.log2(np.e)
        assert ((blocks[..., 1:] - np.maximum.accumulate(blocks, -1)[..., :-1]).max(-1) > 8).mean() > 0.01
    p = np.exp(s - s.max(-1, keepdims=True))
    o = np.einsum("hqk,khd->qhd", p / p.sum(-1, keepdims=True), v.reshape(n, heads, dh)).reshape(n, dim)
    want = _ln(pos + 2.0 ** 6 * o)
    err = np.linalg.norm(out - want) / np.linalg.norm(want)
    assert err < 0.01, err  # roundings of P, O and the tokens to bf16, 2^-9 each
