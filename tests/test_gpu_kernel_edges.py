"""Kernels at the edges of their tiles, through the C ABI against the fp32 oracle: an encoder of
one or two layers encodes a stream in full and incrementally (updated lists bit-exact, tokens
within the parity bars of gpu_util)."""
import os
import re
import subprocess

import numpy as np
import pytest

from tests import gpu_util

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2607_12287_gb300 as p
    p.load()
    return p


def _run(pkg, oracle_mod, grid, views, dim, heads, mlp, depth, change_p, n_frames=3, mlp_tokens=0):
    from paper_2607_12287_gb300 import synth
    shape = synth.EncoderShape(8 * grid[0], 8 * grid[1], 8, dim, depth, heads, mlp, synth.GELU_TANH)
    frames = list(synth.stream_random(shape, views, n_frames, 11, change_p=change_p))
    stats = gpu_util.run_side_by_side(pkg, oracle_mod, shape, synth.make_weights(shape, 3), frames, 1, views,
                                      check_caches=True, cache_layers="all",
                                      mlp_tokens=mlp_tokens)
    assert len(stats) == n_frames and all(np.isfinite(s[0]).all() for s in stats)


# (grid, views, dim, heads, mlp): row counts around the 64-, 128- and 256-row tiles and their
# 32-row halves, feature counts that are no multiple of the pair's 256 (192 = 1.5 x 128, 320,
# 520, 840), one k-block (dim 64), and more tiles than CTA pairs
PAIR_SHAPES = [((5, 13), 1, 192, 3, 520), ((1, 43), 3, 320, 5, 840), ((1, 257), 1, 192, 3, 520),
               ((13, 25), 4, 320, 5, 840), ((10, 10), 1, 64, 1, 264), ((20, 26), 5, 576, 8, 1160)]


@pytest.mark.parametrize("grid,views,dim,heads,mlp", PAIR_SHAPES,
                         ids=[f"n{g[0] * g[1]}x{v}_d{d}_f{f}" for g, v, d, _, f in PAIR_SHAPES])
def test_gemm_tile_edges(pkg, oracle_mod, grid, views, dim, heads, mlp):
    _run(pkg, oracle_mod, grid, views, dim, heads, mlp, 1, 0.4)


# head tiles (tokens x head width x 2 bytes) that are no multiple of the 128 bytes a TMA
# destination needs
@pytest.mark.parametrize("grid,views,dim,heads", [((5, 19), 2, 64, 4), ((1, 1), 2, 64, 8), ((5, 13), 2, 128, 4)],
                         ids=["n95_dh16", "n1_dh8", "n65_dh32"])
def test_persistent_kernel_odd_key_tiles(pkg, oracle_mod, monkeypatch, grid, views, dim, heads):
    monkeypatch.setenv("IVIT_PATH", "persistent")
    _run(pkg, oracle_mod, grid, views, dim, heads, 2 * dim, 2, 0.5)


# (grid, dim, heads, mlp, change): a few updated rows in one to three passes of 32 and in one or
# two 16-row tiles, K of a ragged last chunk (mlp 520, 840), one chunk per two warps (dim 64),
# feature counts that are no multiple of a CTA's
ROW_SHAPES = [((6, 10), 64, 1, 264, 0.05), ((6, 10), 320, 5, 840, 0.25), ((6, 10), 320, 5, 520, 0.5),
              ((8, 12), 576, 8, 1160, 0.95)]


@pytest.mark.parametrize("mlp_tokens", [0, 1], ids=["updated", "all"])
@pytest.mark.parametrize("grid,dim,heads,mlp,change", ROW_SHAPES,
                         ids=[f"d{d}_f{f}_p{int(100 * c)}" for _, d, _, f, c in ROW_SHAPES])
def test_few_row_gemm_edges(pkg, oracle_mod, grid, dim, heads, mlp, change, mlp_tokens):
    _run(pkg, oracle_mod, grid, 1, dim, heads, mlp, 2, change, n_frames=4, mlp_tokens=mlp_tokens)


# wide encoders whose residual GEMMs leave more than 8 splits to the next layer norm, which then
# holds 16 partials per thread of its widest blocks (416 and 512 threads)
@pytest.mark.parametrize("grid,dim,heads", [((16, 16), 1664, 26), ((8, 8), 1664, 13), ((16, 16), 2048, 16), ((8, 8), 2048, 32)],
                         ids=["d1664_n256", "d1664_n64", "d2048_n256", "d2048_n64"])
def test_many_splits_of_wide_rows(pkg, oracle_mod, monkeypatch, capfd, grid, dim, heads):
    monkeypatch.setenv("IVIT_DEBUG", "1")
    _run(pkg, oracle_mod, grid, 1, dim, heads, 8192, 1, 0.05, n_frames=2)
    plans = re.findall(r"^ivit gemm (?:full|inc)\s.*splits=(\d+)$", capfd.readouterr().err, flags=re.M)
    assert len(plans) == 10 and max(map(int, plans)) > 8, plans


# (grid, views, dim, heads): head widths of every padded width (8 -> 16 ... 128), token counts
# one off the key blocks of 64, 96 and 128 and the few-query kernel's 32 and 256, one and several
# query tiles of 16 and 128 per head; on both kernels
ATTN_SHAPES = [((1, 1), 2, 64, 8), ((5, 19), 2, 64, 4), ((3, 33), 1, 128, 4), ((1, 97), 2, 320, 8),
               ((8, 16), 1, 192, 3), ((3, 43), 2, 576, 8), ((1, 193), 1, 320, 4), ((1, 257), 1, 704, 8),
               ((5, 13), 3, 832, 8), ((2, 161), 1, 256, 2),
               # few-query kernel: more 16-query items than SMs, and than twice that
               ((14, 14), 6, 192, 3), ((9, 11), 8, 256, 8)]


@pytest.mark.parametrize("kernel", ["tc", "rows"])
@pytest.mark.parametrize("grid,views,dim,heads", ATTN_SHAPES,
                         ids=[f"n{g[0] * g[1]}x{v}_dh{d // h}" for g, v, d, h in ATTN_SHAPES])
def test_attention_block_edges(pkg, oracle_mod, monkeypatch, grid, views, dim, heads, kernel):
    monkeypatch.setenv("IVIT_ATTN", kernel)
    _run(pkg, oracle_mod, grid, views, dim, heads, 2 * dim, 2, 0.5)


@pytest.mark.parametrize("with_nan", [False, True], ids=["finite", "nan"])
@pytest.mark.parametrize("n_tok", [1, 31, 33, 200, 1024])
def test_topk_selection_ties(pkg, n_tok, with_nan):
    """Scores from a handful of values (-1 ... 1, zero vectors, NaN), so that every k falls into a
    run of equal ones: exactly the order (score, index), a NaN beside the k lowest of the rest."""
    import torch
    from paper_2607_12287_gb300 import synth

    rng = np.random.default_rng(n_tok)
    views, dim = 2, 64
    cos = rng.choice([-1.0, -0.5, 0.0, 0.25, 0.5, 1.0], size=(views, n_tok))
    cur = np.zeros((views, n_tok, dim), np.float32)
    cur[..., 0], cur[..., 1] = cos, np.sqrt(1 - cos ** 2)
    zero = rng.random((views, n_tok)) < 0.1  # a zero vector's score is 0
    cur[zero], cos[zero] = 0, 0.0
    if with_nan:
        nan = rng.random((views, n_tok)) < 0.05
        cur[nan], cos[nan] = np.nan, np.nan
    ref = np.zeros_like(cur)
    ref[..., 0] = 1
    d_cur, d_ref = torch.from_numpy(cur).cuda(), torch.from_numpy(ref).cuda()
    idx = torch.empty(views, n_tok, dtype=torch.int32, device="cuda")
    cnt = torch.empty(views, dtype=torch.int32, device="cuda")
    for k in sorted({0, 1, n_tok // 3, n_tok - 1, n_tok, n_tok + 5}):
        pkg.ivit_select_noalloc(d_cur, d_ref, views, n_tok, dim, synth.SEL_TOPK, 0.0, k, idx, cnt)
        for v in range(views):
            c = cos[v]
            order = [i for i in np.argsort(np.where(np.isnan(c), np.inf, c), kind="stable") if not np.isnan(c[i])]
            want = sorted(order[:k] + [i for i in range(n_tok) if np.isnan(c[i]) and k > 0])
            got = idx[v].cpu().numpy()
            assert int(cnt[v]) == len(want), (k, v)
            assert got[: len(want)].tolist() == want and (got[len(want):] == -1).all(), (k, v)


@pytest.mark.parametrize("bias", [False, True], ids=["nobias", "bias"])
@pytest.mark.parametrize("batch,width", [(1, 1), (1, 3), (5, 1), (7, 2), (9, 3), (33, 5), (11, 7), (4096, 350), (257, 1023)])
def test_action_combine_rows_of_any_width(pkg, batch, width, bias):
    """128-bit accesses over rows that are no multiple of four values: every value is the same two
    fused multiply-adds (and addition) in fp32, whichever loop it takes."""
    import torch

    g = torch.Generator().manual_seed(batch)
    x0, v0, v7, b = (torch.randn(batch, width, generator=g) for _ in range(4))
    al, be = (torch.rand(batch, generator=g) for _ in range(2))
    out = torch.full((batch, width), float("nan"), device="cuda")
    dev = [t.cuda() for t in (x0, v0, v7, al, be, b)]
    pkg.ivit_action_combine(*dev[:5], dev[5] if bias else None, out)
    d = [t.double() for t in (x0, v0, v7, al, be, b)]
    inner = (d[3][:, None] * d[1] + d[0]).float().double()  # fp64 holds the product exactly: fmaf's rounding
    want = (d[4][:, None] * d[2] + inner).float()
    want = (want.double() + (d[5] if bias else 0.0)).float()
    # (an fp64 sum rounds once before the rounding to fp32: at most the last bit in a tie)
    assert torch.allclose(out.cpu(), want, rtol=2 ** -23, atol=2 ** -23)


@pytest.mark.parametrize("offset", [0, 1, 8], ids=["aligned", "2bytes", "16bytes"])
def test_outputs_at_any_alignment(pkg, offset):
    """Tokens into a view that starts `offset` elements into its buffer: the same values, and nothing
    written outside the view."""
    import torch
    from paper_2607_12287_gb300 import synth

    shape = synth.EncoderShape(40, 104, 8, 192, 1, 3, 520, synth.GELU_TANH)
    enc = pkg.IncrementalViT(shape, synth.make_weights(shape, 3), 1, 2)
    frames = [torch.from_numpy(f).cuda() for f in synth.stream_random(shape, 2, 2, 11, change_p=0.4)]
    n = 2 * shape.n_tokens * shape.dim
    for call in (enc.encode_full, enc.encode_incremental):
        frame = frames[call == enc.encode_incremental]
        want = call(frame)
        want = want[0] if isinstance(want, tuple) else want
        buf = torch.full((n + 16,), 7.0, dtype=torch.bfloat16, device="cuda")
        enc.encode_full(frames[0]) if call == enc.encode_incremental else None
        call(frame, buf[offset:offset + n])
        assert torch.equal(buf[offset:offset + n], want.reshape(-1))
        assert (buf[:offset] == 7).all() and (buf[offset + n:] == 7).all()
    enc.close()


def test_pointers_outside_the_gpu_take_the_copy_engine(pkg):
    """Frames, tokens and counts in pinned host memory (which, like another GPU's, the copy engine
    reaches), and frames at an odd address: the results of buffers on the GPU, without the library's
    output copy among the launches."""
    import torch
    from paper_2607_12287_gb300 import synth

    shape = synth.EncoderShape(40, 104, 8, 192, 1, 3, 520, synth.GELU_TANH)
    frames = list(synth.stream_random(shape, 2, 2, 11, change_p=0.4))
    weights = synth.make_weights(shape, 3)

    def encode(where):
        enc = pkg.IncrementalViT(shape, weights, 1, 2)
        host = where == "host"
        out = torch.zeros(2, shape.n_tokens, shape.dim, dtype=torch.bfloat16, device="cpu" if host else "cuda", pin_memory=host)
        cnt = torch.zeros(2, dtype=torch.int32, device=out.device, pin_memory=host)
        got = []
        for call, frame in enumerate(frames):
            f = torch.from_numpy(frame).reshape(-1)
            buf = torch.empty(f.numel() + 1, dtype=torch.uint8, device=out.device, pin_memory=host)
            at = buf[1:] if where == "odd" else buf[:-1]
            at.copy_(f)
            torch.cuda.synchronize()
            if call == 0:
                pkg.ivit_encode_full(enc.h, at.data_ptr(), out.data_ptr())
            else:
                pkg.ivit_encode_incremental(enc.h, at.data_ptr(), out.data_ptr(), cnt.data_ptr())
            torch.cuda.synchronize()
            got.append((out.cpu().clone(), cnt.cpu().clone(), pkg.ivit_last_launch_count(enc.h)))
        assert enc.device_status() == 0
        enc.close()
        return got

    gpu = encode("gpu")
    assert gpu[1][1].sum() > 0
    for where, fewer in (("host", 1), ("odd", 0)):
        for (tok, cnt, n), (tok0, cnt0, n0) in zip(encode(where), gpu):
            assert torch.equal(tok, tok0) and torch.equal(cnt, cnt0), where
            assert n == n0 - fewer, where


@pytest.mark.parametrize("mlp_tokens", [0, 1], ids=["updated", "all"])
@pytest.mark.parametrize("select,topk", [(0, 0), (1, 20)], ids=["threshold", "top20"])
def test_cold_calls_take_the_plans_of_their_rows(pkg, select, topk, mlp_tokens):
    """An incremental call whose views are all cold updates every token, in the launch shapes of a full
    encode and so with its rounding: bit for bit its tokens.  (Those of a tenth of the rows split K
    elsewhere.)"""
    import torch
    from paper_2607_12287_gb300 import synth

    shape = synth.EncoderShape(128, 128, 8, 576, 2, 8, 2328, synth.GELU_TANH)
    weights = synth.make_weights(shape, 3)
    frames = [torch.from_numpy(f).cuda() for f in synth.stream_random(shape, 1, 2, 11, change_p=0.3)]
    enc = pkg.IncrementalViT(shape, weights, 1, 1, select, 0.98, topk, mlp_tokens=mlp_tokens)
    for frame in frames:
        want = enc.encode_full(frame)
        enc.reset()
        got, count = enc.encode_incremental(frame)
        assert int(count[0]) == shape.n_tokens and torch.equal(got, want)
    enc.close()


def test_every_cta_of_both_row_groups_has_its_own_stamp(pkg, tmp_path):
    """Timeline stamps of the few-row GEMM with more rows than one group's pass (stamp_probe.cu)."""
    from paper_2607_12287_gb300 import build as b
    exe = str(tmp_path / "stamp_probe")
    subprocess.run([b.NVCC, *b.ARCH, "-std=c++17", os.path.join(b.ROOT, "tests", "stamp_probe.cu"), b.LIB, "-Xlinker",
                    "-rpath=" + os.path.dirname(b.LIB), "-o", exe], check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split() == ["24", "24", "0"]
