"""GPU parity of obc_score against the CPU checker, element by element, through the C ABI."""
import numpy as np
import pytest
import torch

from oracle import reference as ref
from paper_2510_07651_b200 import api, synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


def _check(case, variants, causal=True, path="auto", tight=None):
    want = H.oracle_scores(case, variants, causal)
    got = H.gpu_scores(case, variants, causal, path)
    own = ("ATTN", "VATP")                            # not on the scale of the three OBCache scores
    mx = max(np.abs(want[n]).max() for n in variants if n not in own) if any(n not in own for n in variants) else None
    for n in variants:
        H.assert_scores_close(got[n], want[n], case.dtype, tight=tight, what=f"{case.name}/{n}/{path}",
                              mx=None if n in own else mx)
        for b in range(case.B):                      # padding beyond each sequence is written as 0
            assert (got[n][b, :, case.seq_lens[b]:] == 0).all()


def test_config1_fp32_all_variants():
    case, run = synth.config(1)
    _check(case, run["variants"] + ["ATTN", "VATP"], tight=2e-5)


@pytest.mark.parametrize("path", ["simt", "auto"])
def test_config2_shape_reduced_length(path):
    case, run = synth.config(2, shrink=8)            # N = 4096: several tiles per split
    _check(case, ["V", "K", "VK"], path=path, tight=2e-2)


@pytest.mark.parametrize("path", ["simt", "auto"])
def test_config3_shape_reduced_length(path):
    case, run = synth.config(3, shrink=32)           # R = 448, N = 4096
    _check(case, run["variants"], path=path, tight=2e-2)


@pytest.mark.parametrize("path", ["simt", "auto"])
def test_config4_ragged_batch_reduced(path):
    case, run = synth.config(4, shrink=16)           # lengths in [512, 4096], ragged tails
    _check(case, run["variants"], path=path, tight=2e-2)


@pytest.mark.parametrize("N,W,Hq,Hkv,dtype,causal", [
    (1, 1, 1, 1, "f32", True),            # single cached token
    (16, 16, 2, 1, "f32", True),          # window == whole cache
    (65, 3, 7, 1, "bf16", True),          # ragged tile tail, odd group
    (200, 1, 4, 1, "bf16", True),         # W = 1 (decode-like), R = 4
    (333, 5, 8, 2, "f32", False),         # non-causal
    (1000, 40, 4, 2, "bf16", True),       # R = 80: not a multiple of the row chunk
    (2333, 5, 8, 2, "bf16", False),       # longer than one kernel takes: pass 1, merge and pass 2, non-causal,
    (2100, 1, 4, 1, "bf16", True),        # W = 1
    (2049, 40, 4, 2, "bf16", True),       # and R = 80 with one token in the last tile
])
def test_small_and_degenerate_shapes(N, W, Hq, Hkv, dtype, causal):
    case = synth.make_prefill("edge", B=2, Hq=Hq, Hkv=Hkv, d=128, W=W, N=N, dtype=dtype, seed=77 + N,
                              hh_frac=0.05)
    _check(case, ["V", "K", "VK", "ATTN", "VATP"], causal=causal, tight=2e-2 if dtype == "bf16" else None)


@pytest.mark.parametrize("lens,W,Hq,Hkv", [
    ([1100, 333], 64, 14, 2),      # R = 448 (row chunks of 64), odd tile counts: the second tile of the last pair is past the end
    ([2900], 40, 5, 1),            # R = 200: padded to 256 rows, 23 tiles
    ([129, 4000, 640], 48, 12, 3), # R = 192, ragged, a unit with two tiles of which the second holds one token
])
def test_more_than_128_window_rows(lens, W, Hq, Hkv):
    case = synth.make_prefill("rows", B=len(lens), Hq=Hq, Hkv=Hkv, d=128, W=W, N=lens, dtype="bf16", seed=101 + W,
                              hh_frac=0.02)
    _check(case, ["V", "K", "VK", "ATTN", "VATP"], tight=2e-2)
    _check(case, ["K", "VK"], tight=2e-2)
    _check(case, ["VK"], tight=2e-2)


@pytest.mark.parametrize("N,W,Hq,Hkv", [(5000, 64, 1, 1), (3001, 16, 8, 2), (257, 128, 1, 1), (4224, 24, 4, 1)])
def test_tensor_core_row_counts(N, W, Hq, Hkv):
    # R = 64, 64, 128, 96 (chunks of 64 / 64 / 128 / 96 rows), token counts with and without a ragged last tile
    case = synth.make_prefill("tc", B=1, Hq=Hq, Hkv=Hkv, d=128, W=W, N=N, dtype="bf16", seed=7 + N, hh_frac=0.02)
    _check(case, ["VK"], path="tc", tight=2e-2)
    _check(case, ["V", "K", "VK", "ATTN", "VATP"], path="tc", tight=2e-2)


@pytest.mark.parametrize("N,W,Hq,Hkv", [
    (1, 1, 2, 2),            # one token, one row: 15 padding rows in the chunk of 16
    (127, 1, 7, 1),          # just under one tile
    (128, 16, 1, 1),         # one whole tile, a chunk without padding
    (129, 17, 1, 1),         # one token in the last tile, chunk of 32
    (3001, 32, 4, 4),        # several tiles per split, no groups
    (1500, 12, 12, 3),       # R = 48: the row halves of pass 2 are 32 and 16
    (700, 63, 1, 1),         # R = 63: the largest row count of this path, one padding row
    (2177, 1, 7, 1),         # the same row counts beyond 2048 tokens, where pass 1, the merge of its splits and pass 2 are kernels of
    (2049, 17, 1, 1),        # their own: 9, 15, 0 and 1 padding rows
    (2500, 12, 12, 3),
    (2305, 63, 1, 1),
])
def test_fewer_than_64_window_rows(N, W, Hq, Hkv):
    """bf16 caches with fewer than 64 window rows: attention weights and outputs travel as two bf16 parts, so the scores
    agree with the double-precision ones as 32-bit sums do.  Bound: the parts leave out 2^-17 of a weight or of an output,
    and 128-term and N-term fp32 sums add a few 2^-24 each; 1e-5 of the largest score covers both with a margin of four."""
    case = synth.make_prefill("fewrows", B=2, Hq=Hq, Hkv=Hkv, d=128, W=W, N=[N, max(W, N - 40)], dtype="bf16", seed=31 + N, hh_frac=0.02)
    for variants in (["VK"], ["V", "K", "VK", "ATTN"], ["V", "K", "VK", "ATTN", "VATP"]):
        want, got = H.oracle_scores(case, variants), H.gpu_scores(case, variants)
        mx = max(np.abs(want[n]).max() for n in variants if n in ("V", "K", "VK"))
        for n in variants:
            H.assert_scores_close(got[n], want[n], "f32", what=f"{case.name}/{n}", mx=None if n in ("ATTN", "VATP") else mx)


@pytest.mark.parametrize("N,Hq,Hkv,dtype,path", [
    (96, 2, 1, "f32", "auto"),            # R = 192 on CUDA cores
    (384, 2, 2, "bf16", "simt"),
    (384, 4, 2, "bf16", "auto"),          # R = 768: twelve row chunks of 64 on tensor cores
    (640, 1, 1, "bf16", "tc"),            # R = 640, five token tiles, every tile needs the mask
])
def test_full_history_window(N, Hq, Hkv, dtype, path):
    """The perturbation window is the whole sequence (w = 1 in Sec. 4.3, the accumulation H2O uses): every
    query position is a window row and row i sees the tokens p <= i."""
    case = synth.make_prefill("history", B=1, Hq=Hq, Hkv=Hkv, d=128, W=N, N=N, dtype=dtype, seed=311 + N,
                              hh_frac=0.02)
    _check(case, ["V", "K", "VK", "ATTN", "VATP"], path=path, tight=2e-2 if dtype == "bf16" else None)


@pytest.mark.parametrize("N,W,Hq,Hkv", [(100, 40, 2, 2), (90, 20, 160, 80), (300, 5, 320, 160), (150, 16, 640, 160), (131, 50, 480, 160),
                                         (100, 40, 170, 170), (90, 20, 340, 170)])
def test_one_cta_per_head_and_chunk(N, W, Hq, Hkv):
    # pass 1 writes the merged rows itself, padding rows included: R = 40 (two bf16 parts), 40, 10, 64, 150 (two chunks), 40 and 40
    # (the first two have all their heads side by side and are scored by one kernel; the last two are more heads than SMs)
    case = synth.make_prefill("direct", B=1, Hq=Hq, Hkv=Hkv, d=128, W=W, N=N, dtype="bf16", seed=N + W, hh_frac=0.02)
    _check(case, ["K", "VK"], tight=2e-2)
    if Hq // Hkv * W < 64:                   # both parts of -2 O: the tolerance of 32-bit sums (see test_fewer_than_64_window_rows)
        want, got = H.oracle_scores(case, ["K", "VK"]), H.gpu_scores(case, ["K", "VK"])
        for n in ("K", "VK"):
            H.assert_scores_close(got[n], want[n], "f32", what=f"{case.name}/{n}", mx=np.abs(want["VK"]).max())


@pytest.mark.parametrize("N,W,Hq,Hkv,lens", [
    (1281, 130, 160, 80, None),           # three chunks, the last pair half empty; one token in the last tile
    (1300, 1300, 26, 26, None),           # whole-sequence window, the chunks of a pair visit different tiles
    (1400, 150, 148, 74, [1400, 333]),    # chunks that straddle heads, two lengths
    (6200, 130, 74, 74, [6200, 100 + 130]),   # two splits of a pair: partial results
])
def test_row_chunks_in_pairs(N, W, Hq, Hkv, lens):
    case = synth.make_prefill("pairs", B=len(lens) if lens else 1, Hq=Hq, Hkv=Hkv, d=128, W=W, N=lens or N, dtype="bf16", seed=N + W, hh_frac=0.02)
    _check(case, ["K", "VK"], tight=2e-2)


@pytest.mark.parametrize("N,W,Hq,Hkv,lens", [
    (1641, 1641, 4, 1, None),             # chunks that straddle heads, a pair shared by many CTAs
    (700, 300, 6, 2, [700, 431]),         # hidden chunks in the last pairs only, two lengths
    (513, 513, 8, 8, None),               # one token in the last pair
    (2300, 130, 5, 1, None),              # three chunks per head and a bit
    (257, 65, 3, 1, [257, 65]),           # the shorter sequence is all window
])
def test_row_chunks_shared_by_several_ctas(N, W, Hq, Hkv, lens):
    case = synth.make_prefill("items", B=len(lens) if lens else 1, Hq=Hq, Hkv=Hkv, d=128, W=W, N=lens or N, dtype="bf16", seed=N + W, hh_frac=0.02)
    _check(case, ["VK"], tight=2e-2)
    _check(case, ["V", "K", "VK", "ATTN"], tight=2e-2)


@pytest.mark.parametrize("N", [2048, 4100])      # one kernel; pass 1, merge and pass 2
def test_peaky_attention_cancellation_case(N):
    # some attention weights approach 1, so ||v_p - o_i||^2 cancels heavily
    case = synth.make_prefill("peaky", B=1, Hq=8, Hkv=2, d=128, W=16, N=N, dtype="bf16", seed=5,
                              hh_frac=0.01, peaky=True)
    _check(case, ["V", "K", "VK"], path="simt")
    _check(case, ["V", "K", "VK"], path="auto")


@pytest.mark.parametrize("N", [700, 2600])       # one kernel; pass 1, merge and pass 2
def test_strided_views_and_split_invariance(N):
    # K/V given as non-contiguous views (token stride 2d) must score like their contiguous copies
    case = synth.make_prefill("strided", B=1, Hq=4, Hkv=2, d=128, W=8, N=N, dtype="bf16", seed=9)
    q, k, v = H.upload(case)
    wide_k = torch.zeros((1, 2, N, 256), dtype=torch.bfloat16, device="cuda")
    wide_v = torch.zeros_like(wide_k)
    wide_k[..., :128] = k
    wide_v[..., :128] = v
    a = api.obc_score(q, k, v, variants=["VK"])
    b = api.obc_score(q, wide_k[..., :128], wide_v[..., :128], variants=["VK"])
    torch.cuda.synchronize()
    assert torch.equal(a, b)


def test_workspace_poison_does_not_leak():
    case = synth.make_prefill("poison", B=1, Hq=4, Hkv=1, d=128, W=4, N=300, dtype="f32", seed=3)
    q, k, v = H.upload(case)
    p = api.score_params(q, k, variants=["VK"])
    ws = torch.full((api.obc_score_workspace(p),), 0xFF, dtype=torch.uint8, device="cuda")   # NaN pattern
    s = api.obc_score(q, k, v, variants=["VK"], workspace=ws)
    want = H.oracle_scores(case, ["VK"])["VK"]
    H.assert_scores_close(s[0].cpu().numpy(), want, "f32", tight=2e-5)


@pytest.mark.parametrize("path", ["simt", "tc"])
def test_ragged_batch_with_poisoned_workspace(path):
    """Splits past the end of a shorter sequence run nothing and write nothing: whatever the workspace held
    there (here a NaN pattern) must not reach the scores."""
    case = synth.make_prefill("ragpoison", B=3, Hq=8, Hkv=2, d=128, W=16, N=[9000, 700, 2500], dtype="bf16", seed=21)
    q, k, v = H.upload(case)
    lens = H.lens_dev(case)
    p = api.score_params(q, k, seq_lens=lens, variants=["VK"], path=path)
    ws = torch.full((api.obc_score_workspace(p),), 0xFF, dtype=torch.uint8, device="cuda")
    s = api.obc_score(q, k, v, seq_lens=lens, variants=["VK"], path=path, workspace=ws)
    api.obc_score_status(ws)
    want = H.oracle_scores(case, ["VK"])["VK"]
    H.assert_scores_close(s[0].cpu().numpy(), want, "bf16", tight=2e-2, what=f"ragged poison {path}")


def test_kernel_spans_are_recorded_and_cleared():
    """Both tensor-core kernels leave a plausible device-side extent in the workspace header; reading
    it zeroes it; the CUDA-core path leaves nothing."""
    case, run = synth.config(2, shrink=8)
    q, k, v = H.upload(case)
    p = api.score_params(q, k, variants=["VK"])
    ws = torch.zeros(api.obc_score_workspace(p), dtype=torch.uint8, device="cuda")
    api.obc_score(q, k, v, variants=["VK"], workspace=ws)
    p1, p2 = api.obc_score_kernel_spans(ws)
    assert 1.0 < p1 < 1e4 and 1.0 < p2 < 1e4
    assert api.obc_score_kernel_spans(ws) == (0.0, 0.0)
    ps = api.score_params(q, k, variants=["VK"], path="simt")
    ws2 = torch.zeros(api.obc_score_workspace(ps), dtype=torch.uint8, device="cuda")
    api.obc_score(q, k, v, variants=["VK"], path="simt", workspace=ws2)
    assert api.obc_score_kernel_spans(ws2) == (0.0, 0.0)


@pytest.mark.parametrize("N", [1500, 2600])      # one kernel; pass 1, merge and pass 2
@pytest.mark.parametrize("Hq,Hkv,W", [(1, 1, 1), (2, 1, 1), (3, 1, 1)])
def test_joint_score_near_its_zero(Hq, Hkv, W, N):
    """Tokens whose scaled logit is close to -1 for every window row: (1 + Z)^2 is then small against 1 + Z^2, and the joint
    score keeps its digits only if the square is taken row by row.  The joint score is the same whatever else is asked for,
    and is off by no more of its own value than a few times what an error of 3e-7 in Z (fp32 logits of magnitude 1, summed
    over 128 channels) does to it: 2 |1 + Z| |v|^2 3e-7 of a score of at least Z^2 |o|^2."""
    scale = 128 ** -0.5
    rng = np.random.default_rng(11)
    q = np.repeat(rng.standard_normal((1, 1, W, 128)), Hq, 1)
    k = rng.standard_normal((1, Hkv, N, 128))
    u = q[0, 0, 0] / np.linalg.norm(q[0, 0, 0])
    near = -1 + 0.05 * rng.standard_normal(N)
    k += ((near / (scale * np.linalg.norm(q[0, 0, 0])) - k @ u)[..., None]) * u
    v = rng.standard_normal((1, Hkv, N, 128))
    bf = lambda x: synth.bf16_round(x.astype(np.float32))  # noqa: E731
    (q, qb), (k, kb), (v, vb) = bf(q), bf(k), bf(v)
    dev = [H.dev_bf16(x) for x in (qb, kb, vb)]
    want = ref.score(q, k, v, want=("VK",))["VK"][0, 0]
    got = [api.obc_score(*dev, variants=names)[at, 0, 0].cpu().numpy() for names, at in
           ((["VK"], 0), (["K", "VK"], 1), (["V", "K", "VK"], 2), (["V", "K", "VK", "ATTN"], 2), (["V", "K", "VK", "ATTN", "VATP"], 2))]
    assert all(np.array_equal(g, got[0]) or np.abs(g / got[0] - 1).max() < 1e-6 for g in got)
    own = np.abs(got[0] / want - 1)
    assert own.max() < 2e-5, own.max()


@pytest.mark.parametrize("Hq,Hkv,W,N", [(4, 2, 20, 300), (2, 2, 5, 700), (6, 2, 24, 500), (6, 2, 70, 400),
                                         (4, 2, 20, 2300), (2, 2, 5, 2700), (6, 2, 24, 2500)])
def test_queries_of_a_neighbour_that_are_not_finite(Hq, Hkv, W, N):
    """Row counts that do not fill the MMA's rows (R = 40, 5, 72 in one kernel, 210 in the multi-chunk pass 2, and 40, 5, 72 again in
    pass 1 and the single-chunk pass 2): what fills them up must not be the queries of the next head or sequence, which may be
    anything (a masked batch item, say)."""
    case = synth.make_prefill("neighbour", B=2, Hq=Hq, Hkv=Hkv, d=128, W=W, N=N, dtype="bf16", seed=N, hh_frac=0.02)
    q, k, v = H.upload(case)
    variants = ["V", "K", "VK", "ATTN"]
    clean = api.obc_score(q, k, v, variants=variants)
    for bad in (float("nan"), float("inf")):
        q2 = q.clone()
        q2[1] = bad
        q2[0, Hq // Hkv:] = bad
        assert torch.equal(api.obc_score(q2, k, v, variants=variants)[:, 0, 0], clean[:, 0, 0])


@pytest.mark.parametrize("N,Hq,Hkv", [(1500, 32, 32), (800, 64, 64)])
def test_fewer_than_64_window_rows_on_many_heads(N, Hq, Hkv):
    # 1024 and 2048 rows of 32 per head: the merge of the splits takes a warp per row (four splits, two), with both parts of -2 O
    case = synth.make_prefill("fewmany", B=1, Hq=Hq, Hkv=Hkv, d=128, W=32, N=N, dtype="bf16", seed=N, hh_frac=0.02)
    case.v, case.v_bits = synth.bf16_round(case.v + 1.0)          # outputs near one in every channel: the cross term weighs more
    for variants in (["VK"], ["V", "K", "VK", "ATTN", "VATP"]):
        want, got = H.oracle_scores(case, variants), H.gpu_scores(case, variants)
        mx = max(np.abs(want[n]).max() for n in variants if n in ("V", "K", "VK"))
        for n in variants:
            H.assert_scores_close(got[n], want[n], "f32", what=f"{case.name}/{n}", mx=None if n in ("ATTN", "VATP") else mx)


@pytest.mark.parametrize("W", [8, 20])                           # 32 rows, two bf16 parts; 80, one
def test_what_stands_past_a_ragged_end_is_not_used(W):
    lens = [2100, 3000, 130]
    case = synth.make_prefill("pastend", B=3, Hq=8, Hkv=2, d=128, W=W, N=lens, dtype="bf16", seed=W, hh_frac=0.02)
    q, k, v = H.upload(case)
    want = api.obc_score(q, k, v, seq_lens=H.lens_dev(case))
    for b, n in enumerate(lens):
        k[b, :, n:] = float("nan")
        v[b, :, n:] = float("nan")
    assert torch.equal(api.obc_score(q, k, v, seq_lens=H.lens_dev(case)), want)
