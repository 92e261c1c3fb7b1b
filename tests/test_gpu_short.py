"""Short caches scored by one kernel (a cluster of CTAs per KV head, one 128-token tile each): GPU parity at the edges of
tiles, clusters and row counts."""
import numpy as np
import pytest
import torch

from paper_2510_07651_b200 import api, synth
from tests import helpers as H

pytestmark = pytest.mark.gpu

_ALL = ["V", "K", "VK", "ATTN", "VATP"]


def _check(got, want, rows, mx, what=""):
    """|gpu - ref| <= tight (|ref| + 1e-3 max|ref|): below 64 rows everything is summed in 32 bits and -2 O enters as two bf16 parts
    (2^-17 of it is left out, of terms that may be ten times their difference): 2e-4; with one part (2^-9) the parity tests' 2e-2.
    (Not their absolute 1e-4: a score that is exactly 0 beside scores of 1e3 is off by their rounding, 2^-23 of 1e3.)"""
    tight = 2e-4 if rows < 64 else 2e-2
    err = np.abs(got.astype(np.float64) - want)
    assert np.isfinite(got).all() and (err <= tight * (np.abs(want) + 1e-3 * mx)).all(), f"{what}: {err.max():.3e} of {mx:.3e}"


@pytest.mark.parametrize("N", [1, 127, 128, 129, 256, 257, 700, 1024, 1025, 2047, 2048, 2049])
@pytest.mark.parametrize("Hq,Hkv,W", [(3, 1, 1), (2, 2, 15), (7, 1, 9), (4, 2, 32), (7, 1, 16), (8, 2, 32)])
def test_one_kernel_edges(N, Hq, Hkv, W):
    W = min(W, N)
    case = synth.make_prefill("short", B=1, Hq=Hq, Hkv=Hkv, d=128, W=W, N=N, dtype="bf16", seed=1000 + N + W, hh_frac=0.02)
    want = H.oracle_scores(case, _ALL)
    for group in (["VK"], ["K", "VK"], _ALL):
        got = H.gpu_scores(case, group)
        mx = max(np.abs(want[n]).max() for n in ("V", "K", "VK"))
        for n in group:
            _check(got[n], want[n], Hq // Hkv * W, np.abs(want[n]).max() if n in ("ATTN", "VATP") else mx, f"{n} of {group}")


@pytest.mark.parametrize("lens,Hkv,causal", [([1, 128, 129, 600], 1, True), ([64, 1500, 900], 2, True), ([300, 40], 3, False)])
def test_one_kernel_ragged(lens, Hkv, causal):
    """CTAs whose tile lies past the end of a sequence merge their rows all the same and write zeros; what stands there is never used."""
    W = min(8, min(lens))
    case = synth.make_prefill("short ragged", B=len(lens), Hq=4 * Hkv, Hkv=Hkv, d=128, W=W, N=lens, dtype="bf16", seed=5, hh_frac=0.02)
    want = H.oracle_scores(case, ["VK"], causal=causal)["VK"]
    q, k, v = H.upload(case)
    for b, n in enumerate(lens):
        k[b, :, n:] = float("nan")
        v[b, :, n:] = float("nan")
    got = api.obc_score(q, k, v, seq_lens=torch.tensor(lens, dtype=torch.int32, device="cuda"), causal=causal)[0].cpu().numpy()
    _check(got, want, 4 * W, np.abs(want).max())
    for b, n in enumerate(lens):
        assert (got[b, :, n:] == 0).all()


def test_one_kernel_rows_of_a_neighbour():
    """A unit whose rows do not fill its chunk is not touched by the next unit's queries, finite or not."""
    case = synth.make_prefill("short rows", B=1, Hq=10, Hkv=2, d=128, W=15, N=500, dtype="bf16", seed=9)
    q, k, v = H.upload(case)
    want = api.obc_score(q, k, v)[0, 0, 0].clone()
    q[:, 5:] = float("inf")
    assert torch.equal(api.obc_score(q, k, v)[0, 0, 0], want)


@pytest.mark.parametrize("B,N", [(7, 2048), (8, 2048), (16, 1024), (40, 500), (148, 100), (149, 100)])
def test_one_kernel_and_three_agree(B, N):
    """On either side of the line (as many units as have their clusters on the chip at once) the scores are the same ones."""
    case = synth.make_prefill("short line", B=1, Hq=4, Hkv=1, d=128, W=8, N=N, dtype="bf16", seed=B)
    q, k, v = (x.expand(B, -1, -1, -1).contiguous() for x in H.upload(case))
    got = api.obc_score(q, k, v)[0]
    want = H.oracle_scores(case, ["VK"])["VK"][0]
    _check(got[0].cpu().numpy(), want, 32, np.abs(want).max())
    assert torch.equal(got, got[:1].expand_as(got))
