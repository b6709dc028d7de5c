"""Tensor-core scorer on contexts whose last work item holds one key tile (9 or 17 tiles in items of eight), with several
items per CTA, so that one MMA issuer has no tile in a job: every head against plain PyTorch, and repetitions bit for bit."""
import pytest
import torch

from gpu_helpers import SCORE_ATOL, SCORE_RTOL
from paper_2602_08585_b200 import lukv

pytestmark = pytest.mark.gpu


def _reference(q, k, T, w, kp):
    """One head: q [M][d] (row g*w + i is the query at position T-w+i), k [T][d] -> pooled scores [T-w]."""
    x = q.float() @ k[:T].float().t() * q.shape[1] ** -0.5
    pos = T - w + torch.arange(q.shape[0], device=q.device) % w
    x.masked_fill_(torch.arange(T, device=q.device)[None, :] > pos[:, None], float("-inf"))
    raw = torch.softmax(x.double(), dim=1).sum(dim=0)[:T - w]
    return torch.nn.functional.max_pool1d(raw[None, None], kp, 1, kp // 2)[0, 0] if kp > 1 else raw


@pytest.mark.parametrize("S,L,H,G,d,w,kp,lens", [
    (3, 27, 8, 4, 128, 32, 7, [1125]), (3, 13, 8, 4, 64, 16, 7, [1100]), (4, 10, 8, 1, 64, 16, 5, [1152]),
    (3, 11, 8, 2, 128, 32, 7, [2125]), (2, 30, 8, 8, 128, 32, 5, [1090]), (2, 30, 8, 8, 64, 32, 5, [2177]),
    (3, 40, 4, 4, 128, 32, 1, [129]), (3, 40, 4, 4, 64, 16, 1, [130]),
    (4, 19, 2, 4, 64, 16, 7, [1000, 3200, 3200, 2400]), (4, 12, 4, 4, 128, 16, 7, [2375, 8000, 7625, 1090]),
])
def test_items_of_one_tile(S, L, H, G, d, w, kp, lens):
    g = torch.Generator(device="cuda").manual_seed(sum(lens))
    T, ragged = max(lens), len(lens) > 1
    q = torch.randn((S, L, H * G, w, d), generator=g, device="cuda").to(torch.bfloat16)
    k = torch.randn((S, L, H, T, d), generator=g, device="cuda").to(torch.bfloat16)
    p = lukv.make_params(S, L, H, G, d, T, w, kp, "bf16", 2)
    ws = lukv.alloc_workspace(p)
    first, again = (torch.zeros((S, L * H, T - w), device="cuda") for _ in range(2))

    def score(out):
        if ragged:
            lukv.lukv_score_ragged(p, lens, q, k, out, ws)
        else:
            lukv.lukv_score(p, q, k, out, ws)

    score(first)
    for rep in range(30):
        score(again)
        assert torch.equal(again, first), rep
    for s in range(S):
        n = (lens[s] if ragged else T) - w
        for u in range(L * H):
            ref = _reference(q[s].reshape(L * H, G * w, d)[u], k[s].reshape(L * H, T, d)[u], n + w, w, kp)
            err = (first[s, u, :n].double() - ref).abs()
            assert bool((err <= SCORE_RTOL * ref + SCORE_ATOL).all()), (s, u, float((err / ref).max()))


@pytest.mark.parametrize("S,L,H,G,d,w,kp,lens", [
    (1, 1, 2, 4, 128, 32, 7, [300]),          # three tiles in items of two: a job of one tile
    (1, 1, 8, 4, 128, 32, 7, [8192]),         # 64 tiles in items of four
    (1, 3, 8, 4, 64, 32, 7, [8320]),          # 65 tiles in eleven items of five or six
    (1, 2, 4, 8, 128, 32, 5, [1999]),         # two row blocks, 16 tiles
    (1, 1, 2, 4, 128, 16, 5, [40000]),        # 313 tiles of two heads, items of different sizes
    (3, 1, 4, 4, 128, 32, 7, [3000, 640, 1000]), (5, 3, 8, 2, 64, 16, 7, [9000, 4125, 250, 7000, 875]),
])
def test_items_of_a_small_call(S, L, H, G, d, w, kp, lens):
    """Calls with few heads share a head out over more and smaller items; with several lengths their sizes differ by one tile."""
    test_items_of_one_tile(S, L, H, G, d, w, kp, lens)
