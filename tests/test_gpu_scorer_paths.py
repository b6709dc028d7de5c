"""GPU parity of the tensor-core scorers on inputs built to reach their rare branches, of the
single-sweep variant on ordinary shapes, and of the bounded-wait expiry path.

Both scorers evaluate a chunk of logits against a running reference and fall back to an exact
re-referencing when the result leaves a safe range; the fold of the per-item partial results has
the same two tiers.  Random benchmark inputs never leave the safe range, so these cases plant
keys whose logits sit hundreds of binary orders above the rest:
  - a dominant key in the last key tile, and one in the first tile only;
  - a first work item of tiny logits followed by a huge key in a later item (the exact fold);
  - a huge key in a slot that is evaluated by the FMA-pipe polynomial, whose exponent arithmetic
    would wrap without the range gate;
  - the same inside a tile, after chunks that were already turned into exponentials (the
    single-sweep kernel rescales what it has stored).
Every case is compared with the oracle at the score tolerance (Eq. 1, Sec. 3.1).
"""
import numpy as np
import pytest
import torch

from paper_2602_08585_b200 import lukv, synth
from gpu_helpers import assert_scores_close, bits, gpu_compress, gpu_score, params_of

pytestmark = pytest.mark.gpu

G, W, D = 4, 32, 128


def _planted(T, huge_at, tiny_upto=0, seed=0, huge=200.0, heads=1):
    """One layer of `heads` KV heads.  All queries share a strong common direction `base`; a planted key
    is `huge` times that direction, so its logit exceeds every other key's by about huge*10*scale*log2(e)
    (~255 binary orders at huge=200) in every row.  Keys below `tiny_upto` are scaled down to near zero."""
    g = torch.Generator().manual_seed(seed)
    base = torch.randn(D, generator=g)
    base = base / base.norm() * 10.0
    q = (torch.randn((1, 1, heads * G, W, D), generator=g) * 0.5 + base).to(torch.bfloat16)
    k = (torch.randn((1, 1, heads, T, D), generator=g) * 0.5).to(torch.bfloat16)
    if tiny_upto:
        k[:, :, :, :tiny_upto] = (k[:, :, :, :tiny_upto].float() * 0.01).to(torch.bfloat16)
    for j in huge_at:
        k[:, :, :, j] = (base / 10.0 * huge).to(torch.bfloat16)
    return q, k


CASES = {
    # name: (T, positions of planted keys, keys scaled to ~0)
    "dominant_key_in_last_prefix_tile": (4096 + W, [4096 - 5], 0),
    "dominant_key_in_first_tile_only": (4096 + W, [3], 0),
    "tiny_first_item_then_huge_key_in_a_later_item": (16384 + W, [9000], 1024),
    "huge_key_in_a_polynomial_slot": (4096 + W, [32 * 10 + 2], 0),           # chunk element 2 goes through the polynomial
    "huge_key_after_stored_chunks_of_its_tile": (4096 + W, [256 + 64 + 19], 0),  # third chunk of its tile, element 19
    "two_planted_keys_of_different_height": (8192 + W, [100, 7000], 0),
    "ragged_tail_with_a_dominant_window_key": (1300, [1300 - 3], 0),           # the planted key is a window key
}


@pytest.mark.parametrize("scorer", ["twosweep", "onesweep"])
@pytest.mark.parametrize("name", list(CASES))
def test_rare_branches_match_oracle(oracle, monkeypatch, scorer, name):
    monkeypatch.setenv("LUKV_SCORER", scorer)
    T, huge_at, tiny = CASES[name]
    q, k = _planted(T, huge_at, tiny, seed=len(name))
    if name == "two_planted_keys_of_different_height":
        k[:, :, :, huge_at[0]] = (k[:, :, :, huge_at[1]].float() * 0.5).to(torch.bfloat16)
    p = lukv.make_params(1, 1, 1, G, D, T, W, 7, torch.bfloat16, 2)
    got = gpu_score(p, q.cuda(), k.cuda()).cpu().numpy()
    ref = oracle.score(bits(q), bits(k), G, 7)
    assert_scores_close(got, ref)
    # the planted prefix key holds (nearly) all of the probability mass of every row
    prefix = [j for j in huge_at if j < T - W]
    if prefix and name != "two_planted_keys_of_different_height":
        assert ref[0, 0, prefix[0]] > 0.99 * G * W


ONE_SWEEP_SHAPES = [
    # S, L, H, G, T, w, kp: bf16, head_dim 128 (the shapes the tensor-core scorers take)
    (1, 2, 1, 4, 1300, 32, 7),      # 128 rows, ragged tail, an item with a single key tile
    (1, 1, 1, 7, 2048, 32, 7),      # 224 rows: two row blocks, the second partly padding
    (1, 1, 1, 4, 1111, 64, 5),      # 256 rows
    (2, 1, 3, 2, 3000, 16, 3),      # 32 rows: most of the row block is padding
    (1, 1, 2, 1, 4096 + 33, 33, 1),  # window not a multiple of anything
    (1, 1, 5, 4, 8192, 32, 7),      # 32 items per head, every CTA folds four rows
]


@pytest.mark.parametrize("shape", ONE_SWEEP_SHAPES)
def test_single_sweep_scorer_matches_oracle(oracle, monkeypatch, shape):
    monkeypatch.setenv("LUKV_SCORER", "onesweep")
    S, L, H, Gq, T, w, kp = shape
    g = torch.Generator().manual_seed(T + w)
    q = (torch.randn((S, L, H * Gq, w, D), generator=g) * 2.0).to(torch.bfloat16)
    k = (torch.randn((S, L, H, T, D), generator=g) * 2.0).to(torch.bfloat16)
    p = lukv.make_params(S, L, H, Gq, D, T, w, kp, torch.bfloat16, 2)
    got = gpu_score(p, q.cuda(), k.cuda()).cpu().numpy()
    assert_scores_close(got, oracle.score(bits(q), bits(k), Gq, kp))


def test_single_sweep_scorer_on_benchmark_config_and_repeats(oracle, monkeypatch):
    wl = synth.CONFIGS["llama8b_1layer_8k"]
    q, k, _ = synth.gen_tensors(wl, "cuda")
    p = params_of(wl)
    two = gpu_score(p, q, k)
    monkeypatch.setenv("LUKV_SCORER", "onesweep")
    one = gpu_score(p, q, k)
    ref = oracle.score(bits(q), bits(k), wl.G, wl.kp)
    assert_scores_close(one.cpu().numpy(), ref)
    assert_scores_close(two.cpu().numpy(), ref)
    for _ in range(20):                                 # every reduction has a fixed order: identical bits
        assert torch.equal(gpu_score(p, q, k), one)
    # the variant really is the kernel that ran
    _, _, v = synth.gen_tensors(wl, "cuda")
    Bs = wl.budgets()
    out = lukv.Outputs(p, Bs)
    names = [nm for nm, _ in lukv.lukv_compress_profile(p, q, k, v, torch.from_numpy(synth.gen_curves(wl)).cuda(), Bs,
                                                        out.k_out, out.v_out, out.kept_idx, out.budgets, out.offsets,
                                                        out.rows, out.dev_status, lukv.alloc_workspace(p))]
    assert "score_onepass" in names and "score_fused" not in names


@pytest.mark.parametrize("scorer", ["twosweep", "onesweep"])
def test_bounded_wait_expiry_is_reported_and_leaves_the_library_usable(monkeypatch, scorer):
    """The CTAs of the scorers wait for one another's partial results.  With the test hooks one work item's
    partials never arrive and the wait limit is short: the call must return, report LUKV_ERR_TIMEOUT in
    dev_status, and the next ordinary call with the same workspace must give the bits of a fresh run."""
    monkeypatch.setenv("LUKV_SCORER", scorer)
    wl = synth.scaled(synth.CONFIGS["llama8b_1layer_8k"], H=2, T=4096, P=33, needles=16)
    p = params_of(wl)
    q, k, v = synth.gen_tensors(wl, "cuda")
    curves = torch.from_numpy(synth.gen_curves(wl)).cuda()
    Bs = wl.budgets()
    ws = lukv.alloc_workspace(p)
    out = lukv.Outputs(p, Bs)

    def call(o):
        lukv.lukv_compress(p, q, k, v, curves, Bs, o.k_out, o.v_out, o.kept_idx, o.budgets, o.offsets, o.rows,
                           o.dev_status, ws)
        torch.cuda.synchronize()
        return int(o.dev_status.item())

    monkeypatch.setenv("LUKV_TEST_SPIN_LIMIT", "20000")
    monkeypatch.setenv("LUKV_TEST_DROP_ITEM", "0")
    assert call(out) == lukv.ERR_TIMEOUT
    monkeypatch.delenv("LUKV_TEST_SPIN_LIMIT")
    monkeypatch.delenv("LUKV_TEST_DROP_ITEM")
    assert call(out) == 0
    fresh = gpu_compress(p, q, k, v, synth.gen_curves(wl), Bs)
    assert torch.equal(out.kept_idx, fresh.kept_idx)
    assert torch.equal(out.k_out.view(torch.int16), fresh.k_out.view(torch.int16))
    assert torch.equal(out.v_out.view(torch.int16), fresh.v_out.view(torch.int16))


# Rows of logits that rise by so many binary orders above the reference (the first 32 keys' maximum): below, at and above the range
# of the tile's sum (80) and of the polynomial's arguments (100), in a slot of either kind; one and two row blocks, the last of
# them with all its 128 rows or fewer, both head sizes, a first tile with hidden keys.
@pytest.mark.parametrize("rise", [40, 79, 82, 99, 102, 140])
@pytest.mark.parametrize("shape", [(1, 16, 128, 700), (4, 32, 64, 2100), (5, 32, 128, 1500), (7, 32, 64, 1111), (4, 64, 128, 1300),
                                   (4, 32, 128, 150)])
def test_sums_that_rise_within_an_item(oracle, shape, rise):
    Gq, w, d, T = shape
    g = torch.Generator().manual_seed(1000 * rise + T)
    base = torch.randn(d, generator=g)
    base = base / base.norm()
    q = (torch.randn((1, 1, 2 * Gq, w, d), generator=g) * 0.05 + 10.0 * base).to(torch.bfloat16)
    k = (torch.randn((1, 1, 2, T, d), generator=g) * 0.05).to(torch.bfloat16)
    height = rise / (10.0 * 1.4426950408889634) * d ** 0.5  # logit = height * 10 / sqrt(d)
    last = T - w - 1
    for h, j in ((0, min(last, 128 + 34)), (1, min(last, 128 + 37))):  # element 2 of a chunk goes through the polynomial, 5 does not
        k[0, 0, h, j] = (height * base).to(torch.bfloat16)
    p = lukv.make_params(1, 1, 2, Gq, d, T, w, 7, torch.bfloat16, 2)
    got = gpu_score(p, q.cuda(), k.cuda()).cpu().numpy()
    assert_scores_close(got, oracle.score(bits(q), bits(k), Gq, 7))
