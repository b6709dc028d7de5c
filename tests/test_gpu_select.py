"""Selection at the branches of its threshold search, bit-exact against the oracle: scores given directly, so that the
keys around the cut are chosen."""
import numpy as np
import pytest
import torch

from gpu_helpers import gpu_compress, gpu_select_gather, params_of
from paper_2602_08585_b200 import lukv, synth

pytestmark = pytest.mark.gpu


def _case(S, N, T, w, budgets, n_sink=0):
    """Parameters, budgets and offsets on the device, K and V (K's first channel tells the position) and the rows."""
    p = lukv.make_params(S, 1, N, 1, 64, T, w, 1, "bf16", 2, n_sink=n_sink)
    b = np.asarray(budgets, np.int32).reshape(-1)
    off = np.concatenate([[0], np.cumsum(b + w)]).astype(np.int32)
    k = torch.zeros((S, 1, N, T, 64), dtype=torch.bfloat16, device="cuda")
    k[..., 0] = (torch.arange(T, device="cuda") % 251).to(torch.bfloat16)
    k[..., 1] = (torch.arange(T, device="cuda") // 251).to(torch.bfloat16)
    return p, torch.from_numpy(b).cuda(), torch.from_numpy(off).cuda(), off, k, int(off[-1])


def _resplit_scores(rng, n, kind):
    """Signed scores over the whole key range whose cut lies in a bin of more keys than are ranked directly."""
    x = rng.uniform(-1.0, 1.0, n).astype(np.float32)
    base = np.float32(0.5).view(np.uint32)
    dense = rng.permutation(n)[: n * 3 // 4]
    m = dense.size
    if kind == "one":       # distinct keys, 16 apart: a second split leaves a few per bin
        bits = base + 16 * np.arange(m, dtype=np.uint32)
    elif kind == "two":     # runs of 700 equal keys in neighbouring key values: down to bins of one key value
        bits = base + (np.arange(m, dtype=np.uint32) // 700)
    else:                   # one value
        bits = np.full(m, base, np.uint32)
    x[dense] = bits.astype(np.uint32).view(np.float32)
    return x


@pytest.mark.parametrize("kind", ["one", "two", "tied"])
@pytest.mark.parametrize("n", [3001, 7000, 16000, 32700, 60001, 120000, 250000])
def test_cut_in_a_bin_that_is_split_again(oracle, n, kind):
    rng = np.random.default_rng(n)
    w, heads = 4, 6
    scores = np.stack([_resplit_scores(rng, n, kind) for _ in range(heads)])
    budgets = [n // 8, n // 4, n // 2, n * 3 // 4, 1, n - 1]
    p, b, o, off, k, rows = _case(1, heads, n + w, w, budgets, n_sink=3)
    _, _, kept = gpu_select_gather(p, torch.from_numpy(scores).cuda(), b, o, k, k, rows)
    kept = kept.cpu().numpy()
    for h in range(heads):
        got = kept[off[h]:off[h + 1]]
        np.testing.assert_array_equal(got[:budgets[h]], oracle.select(scores[h], budgets[h], 3))
        np.testing.assert_array_equal(got[budgets[h]:], np.arange(n, n + w))


@pytest.mark.parametrize("d,dtype,T", [(64, "bf16", 600), (128, "bf16", 2064), (128, "fp32", 600), (64, "bf16", 100016)])
def test_slices_of_a_larger_calls_offsets(d, dtype, T):
    """Layer by layer on slices of one allocation's budgets and offsets, into outputs of the whole: from the third layer on
    the slice's rows lie beyond the rows that its own heads could fill."""
    L, H, w = 8, 2, 16
    n = T - w
    g = torch.Generator(device="cuda").manual_seed(T)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    k, v = (torch.randn((1, L, H, T, d), generator=g, device="cuda").to(dt) for _ in range(2))
    scores = torch.randn((1, L * H, n), generator=g, device="cuda")
    budgets = torch.from_numpy((n // 2 + 5 * np.arange(L * H)).astype(np.int32)).cuda()
    offsets = torch.cat([torch.zeros(1, dtype=torch.int32, device="cuda"), torch.cumsum(budgets + w, 0).to(torch.int32)])
    rows = int(offsets[-1])
    whole = gpu_select_gather(lukv.make_params(1, L, H, 1, d, T, w, 1, dtype, 2), scores, budgets, offsets, k, v, rows)
    assert rows > 3 * H * T
    p = lukv.make_params(1, 1, H, 1, d, T, w, 1, dtype, 2)
    ws = lukv.alloc_workspace(p)
    k_out, v_out = (torch.zeros((rows, d), dtype=dt, device="cuda") for _ in range(2))
    kept = torch.full((rows,), -1, dtype=torch.int32, device="cuda")
    for layer in range(L):
        lukv.lukv_select_gather(p, scores[0, layer * H:], budgets[layer * H:], offsets[layer * H:], k[0, layer], v[0, layer],
                                k_out, v_out, kept, rows, ws)
    torch.cuda.synchronize()
    for got, want in zip((k_out, v_out, kept), whole):
        assert torch.equal(got, want)


@pytest.mark.parametrize("n,n_sink", [(1500, 4), (32700, 0), (60001, 4)])
@pytest.mark.parametrize("bits,share", [(0x7FFFFFFF, 1.0), (0xFFFFFFFF, 1.0), (0x7FFFFFFF, 0.6), (0xFFFFFFFF, 0.6)])
def test_scores_that_are_no_numbers_stay_in_their_head(oracle, n, n_sink, bits, share):
    """A head with NaN scores still fills exactly its own rows (where they rank is left open, but equal ones tie: the lower
    position first); the heads around it are not touched."""
    rng = np.random.default_rng(n)
    w, heads = 8, 5
    scores = rng.standard_normal((heads, n)).astype(np.float32)
    budgets = [n // 3, n // 2, n // 3, n - 2, 7]
    nan_at = rng.random(n) < share
    for h in (1, 3):
        scores.view(np.uint32)[h, nan_at] = bits
    p, b, o, off, k, rows = _case(1, heads, n + w, w, budgets, n_sink=n_sink)
    _, _, kept = gpu_select_gather(p, torch.from_numpy(scores).cuda(), b, o, k, k, rows)
    kept = kept.cpu().numpy()
    for h in range(heads):
        got, tail = np.split(kept[off[h]:off[h + 1]], [budgets[h]])
        np.testing.assert_array_equal(tail, np.arange(n, n + w))
        if h not in (1, 3):
            np.testing.assert_array_equal(got, oracle.select(scores[h], budgets[h], n_sink))
            continue
        assert np.all(np.diff(got) > 0) and got[0] >= 0 and got[-1] < n
        np.testing.assert_array_equal(got[:n_sink], np.arange(n_sink))
        for part in (nan_at, ~nan_at):   # of either kind those that rank first
            at = np.flatnonzero(part[n_sink:]) + n_sink
            mine = np.intersect1d(got, at)
            x = scores[h][at] if part is not nan_at else np.zeros(at.size, np.float32)
            np.testing.assert_array_equal(np.searchsorted(at, mine), oracle.select(x, mine.size))


def test_a_query_that_is_no_number_stays_in_its_head():
    """One NaN in a query spoils all scores of its head: it still fills its own rows with positions in ascending order, and
    every other head's rows are those of the call without the NaN."""
    wl = synth.scaled(synth.CONFIGS["llama8b_1layer_8k"], H=4, T=4096, P=65)
    q, k, v = synth.gen_tensors(wl, "cuda")
    p, curves, Bs = params_of(wl), synth.gen_curves(wl), wl.budgets()
    ref = gpu_compress(p, q, k, v, curves, Bs)
    q[0, 0, 1 * wl.G, 3, 5] = float("nan")
    out = gpu_compress(p, q, k, v, curves, Bs)
    off, b = ref.offsets.cpu().numpy(), ref.budgets.cpu().numpy().reshape(-1)
    assert torch.equal(out.offsets, ref.offsets) and 0 < b[1] < wl.n
    for h in range(wl.N):
        rows = slice(int(off[h]), int(off[h + 1]))
        if h != 1:
            assert torch.equal(out.kept_idx[rows], ref.kept_idx[rows])
            assert torch.equal(out.k_out[rows], ref.k_out[rows]) and torch.equal(out.v_out[rows], ref.v_out[rows])
    got = out.kept_idx[int(off[1]):int(off[2])].cpu().numpy()
    assert np.all(np.diff(got) > 0) and got[0] >= 0 and got[b[1] - 1] < wl.n
    np.testing.assert_array_equal(got[b[1]:], np.arange(wl.n, wl.T))


@pytest.mark.parametrize("T,w", [(13, 5), (1024, 16), (1031, 7), (2050, 3), (4090, 9), (8195, 2), (16391, 6), (32774, 6),
                                 (40003, 4), (100001, 3), (200002, 8), (262145, 2)])
def test_pooling_inside_the_selection(oracle, T, w):
    """The whole path pools on the way into the selection (up to nine positions; a separate pass beyond): its kept positions
    are those of lukv_score, whose pooled scores are exactly the maxima of the un-pooled ones, and the oracle's selection.
    Every register layout, thread count and cluster size, rows of every remainder modulo 4."""
    H, G, d, n = 3, 1, 64, T - w
    g = torch.Generator(device="cuda").manual_seed(T)
    q = torch.randn((1, 1, H * G, w, d), generator=g, device="cuda")
    k = torch.randn((1, 1, H, T, d), generator=g, device="cuda")
    curves = np.array([[0.0, 3.0], [0.0, 2.0], [0.0, 1.0]], np.float32)
    raw = None
    for kp in (1, 3, 5, 7, 9, 11):
        p = lukv.make_params(1, 1, H, G, d, T, w, kp, "fp32", 2, n_sink=min(4, n) if kp in (5, 11) else 0)
        ws = lukv.alloc_workspace(p)
        scores = torch.empty((1, H, n), device="cuda")
        lukv.lukv_score(p, q, k, scores, ws)
        raw = scores.clone() if raw is None else raw
        assert torch.equal(scores, torch.nn.functional.max_pool1d(raw, kp, 1, kp // 2))
        Bs = [n + n // 3]    # one head whole, a third of the next, nothing of the last
        out = gpu_compress(p, q, k, k, curves, Bs)
        off, b, kept = out.offsets.cpu().numpy(), out.budgets.cpu().numpy()[0], out.kept_idx.cpu().numpy()
        for h in range(H):
            got, tail = np.split(kept[off[h]:off[h + 1]], [b[h]])
            np.testing.assert_array_equal(got, oracle.select(scores[0, h].cpu().numpy(), int(b[h]), p.n_sink))
            np.testing.assert_array_equal(tail, np.arange(n, T))
