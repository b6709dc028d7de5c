"""GPU parity of the exact allocation solver (Sec. 4.2, Eq. "combinatorial_optimization") against the oracle.
The optimum is unique, the optimal budgets need not be: the optimum is compared (fp32 accumulation over N
heads against the oracle's fp64: relative 1e-5), the budgets are checked to be feasible and to reach it."""
import numpy as np
import pytest
import torch

from paper_2602_08585_b200 import lukv, synth

pytestmark = pytest.mark.gpu
RTOL = 1e-5


def gpu_exact(N, T, w, U, Bs, L=1):
    p = lukv.make_params(len(Bs), L, N // L, 1, 64, T, w, 1, "fp32", T + 1)
    ws = torch.empty(lukv.lukv_exact_workspace_bytes(p, max(Bs)), dtype=torch.uint8, device="cuda")
    budgets = torch.full((len(Bs), N), -7, dtype=torch.int32, device="cuda")
    offsets = torch.full((len(Bs) * N + 1,), -7, dtype=torch.int32, device="cuda")
    values = torch.zeros(len(Bs), dtype=torch.float64, device="cuda")
    lukv.lukv_exact_allocate(p, torch.from_numpy(np.ascontiguousarray(U, np.float32)).cuda(), Bs, budgets, offsets,
                             values, ws)
    torch.cuda.synchronize()
    return budgets.cpu().numpy(), offsets.cpu().numpy(), values.cpu().numpy()


def _value(U, b):
    return float(np.take_along_axis(U.astype(np.float64), b.astype(np.int64)[:, None], axis=1).sum())


def _check(oracle, N, T, w, U, Bs, L=1):
    n = T - w
    b, off, val = gpu_exact(N, T, w, U, Bs, L)
    _, val_ref = oracle.exact_allocate(U, T, w, Bs)
    for q, B in enumerate(Bs):
        tol = RTOL * max(1.0, abs(val_ref[q]))
        assert abs(val[q] - val_ref[q]) <= tol, (q, val[q], val_ref[q])
        assert b[q].sum() == B and b[q].min() >= 0 and b[q].max() <= n
        assert abs(_value(U, b[q]) - val_ref[q]) <= tol
    np.testing.assert_array_equal(off, np.concatenate([[0], np.cumsum(b.reshape(-1) + w)]))


def _rough(rng, N, P):
    inc = rng.exponential(size=(N, P - 1)) * np.where(rng.random((N, P - 1)) < 0.2, 3.0, 1.0)
    U = np.zeros((N, P), np.float32)
    U[:, 1:] = np.cumsum(inc, axis=1)
    return U


def test_small_cases_and_edges(oracle):
    rng = np.random.default_rng(80)
    N, T, w = 5, 40, 4
    U = _rough(rng, N, T + 1)
    U[:, 1:] -= rng.random((N, T)).astype(np.float32)            # not monotone
    _check(oracle, N, T, w, U, [0, 1, 17, 36, 100, N * (T - w) - 1, N * (T - w)])
    _check(oracle, 1, 16, 3, _rough(rng, 1, 17), [0, 5, 13])       # one head: b = B
    _check(oracle, 3, 8, 7, _rough(rng, 3, 9), [0, 2, 3])          # one rankable position per head


def test_medium_size_spans_many_tiles(oracle):
    rng = np.random.default_rng(81)
    N, T, w = 64, 1024, 32                                          # n = 992; budgets beyond one tile of 1024
    U = synth.gen_calibration_curves(81, 1, N, T)[0]
    _check(oracle, N, T, w, U, [5000, 30000], L=8)


def test_calibration_size_sandwich(oracle):
    # 256 heads x 3968 tokens: the oracle's recursion would take minutes; instead
    # value(greedy budgets on the raw curves) <= exact optimum <= optimum of the relaxed problem
    N, T, w = 256, 4000, 32
    n = T - w
    U = synth.gen_calibration_curves(synth.BASE_SEED, 1, N, T)[0]
    B = int(0.3 * N * n)
    b, off, val = gpu_exact(N, T, w, U, [B], L=32)
    assert b[0].sum() == B and b[0].min() >= 0 and b[0].max() <= n
    assert abs(_value(U, b[0]) - val[0]) <= RTOL * val[0]
    bg, _ = oracle.allocate(U, T, w, [B])
    g64, _ = oracle.hull(U)
    Hc = np.concatenate([np.zeros((N, 1)), np.cumsum(g64, axis=1)], axis=1)
    raw = _value(U, bg[0])
    relaxed = float(np.take_along_axis(Hc, bg[0].astype(np.int64)[:, None], axis=1).sum())
    assert raw <= val[0] * (1 + RTOL) and val[0] <= relaxed * (1 + RTOL)
    # the paper's point: the relaxation gives up very little
    assert (val[0] - raw) / val[0] < 0.01


def _recursion(U, B, n):
    """The recursion as defined, fp32, smallest b on ties: (budgets, optimum)."""
    f = np.full(B + 1, -np.inf, np.float32)
    f[0] = 0
    choice = []
    for row in U:
        g, arg = np.full(B + 1, -np.inf, np.float32), np.zeros(B + 1, np.int64)
        for b in range(min(n, B) + 1):
            c = f[:B + 1 - b] + row[b]
            better = c > g[b:]
            g[b:][better], arg[b:][better] = c[better], b
        f = g
        choice.append(arg)
    x, out = B, []
    for arg in reversed(choice):
        out.append(int(arg[x]))
        x -= out[-1]
    return out[::-1], f[B]


@pytest.mark.parametrize("kind", ["rough", "steps", "decay", "falling"])
@pytest.mark.parametrize("N,T,w,Bs", [(7, 130, 3, [1, 63, 64, 65, 128, 500, 7 * 127 - 1]),   # block and tile edges
                                      (3, 4096, 1, [4095, 4096, 8191])])                      # the longest curves
def test_budgets_of_the_full_recursion(kind, N, T, w, Bs):
    """Blocks are skipped on a bound: the budgets and the optimum stay those of the full recursion, bit for bit, on
    curves with and without a single maximum, with equal increments (ties) and falling ones."""
    rng = np.random.default_rng(82)
    inc = rng.exponential(size=(N, T)).astype(np.float32)
    if kind == "rough":
        inc -= 0.9
    elif kind == "steps":
        inc = np.floor(2 * inc)
    elif kind == "decay":
        inc *= (np.arange(1, T + 1) ** -rng.uniform(0.2, 1.6, size=(N, 1))).astype(np.float32)
    else:
        inc = -inc
    U = np.zeros((N, T + 1), np.float32)
    U[:, 1:] = np.cumsum(inc, axis=1)
    b, _, val = gpu_exact(N, T, w, U, Bs)
    for q, B in enumerate(Bs):
        ref, best = _recursion(U, B, T - w)
        assert list(b[q]) == ref and np.float32(val[q]) == best


def test_unsupported_shapes():
    f = torch.empty(1, device="cuda")
    p = lukv.make_params(1, 1, 4, 1, 64, 64, 8, 1, "fp32", 33)      # 2 tokens per segment
    assert lukv.lukv_exact_allocate(p, f, [10], f, f, f, f, check=False) == lukv.ERR_UNSUPPORTED
    p = lukv.make_params(1, 1, 4, 1, 64, 64, 8, 1, "fp32", 65, min_keep=0.1)
    assert lukv.lukv_exact_allocate(p, f, [40], f, f, f, f, check=False) == lukv.ERR_UNSUPPORTED


def test_curves_with_jumps_near_the_end_of_fp32():
    """Jumps of 1e37 to 3e37: a slope over 64 budgets, times the distance to a block, is beyond fp32, and the bound that
    skips blocks must not take that for "cannot matter"."""
    T, w = 2400, 16
    U = np.zeros((3, T + 1), np.float32)
    U[0, 2230:] = 1.5e37
    U[1, 2200:] = 1e37
    U[2, 90:] = 3e37
    Bs = [2210, 2295, 2300, 4600]
    b, _, val = gpu_exact(3, T, w, U, Bs)
    for q, B in enumerate(Bs):
        ref, best = _recursion(U, B, T - w)
        assert list(b[q]) == ref and np.float32(val[q]) == best


def _curves(kind, N, T):
    rng = np.random.default_rng(N + T)
    inc = rng.exponential(size=(N, T)) * np.arange(1, T + 1) ** -rng.uniform(0.2, 1.6, (N, 1))
    if kind == "rough":
        inc = rng.exponential(size=(N, T)) * np.where(rng.random((N, T)) < 0.2, 3.0, 1.0)
    elif kind == "falling":
        inc = rng.normal(size=(N, T))
    elif kind == "ties":
        inc = rng.integers(0, 3, (N, T)).astype(np.float64)
    elif kind == "zero":
        inc = np.zeros((N, T))
    elif kind == "steep":
        inc *= 1e33
    U = np.zeros((N, T + 1), np.float32)
    U[:, 1:] = np.cumsum(inc, axis=1)
    if kind in ("nan", "-inf", "inf"):  # no number at some tokens of every other head, its last ones among them
        U[::2, 1:][rng.random(U[::2, 1:].shape) < (0.3 if kind != "inf" else 0.01)] = float(kind)
        U[::4, -T // 2:] = float(kind)
    return U


@pytest.mark.parametrize("kind", ["utility", "rough", "falling", "ties", "zero", "steep", "nan", "-inf", "inf"])
@pytest.mark.parametrize("N,T,w,Bs,reduced", [
    (40, 300, 20, [1500, 0, 40 * 280, 7001], False),   # several sequences, no budget, all of it
    (24, 497, 50, [24 * 447 - 1, 63, 5000], False),    # more than six blocks of tokens on curves that leave them all
    (17, 130, 2, [640, 1087], False),                  # tokens up to a block's edge
    # from here on tokens and budgets are left out
    (40, 404, 20, [2300, 0, 40 * 384, 64, 40 * 384 - 1, 9001], True),
    (300, 100, 12, [300 * 88 // 3, 2000], True),      # more heads than the threads that add up their tokens
    (48, 700, 28, [48 * 672 // 4], True),              # eleven blocks on curves that leave all tokens; long curves' hulls
])
def test_same_solution_as_the_full_recursion(kind, N, T, w, Bs, reduced):
    """To the bit: the same smallest solution and the same sum, on curves that leave few tokens (utility), on curves that
    leave all (ties, zero), and where some values are no numbers, which no solution takes, or infinite."""
    n, U = T - w, _curves(kind, N, T)
    b, off, val = gpu_exact(N, T, w, U, Bs)
    # one kernel and three a sequence, or the hulls, the greedy solution and two more a sequence before the rows
    assert (lukv.lukv_last_launch_count() > 1 + 3 * len(Bs)) == reduced
    for q, B in enumerate(Bs):
        with np.errstate(invalid="ignore"):
            ref, best = _recursion(U, B, n)
        assert np.float32(val[q]) == best
        if best > -np.inf:  # else no solution: every one is as good
            assert list(b[q]) == ref
    if kind not in ("-inf", "nan"):
        np.testing.assert_array_equal(off, np.concatenate([[0], np.cumsum(b.reshape(-1) + w)]))


@pytest.mark.parametrize("kind", ["utility", "rough", "ties", "nan"])
@pytest.mark.parametrize("N,T,w,Bs", [
    (16, 2400, 32, [16 * 2368 // 5]),                  # fewest heads; rows of more blocks than a narrow step has, between narrow ones
    (33, 600, 24, [33 * 576 // 3, 33 * 576 - 5, 70]),  # an odd number of heads: the last one has a step of its own
    (150, 100, 36, [150 * 64 // 2, 1]),                # bands of few budgets, tokens up to a block's edge
])
def test_bands_and_narrow_steps(kind, N, T, w, Bs):
    """To the bit, where budgets are left out by the bounds at neighbouring slopes and narrow rows are made two at a time."""
    n, U = T - w, _curves(kind, N, T)
    b, off, val = gpu_exact(N, T, w, U, Bs)
    assert lukv.lukv_last_launch_count() > 1 + 3 * len(Bs)  # the greedy solution came first
    for q, B in enumerate(Bs):
        with np.errstate(invalid="ignore"):
            ref, best = _recursion(U, B, n)
        assert np.float32(val[q]) == best
        if best > -np.inf:
            assert list(b[q]) == ref


@pytest.mark.parametrize("seed", [3, 10, 17])
def test_values_that_are_no_numbers_bound_nothing(seed):
    """Where some values are no numbers the greedy solution need not have the sum of the budget (seed 10: 12189 instead of
    12117), and its value is no bound for leaving tokens out."""
    rng = np.random.default_rng(seed)
    N, T, w = 40, 404, 20
    inc = rng.exponential(size=(N, T)) * np.arange(1, T + 1) ** -rng.uniform(0.2, 1.6, (N, 1))
    U = np.zeros((N, T + 1), np.float32)
    U[:, 1:] = np.cumsum(inc, axis=1)
    none = rng.random(U[:, 1:].shape) < 10 ** rng.uniform(-4, -0.2)
    none[rng.random(N) < rng.uniform(0, 0.8)] = False
    U[:, 1:][none] = np.nan
    B = int(rng.integers(1, N * (T - w)))
    b, _, val = gpu_exact(N, T, w, U, [B])
    with np.errstate(invalid="ignore"):
        ref, best = _recursion(U, B, T - w)
    assert list(b[0]) == ref and np.float32(val[0]) == best


@pytest.mark.parametrize("N,T,w", [(32, 300, 20), (40, 404, 20)])  # all tokens; those that can matter
def test_a_wait_that_runs_out_leaves_no_solution(monkeypatch, N, T, w):
    """With the test hooks one CTA stores nothing and the wait limit is short: the optimum is no number and the budgets are
    zero.  The next ordinary call gives the same as a fresh one."""
    B = N * (T - w) // 2
    U = _rough(np.random.default_rng(9), N, T + 1)
    ref = gpu_exact(N, T, w, U, [B])
    monkeypatch.setenv("LUKV_TEST_SPIN_LIMIT", "20000")
    monkeypatch.setenv("LUKV_TEST_DROP_ITEM", "0")
    b, off, val = gpu_exact(N, T, w, U, [B])
    assert np.isnan(val).all() and not b.any()
    np.testing.assert_array_equal(off, w * np.arange(N + 1))
    monkeypatch.delenv("LUKV_TEST_SPIN_LIMIT")
    monkeypatch.delenv("LUKV_TEST_DROP_ITEM")
    for x, y in zip(gpu_exact(N, T, w, U, [B]), ref):
        np.testing.assert_array_equal(x, y)
