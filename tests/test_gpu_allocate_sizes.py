"""GPU parity of stage (b) at the sizes where its kernels change: points per lane of the hull walk, curves in registers or
shared memory, one launch or two, heads per thread, lists staged or in place.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from gpu_helpers import gpu_allocate, gpu_compress
from paper_2602_08585_b200 import lukv

pytestmark = pytest.mark.gpu


def _curves(rng, N, P, kind):
    inc = rng.exponential(size=(N, P - 1)) * np.where(rng.random((N, P - 1)) < 0.2, 3.0, 1.0)
    if kind == "concave":
        inc = -np.sort(-inc, axis=1)                       # every point is a vertex
    elif kind == "ties":
        inc = -np.sort(-np.floor(inc * 2), axis=1)         # equal slopes inside and across heads
    elif kind == "mixed":
        inc = inc * np.arange(1, P) ** -0.7 - 0.02         # few vertices, falling tails
    U = np.zeros((N, P), np.float32)
    U[:, 1:] = np.cumsum(inc, axis=1)
    return U


@pytest.mark.parametrize("kind", ["rough", "concave", "ties", "mixed"])
@pytest.mark.parametrize("N,P", [(1, 2), (4, 65), (7, 97), (32, 161), (3, 289), (32, 544), (5, 545), (33, 98), (40, 1025),
                                 (3, 2049), (2, 4097), (300, 257), (1025, 5), (2100, 9)])
def test_allocation_at_the_edges(oracle, N, P, kind):
    rng = np.random.default_rng(1000 * N + P)
    s, w = (3, 4) if P < 1000 else (1, 2)
    T = s * (P - 1)
    if T <= w:
        T, w = 8 * (P - 1), 3
    U = _curves(rng, N, P, kind)
    most = N * (T - w)
    Bs = [0, 1, most // 5, most // 2 + 1, most - 1, most]
    p = lukv.make_params(len(Bs), 1, N, 1, 64, T, w, 1, "bf16", P)
    b, o = gpu_allocate(p, U, Bs)
    b_ref, o_ref = oracle.allocate(U, T, w, Bs)
    np.testing.assert_array_equal(b, b_ref)
    np.testing.assert_array_equal(o, o_ref)


@pytest.mark.parametrize("N,P", [(18944, 5), (18751, 9)])
def test_largest_head_counts(oracle, N, P):
    """As many heads as the greedy's shared memory holds: the allocation, the whole path and the profile build."""
    rng = np.random.default_rng(N)
    T, w = 8 * (P - 1), 4
    U = _curves(rng, N, P, "mixed")
    most = N * (T - w)
    Bs = [0, most // 3, most - 1]
    p = lukv.make_params(len(Bs), N, 1, 1, 64, T, w, 1, "bf16", P)
    b, o = gpu_allocate(p, U, Bs)
    b_ref, o_ref = oracle.allocate(U, T, w, Bs)
    np.testing.assert_array_equal(b, b_ref)
    np.testing.assert_array_equal(o, o_ref)

    p1 = lukv.make_params(1, N, 1, 1, 64, T, w, 1, "bf16", P)
    g = torch.Generator(device="cuda").manual_seed(N)
    q = torch.randn((1, N, 1, w, 64), generator=g, device="cuda").to(torch.bfloat16)
    k = torch.randn((1, N, 1, T, 64), generator=g, device="cuda").to(torch.bfloat16)
    out = gpu_compress(p1, q, k, k, U, Bs[1:2])
    np.testing.assert_array_equal(out.budgets.cpu().numpy(), b_ref[1:2])

    ratios = [0.25, 0.5]
    curves = np.stack([U, _curves(rng, N, P, "concave")])
    profile = torch.empty((2, N), device="cuda")
    ws = torch.empty(lukv.lukv_profile_workspace_bytes(p1, 2, 2), dtype=torch.uint8, device="cuda")
    lukv.lukv_profile_build(p1, torch.from_numpy(curves).cuda(), 2, ratios, profile, ws)
    np.testing.assert_array_equal(profile.cpu().numpy(), oracle.profile_build(curves, T, w, ratios))


@pytest.mark.parametrize("N,points", [(16, range(417, 513, 8)), (32, range(209, 257, 4)), (33, range(177, 241, 8)),
                                      (56, (113, 121, 129, 137)), (200, (29, 33, 37, 41))])
def test_shared_memory_around_48_kilobytes(oracle, N, points):
    """Curves whose staging, with the kernels' static arrays, comes to just under and just over what a kernel gets without
    asking."""
    rng = np.random.default_rng(N)
    for P in points:
        T, w = 2 * (P - 1), 2
        U = _curves(rng, N, P, "mixed")
        Bs = [N * (T - w) // 3, N * (T - w) - 5]
        p = lukv.make_params(len(Bs), 1, N, 1, 64, T, w, 1, "bf16", P)
        b, o = gpu_allocate(p, U, Bs)
        b_ref, o_ref = oracle.allocate(U, T, w, Bs)
        np.testing.assert_array_equal(b, b_ref)
        np.testing.assert_array_equal(o, o_ref)


@pytest.mark.parametrize("kind", ["concave", "noisy", "hump", "scallops"])
@pytest.mark.parametrize("N,P", [(8, 18), (8, 65), (32, 129), (4, 257), (8, 513), (5, 544), (40, 257), (33, 513)])
def test_curves_of_many_vertices(oracle, N, P, kind):
    """Curves with more vertices than are walked to: the rest goes through passes over its points, in the lists of one
    launch and of two; `hump` loses its points a few at a time, in dozens of passes."""
    rng = np.random.default_rng(N + P)
    t = np.arange(1, P)[None, :]
    inc = np.exp(-t / (P * rng.uniform(0.2, 1.0, (N, 1))))
    if kind == "noisy":
        inc = inc * (1 + 0.1 * rng.standard_normal((N, P - 1)))
    elif kind == "hump":      # a concave start, then a smooth convex stretch that turns concave
        inc = np.maximum(3 - 0.1 * t, 0) + np.exp(-((t - 0.6 * P) / (P / 5)) ** 2)
        inc = inc * rng.uniform(0.5, 2.0, (N, 1))
    elif kind == "scallops":
        inc = inc * (1 + 0.5 * np.sin(t / rng.uniform(0.5, 6.0, (N, 1))))
    U = np.zeros((N, P), np.float32)
    U[:, 1:] = np.cumsum(inc, axis=1)
    T, w = 3 * (P - 1), 4
    most = N * (T - w)
    Bs = [most // 7, most // 3 + 1, most * 4 // 5]
    p = lukv.make_params(len(Bs), 1, N, 1, 64, T, w, 1, "bf16", P)
    b, o = gpu_allocate(p, U, Bs)
    b_ref, o_ref = oracle.allocate(U, T, w, Bs)
    np.testing.assert_array_equal(b, b_ref)
    np.testing.assert_array_equal(o, o_ref)


@pytest.mark.parametrize("noise", [0.0, 0.003, 0.01, 0.02, 0.03, "half", "late"])
@pytest.mark.parametrize("N,P", [(40, 545), (40, 1030), (36, 4001), (33, 4097)])
def test_long_curves_whose_first_pass_leaves_many_points(oracle, N, P, noise):
    """Long curves that are smooth but for a little noise: between all points and a fifth of them are left by the first pass
    (at 4001 points 0.65, 0.45, 0.35, 0.29 and 0.27 of them), more than the shared memory of a curve holds at once.  "half":
    smooth up to the middle, rough behind it; "late": the other way round."""
    rng = np.random.default_rng(P)
    t = np.arange(1, P)[None, :]
    sigma = np.full((1, P - 1), 0.8 if isinstance(noise, str) else noise)
    if isinstance(noise, str):
        sigma[:, slice(0, P // 2) if noise == "half" else slice(P // 2, P)] = 0.0
    inc = t ** -rng.uniform(0.5, 0.9, (N, 1)) * (1 + sigma * rng.standard_normal((N, P - 1)))
    U = np.zeros((N, P), np.float32)
    U[:, 1:] = np.cumsum(inc, axis=1)
    T, w = 2 * (P - 1), 4
    most = N * (T - w)
    Bs = [most // 7, most // 3 + 1, most * 4 // 5]
    p = lukv.make_params(len(Bs), 1, N, 1, 64, T, w, 1, "bf16", P)
    b, o = gpu_allocate(p, U, Bs)
    b_ref, o_ref = oracle.allocate(U, T, w, Bs)
    np.testing.assert_array_equal(b, b_ref)
    np.testing.assert_array_equal(o, o_ref)


@pytest.mark.parametrize("exponent", [-105, -90, 90, 112, 117])
@pytest.mark.parametrize("kind", ["rough", "concave", "mixed"])
@pytest.mark.parametrize("N,P", [(6, 513), (40, 257), (6, 1025), (3, 4001)])
def test_curves_far_from_one(oracle, N, P, kind, exponent):
    """Curves scaled by a power of two that leaves every value and gain a normal number have the budgets of the unscaled
    curves: fp32 products that overflow or flush to zero decide nothing."""
    rng = np.random.default_rng(P)
    U = _curves(rng, N, P, kind)
    assert U.max() < 2.0 ** 13
    if exponent > 114:
        U *= np.float32(2.0 ** -4)    # up to the last factor of four below the largest number
    T, w = 2 * (P - 1), 2
    Bs = [N * (T - w) // 9, N * (T - w) // 3, N * (T - w) * 3 // 4]
    p = lukv.make_params(len(Bs), 1, N, 1, 64, T, w, 1, "bf16", P)
    b, o = gpu_allocate(p, U * np.float32(2.0 ** exponent), Bs)
    b_ref, o_ref = oracle.allocate(U, T, w, Bs)
    np.testing.assert_array_equal(b, b_ref)
    np.testing.assert_array_equal(o, o_ref)


@pytest.mark.parametrize("kind", ["rough", "concave", "mixed"])
@pytest.mark.parametrize("P,shift", [(545, 1), (607, 2), (640, 3), (641, 0), (673, 1), (801, 3), (1281, 2), (3997, 1)])
def test_long_curves_at_any_alignment(oracle, kind, P, shift):
    """The first pass over a long curve reads aligned groups of four points, 128 a turn: curves that start anywhere in a group
    and end anywhere in a turn, of which some leave all their points."""
    rng = np.random.default_rng(P)
    N, w = 6, 2
    T = P - 1
    U = _curves(rng, N, P, kind)
    Bs = [0, N * (T - w) // 3, N * (T - w) - 1]
    p = lukv.make_params(len(Bs), 1, N, 1, 64, T, w, 1, "bf16", P)
    store = torch.full((N * P + 8,), float("nan"), device="cuda")
    curves = store[shift:shift + N * P].view(N, P)
    curves.copy_(torch.from_numpy(U))
    b = torch.empty((len(Bs), N), dtype=torch.int32, device="cuda")
    o = torch.empty(len(Bs) * N + 1, dtype=torch.int32, device="cuda")
    lukv.lukv_allocate(p, curves, Bs, b, o, lukv.alloc_workspace(p))
    b_ref, o_ref = oracle.allocate(U, T, w, Bs)
    np.testing.assert_array_equal(b.cpu().numpy(), b_ref)
    np.testing.assert_array_equal(o.cpu().numpy(), o_ref)
