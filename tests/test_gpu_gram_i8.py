"""GPU: the integer Gram kernel (bf16 queries, 49152 stacked rows or more over all heads, twice that above 49 heads) against exact
sums, where it can go wrong: ragged rows, stacked heads, one wave of parts and two, channels of zeros, elements far below their
channel's largest (listed remainders, a full list, an overfull one)."""
import numpy as np
import pytest
import torch

import paper_2503_24358_b200 as sq

pytestmark = pytest.mark.gpu
D = 128


def _gram(x):
    """x^T x of bf16 numbers [rows, D]: sums over 16 rows in float64 (products of bf16 numbers are exact, so these are within
    16 x 2^-53 of sum |x_i x_j|), added up in extended precision."""
    ref = np.zeros((D, D), np.longdouble)
    for n in range(0, len(x), 4096):
        y = x[n:n + 4096]
        y = np.concatenate([y, np.zeros((-len(y) % 16, D))]).reshape(-1, 16, D)
        ref += (y.transpose(0, 2, 1) @ y).sum(0, dtype=np.longdouble)
    return ref


def _tiny(q, H, n, g):
    """n elements of each KV head's queries far below their channel's largest (none of the others is); 1.5 and 1.25 alternate"""
    q.copy_(q.sign() * q.abs().clamp(0.01, 4.0))
    rows = q.view(H, -1, D)
    for h in range(H):
        at = torch.randperm(rows[h].numel(), generator=g)[:n]
        rows[h].view(-1)[at] = 2.0 ** -26 * (1.25 + 0.25 * (torch.arange(n) % 2))


@pytest.mark.parametrize("H,qpk,T,data", [
    (32, 1, 1600, "normal"), (32, 1, 7001, "normal"), (8, 4, 1600, "normal"), (1, 1, 49153, "normal"), (2, 2, 12289, "zeros"),
    (40, 1, 1300, "normal"), (18, 1, 21001, "normal"), (64, 1, 1601, "normal"), (8, 1, 6200, "outliers"), (2, 1, 24600, "wide"),
    (4, 2, 6200, "normal"), (2, 1, 24600, "listed"), (3, 2, 8200, "full list"), (3, 2, 8200, "one head"), (1, 4, 12301, "wide")])
def test_gram_is_exact(H, qpk, T, data):
    g = torch.Generator().manual_seed(7)
    q = torch.randn((H * qpk, T, D), generator=g)
    if data == "zeros":
        q[:, :, 5] = 0.0
        q[:, 1:, 9] = 0.0
    elif data == "outliers":                             # two tokens far above the rest: some remainders below their digits
        q[:, 3] *= 3000.0
        q[:, T - 1] *= 1000.0
        q[:, 17, :4] = 1e-6
    elif data == "wide":                                 # every exponent of a wide range: the list of remainders overflows
        q *= torch.exp2(torch.randint(-40, 8, q.shape, generator=g).float())
    elif data in ("listed", "full list"):                # many remainders, then exactly as many as the list holds
        _tiny(q, H, 200 if data == "listed" else 256, g)
    elif data == "one head":                             # one more than it holds, in one head
        _tiny(q[2:4], 1, 257, g)
    q = q.to(torch.bfloat16)
    s = sq.Subspace(H, D)
    sq.squat_build_subspace(s, q.cuda(), 8, 1e-3)
    a = sq.squat_subspace_export(s, ("gram",))["gram"]
    sq.squat_build_subspace(s, q.cuda(), 8, 1e-3)
    assert np.array_equal(a, sq.squat_subspace_export(s, ("gram",))["gram"])           # the same bits every time
    for h in {0, H // 2, H - 1}:
        x = q[h * qpk:(h + 1) * qpk].double().numpy().reshape(-1, D)
        ref = _gram(x)
        size = np.sqrt(np.outer(np.diag(ref), np.diag(ref))).astype(np.float64)
        err = np.abs((a[h] - ref).astype(np.float64))
        assert np.all(err <= 4e-15 * size + 0.0), (err / np.maximum(size, 1e-300)).max()
    assert sq.squat_get_device_status(clear=True) & ~sq.FLAG_ZERO_RANGE == 0
    s.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_elements_that_are_not_finite_stay_in_their_head_and_channel(bad):
    H, T = 2, 24600
    q = torch.randn((H, T, D), generator=torch.Generator().manual_seed(9)).to(torch.bfloat16)
    q[0, 777, 5] = bad
    s = sq.Subspace(H, D)
    sq.squat_build_subspace(s, q.cuda(), 8, 1e-3)
    a = sq.squat_subspace_export(s, ("gram",))["gram"]
    x = q.double().numpy()
    x[0, 777, 5] = 0.0
    ok = np.ones((H, D, D), bool)
    ok[0, 5] = ok[0, :, 5] = False
    assert not np.isfinite(a[~ok]).any()
    for h in range(H):
        ref = _gram(x[h])
        size = np.sqrt(np.outer(np.diag(ref), np.diag(ref))).astype(np.float64)
        assert np.all((np.abs((a[h] - ref).astype(np.float64)) <= 4e-15 * size)[ok[h]])
    sq.squat_get_device_status(clear=True)
    s.close()


@pytest.mark.parametrize("H,qpk,T,stride_h,stride_t", [
    (1, 1, 49200, 0, 1 << 19), (1, 2, 24700, 24700 << 19, 1 << 19), (1, 3, 16500, 1 << 33, 128), (2, 1, 24700, 1 << 34, 128)])
def test_views_spread_over_more_than_32_gigabytes(H, qpk, T, stride_h, stride_t):
    size = (H * qpk - 1) * stride_h + (T - 1) * stride_t + D
    if torch.cuda.mem_get_info()[0] < 2 * size + (4 << 30):
        pytest.skip("not enough free device memory")
    x = torch.randn((H * qpk, T, D), generator=torch.Generator().manual_seed(5)).to(torch.bfloat16)
    q = torch.empty(size, dtype=torch.bfloat16, device="cuda").as_strided((H * qpk, T, D), (stride_h, stride_t, 1))
    q.copy_(x)
    s = sq.Subspace(H, D)
    sq.squat_build_subspace(s, q, 8, 1e-3)
    a = sq.squat_subspace_export(s, ("gram",))["gram"]
    for h in range(H):
        y = x[h * qpk:(h + 1) * qpk].double().numpy().reshape(-1, D)
        ref = _gram(y)
        size = np.sqrt(np.outer(np.diag(ref), np.diag(ref))).astype(np.float64)
        assert np.all(np.abs((a[h] - ref).astype(np.float64)) <= 4e-15 * size)
    s.close()
    del q
    torch.cuda.empty_cache()


def _us(s, q, passes=5):
    """Median time of a build from q, GPU events."""
    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(2)] for _ in range(passes)]
    for a, b in [ev[0]] + ev:
        a.record()
        sq.squat_build_subspace(s, q, 32, 1e-3)
        b.record()
    torch.cuda.synchronize()
    return 1e3 * sorted(a.elapsed_time(b) for a, b in ev)[passes // 2]


@pytest.mark.parametrize("H,T,data", [(8, 32768, "one token"), (32, 16384, "one token"), (8, 32768, "listed"), (32, 16384, "one head")])
def test_time_does_not_hang_on_the_data(H, T, data):
    # The digits can be no help with such queries: a build may then cost the integer kernel's pass and the fp64 kernel's, which
    # is what the same queries in float32 take, and no more (half as much again for clocks and noise).
    g = torch.Generator().manual_seed(3)
    q = torch.randn((H, T, D), generator=g)
    s = sq.Subspace(H, D)
    usual, fp64 = _us(s, q.to(torch.bfloat16).cuda()), _us(s, q.cuda())
    if data == "one token":
        q[:, T // 3] *= 1000.0
    elif data == "one head":
        q[0, T // 3] *= 1000.0
    else:
        _tiny(q, H, 250, g)
    took = _us(s, q.to(torch.bfloat16).cuda())
    print(f"usual {usual:.0f} us, float32 {fp64:.0f} us, these {took:.0f} us")
    assert took <= 1.5 * (usual + fp64)
    s.close()
