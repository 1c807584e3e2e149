"""GPU: the integer Gram kernel (bf16 queries, 1024 stacked rows or more) against exact sums, where it can go wrong: ragged
rows, stacked heads, channels of zeros, elements far below their channel's largest (listed remainders, then a full list)."""
import numpy as np
import pytest
import torch

import paper_2503_24358_b200 as sq

pytestmark = pytest.mark.gpu
D = 128


@pytest.mark.parametrize("H,qpk,T,data", [
    (32, 1, 1024, "normal"), (8, 4, 300, "normal"), (1, 1, 4097, "normal"), (2, 2, 2049, "zeros"), (40, 1, 1100, "normal"),
    (8, 1, 1500, "outliers"), (2, 1, 1024, "wide"), (4, 2, 5000, "normal")])
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
    q = q.to(torch.bfloat16)
    s = sq.Subspace(H, D)
    sq.squat_build_subspace(s, q.cuda(), 8, 1e-3)
    a = sq.squat_subspace_export(s, ("gram",))["gram"]
    sq.squat_build_subspace(s, q.cuda(), 8, 1e-3)
    assert np.array_equal(a, sq.squat_subspace_export(s, ("gram",))["gram"])           # the same bits every time
    for h in {0, H // 2, H - 1}:
        x = q[h * qpk:(h + 1) * qpk].double().numpy().reshape(-1, D)
        ref = x.astype(np.longdouble).T @ x.astype(np.longdouble)
        size = np.sqrt(np.outer(np.diag(ref), np.diag(ref))).astype(np.float64)
        err = np.abs((a[h] - ref).astype(np.float64))
        assert np.all(err <= 4e-15 * size + 0.0), (err / np.maximum(size, 1e-300)).max()
    assert sq.squat_get_device_status(clear=True) & ~sq.FLAG_ZERO_RANGE == 0
    s.close()
