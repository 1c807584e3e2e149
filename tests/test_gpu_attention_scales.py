"""GPU: the reader's accuracy does not depend on how far the value scales of a cache lie apart -- between channel groups, or
between a token that carries weight and one that carries none -- as a float32 sum's does not.

Reference: float64 on the stored codes and grids.  Bound, per output element: sum_t w_t (|zero_t| + scale_t code_t) times the
relative error of a weight and of its sum.  A float32 score is off by up to about 2^-24 A, A = scale * sum_c |q_c k_tc|
(products and sum), both for the token and for the maximum; twice that is allowed (four times with the rotary table, whose
entries are rounded to float32 and multiplied), plus 2^-20 for the exponential, the products and the sums."""
import numpy as np
import pytest
import torch

import paper_2503_24358_b200 as sq

pytestmark = pytest.mark.gpu
D = 128


def _bytes(codes, bits):
    c = codes.reshape(*codes.shape[:-1], -1, 8 // bits).astype(np.uint32)
    return sum(c[..., i] << (bits * i) for i in range(8 // bits)).astype(np.uint8)


def _turned(k, first):
    """Channel pairs (i, i + 64) of row t turned by (first + t) 10000^(-2 i / 128)."""
    ang = (first + np.arange(len(k)))[:, None] * 10000.0 ** (-2.0 * np.arange(64) / 128)
    a, b = k[:, :64], k[:, 64:]
    return np.concatenate([a * np.cos(ang) - b * np.sin(ang), a * np.sin(ang) + b * np.cos(ang)], 1)


def _data(rng, bits, G, qpk, T, H):
    NG, L = D // G, 2 ** bits - 1
    codes = [rng.integers(0, L + 1, (H, T, D)) for _ in range(2)]
    ks, kz = rng.uniform(0.3, 0.9, (H, T // G, D)) * 3 / L, rng.normal(-0.9, 0.1, (H, T // G, D))
    vs, vz = rng.uniform(0.3, 0.9, (H, T, NG)) * 3 / L, rng.normal(-0.9, 0.3, (H, T, NG))
    q = (6.0 * rng.standard_normal((H * qpk, D))).astype(np.float32)           # few tokens of a chunk carry weight
    return codes[0], codes[1], ks, kz, vs, vz, q


def _read(q, kcode, ks, kz, vcode, vs, vz, bits, G, rope, first):
    """The reader's output [query heads, D] for one sample, as float64."""
    H, T = kcode.shape[:2]
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)[None]).cuda()
    cache = [dev(x) for x in (_bytes(kcode, bits), ks, kz, _bytes(vcode, bits), vs, vz)]
    out = torch.empty((1, len(q), D), device="cuda")
    ws = torch.empty(sq.squat_decode_attention_workspace_bytes(1, len(q), T), dtype=torch.uint8, device="cuda")
    if rope:
        sq.squat_decode_attention_pre_rope(dev(q), *cache, H, T, bits, G, out, ws, sq.squat_rope_table(first + T).cuda(), first + T, first)
    else:
        sq.squat_decode_attention(dev(q), *cache, H, T, bits, G, out, ws)
    return out[0].double().cpu().numpy()


SHAPES = [(2, 32, 1, 1024, np.float32, False), (2, 32, 4, 1184, np.float16, False), (4, 64, 2, 640, np.float32, False),
          (4, 32, 4, 320, np.float32, True), (2, 128, 1, 2048, np.float32, False), (2, 64, 1, 768, np.float16, True)]


@pytest.mark.parametrize("bits,G,qpk,T,meta,rope", SHAPES)
@pytest.mark.parametrize("where,apart", [("groups", 6.0), ("groups", 1e3), ("groups", 3e4), ("tokens", 6.0), ("tokens", 1e3), ("tokens", 3e4), ("zeros", 1.0)])
def test_value_scales_far_apart(bits, G, qpk, T, meta, rope, where, apart):
    H, NG, L, first = 2, D // G, 2 ** bits - 1, 64
    rng = np.random.default_rng(int(apart) + bits + G + qpk)
    kcode, vcode, ks, kz, vs, vz, q = _data(rng, bits, G, qpk, T, H)
    if where == "groups":                                # the first group far above the others (one group: the first half of the heads)
        f = np.ones((H, 1, NG))
        f[:1 if NG == 1 else H, :, 1 if NG > 1 else 0:] = 1.0 / apart
        vs, vz = vs * f, vz * f
    elif where == "tokens":                              # one token per 256 far above the others, of almost no weight for any head
        for h in range(H):
            toward = q[h * qpk:(h + 1) * qpk].mean(0)
            at = np.arange(100, T, 256)
            kcode[h, at] = np.where(toward > 0, 0, L)
            vs[h, at] *= apart
    else:                                                # constant groups: scale 0
        vs[:, ::3] = 0.0
        vs[0] = 0.0
    ks, kz, vs, vz = (x.astype(meta) for x in (ks, kz, vs, vz))
    got = _read(q, kcode, ks, kz, vcode, vs, vz, bits, G, rope, first)
    f64 = lambda x: x.astype(np.float64)
    worst = 0.0
    for h in range(H):
        k = kcode[h] * np.repeat(f64(ks[h]), G, 0) + np.repeat(f64(kz[h]), G, 0)
        if rope:
            k = _turned(k, first)
        sc, z = np.repeat(f64(vs[h]), G, 1) * vcode[h], np.repeat(f64(vz[h]), G, 1)
        for j in range(h * qpk, (h + 1) * qpk):
            s = k @ f64(q[j]) / np.sqrt(D)
            w = np.exp(s - s.max())
            w /= w.sum()
            if where == "tokens" and not rope:
                assert (w[100::256] * apart).max() <= 1e-3      # (those tokens are no part of the result)
            A = (np.abs(k) @ np.abs(f64(q[j]))).max() / np.sqrt(D)
            bound = ((8 if rope else 4) * 2.0 ** -24 * A + 2.0 ** -20) * (w @ (np.abs(z) + sc))
            worst = max(worst, (np.abs(got[j] - w @ (sc + z)) / bound).max())
    print(f"worst error / bound {worst:.3f}")
    assert worst <= 1.0
    assert sq.squat_get_device_status(clear=True) & ~sq.FLAG_ZERO_RANGE == 0


@pytest.mark.parametrize("bits,G,qpk,T,meta,rope", SHAPES)
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_value_scale_that_is_not_finite_shows_in_its_group(bits, G, qpk, T, meta, rope, bad):
    H, NG = 2, D // G
    kcode, vcode, ks, kz, vs, vz, q = _data(np.random.default_rng(5), bits, G, qpk, T, H)
    q *= 0.1                                             # (every token carries weight)
    vs[1, T - 3, NG - 1] = bad
    got = _read(q, kcode, *(x.astype(meta) for x in (ks, kz)), vcode, *(x.astype(meta) for x in (vs, vz)), bits, G, rope, 64)
    assert np.isfinite(got[:qpk]).all()
    assert not np.isfinite(got[qpk:, D - G:]).any()
