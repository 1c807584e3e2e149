"""The dense key kernels' units of work: one token per lane (groups of 32, and of 128 in small calls), two or four tokens per lane (groups of 64
and 128), ragged units, heads that change inside a CTA's range, and the blocks that are decided exactly."""
import numpy as np
import pytest
import torch

import oracle
import squat_inputs as si
import paper_2503_24358_b200 as sq
from parity import alloc_key_outputs, compare_key_unit, to_torch

pytestmark = pytest.mark.gpu

D = 128


@pytest.mark.parametrize("G,bits,dtype,m16,B,H,T", [
    (32, 2, torch.bfloat16, False, 1, 37, 512),      # 148 tiles: one per CTA on 148 SMs
    (32, 2, torch.bfloat16, False, 1, 149, 128),     # 149 tiles: the first size at which a CTA has two
    (32, 4, torch.float32, True, 3, 5, 224),         # 21 groups per head: ragged tiles and units
    (64, 2, torch.bfloat16, True, 5, 60, 192),       # 15 groups per head, 4 a unit: ragged, several heads per CTA
    (64, 4, torch.float32, False, 1, 3, 64),
    (128, 2, torch.float32, False, 7, 50, 128),      # 7 groups per head, 4 a unit; a sample alone (50 tiles): one token per lane
    (128, 4, torch.bfloat16, True, 2, 74, 128),      # 148 tiles: the last size with one token per lane
    (128, 4, torch.bfloat16, True, 3, 50, 128),      # 150: the first with four
    (128, 4, torch.bfloat16, False, 1, 2, 384),
    (128, 2, torch.bfloat16, True, 1, 1, 128),
])
def test_whole_and_window_calls_and_head_batches_agree(G, bits, dtype, m16, B, H, T):
    """Every group's result depends on its own tokens and its head's W alone, so however a call is cut into tiles, units and
    CTAs the bytes are the same: whole against one window per group against one call per sample."""
    gen = torch.Generator().manual_seed(G + H)
    W = torch.tril(0.3 * torch.randn((H, D, D), generator=gen), -1).numpy()
    k = torch.randn((B, H, T, D), generator=gen)
    k[..., ::31] *= 10
    k = k.to(dtype).cuda()
    s = sq.Subspace(H, D)
    sq.squat_subspace_import(s, W)
    meta = torch.float16 if m16 else torch.float32
    new = lambda b: [t if t.dtype == torch.uint8 else t.to(meta) for t in alloc_key_outputs(b, H, T, D, bits, G)]
    sq.squat_get_device_status(clear=True)
    whole = new(B)
    sq.squat_quantize_keys(s, k, bits, G, *whole)
    windows = [torch.zeros_like(t) for t in whole]
    for lo in range(0, T, G):
        sq.squat_quantize_keys(s, k[:, :, lo:lo + G], bits, G, windows[0][:, :, lo:], windows[1][:, :, lo // G:], windows[2][:, :, lo // G:],
                               out_stride_b=H * T, out_stride_h=T)
    samples = [new(1) for _ in range(B)]
    for b in range(B):
        sq.squat_quantize_keys(s, k[b:b + 1], bits, G, *samples[b])
    torch.cuda.synchronize()
    for i, w in enumerate(whole):
        assert torch.equal(w, windows[i])
        assert torch.equal(w, torch.cat([x[i] for x in samples]))
    assert sq.squat_get_device_status(clear=True) & ~sq.FLAG_ZERO_RANGE == 0
    s.close()


@pytest.mark.parametrize("uncorrected", [1, 2, 16, 17, 128])
@pytest.mark.parametrize("G", [32, 128])
def test_uncorrected_channels_are_decided_exactly(uncorrected, G):
    """The leading channels that nothing corrects hold raw values, where exact ties are structural: keys on a coarse grid, so
    that every third code is a tie; against the oracle, whose decisions on the stored scale they must equal bit for bit."""
    H, T, bits = 2, 1024, 2
    gen = torch.Generator().manual_seed(uncorrected)
    W = torch.tril(0.2 * torch.randn((H, D, D), generator=gen), -1)
    W[:, :uncorrected] = 0                               # row j' of W: what is pushed onto channel j'
    k = torch.randint(-6, 7, (1, H, T, D), generator=gen).float().to(torch.bfloat16)
    s = sq.Subspace(H, D)
    sq.squat_subspace_import(s, W.numpy())
    kc, ks, kz = alloc_key_outputs(1, H, T, D, bits, G)
    sq.squat_quantize_keys(s, k.cuda(), bits, G, kc, ks, kz)
    torch.cuda.synchronize()
    n = uncorrected
    for h in range(H):
        x = k[0, h].double().numpy().reshape(T // G, G, D)[:, :, :n]
        scale, zero = ks[0, h].cpu().numpy()[:, None, :n], kz[0, h].cpu().numpy()[:, None, :n]
        assert np.array_equal(zero[:, 0], x.min(1).astype(np.float32))
        assert np.array_equal(scale[:, 0], ((x.max(1) - x.min(1)).astype(np.float32) / np.float32(3)))
        want = np.rint((x - zero.astype(np.float64)) / scale.astype(np.float64))      # ties to even, in real arithmetic on the stored scale
        got = oracle.unpack(kc[0, h].cpu().numpy(), D, bits).reshape(T // G, G, D)[:, :, :n]
        assert np.array_equal(got, want)
    s.close()


@pytest.mark.parametrize("constant", [1, 15, 16, 17, 31])
@pytest.mark.parametrize("G,bits,m16", [(32, 2, False), (64, 4, False), (128, 2, False), (128, 4, True), (32, 4, True)])
def test_channel_behind_constant_ones_is_decided_exactly(constant, G, bits, m16):
    """Constant leading channels leave no error, so under a full W the channel behind them holds raw values like an uncorrected one: in
    the first block of 32 channels, all of which are decided exactly, its codes and grid are those of plain rounding.  Every third
    group is such a one; the others are ordinary, and which groups share a warp or a call changes no byte."""
    H, T, L, n = 2, 9 * 128, 2 ** bits - 1, constant
    gen = torch.Generator().manual_seed(100 * constant + G)
    W = torch.tril(0.2 * torch.randn((H, D, D), generator=gen), -1)
    k = torch.randint(-6, 7, (1, H, T // G, G, D), generator=gen).float()
    k[:, :, ::3, :, :n] = 1.5
    k = k.view(1, H, T, D).to(torch.bfloat16).cuda()
    s = sq.Subspace(H, D)
    sq.squat_subspace_import(s, W.numpy())
    meta = torch.float16 if m16 else torch.float32
    out = [t if t.dtype == torch.uint8 else t.to(meta) for t in alloc_key_outputs(1, H, T, D, bits, G)]
    sq.squat_quantize_keys(s, k, bits, G, *out)
    windows = [torch.zeros_like(t) for t in out]
    for lo in range(0, T, G):
        sq.squat_quantize_keys(s, k[:, :, lo:lo + G], bits, G, windows[0][:, :, lo:], windows[1][:, :, lo // G:], windows[2][:, :, lo // G:],
                               out_stride_b=H * T, out_stride_h=T)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(out, windows))
    assert sq.squat_get_device_status(clear=True) == sq.FLAG_ZERO_RANGE      # the constant groups are reported
    x = k[0].double().cpu().numpy().reshape(H, T // G, G, D)[:, ::3, :, n]
    scale, zero = (t[0].float().cpu().numpy()[:, ::3, n] for t in out[1:])
    want = (x.max(2) - x.min(2)).astype(np.float32) / np.float32(L)
    assert np.array_equal(zero, x.min(2).astype(np.float32))
    assert np.array_equal(scale, want.astype(np.float16).astype(np.float32) if m16 else want)
    code = np.clip(np.rint((x - zero[..., None]) / scale[..., None].astype(np.float64)), 0, L)
    got = oracle.unpack(out[0][0].cpu().numpy().reshape(H * T, -1), D, bits).reshape(H, T // G, G, D)[:, ::3, :, n]
    assert np.array_equal(got, code)
    s.close()


@pytest.mark.parametrize("H", [2, 32])           # 10 tiles: one token per lane; 160: two pairs
def test_units_match_the_oracle_for_two_pairs_per_lane(H):
    # 5 groups of 128 per head: a ragged second unit; element by element under the replay protocol
    cfg = si.get_config(1).with_(batch=1, n_kv_heads=H, n_q_heads=H, n_tokens=640)
    gen = np.random.default_rng(3)
    W = np.tril(0.1 * gen.standard_normal((H, D, D)), -1).astype(np.float32)
    k_np = si.gen_keys(cfg)
    s = sq.Subspace(H, D)
    sq.squat_subspace_import(s, W)
    kc, ks, kz = alloc_key_outputs(1, H, 640, D, 4, 128)
    sq.squat_quantize_keys(s, to_torch(k_np, cfg.dtype), 4, 128, kc, ks, kz)
    torch.cuda.synchronize()
    for h in (0, H - 1):
        compare_key_unit(si.to_f32(k_np[0, h], cfg.dtype).astype(np.float64), W[h].astype(np.float64), 128, 4,
                         oracle.unpack(kc[0, h].cpu().numpy(), D, 4), ks[0, h].cpu().numpy(), kz[0, h].cpu().numpy())
    s.close()
