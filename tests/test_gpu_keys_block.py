"""GPU parity of the key quantizer for block updates (g = 32, 64): the subspace is built on the GPU, squat_quantize_keys then
runs the kernel for block updates, and the result is compared with the oracle under the protocol of parity.py and with the
dense kernel on the same handle."""
import numpy as np
import pytest
import torch

import oracle
import squat_inputs as si
import paper_2503_24358_b200 as sq
from parity import alloc_key_outputs, compare_key_unit, oracle_mats, to_torch

pytestmark = pytest.mark.gpu

D = 128


def _build(cfg, r, g):
    s = sq.Subspace(cfg.n_kv_heads, D)
    q = to_torch(si.gen_queries(cfg, n_tokens=max(cfg.n_tokens, 256)), cfg.dtype)
    sq.squat_build_subspace(s, q, r, cfg.lam, g)
    return s


def _quantize(s, cfg, k, bits, G, m16=False):
    B, H, T = cfg.batch, cfg.n_kv_heads, cfg.n_tokens
    kc, ks, kz = alloc_key_outputs(B, H, T, D, bits, G)
    if m16:
        ks, kz = ks.to(torch.float16), kz.to(torch.float16)
    sq.squat_quantize_keys(s, k, bits, G, kc, ks, kz)
    return kc, ks, kz


def _deq(cfg, kc, ks, kz, bits, G):
    B, H, T = cfg.batch, cfg.n_kv_heads, cfg.n_tokens
    deq = torch.empty((B, H, T, D), dtype=torch.float32, device="cuda")
    sq.squat_dequantize(sq.SQUAT_KEYS, kc, ks, kz, B, H, T, D, bits, G, deq)
    torch.cuda.synchronize()
    return deq


@pytest.mark.parametrize("g,r,bits,G,dtype,m16", [
    (64, 32, 2, 32, "bf16", False), (64, 64, 4, 128, "bf16", True), (64, 8, 2, 64, "f32", False), (64, 32, 2, 32, "bf16", True),
    (32, 32, 2, 32, "bf16", False), (32, 40, 4, 64, "bf16", True), (32, 8, 2, 128, "f32", False), (32, 16, 4, 32, "f32", True),
])
def test_block_keys_match_the_oracle(g, r, bits, G, dtype, m16):
    # 3 heads x batch 2 x 1024 tokens; the 99.9 % bar on the raw identical fraction as for the other two kernels
    cfg = si.get_config(1 if dtype == "bf16" else 0).with_(batch=2, n_kv_heads=3, n_q_heads=3, n_tokens=1024)
    B, H, T = cfg.batch, cfg.n_kv_heads, cfg.n_tokens
    k_np = si.gen_keys(cfg)
    k = to_torch(k_np, cfg.dtype)
    sq.squat_get_device_status(clear=True)
    s = _build(cfg, r, g)
    kc, ks, kz = _quantize(s, cfg, k, bits, G, m16)
    deq = _deq(cfg, kc, ks, kz, bits, G)
    un = oracle.unpack(kc.cpu().numpy().reshape(B * H * T, -1), D, bits).reshape(B, H, T, D)
    tot = {"elements": 0, "raw_equal": 0, "ties": 0}
    for h in range(H):
        m = oracle_mats(cfg, h, rank_r=r, g=g)
        for b in range(B):
            st = compare_key_unit(si.to_f32(k_np[b, h], cfg.dtype).astype(np.float64), m["W"], G, bits, un[b, h],
                                  ks[b, h].float().cpu().numpy(), kz[b, h].float().cpu().numpy(), deq[b, h].cpu().numpy(),
                                  m["Qhat"], meta16=m16)
            for key in tot:
                tot[key] += st[key]
    print(f"block kernel g={g} r={r} bits={bits} G={G} {dtype} m16={m16}:", tot)
    assert tot["raw_equal"] >= 0.999 * tot["elements"], tot
    # channels of the first block are uncorrected: both kernels decide them exactly, so they agree bit for bit
    sq.squat_subspace_select_key_kernel(s, True)
    kd, sd, zd = _quantize(s, cfg, k, bits, G, m16)
    torch.cuda.synchronize()
    nb = g * bits // 8
    assert torch.equal(kd[..., :nb], kc[..., :nb]) and torch.equal(sd[..., :g], ks[..., :g]) and torch.equal(zd[..., :g], kz[..., :g])
    assert (kd == kc).float().mean().item() >= 0.998
    assert sq.squat_get_device_status(clear=True) & ~sq.FLAG_ZERO_RANGE == 0
    s.close()


@pytest.mark.parametrize("g,G,B,H,T", [(64, 32, 3, 2, 160), (32, 32, 3, 3, 96), (64, 64, 1, 3, 192), (32, 64, 5, 1, 64),
                                       (64, 128, 1, 400, 128), (32, 128, 3, 2, 128), (32, 32, 1, 5, 32)])
def test_block_keys_ragged_tiles_strides_and_windows(g, G, B, H, T):
    # ragged tiles and units, heads that change inside a CTA's range, keys as a view of a fused projection, a prompt cut into
    # window calls written into a larger cache: identical bytes, and nothing outside the window touched
    cfg = si.get_config(1).with_(batch=B, n_kv_heads=H, n_q_heads=H, n_tokens=T)
    fused = torch.randn((B, T, H, 2, D), generator=torch.Generator().manual_seed(g + T)).to(torch.bfloat16).cuda()
    k = fused[:, :, :, 1].transpose(1, 2)
    s = _build(si.get_config(1).with_(n_kv_heads=H, n_q_heads=H, n_tokens=256), 16, g)
    kc, ks, kz = _quantize(s, cfg, k.contiguous(), 2, G)
    sq.squat_subspace_select_key_kernel(s, True)
    kd, sd, zd = _quantize(s, cfg, k.contiguous(), 2, G)
    sq.squat_subspace_select_key_kernel(s, False)
    assert (kc == kd).float().mean().item() >= 0.995       # a tie at this size moves up to 32 bytes of each of G tokens
    Tc = T + 2 * G
    parts = [torch.full((B, H, Tc, D // 4), 7, dtype=torch.uint8, device="cuda")] + [torch.full((B, H, Tc // G, D), 7.0, device="cuda") for _ in range(2)]
    cuts = [0, G, T] if T > G else [0, T]
    for lo, hi in zip(cuts, cuts[1:]):
        at = lo + G
        sq.squat_quantize_keys(s, k[:, :, lo:hi], 2, G, parts[0][:, :, at:], parts[1][:, :, at // G:], parts[2][:, :, at // G:],
                               out_stride_b=H * Tc, out_stride_h=Tc)
    torch.cuda.synchronize()
    for whole, part, n in ((kc, parts[0], G), (ks, parts[1], 1), (kz, parts[2], 1)):
        assert torch.equal(whole, part[:, :, n:-n])
        assert (part[:, :, :n] == 7).all() and (part[:, :, -n:] == 7).all()
    s.close()


@pytest.mark.parametrize("g,G,bits", [(64, 32, 2), (64, 128, 4), (32, 64, 2), (32, 32, 4)])
def test_block_keys_clamp_where_a_16_bit_grid_leaves_the_extremes_outside(g, G, bits):
    """Channels far from 0 against their range: the binary16 zero-point lies up to an eighth above or below the minimum, more than half a
    step of the grid.  In uncorrected channels (the exact decision), in the middle and in the last block; every third group is
    ordinary, so that one call holds both instances.  Algorithm 1 is replayed in float64 with the kernel's own codes and grids: a code is the
    clamped nearest one but for what float32 leaves open, half a unit in the last place of the key's and of the
    correction's sum (2^-24 of the value each) and 1e-6 L for the reciprocal; in uncorrected channels it is the nearest one."""
    cfg = si.get_config(0).with_(batch=1, n_kv_heads=2, n_q_heads=2, n_tokens=9 * 128)
    gen = torch.Generator().manual_seed(g + G)
    k = torch.randn((1, 2, cfg.n_tokens // 128, 128, D), generator=gen)
    far = [3, 31, 40, 63, 64, 100, 127]
    for grp in range(9):
        if grp % 3:
            k[:, :, grp, :, far] = 300 + 0.07 * grp + 0.3 * torch.rand((1, 2, 128, len(far)), generator=gen)
    k = k.view(1, 2, -1, D)
    sq.squat_get_device_status(clear=True)
    s = _build(cfg, 16, g)
    kc, ks, kz = _quantize(s, cfg, k.cuda(), bits, G, True)
    torch.cuda.synchronize()
    L, T = 2 ** bits - 1, cfg.n_tokens
    codes = torch.from_numpy(oracle.unpack(kc.cpu().numpy().reshape(2 * T, -1), D, bits)).view(2, T // G, G, D).double()
    scale, zero = ks[0].double().cpu().unsqueeze(2), kz[0].double().cpu().unsqueeze(2)
    deq = (codes * scale + zero).view(2, T, D)
    W = torch.from_numpy(sq.squat_subspace_export(s)["W"]).double()
    x = k[0].double().clone()
    for j in range(D - 1):
        x[:, :, j + 1:] += (deq[:, :, j] - x[:, :, j]).unsqueeze(2) * W[:, None, j + 1:, j]
    x = x.view(2, T // G, G, D)
    t = (x - zero) / scale
    outside = (t < -0.5) | (t > L + 0.5)                 # the case is met: on both sides in uncorrected channels, and in corrected ones, whose
    assert all((t[..., n] < -0.5).any() and (t[..., n] > L + 0.5).any() for n in far if n < g)         # ranges are wider
    assert outside[..., g:].any() and not outside[:, ::3 * 128 // G].any()
    off = (codes - t.clamp(0, L)).abs() - 0.5
    assert off[..., :g].max() <= 0
    assert (off <= 2 ** -23 * x.abs() / scale + 1e-6 * L).all()
    low, high = x.amin(2, keepdim=True), x.amax(2, keepdim=True)
    noise = 2 ** -22 * torch.maximum(low.abs(), high.abs())
    assert ((zero - low).abs() <= 2 ** -11 * low.abs() + noise).all()                      # one rounding to binary16
    assert ((scale - (high - low) / L).abs() <= 2 ** -11 * scale + 2 * noise / L).all()
    assert sq.squat_get_device_status(clear=True) == 0
    s.close()


@pytest.mark.parametrize("g,G,bits,dtype,m16,B,H,T", [
    (64, 32, 4, "f32", True, 3, 2, 160), (32, 64, 4, "bf16", True, 5, 3, 64), (64, 128, 4, "f32", False, 1, 310, 128), (32, 128, 2, "f32", True, 3, 2, 384)])
def test_block_keys_windows_of_other_forms(g, G, bits, dtype, m16, B, H, T):
    """The ragged units and window calls of the test above for 4 bits, float32 keys and 16-bit grids: identical bytes however a call is cut;
    grids of the uncorrected channels equal to the dense kernel's, and codes but for what ties move."""
    cfg = si.get_config(1).with_(batch=B, n_kv_heads=H, n_q_heads=H, n_tokens=T)
    k = torch.randn((B, H, T, D), generator=torch.Generator().manual_seed(g + T)).to(torch.float32 if dtype == "f32" else torch.bfloat16).cuda()
    s = _build(si.get_config(1).with_(n_kv_heads=H, n_q_heads=H, n_tokens=256), 16, g)
    whole = _quantize(s, cfg, k, bits, G, m16)
    parts = [torch.zeros_like(t) for t in whole]
    for b in range(B):
        for lo in range(0, T, G):
            sq.squat_quantize_keys(s, k[b:b + 1, :, lo:lo + G], bits, G, parts[0][b:b + 1, :, lo:], parts[1][b:b + 1, :, lo // G:], parts[2][b:b + 1, :, lo // G:],
                                   out_stride_b=H * T, out_stride_h=T)
    sq.squat_subspace_select_key_kernel(s, True)
    dense = _quantize(s, cfg, k, bits, G, m16)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(whole, parts))
    assert all(torch.equal(a[..., :n], b[..., :n]) for a, b, n in zip(whole, dense, (g * bits // 8, g, g)))
    assert (whole[0] == dense[0]).float().mean().item() >= 0.99
    s.close()


@pytest.mark.parametrize("captured,rebuilt", [(64, 1), (64, 32), (32, 64), (32, 16), (1, 64)])
def test_a_captured_key_call_follows_the_handle(captured, rebuilt):
    """A graph that holds a key call quantizes by the matrices that its handle has when the graph is launched, whatever block size they were
    built with: the dense kernel's bytes for matrices that are not the captured kernel's."""
    cfg = si.get_config(1).with_(batch=2, n_kv_heads=3, n_q_heads=3, n_tokens=256)
    q = to_torch(si.gen_queries(cfg, n_tokens=256), cfg.dtype)
    k = to_torch(si.gen_keys(cfg), cfg.dtype)
    s = _build(cfg, 32, captured)
    want_first = _quantize(s, cfg, k, 2, 32)
    out = [torch.zeros_like(t) for t in want_first]
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        sq.squat_quantize_keys(s, k, 2, 32, *out)
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(out, want_first))
    sq.squat_build_subspace(s, q, 32, cfg.lam, rebuilt)
    sq.squat_subspace_select_key_kernel(s, True)
    want = _quantize(s, cfg, k, 2, 32)
    for t in out:
        t.zero_()
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(out, want))
    assert not torch.equal(out[0], want_first[0])
    s.close()


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("g,channel", [(64, 5), (64, 70), (32, 40)])
def test_block_keys_nonfinite_stays_in_its_group_and_later_blocks(g, channel, value):
    cfg = si.get_config(1).with_(batch=1, n_kv_heads=2, n_q_heads=2, n_tokens=256)
    s = _build(cfg, 16, g)
    k = to_torch(si.gen_keys(cfg), cfg.dtype)
    ref = _quantize(s, cfg, k, 2, 32)
    torch.cuda.synchronize()
    sq.squat_get_device_status(clear=True)
    k[0, 1, 71, channel] = value
    got = _quantize(s, cfg, k, 2, 32)
    torch.cuda.synchronize()
    assert sq.squat_get_device_status(clear=True) & sq.FLAG_NONFINITE
    first = channel // g * g                                # of the group, this block and the later ones may differ
    for a, b, rows in zip(ref, got, (slice(64, 96), slice(2, 3), slice(2, 3))):
        keep = torch.ones_like(a, dtype=torch.bool)
        keep[0, 1, rows, (first // 4 if a.dtype == torch.uint8 else first):] = False
        assert torch.equal(a[keep], b[keep])
    s.close()


def test_zero_update_with_a_block_size_is_round_to_nearest():
    # W = 0 (rank 0) with a block size: the dense kernel's exact form, plain round-to-nearest as before
    cfg = si.get_config(0).with_(n_tokens=256)
    k = to_torch(si.gen_keys(cfg), cfg.dtype)
    out = []
    for g in (1, 64):
        s = _build(cfg, 0, g)
        out.append(_quantize(s, cfg, k, 2, 32))
        torch.cuda.synchronize()
        s.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
