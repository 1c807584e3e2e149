"""The dense key kernels' results, byte for byte.  Near-ties and the order in which a value takes its corrections decide bytes far down a
token's channels, so a kernel that rounds otherwise is seen here though it may lie as close to real arithmetic.  Inputs are whole
numbers times powers of two, made by numpy; the digests are those of the kernel with one token per lane (keys_lane.cu), which all
sizes ran before there was another."""
import hashlib

import numpy as np
import pytest
import torch

import paper_2503_24358_b200 as sq
from parity import alloc_key_outputs

pytestmark = pytest.mark.gpu

D = 128

# group, bits, keys, 16-bit grids, batch, heads, tokens, channels that W leaves uncorrected, digest
CASES = [
    (32, 2, "bf16", False, 1, 5, 416, 1, "aa27a05ad6307754"),
    (32, 4, "f32", True, 2, 3, 224, 17, "40a2d106a23d3783"),
    (64, 2, "bf16", False, 1, 3, 1088, 1, "b2b17cbd0d6ca0b5"),
    (64, 4, "f32", False, 2, 2, 192, 5, "acfd8b2133944da2"),
    (64, 2, "bf16", True, 1, 2, 320, 33, "8a27c21caf116526"),
    (64, 4, "f32", True, 3, 100, 64, 1, "0738b4fc9e5e2e3b"),           # two units per CTA, several heads
    (128, 4, "bf16", False, 2, 80, 256, 1, "e7838dc2af23df77"),        # 320 tiles: four tokens per lane
    (128, 2, "f32", True, 3, 60, 128, 1, "6c8fd15203b9f1dc"),
    (128, 4, "bf16", True, 1, 150, 128, 64, "82ba9cd0a14a032f"),
    (128, 4, "bf16", False, 1, 2, 384, 1, "c62da23f20b06714"),         # 6 tiles: one token per lane
    (64, 2, "bf16", False, 1, 3, 256, 128, "7372d6c77882c383"),        # W = 0
    (128, 2, "bf16", False, 1, 150, 128, 128, "6b6e5b4df51c33e3"),
    (64, 4, "bf16", True, 1, 3, 256, 0, "76478f6db04c3cdb"),           # entries that are never applied, but the first block is not decided exactly
    (128, 2, "f32", False, 1, 150, 128, 0, "9ea59e97ea437615"),
    (64, 2, "ties", False, 1, 3, 640, 1, "6e4ce3bbc05e452f"),          # channels that hold raw values behind constant ones: exact ties where W corrects
    (64, 4, "ties", True, 1, 3, 640, 1, "9e1dd4054d8f4bc9"),
    (128, 2, "ties", False, 2, 75, 256, 1, "e6da49f205675825"),
]


def digest(G, bits, keys, m16, B, H, T, uncorrected):
    rng = np.random.default_rng([G, bits, B, H, T, uncorrected])
    W = np.tril(rng.integers(-60, 61, (H, D, D)), -1).astype(np.float32) / 256
    W[:, :uncorrected] = 0                              # row j' of W: what is pushed onto channel j'
    if uncorrected == 0:
        W[:, 0, 1] = 1
    if keys == "ties":
        k = rng.integers(-6, 7, (B, H, T // G, G, D))
        k[:, :, ::2, :, :1] = 2
        k[:, :, ::3, :, :20] = 2
        k = k.reshape(B, H, T, D).astype(np.float32)
    else:
        k = rng.integers(-(1 << 20), (1 << 20) + 1, (B, H, T, D)).astype(np.float32) / 2 ** 18
        k[..., ::31] *= 8
    k = torch.from_numpy(k).to(torch.float32 if keys == "f32" else torch.bfloat16).cuda()
    s = sq.Subspace(H, D)
    sq.squat_subspace_import(s, W)
    out = [t if t.dtype == torch.uint8 else t.to(torch.float16 if m16 else torch.float32) for t in alloc_key_outputs(B, H, T, D, bits, G)]
    sq.squat_quantize_keys(s, k, bits, G, *out)
    torch.cuda.synchronize()
    s.close()
    assert sq.squat_get_device_status(clear=True) & ~sq.FLAG_ZERO_RANGE == 0
    return hashlib.sha256(b"".join(t.cpu().numpy().tobytes() for t in out)).hexdigest()[:16]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c[:-1])))
def test_bytes(case):
    assert digest(*case[:-1]) == case[-1]
