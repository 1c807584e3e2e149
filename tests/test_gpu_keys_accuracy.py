"""How far the float32 values that the key kernels correct lie from float64: Algorithm 1 is replayed in float64 with the kernel's own
codes and stored grids, so that no rounding decision differs, and a group's stored zero-point is compared with the minimum of the
replayed values."""
import numpy as np
import pytest
import torch

import oracle
import paper_2503_24358_b200 as sq
from parity import alloc_key_outputs

pytestmark = pytest.mark.gpu

D = 128


def _replay(H, T, rank, bits, G, g, dtype, spread, seed=5):
    """(error of each group's zero-point, the group's range), each [H, groups, D]; float64."""
    gen = torch.Generator().manual_seed(seed)
    q = torch.randn((H, 1024, 16), generator=gen) @ torch.randn((H, 16, D), generator=gen) + 0.1 * torch.randn((H, 1024, D), generator=gen)
    k = torch.randn((1, H, T, D), generator=gen)
    k[..., ::32] *= 10
    k *= torch.exp(0.5 * np.log(spread) * torch.randn((1, H, 1, D), generator=gen))
    k = k.to(dtype)
    s = sq.Subspace(H, D)
    sq.squat_build_subspace(s, q.to(dtype).cuda(), rank, 1e-3, g)
    W = torch.from_numpy(sq.squat_subspace_export(s)["W"]).double()
    kc, ks, kz = alloc_key_outputs(1, H, T, D, bits, G)
    sq.squat_quantize_keys(s, k.cuda(), bits, G, kc, ks, kz)
    torch.cuda.synchronize()
    s.close()
    codes = torch.from_numpy(oracle.unpack(kc[0].cpu().numpy().reshape(H * T, -1), D, bits)).view(H, T // G, G, D).double()
    scale, zero = ks[0].cpu().double(), kz[0].cpu().double()
    deq = (codes * scale.unsqueeze(2) + zero.unsqueeze(2)).view(H, T, D)
    x = k[0].double().clone()
    for j in range(D - 1):
        x[:, :, j + 1:] += (deq[:, :, j] - x[:, :, j]).unsqueeze(2) * W[:, None, j + 1:, j]
    xg = x.view(H, T // G, G, D)
    low = xg.amin(2)
    return zero - low, xg.amax(2) - low


# Bounds: 1.05 times what the kernel of keys_lane.cu, which every handle ran before there was another, shows on these inputs: 0.929, 0.771, 0.896 and 3.34e-7
# with element-wise updates (here too: the dense kernels give the same bytes); 0.321, 0.545, 0.296 and 1.84e-7 with blocks of 32 or 64 channels (keys_block.cu:
# 0.204, 0.545, 0.296, 1.84e-7).
@pytest.mark.parametrize("rank,bits,G,dtype,spread,bound", [
    (32, 2, 32, torch.bfloat16, 1.0, 0.976e-7),
    (64, 4, 128, torch.bfloat16, 1.0, 0.810e-7),
    (32, 2, 64, torch.float32, 1.0, 0.941e-7),
    (32, 2, 32, torch.float32, 1000.0, 3.51e-7),         # channels a factor of 1000 apart
])
def test_corrected_values_of_the_dense_kernels(rank, bits, G, dtype, spread, bound):
    err, rng = _replay(4, 2048, rank, bits, G, 1, dtype, spread)
    assert (err / rng).square().mean().sqrt() <= bound


@pytest.mark.parametrize("rank,bits,G,g,dtype,spread,bound", [
    (32, 2, 32, 64, torch.bfloat16, 1.0, 0.337e-7),
    (32, 2, 32, 32, torch.bfloat16, 1.0, 0.572e-7),
    (64, 4, 128, 32, torch.float32, 1.0, 0.311e-7),
    (32, 2, 32, 32, torch.float32, 1000.0, 1.93e-7),
])
def test_corrected_values_of_the_block_kernel(rank, bits, G, g, dtype, spread, bound):
    err, rng = _replay(4, 2048, rank, bits, G, g, dtype, spread)
    assert (err / rng).square().mean().sqrt() <= bound
