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


def _replay(H, T, rank, bits, G, g, dtype, spread, dense=False, seed=5):
    """(error of each group's zero-point, the group's range, what channels of earlier blocks of `unit` channels have pushed onto the
    element that is the minimum), each [H, groups, D]; float64."""
    gen = torch.Generator().manual_seed(seed)
    q = torch.randn((H, 1024, 16), generator=gen) @ torch.randn((H, 16, D), generator=gen) + 0.1 * torch.randn((H, 1024, D), generator=gen)
    k = torch.randn((1, H, T, D), generator=gen)
    k[..., ::32] *= 10
    k *= torch.exp(0.5 * np.log(spread) * torch.randn((1, H, 1, D), generator=gen))
    k = k.to(dtype)
    s = sq.Subspace(H, D)
    sq.squat_build_subspace(s, q.to(dtype).cuda(), rank, 1e-3, g)
    if dense:
        sq.squat_subspace_select_key_kernel(s, 1)
    W = torch.from_numpy(sq.squat_subspace_export(s)["W"]).double()
    kc, ks, kz = alloc_key_outputs(1, H, T, D, bits, G)
    sq.squat_quantize_keys(s, k.cuda(), bits, G, kc, ks, kz)
    torch.cuda.synchronize()
    s.close()
    codes = torch.from_numpy(oracle.unpack(kc[0].cpu().numpy().reshape(H * T, -1), D, bits)).view(H, T // G, G, D).double()
    scale, zero = ks[0].cpu().double(), kz[0].cpu().double()
    deq = (codes * scale.unsqueeze(2) + zero.unsqueeze(2)).view(H, T, D)
    x, far = k[0].double().clone(), torch.zeros((H, T, D), dtype=torch.float64)
    unit = max(g, 16)
    for j in range(D - 1):
        push = (deq[:, :, j] - x[:, :, j]).unsqueeze(2) * W[:, None, j + 1:, j]
        x[:, :, j + 1:] += push
        first = (j // unit + 1) * unit
        far[:, :, first:] += push[:, :, first - j - 1:]
    xg = x.view(H, T // G, G, D)
    low, at = xg.min(2)
    return zero - low, xg.amax(2) - low, far.view(H, T // G, G, D).gather(2, at.unsqueeze(2)).squeeze(2)


@pytest.mark.parametrize("rank,bits,G,dtype,spread,bound", [
    (32, 2, 32, torch.bfloat16, 1.0, 1),
    (64, 4, 128, torch.bfloat16, 1.0, 1),
    (32, 2, 64, torch.float32, 1.0, 1),
    (32, 2, 32, torch.float32, 1000.0, 1),
])
def test_corrected_values_of_the_dense_kernel(rank, bits, G, dtype, spread, bound):
    err, rng, far = _replay(4, 2048, rank, bits, G, 1, dtype, spread)
    rms = (err / rng).square().mean().sqrt().item()
    slope = [2 ** 24 * ((err * far)[..., c:c + 16].sum() / far.square()[..., c:c + 16].sum()).item() for c in range(16, D, 16)]
    print(f"DENSE r{rank} b{bits} G{G} {dtype} spread {spread}: rms {rms * 1e7:.3f}e-7; slopes {[round(v, 2) for v in slope]}")


@pytest.mark.parametrize("rank,bits,G,g,dtype,spread,bound", [
    (32, 2, 32, 64, torch.bfloat16, 1.0, 1),
    (32, 2, 32, 32, torch.bfloat16, 1.0, 1),
    (64, 4, 128, 32, torch.float32, 1.0, 1),
    (32, 2, 32, 32, torch.float32, 1000.0, 1),
])
def test_corrected_values_of_the_block_kernel(rank, bits, G, g, dtype, spread, bound):
    for dense in (False, True):
        err, rng, far = _replay(4, 2048, rank, bits, G, g, dtype, spread, dense)
        rms = (err / rng).square().mean().sqrt().item()
        slope = [2 ** 24 * ((err * far)[..., c:c + g].sum() / far.square()[..., c:c + g].sum()).item() for c in range(g, D, g)]
        print(f"BLOCK dense={dense} r{rank} b{bits} G{G} g{g} {dtype} spread {spread}: rms {rms * 1e7:.3f}e-7; slopes {[round(v, 2) for v in slope]}")
