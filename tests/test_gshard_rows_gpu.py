"""GPU parity of the GShard gradient where its lanes hold three or four chunks
of a row, at the edges of those widths, and of the rank average with more
shards than fit a kernel argument."""
import numpy as np
import pytest
import torch

import brute
import oracle
import paper_2609_28053_gb300 as eqb
from gpu_harness import Guarded, bits_f32, to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ok):
    eqb.load()


@pytest.mark.parametrize("T,E", [(1, 264), (63, 384), (700, 392), (1300, 520), (900, 1024), (257, 8), (5000, 8), (1290, 16)])
def test_gshard_rows(T, E):
    K, M, alpha = min(8, E // 4), 3, 50.0
    rng = np.random.default_rng(T + E)
    z = brute.bf16_bits_from_f32((rng.standard_normal((T, E)) * 2).astype(np.float32))
    off = np.array([0, T // 3, T // 3, T], np.int64)
    _, _, loads = oracle.route(z, np.zeros(E, np.float32), K, off)
    g = (rng.standard_normal((T, E)) * 0.1).astype(np.float32)
    want = oracle.gshard(g, z, loads, off, K, alpha)
    G = Guarded((T, E), torch.float32)
    G.view.copy_(torch.from_numpy(g))
    eqb.gshard_inject_grad(G.view, to_dev_bf16(z), torch.from_numpy(loads).cuda(), torch.from_numpy(off).cuda(), K,
                           alpha)
    torch.cuda.synchronize()
    assert G.intact()
    # the term is coef (r - mean) with |r| <= 1: coef = alpha / (n d) <= alpha / (n min d), each of its fp32 factors
    # within (E + 8) 2^-24 of its value (the sums over E experts), plus the final addition's rounding of g + term
    n = np.maximum(np.diff(off)[np.searchsorted(off[1:], np.arange(T), side="right")], 1)
    d = (1.0 / (1.0 + np.exp(-(z.astype(np.uint32) << 16).view(np.float32).astype(np.float64)))).sum(axis=1)
    term = (alpha / (n * d))[:, None]
    tol = term * 3.0 * (E + 8) * 2.0**-24 + np.abs(want) * 2.0**-23
    assert np.all(np.abs(G.view.cpu().numpy().astype(np.float64) - want) <= tol)


@pytest.mark.parametrize("E", [16, 64, 264])
@pytest.mark.parametrize("P", [128, 129])
def test_rank_average_of_many_shards(P, E):
    T, K = 3000, min(8, E // 4)
    rng = np.random.default_rng(P)
    z = brute.bf16_bits_from_f32(rng.standard_normal((T, E)).astype(np.float32))
    _, tau, _ = oracle.route(z, (0.1 * rng.standard_normal(E)).astype(np.float32), K)
    shards = [0] + sorted(rng.integers(0, T, P - 1).tolist()) + [T]
    want, _ = oracle.rank_averaged_bias(z, tau, K, shards)
    B = Guarded((E,), torch.float32)
    ws = torch.full((eqb.eqb_rank_averaged_workspace_bytes(E, P),), 0x5a, dtype=torch.uint8, device="cuda")
    eqb.eqb_rank_averaged_bias(to_dev_bf16(z), torch.from_numpy(tau).cuda(), K, np.array(shards), ws, b_out=B.view)
    torch.cuda.synchronize()
    assert B.intact()
    assert np.array_equal(bits_f32(B.view.cpu().numpy()), bits_f32(want))
