"""GPU parity of the histogram passes at the edges of how they are cut into
blocks: expert counts whose last tile is narrower than the others or whose
tokens straddle warps, and token counts on both sides of the lines between
tiles of 8 and 16 chunks and between rows of bins and bins banked by lane.
Counts are whole numbers: every bin equals the oracle's."""
import numpy as np
import pytest
import torch

import brute
import oracle
import paper_2609_28053_gb300 as eqb
from gpu_harness import Guarded, bits_f32, to_dev_bf16

pytestmark = pytest.mark.gpu

# Chunks of z per SM (T E / 8 / 152): the lines lie at 5,000 (banked bins) and
# 10,000 (16-chunk tiles).
CUTS = [(1, 8, 2),           # one thread's work
        (130, 264, 8),       # 33 chunks in tiles of 7, the last of 5
        (500, 264, 8),       # one chunk a tile, 512 threads
        (600, 1024, 8),      # 505: two, or five where the tiles are counted
        (1700, 264, 8),      # 369: 512 threads, several ranges
        (2600, 264, 8),      # 564: 1,024
        (14000, 200, 8),     # 2,302: two chunks a tile in pass 2
        (60000, 24, 4),      # 1,184: one
        (5000, 104, 3),      # 13 chunks: 7 and 6
        (23500, 256, 4),     # 4,947: rows
        (24500, 264, 4),     # 5,319: banked, tiles of 7 and 5 chunks
        (35000, 264, 8),     # 7,598
        (47000, 264, 4),     # 10,203: tiles of 11
        (32000, 392, 8),     # 10,315: 13, 13, 13 and 10 chunks, two columns each
        (200000, 64, 8),     # 10,526: one 8-chunk tile, four columns each
        (1600000, 8, 2)]     # 10,526: one chunk, 32 columns


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ok):
    eqb.load()


@pytest.mark.parametrize("T,E,K", CUTS)
def test_passes_and_step_match_oracle(T, E, K):
    rng = np.random.default_rng(T + E)
    z = brute.bf16_bits_from_f32(rng.standard_normal((T, E), dtype=np.float32))
    b = (rng.standard_normal(E) * 0.3).astype(np.float32)
    _, tau, _ = oracle.route(z, b, K)
    H_ref = oracle.hist_hi(z, tau)
    u, rho = oracle.select_hi(H_ref, oracle.target_rank(T, E, K))
    L_ref = oracle.hist_lo(z, tau, u)
    b_ref = oracle.bias_update(oracle.select_lo(L_ref, u, rho))
    zd, td = to_dev_bf16(z), torch.from_numpy(tau).cuda()
    H, L = Guarded((E, 256), torch.int32), Guarded((E, 256), torch.int32)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    eqb.eqb_margin_hist_pass1(zd, td, H.view, err)
    eqb.eqb_margin_hist_pass2(zd, td, torch.from_numpy(u).cuda(), L.view)
    torch.cuda.synchronize()
    assert H.intact() and L.intact() and err.item() == 0
    assert np.array_equal(H.view.cpu().numpy(), H_ref)
    assert np.array_equal(L.view.cpu().numpy(), L_ref)
    # pass 1 beside an injection of half of the tokens: the same counts
    H2, g = Guarded((E, 256), torch.int32), torch.zeros((T, E), device="cuda")
    off, coef = torch.tensor([0, T], device="cuda"), torch.rand((1, E), device="cuda")
    eqb.eqb_margin_hist_lei(zd, td, 1, H2.view, g, coef, off, 0, (T + 1) // 2)
    torch.cuda.synchronize()
    assert H2.intact() and np.array_equal(H2.view.cpu().numpy(), H_ref)
    assert torch.equal(g[:(T + 1) // 2], coef.expand((T + 1) // 2, E)) and not g[(T + 1) // 2:].any()
    # the one-call step, whose fine pass selects by tiles
    loads = torch.zeros((1, E), dtype=torch.int32, device="cuda")
    bn = Guarded((E,), torch.float32)
    ws = torch.full((eqb.eqb_layer_workspace_bytes(E),), 0x5a, dtype=torch.uint8, device="cuda")
    eqb.eqb_layer_step(zd, torch.from_numpy(b).cuda(), K, off, loads, bn.view, ws, err_flag=err)
    torch.cuda.synchronize()
    assert bn.intact() and err.item() == 0
    assert np.array_equal(bits_f32(bn.view.cpu().numpy()), bits_f32(b_ref))
    # what the step leaves in its workspace: H, L, 256 bytes of counters, u, rho
    wb = ws.cpu().numpy()
    at = 2 * E * 1024 + 256
    assert np.array_equal(wb[:E * 1024].view(np.int32).reshape(E, 256), H_ref)
    assert np.array_equal(wb[E * 1024:2 * E * 1024].view(np.int32).reshape(E, 256), L_ref)
    assert np.array_equal(wb[at:at + E], u)
    at += (E + 255) // 256 * 256
    assert np.array_equal(wb[at:at + 4 * E].view(np.int32), rho)
