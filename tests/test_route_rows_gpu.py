"""GPU parity of routing at the edges of its kernels: row widths on both sides
of every compile-time width, token counts on both sides of the line between a
warp per token and tiles, list lengths on both sides of theirs, and rows with
more candidates than a warp collects (all scores equal).  tau, indices and
loads equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import brute
import oracle
import paper_2609_28053_gb300 as eqb
from eqb_workloads import ragged_offsets
from gpu_harness import Guarded, bits_f32, to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ok):
    eqb.load()


def check(z, b, K, M, seed):
    T, E = z.shape
    off = ragged_offsets(T, M, seed=seed) if M > 1 else np.array([0, T], np.int64)
    idx_ref, tau_ref, loads_ref = oracle.route(z, b, K, off)
    idx, tau, loads = Guarded((T, K), torch.int32), Guarded((T,), torch.float32), Guarded((M, E), torch.int32)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    eqb.eqb_route_topk(to_dev_bf16(z), torch.from_numpy(b).cuda(), K, torch.from_numpy(off).cuda(), idx.view,
                       tau.view, loads.view, err_flag=err)
    torch.cuda.synchronize()
    assert idx.intact() and tau.intact() and loads.intact() and err.item() == 0
    assert np.array_equal(idx.view.cpu().numpy(), idx_ref)
    assert np.array_equal(bits_f32(tau.view.cpu().numpy()), bits_f32(tau_ref))
    assert np.array_equal(loads.view.cpu().numpy(), loads_ref)


WIDTHS = [8, 32, 40, 64, 72, 96, 104, 128, 136, 160, 168, 192, 200, 224, 232, 256, 264, 320, 328, 384, 392, 512, 520,
          640, 648, 1024]


@pytest.mark.parametrize("E", [128, 512, 1024])
@pytest.mark.parametrize("T,M", [(40, 1), (1000, 1), (3000, 3), (3001, 40), (8192, 1)])
def test_loads_of_few_tokens(T, E, M):
    """A warp per token, on both sides of the line between each token's adds
    and the block's counters (an average load of 40)."""
    rng = np.random.default_rng(T + E)
    z = brute.bf16_bits_from_f32(rng.standard_normal((T, E), dtype=np.float32))
    check(z, (rng.standard_normal(E) * 0.3).astype(np.float32), 8, M, seed=E)


@pytest.mark.parametrize("E", WIDTHS)
@pytest.mark.parametrize("side", ["one", "warp", "tile"])
def test_row_widths(E, side):
    K = min(8, E // 4)
    line = min(32 * E, 8192)  # between a warp per token and tiles
    T = {"one": 1, "warp": line, "tile": line + 1}[side]
    rng = np.random.default_rng(E)
    z = brute.bf16_bits_from_f32(rng.standard_normal((T, E), dtype=np.float32))
    check(z, (rng.standard_normal(E) * 0.3).astype(np.float32), K, 1 if T < 3 else 5, seed=E)


@pytest.mark.parametrize("E", [8, 64, 256, 1024])
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 6, 7, 8, 15, 16, 31])
def test_list_lengths(E, K):
    if K >= E:
        pytest.skip("K < E")
    rng = np.random.default_rng(K)
    for T in (70, 2100, 32 * E + 40):
        z = brute.bf16_bits_from_f32(rng.standard_normal((T, E), dtype=np.float32))
        check(z, (rng.standard_normal(E) * 0.3).astype(np.float32), K, 3, seed=K)


@pytest.mark.parametrize("E,K", [(24, 4), (72, 8), (128, 8), (264, 12), (512, 8), (1024, 15)])
@pytest.mark.parametrize("kind", ["constant", "two values", "zeros"])
def test_equal_scores(E, K, kind):
    rng = np.random.default_rng(E)
    for T in (9, 32 * E + 3):
        z = np.full((T, E), 1.5, np.float32)
        if kind == "two values":
            z = np.where(rng.random((T, E)) < 0.5, np.float32(0.25), np.float32(-0.75))
        if kind == "zeros":  # -0 and +0 are equal scores
            z = np.where(rng.random((T, E)) < 0.5, np.float32(0.0), np.float32(-0.0))
        b = np.where(np.arange(E) % 3 == 0, np.float32(-0.0), np.float32(0.0)).astype(np.float32)
        check(brute.bf16_bits_from_f32(z), b, K, 2, seed=E)


@pytest.mark.parametrize("E,K", [(8, 7), (24, 15), (136, 15), (200, 4)])
@pytest.mark.parametrize("pattern", [0xff800001, 0x7f800001, 0xffffffff])
def test_nan_bias_of_a_padded_row(E, K, pattern):
    """A NaN bias whose payload lies in the bits that bf16 drops, on a row
    padded to a wider kernel, with more list entries than groups of finite
    experts: the call is flagged, and no expert past E is listed or counted
    (tokens of the last microbatch inside a tile of the one before)."""
    T = 32 * E + 70
    rng = np.random.default_rng(E)
    z = brute.bf16_bits_from_f32(rng.standard_normal((T, E), dtype=np.float32))
    z[:, K // 2 + 1:E - 1] = 0xff80  # -inf: no more than K finite scores
    b = np.zeros(E, np.float32)
    b.view(np.uint32)[E - 1] = pattern
    off = torch.tensor([0, T - 45, T - 13, T], device="cuda")
    idx, tau, loads = Guarded((T, K), torch.int32, fill=-7), Guarded((T,), torch.float32), Guarded((3, E), torch.int32)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    eqb.eqb_route_topk(to_dev_bf16(z), torch.from_numpy(b).cuda(), K, off, idx.view, tau.view, loads.view, err_flag=err)
    torch.cuda.synchronize()
    assert err.item() == 4  # EQB_ERR_NONFINITE
    assert idx.intact() and tau.intact() and loads.intact()
    assert int(idx.view.min()) >= 0 and int(idx.view.max()) < E
    assert torch.equal(loads.view.sum(dim=1).cpu(), K * (off[1:] - off[:-1]).cpu().to(torch.int32))


def check_flagged(idx, tau, err, E, nan_rows, idx_ref, tau_ref):
    """A call with NaN scores: flagged, every output written and every index
    in range, distinct in its row; the other rows as the oracle has them."""
    idx, tau = idx.cpu().numpy(), tau.cpu().numpy()
    assert err.item() == 4  # EQB_ERR_NONFINITE
    assert idx.min() >= 0 and idx.max() < E and not (tau == -7).any()
    assert all(len(set(row)) == len(row) for row in idx)
    assert np.array_equal(idx[~nan_rows], idx_ref[~nan_rows])
    assert np.array_equal(bits_f32(tau[~nan_rows]), bits_f32(tau_ref[~nan_rows]))


@pytest.mark.parametrize("E", [256, 512, 1000])
def test_nan_scores_of_a_warp(E):
    T, K = 500, 8
    rng = np.random.default_rng(E)
    z = brute.bf16_bits_from_f32(rng.standard_normal((T, E), dtype=np.float32))
    b = (rng.standard_normal(E) * 0.3).astype(np.float32)
    idx_ref, tau_ref, _ = oracle.route(z, b, K)
    nan_rows = np.arange(T) % 3 == 0
    for t in np.flatnonzero(nan_rows):  # one, two or many NaN
        z[t, rng.choice(E, [1, 2, 20][t // 3 % 3], replace=False)] = [0x7fc0, 0xffc1][t % 2]
    idx, tau = Guarded((T, K), torch.int32, fill=-7), Guarded((T,), torch.float32, fill=-7.0)
    loads, err = Guarded((2, E), torch.int32), torch.zeros(1, dtype=torch.int32, device="cuda")
    off = torch.tensor([0, 200, T], device="cuda")
    eqb.eqb_route_topk(to_dev_bf16(z), torch.from_numpy(b).cuda(), K, off, idx.view, tau.view, loads.view, err_flag=err)
    torch.cuda.synchronize()
    assert idx.intact() and tau.intact() and loads.intact()
    check_flagged(idx.view, tau.view, err, E, nan_rows, idx_ref, tau_ref)
    assert torch.equal(loads.view.sum(dim=1).cpu(), torch.tensor([200 * K, (T - 200) * K], dtype=torch.int32))


@pytest.mark.parametrize("E", [64, 128])
@pytest.mark.parametrize("n", [1, 2])
def test_nan_scores_of_the_split_projection(E, n):
    T, d, K = 200, 1024, 8
    x, W = torch.randn((T, d), device="cuda").to(torch.bfloat16), torch.randn((E, d), device="cuda").to(torch.bfloat16)
    W[5:5 + n] = float("nan")  # n experts of every token
    idx, tau = Guarded((T, K), torch.int32, fill=-7), Guarded((T,), torch.float32, fill=-7.0)
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    eqb.eqb_router_route(x, W, torch.zeros(E, device="cuda"), K, topk_idx=idx.view, tau=tau.view, err_flag=err)
    torch.cuda.synchronize()
    assert idx.intact() and tau.intact()
    check_flagged(idx.view, tau.view, err, E, np.ones(T, bool), idx.view.cpu().numpy(), tau.view.cpu().numpy())


def test_microbatches_of_a_warp():
    """More boundaries than a warp loads at once (two and three rounds of
    loads), many of them equal, and enough tokens of a wide row for the loads to be counted by segments."""
    E, K = 520, 4
    for T, M in ((700, 200), (1500, 1104), (1500, 9000), (130000, 90)):
        rng = np.random.default_rng(M)
        z = brute.bf16_bits_from_f32(rng.standard_normal((T, E), dtype=np.float32))
        b = (rng.standard_normal(E) * 0.3).astype(np.float32)
        off = np.sort(np.concatenate([[0] * 40, rng.integers(0, T, M - 79), [T] * 40])).astype(np.int64)
        _, _, ref = oracle.route(z, b, K, off)
        loads = torch.zeros((len(off) - 1, E), dtype=torch.int32, device="cuda")
        eqb.eqb_route_topk(to_dev_bf16(z), torch.from_numpy(b).cuda(), K, torch.from_numpy(off).cuda(), None, None,
                           loads)
        torch.cuda.synchronize()
        assert np.array_equal(loads.cpu().numpy(), ref)
