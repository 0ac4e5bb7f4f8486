"""GPU parity of the router projection for few tokens, where a cluster of 2, 4
or 8 blocks shares each 128-token tile: on integer-valued inputs (every sum is
exact in fp32, in any order) z equals the rounded exact product bit for bit,
and the routed outputs equal routing those logits; T lies on both sides of the
lines between cluster sizes."""
import numpy as np
import pytest
import torch

import paper_2609_28053_gb300 as eqb
from eqb_workloads import ragged_offsets
from gpu_harness import Guarded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ok):
    eqb.load()


def inputs(T, d, E, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randint(-8, 9, (T, d), generator=g, device="cuda").to(torch.bfloat16)
    W = torch.randint(-4, 5, (E, d), generator=g, device="cuda").to(torch.bfloat16)
    z = (x.double() @ W.double().t()).to(torch.float32).to(torch.bfloat16)  # |sums| < 2^17: exact in fp32
    return x, W, z


@pytest.mark.parametrize("T", [1, 8, 127, 129, 1024, 1025, 1153, 4096, 4225, 8192, 8449])
@pytest.mark.parametrize("d,E,M", [(1024, 128, 5), (4096, 64, 5), (1088, 64, 100)])
def test_route(T, d, E, M):
    """Few microbatches, where a tile's loads are counted together, and more than
    a tile has tokens of one."""
    K, M = (8, M) if T > 8 else (3, 1)
    x, W, z_ref = inputs(T, d, E, seed=T + E)
    b = torch.randn(E, device="cuda") * 30.0
    off = torch.from_numpy(ragged_offsets(T, M, seed=T) if M > 1 else np.array([0, T], np.int64)).cuda()
    z, idx, tau, loads = (Guarded((T, E), torch.bfloat16), Guarded((T, K), torch.int32), Guarded((T,), torch.float32),
                          Guarded((M, E), torch.int32))
    hist, err = Guarded((E, 256), torch.int32), torch.zeros(1, dtype=torch.int32, device="cuda")
    eqb.eqb_router_route(x, W, b, K, off, z=z.view, topk_idx=idx.view, tau=tau.view, loads=loads.view, err_flag=err,
                         hist_hi=hist.view)
    idx2, tau2 = torch.empty((T, K), dtype=torch.int32, device="cuda"), torch.empty(T, device="cuda")
    loads2, hist2 = torch.zeros((M, E), dtype=torch.int32, device="cuda"), torch.zeros((E, 256), dtype=torch.int32,
                                                                                     device="cuda")
    eqb.eqb_route_topk(z_ref, b, K, off, idx2, tau2, loads2, hist_hi=hist2)
    torch.cuda.synchronize()
    assert all(g.intact() for g in (z, idx, tau, loads, hist)) and err.item() == 0
    assert torch.equal(z.view.view(torch.int16), z_ref.view(torch.int16))
    assert torch.equal(idx.view, idx2) and torch.equal(tau.view, tau2)
    assert torch.equal(loads.view, loads2) and torch.equal(hist.view, hist2)


@pytest.mark.parametrize("E", [64, 128])
@pytest.mark.parametrize("kind", ["constant", "two values", "zeros"])
def test_equal_scores(E, kind):
    """More candidates than a warp lists: scores from the bias alone, all equal,
    of two values, or zeros of both signs (equal scores)."""
    T, d, K = 300, 1024, 8
    x, W = torch.zeros((T, d), dtype=torch.bfloat16, device="cuda"), torch.ones((E, d), dtype=torch.bfloat16, device="cuda")
    odd = torch.arange(E, device="cuda") % 3 == 0
    b = {"constant": torch.full((E,), 1.5), "two values": torch.where(odd.cpu(), 0.25, -0.75),
         "zeros": torch.where(odd.cpu(), -0.0, 0.0)}[kind].cuda()
    z, idx, tau = eqb.eqb_router_route(x, W, b, K, topk_idx=torch.full((T, K), -7, dtype=torch.int32, device="cuda"))
    idx2, tau2 = eqb.eqb_route_topk(z, b, K, topk_idx=torch.empty_like(idx))
    assert torch.equal(idx, idx2) and torch.equal(tau, tau2)
    best = torch.sort(b, descending=True, stable=True).indices[:K].to(torch.int32)  # ties to the lower index
    assert torch.equal(idx, best.expand(T, K))


@pytest.mark.parametrize("E,d", [(64, 1024), (64, 3008), (64, 3072), (128, 1472), (128, 1536)])
@pytest.mark.parametrize("T", [100, 3000, 6000, 9000])
def test_logits_do_not_depend_on_routing(T, d, E):
    """On inputs whose sums depend on their order, the logits of the call that
    routes are those of the call that does not, bit for bit."""
    x, W = (torch.randn(s, device="cuda").to(torch.bfloat16) for s in ((T, d), (E, d)))
    z, _, _ = eqb.eqb_router_route(x, W, torch.zeros(E, device="cuda"), 8)
    assert torch.equal(z.view(torch.int16), eqb.eqb_router_logits(x, W).view(torch.int16))


@pytest.mark.parametrize("T,d,E", [(5, 1024, 16), (300, 1088, 48), (130, 2048, 240), (1100, 1024, 256), (4300, 1600, 256),
                                   (4300, 1024, 144)])
def test_logits(T, d, E):
    """Expert counts that fill no whole run of lanes, columns that the blocks
    of a cluster share unevenly."""
    x, W, z_ref = inputs(T, d, E, seed=T)
    z, err = Guarded((T, E), torch.bfloat16), torch.zeros(1, dtype=torch.int32, device="cuda")
    eqb.eqb_router_logits(x, W, z=z.view, err_flag=err)
    torch.cuda.synchronize()
    assert z.intact() and err.item() == 0
    assert torch.equal(z.view.view(torch.int16), z_ref.view(torch.int16))
