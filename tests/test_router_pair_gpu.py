"""GPU parity of the router projection by pairs of SMs (224 or 256 experts): on
integer-valued inputs, whose sums are exact in fp32 in any order, z equals
the rounded exact product bit for bit.  T lies at the edges of the 256-token
pairs (a second tile that is full, empty, of one row) and past one and two
rounds of the persistent pairs; d fills the ring of stages unevenly."""
import pytest
import torch

import paper_2609_28053_gb300 as eqb
from gpu_harness import Guarded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ok):
    eqb.load()


@pytest.mark.parametrize("T", [16384, 16385, 16513, 19457, 40000])
@pytest.mark.parametrize("d,E", [(2048, 224), (3072, 224), (2112, 256), (4096, 256)])
def test_logits(T, d, E):
    g = torch.Generator(device="cuda").manual_seed(T + E)
    x = torch.randint(-8, 9, (T, d), generator=g, device="cuda").to(torch.bfloat16)
    W = torch.randint(-4, 5, (E, d), generator=g, device="cuda").to(torch.bfloat16)
    z_ref = (x.double() @ W.double().t()).to(torch.float32).to(torch.bfloat16)
    z, err = Guarded((T, E), torch.bfloat16), torch.zeros(1, dtype=torch.int32, device="cuda")
    eqb.eqb_router_logits(x, W, z=z.view, err_flag=err)
    torch.cuda.synchronize()
    assert z.intact() and err.item() == 0
    assert torch.equal(z.view.view(torch.int16), z_ref.view(torch.int16))


@pytest.mark.parametrize("d,E", [(3072, 224), (2112, 256), (4096, 256)])
def test_logits_equal_the_one_sm_kernel(d, E):
    """On inputs whose sums depend on their order: parts of fewer than 16,384
    tokens (and more than the split projection takes) go through the one-SM
    kernel, and the pairs give the same bits."""
    T, part = 26000, 13000
    g = torch.Generator(device="cuda").manual_seed(E)
    x = torch.randn((T, d), generator=g, device="cuda").to(torch.bfloat16)
    W = torch.randn((E, d), generator=g, device="cuda").to(torch.bfloat16)
    z = eqb.eqb_router_logits(x, W)
    parts = [eqb.eqb_router_logits(x[t:t + part], W) for t in (0, part)]
    assert torch.equal(z.view(torch.int16), torch.cat(parts).view(torch.int16))
