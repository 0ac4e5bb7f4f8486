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
@pytest.mark.parametrize("d,E", [(2048, 224), (2112, 256), (4096, 256)])
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
