"""GPU parity of calls made from two host threads at once, each on its own
stream with its own shape: the kernels' launch settings are shared by all
threads, so neither shape's may depend on the other's call."""
import threading

import pytest
import torch

import paper_2609_28053_gb300 as eqb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(cuda_ok):
    eqb.load()


def step(T, E, K):
    """The one-call step of one batch: a call to repeat, and its outputs."""
    g = torch.Generator(device="cuda").manual_seed(T + E)
    z = torch.randn((T, E), generator=g, device="cuda").to(torch.bfloat16)
    b, off = torch.zeros(E, device="cuda"), torch.tensor([0, T // 3, T], device="cuda")
    out = [torch.zeros((T, K), dtype=torch.int32, device="cuda"), torch.zeros(T, device="cuda"),
           torch.zeros((2, E), dtype=torch.int32, device="cuda"), torch.zeros(E, device="cuda")]
    ws = torch.zeros(eqb.eqb_layer_workspace_bytes(E), dtype=torch.uint8, device="cuda")
    return out, lambda: eqb.eqb_layer_step(z, b, K, off, out[2], out[3], ws, tau=out[1], topk_idx=out[0])


def logits(T, d, E):
    g = torch.Generator(device="cuda").manual_seed(T + E)
    x = torch.randn((T, d), generator=g, device="cuda").to(torch.bfloat16)
    W = torch.randn((E, d), generator=g, device="cuda").to(torch.bfloat16)
    out = [torch.zeros((T, E), dtype=torch.bfloat16, device="cuda")]
    return out, lambda: eqb.eqb_router_logits(x, W, z=out[0])


def route(T, E, K):
    g = torch.Generator(device="cuda").manual_seed(T + E)
    z = torch.randn((T, E), generator=g, device="cuda").to(torch.bfloat16)
    b = torch.zeros(E, device="cuda")
    out = [torch.zeros((T, K), dtype=torch.int32, device="cuda"), torch.zeros(T, device="cuda")]
    return out, lambda: eqb.eqb_route_topk(z, b, K, None, out[0], out[1])


def maxvio(M, E):
    loads = torch.randint(0, 99, (M, E), dtype=torch.int32, device="cuda")
    off = torch.arange(M + 1, device="cuda") * 7
    out = [torch.zeros(2, dtype=torch.float64, device="cuda")]
    return out, lambda: eqb.eqb_maxvio(loads, off, 1, out=out[0])


@pytest.mark.parametrize("T,d,E", [(100, 1024, 64), (100, 512, 64), (16384, 2048, 256)])
def test_first_call_of_a_thread(T, d, E):
    """A projection as the first CUDA work of a thread: the context is not
    current there yet when the call prepares its tensor maps."""
    out, f = logits(T, d, E)
    f()
    torch.cuda.synchronize()
    ref, failed = out[0].clone(), []

    def work():
        try:
            f()
        except Exception as e:
            failed.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    assert torch.equal(out[0], ref)


@pytest.mark.parametrize("make,small,large", [
    (step, (9000, 256, 8), (120000, 256, 8)),         # tiles of routing, tiles of bins
    (step, (3000, 64, 8), (120000, 64, 8)),
    (logits, (100, 1024, 16), (100, 4096, 256)),      # the split projection's stages
    (logits, (100, 512, 16), (100, 512, 256)),        # the one-SM projection's
    (logits, (16384, 3072, 224), (16384, 3072, 256)),
    (route, (300, 32, 20), (300, 256, 20)),           # long lists
    (maxvio, (6200, 8), (16384, 8))])
def test_two_shapes_from_two_threads(make, small, large):
    calls = [make(*small), make(*large)]
    refs = []
    for out, f in calls:
        f()
        torch.cuda.synchronize()
        refs.append([t.clone() for t in out])
        for t in out:
            t.zero_()
    torch.cuda.synchronize()
    failed = []

    def work(f):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(1500):
                    f()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # an EqbError of a refused launch
            failed.append(e)

    threads = [threading.Thread(target=work, args=(f,)) for _, f in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for (out, _), ref in zip(calls, refs):
        assert all(torch.equal(x, y) for x, y in zip(out, ref))
