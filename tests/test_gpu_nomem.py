"""A device allocation that fails inside a call is reported by that call
(PEPSI_E_NOMEM), and the context works again once there is memory: the
relinearisation digits, the last scratch a relinearisation or an evaluation
allocates, do not fit while a test buffer holds the rest of the memory."""
import numpy as np
import pytest

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _hold(torch, leave):
    """A buffer that leaves about `leave` bytes of device memory."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(max(0, free - leave), dtype=torch.uint8, device="cuda")


def test_relin_without_room_for_the_digits():
    torch = torch_cuda()
    import paper_2310_14565_gb300 as pepsi

    n, k, N = 512, 8, 16384
    gc = pepsi.Context(N=N, prime_bits=[55] * 6 + [54] * 2, h=2, lambda_bar=12, ell=128)
    ct3 = torch.stack([torch.randint(0, gc.q[i], (n, 3, N), dtype=torch.int64, device="cuda") for i in range(k)], 2)
    ct3 = ct3.contiguous()
    out = torch.zeros((n, 2, k, N), dtype=torch.int64, device="cuda")
    result = out.numel() * 8  # the result rows (1.1 GB) fit beside the buffer, the digits (5.4 GB) do not
    held = _hold(torch, result + (2 << 30))
    with pytest.raises(pepsi.PepsiError) as e:
        gc.relin(ct3, n, out)
    assert e.value.code == pepsi.E_NOMEM
    del held
    torch.cuda.empty_cache()
    gc.relin(ct3, n, out)
    few = torch.zeros((1, 2, k, N), dtype=torch.int64, device="cuda")
    gc.relin_noalloc(ct3[-1:], 1, few)
    torch.cuda.synchronize()
    assert torch.equal(out[-1:], few)


@pytest.mark.parametrize("fused", [1, 0])
def test_evaluation_without_room_for_the_digits(fused):
    torch = torch_cuda()
    import paper_2310_14565_gb300 as pepsi
    from paper_2310_14565_gb300.workload import make_sets

    N, k, chunk = 8192, 4, 64
    sets = make_sets(256, 1 << 15, 20, bits=64)

    def load():
        c = pepsi.Context(N=N, prime_bits=[55, 55, 54, 54], h=4, lambda_bar=16, mu=chunk)
        c.set_schedule(relin_fused=fused)
        return c, c.server_load(sets.server)

    first, s0 = load()
    request, _ = first.query(sets.client, 4)
    torch.cuda.synchronize()
    before, _ = torch.cuda.mem_get_info()
    want = first.eval(s0, request)
    scratch = before - torch.cuda.mem_get_info()[0]  # what one evaluation allocates
    digits = (k + 2) * k * N * 8 * chunk             # the relinearisation digits, allocated last (100 MB)
    gc, sid = load()
    held = _hold(torch, scratch - digits // 2)
    with pytest.raises(pepsi.PepsiError) as e:
        gc.eval(sid, request)
    assert e.value.code == pepsi.E_NOMEM
    del held
    torch.cuda.empty_cache()
    assert np.array_equal(gc.eval(sid, request), want)
