"""The autotuner compares the default threads per transform block with half and
twice as many: a count it settles on is never the default again (that is 0) nor
one it should not have tried."""
import pytest

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,bits,default", [(4096, [36, 36, 37], 256), (8192, [55, 55, 54, 54], 512),
                                            (16384, [55] * 6 + [54] * 2, 1024)])
def test_autotuned_threads(N, bits, default):
    torch = torch_cuda()
    import paper_2310_14565_gb300 as pepsi
    from paper_2310_14565_gb300.workload import make_sets

    sets = make_sets(200, 3000, 20, bits=64)
    gc = pepsi.Context(N=N, prime_bits=bits, h=2, lambda_bar=16, mu=33)
    sid = gc.server_load(sets.server)
    cts = torch.empty((gc.ell, 2, gc.k, N), dtype=torch.int64, device="cuda")
    gc.query(sets.client, 4, out=cts)
    for _ in range(4):
        gc.autotune(sid, cts)
        assert gc.schedule()["ntt_threads"] in {0, default // 2, min(1024, 2 * default)} - {default}
