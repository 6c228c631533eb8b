"""Rings below 4096 run the transform kernels without the named barriers of the
larger ones (which would limit their small blocks to a few per SM): many rows at
once, every arithmetic, every block size, against the oracle's products and the
inverse of the transform."""
import numpy as np
import pytest

from gpu_helpers import T, to_dev, to_host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 256, 1024, 2048])
@pytest.mark.parametrize("bits", [[55, 54], [36, 37], [60, 55], [58, 40]])
def test_small_ring_products_match_oracle(N, bits):
    torch = torch_cuda()
    import oracle
    import paper_2310_14565_gb300 as pepsi

    n, k, t = 40, len(bits), T
    oc = oracle.Ctx(N=N, t=t, prime_bits=bits, h=2, lambda_bar=6, mu=4, hash_key=1)
    gc = pepsi.Context(N=N, t=t, prime_bits=bits, h=2, lambda_bar=6, mu=4, hash_key=1, key_seed=3)
    s, rlk = oc.keygen(3)
    rng = np.random.default_rng(N)
    a, b = [np.stack([rng.integers(0, q, (n, 2, N), dtype=np.uint64) for q in gc.q], 2) for _ in range(2)]
    want = np.stack([oc.relin(rlk, oc.ct_mult(a[i], b[i])) for i in (0, n - 1)])
    da, db = to_dev(a), to_dev(b)
    out = torch.zeros((n, 2, k, N), dtype=torch.int64, device="cuda")
    for nt in (0, 64, 256, 1024):
        gc.set_schedule(ntt_threads=nt)
        gc.ct_mult(da, db, n, out, relin=True)
        torch.cuda.synchronize()
        got = to_host(out)
        assert np.array_equal(got[[0, -1]], want), nt
        rows = to_dev(a)
        gc.ntt(rows, 2 * n)
        gc.ntt(rows, 2 * n, inverse=True)
        torch.cuda.synchronize()
        assert np.array_equal(to_host(rows).reshape(a.shape), a), nt
