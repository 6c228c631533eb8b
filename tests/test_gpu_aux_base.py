"""The auxiliary base of the exact products: how many primes a context takes, and the
words of the conversions at the largest counts in use."""
import numpy as np
import pytest

from gpu_helpers import T, torch_cuda

pytestmark = pytest.mark.gpu

ALL = 0xFFFFFFFF


@pytest.mark.parametrize("kw,kb", [
    # 57-bit primes where as few of them do as of 61 bits, or one more where the conversions fold with them
    (dict(N=4096, prime_bits=[36, 36, 37], h=2, lambda_bar=16), 3),
    (dict(N=8192, prime_bits=[55, 55, 54, 54], h=4, lambda_bar=32, ell=600, mu=526, rescale_group=ALL), 5),
    (dict(N=8192, prime_bits=[55, 55, 54, 54], h=4, lambda_bar=32, ell=600, mu=526, rescale_group=ALL,
          server_values=1), 6),
    (dict(N=16384, prime_bits=[55] * 6 + [54] * 2, h=8, lambda_bar=40, ell=128, mu=3487, rescale_group=ALL), 9),
    # primes whose conversions do not fold: no prime more than the bound asks for
    (dict(N=16384, prime_bits=[50] * 5, h=4, lambda_bar=32, mu=100, rescale_group=ALL), 5),
    (dict(N=4096, prime_bits=[36, 36, 37], h=2, lambda_bar=16, mu=20, rescale_group=ALL, server_values=1), 3),
])
def test_auxiliary_primes(kw, kb):
    torch_cuda()
    import paper_2310_14565_gb300 as pepsi

    gc = pepsi.Context(**kw)
    assert gc.kb == kb
    gc.close()


def test_ten_auxiliary_primes_match_oracle():
    """Eight 56-bit primes, values, runs of up to 40000 layers: ten auxiliary
    primes, the conversions' largest instantiated form.  Labels and masked sum
    against the oracle word for word."""
    torch_cuda()
    import oracle
    import paper_2310_14565_gb300 as pepsi
    from paper_2310_14565_gb300.workload import make_sets

    N, bits, h, lb, mu = 256, [56] * 8, 4, 10, 8
    sets = make_sets(20, 70, 5, bits=32)
    values = np.arange(1, 71, dtype=np.uint32)
    oc = oracle.Ctx(N=N, t=T, prime_bits=bits, h=h, lambda_bar=lb, mu=mu, hash_key=0x5EED)
    gc = pepsi.Context(N=N, t=T, prime_bits=bits, h=h, lambda_bar=lb, mu=mu, hash_key=0x5EED, key_seed=3,
                       rescale_group=40000, server_values=1)
    assert gc.kb == 10
    s, rlk = oc.keygen(3)
    rc, Ts, V, _ = oc.server_table_values(sets.server, values)
    assert rc == 0
    sid = gc.server_load_values(sets.server, values)
    cts, _ = gc.query(sets.client, 4)
    for mode in (2, 3):
        want = oc.eval(rlk, cts, Ts, mode=mode, mask_seed=7, V=V, group=mu)
        assert np.array_equal(gc.eval(sid, cts, mode=mode, mask_seed=7), want), mode
    assert np.array_equal(gc.eval(sid, cts), oc.eval(rlk, cts, Ts, group=mu))
