"""The auxiliary base of the exact products: how many primes a context takes."""
import pytest

from gpu_helpers import torch_cuda

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
