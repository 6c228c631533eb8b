"""Products modulo q = 2^n - d by folding (transforms of the primes just below
a power of two, n = 40..57): their bounds with Python integers, and the
transforms' words at every fused ring size and block size."""
import random

import numpy as np
import pytest


def _prime(bits, N, skip):
    from test_arith_bounds import is_prime

    q = (1 << bits) - ((1 << bits) - 1) % (2 * N)
    while True:
        if q < 1 << bits and is_prime(q):
            if skip == 0:
                return q
            skip -= 1
        q -= 2 * N


def _mul(x, w, q, n, s):
    """The device's product, with the width of every intermediate checked."""
    d, v = (1 << n) - q, (w << s) % q
    lo, m32 = (1 << s) - 1, (1 << 32) - 1
    x0, x1 = x & lo, x >> s
    assert x1 <= m32
    L = x0 * (w & m32) + x1 * (v & m32)
    assert L < 1 << 64
    M = x0 * (w >> 32) + x1 * (v >> 32) + (L >> 32)
    assert M < 1 << 64 and M >> (n - 32) <= m32
    r = (M >> (n - 32)) * d + ((M & ((1 << (n - 32)) - 1)) << 32 | L & m32)
    assert r < 2 * q and r % q == x * w % q
    return r


@pytest.mark.parametrize("n", [40, 41, 48, 51, 54, 55, 56, 57])
@pytest.mark.parametrize("N,skip", [(4096, 0), (16384, 5)])
def test_bounds(n, N, skip):
    q = _prime(n, N, skip)
    d, s = (1 << n) - q, (n + 6) // 2
    if not (d < 1 << 27 and (d << (s + 1)) + 2 * d < 1 << n):
        pytest.skip("the library keeps Shoup products for this prime")
    rng = random.Random(n * N)
    top = (1 << (n + 5)) - 1
    for w in [0, 1, q - 1, q // 2, (1 << (n - 1)) - 1] + [rng.randrange(q) for _ in range(50)]:
        for x in [0, 1, q, 32 * q - 1, top, (1 << s) - 1, top - ((1 << s) - 1)] + [rng.randrange(top + 1) for _ in range(20)]:
            _mul(x, w, q, n, s)
    for x in (0, q - 1, 32 * q - 1, top):  # the fold of a grown value
        h = x >> n
        assert h * d < 1 << 32 and (x & ((1 << n) - 1)) + h * d < 2 * q
    assert 32 * q <= top + 1  # (4 + 2 log2 N) q at N = 16384, and three doublings of 4 q


@pytest.mark.gpu
@pytest.mark.parametrize("N", [1024, 4096, 8192, 16384])
@pytest.mark.parametrize("bits", [[57, 40], [55, 54], [41, 58, 60]])
def test_transforms_at_every_block_size(N, bits):
    import oracle
    from gpu_helpers import pair, to_dev, to_host, torch_cuda

    torch_cuda()
    oc, gc, _, _ = pair(N, bits, 2, 8, mu=1)
    rng = np.random.default_rng(N)
    x = np.stack([np.stack([rng.integers(0, q, N, dtype=np.uint64) for q in oc.q]) for _ in range(2)])
    x[0, :, :] = np.array(oc.q, dtype=np.uint64)[:, None] - 1
    want = np.stack([np.stack([oracle.ntt_fwd(x[c, p], N, oc.q[p], oc.psi[p]) for p in range(len(bits))])
                     for c in range(2)])
    for nt in (0, 64, 128, 256, 512, 1024):
        gc.set_schedule(ntt_threads=nt)
        d = to_dev(x)
        gc.ntt(d, 2)
        assert np.array_equal(to_host(d).reshape(x.shape), want), nt
        gc.ntt(d, 2, inverse=True)
        assert np.array_equal(to_host(d).reshape(x.shape), x), nt
