"""The multiply-accumulate on byte planes (resident tables): the exactness of
its sums, and its words at the edges of its tiles (16 layers), steps (16 code
bits), runs between moves to the integer sums (128 code bits) and plane counts
(4 to 8 bytes per word)."""
import numpy as np
import pytest


def test_byte_products_are_exact_in_f32_from_the_bias():
    """Bytes read as f16 subnormals are byte * 2^-24; 128 products of two
    bytes on top of 2^23 units of 2^-48 stay below 2^24 units, where f32 holds
    every integer; 65535 products of two bytes fit 32 bits."""
    b = np.arange(256, dtype=np.uint16)
    assert np.array_equal(b.view(np.float16).astype(np.float64), b * 2.0 ** -24)
    assert (1 << 23) + 128 * 255 * 255 < 1 << 24
    assert 65535 * 255 * 255 < 1 << 32
    acc = np.float32(2.0 ** -25)  # 2^23 units
    want = 0
    rng = np.random.default_rng(7)
    for a, c in [(255, 255)] * 96 + [tuple(rng.integers(0, 256, 2)) for _ in range(32)]:
        x, y = np.uint16(a).view(np.float16), np.uint16(c).view(np.float16)
        acc = np.float32(acc + np.float32(x) * np.float32(y))
        want += int(a) * int(c)
    assert int(acc.view(np.uint32)) - 0x33000000 == want


@pytest.mark.gpu
@pytest.mark.parametrize("bits,ell,mu", [
    ([30, 31], 16, 17),        # tables kept in words
    ([36, 36, 37], 17, 16),
    ([36, 36, 37], 32, 16),
    ([30, 31], 32, 17),        # 4 planes, two steps, one layer beyond a tile
    ([36, 36, 37], 42, 16),    # the last length of 5 planes in words and the first in planes
    ([36, 36, 37], 43, 33),
    ([55, 54], 79, 16),        # the same with 7 planes
    ([55, 54], 80, 17),
    ([45, 46], 129, 15),       # 6 planes, one bit beyond the run of 128
    ([55, 54], 128, 33),       # 7 planes, whole runs
    ([55, 54], 300, 18),
    ([60, 60], 127, 16),       # words
    ([58, 57], 144, 16),       # 8 planes
    ([59], 257, 9),
])
def test_planes_match_the_oracle(bits, ell, mu):
    from gpu_helpers import to_dev, to_host, torch_cuda
    from test_gpu_parity import _psi_case

    torch = torch_cuda()
    oc, gc, s, rlk, sets, Ts, cts, where, sid = _psi_case(64, bits, 2, 6, mu=mu, m=20, n=80, planted=5, ell=ell)
    mu = Ts.shape[0]
    want, dh, de = oc.eval(rlk, cts, Ts, debug=True)
    gh, _ = gc.eval_layers(sid, cts, 0, mu)  # host request: in two pieces from 128 bits on
    assert np.array_equal(gh, dh)
    dev = to_dev(cts)
    for l0, nl in ((0, 1), (mu - 1, 1), (mu // 2, mu - mu // 2), (3, min(15, mu - 3))):  # parts of tiles
        assert np.array_equal(gc.eval_layers(sid, dev, l0, nl)[0], dh[l0:l0 + nl]), (l0, nl)
    P = gc.server_plaintexts(sid, mu - 2, 2)
    assert np.array_equal(P[1, ell - 1], oc.server_plaintext(Ts, mu - 1, ell - 1))
    other = oc.query(s, sets.client[::-1], 9)[1]
    want2 = oc.eval(rlk, other, Ts)
    gc.set_schedule(batch_requests=4)
    for n in (2, 3, 4):  # requests sharing one read of the table
        outs = gc.eval_batch([sid] * n, [cts, other, cts, other][:n])
        for q in range(n):
            assert np.array_equal(outs[q], (want, want2)[q & 1]), (n, q)
