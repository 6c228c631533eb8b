"""The form of a resident table (64-bit words or byte planes) follows the
budget: where the faster form does not hold every layer but the smaller one does,
no layer is regenerated; a caller that asks for seven bytes gets the smaller
form throughout.  The words are those of a wholly regenerated table."""
import numpy as np
import pytest

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,ell,plaintext_bytes,bytes_per_point", [
    ([55, 54], 61, 0, 64 * 7),      # faster as words (61 * 8), smaller in planes
    ([55, 54], 61, 7, 64 * 7),
    ([58, 58], 250, 0, 250 * 8),    # faster in planes (256 * 8), smaller as words
    ([36, 37], 34, 7, 48 * 5),      # faster as words (34 * 8), smaller in planes
    ([55, 54], 24, 7, 24 * 8),      # two steps in planes (32 * 7) are more than the words
])
def test_every_layer_is_resident_where_either_form_holds_it(bits, ell, plaintext_bytes, bytes_per_point):
    torch_cuda()
    import paper_2310_14565_gb300 as pepsi
    from paper_2310_14565_gb300.workload import make_sets

    N, mu = 4096, 37
    kw = dict(N=N, prime_bits=bits, h=2, lambda_bar=8, ell=ell, mu=mu, hash_key=5)
    sets = make_sets(300, 20000, 30, bits=64)
    gc = pepsi.Context(resident_bytes=mu * bytes_per_point * len(bits) * N, plaintext_bytes=plaintext_bytes, **kw)
    sid = gc.server_load(sets.server)
    cts, _ = gc.query(sets.client, 4)
    gc.profile(True)
    got = gc.eval(sid, cts)
    assert gc.profile_read()["ptgen"][0] == 0  # no layer regenerated
    gc.profile(False)
    ref = pepsi.Context(resident_bytes=(1 << 64) - 1, **kw)
    assert np.array_equal(got, ref.eval(ref.server_load(sets.server), cts))
    # one byte less: the last layer is regenerated, the words stay
    less = pepsi.Context(resident_bytes=mu * bytes_per_point * len(bits) * N - 1, plaintext_bytes=plaintext_bytes,
                         **kw)
    ls = less.server_load(sets.server)
    less.profile(True)
    assert np.array_equal(less.eval(ls, cts), got)
    assert less.profile_read()["ptgen"][0] == 1
