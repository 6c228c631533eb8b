"""Resident tables in byte planes against the same plaintexts regenerated at
evaluation (64-bit words, another kernel): equal words, at sizes where every
team of the byte-plane kernel takes many items through its ring of stages.
Whole stages, stages cut short by the code's end and by the two pieces of a
host request, tables that end within a tile, layer ranges that start and end
within one, and batches that share a read."""
import numpy as np
import pytest

from gpu_helpers import to_dev, to_host, torch_cuda

pytestmark = pytest.mark.gpu

ALL = 0xFFFFFFFF
REGENERATED = (1 << 64) - 1


def _contexts(N, bits, ell, mu, resident):
    import paper_2310_14565_gb300 as pepsi
    from paper_2310_14565_gb300.workload import make_sets

    npl = max(4, (max(bits) + 7) // 8)
    layer_bytes = (ell + 15) // 16 * 16 * len(bits) * N * npl
    kw = dict(N=N, prime_bits=bits, h=2, lambda_bar=12, mu=mu, ell=ell, hash_key=5, rescale_group=ALL)
    planes = pepsi.Context(resident_bytes=resident * layer_bytes, **kw)
    words = pepsi.Context(resident_bytes=REGENERATED, **kw)
    n = mu * N // 6  # half the table's layers on average
    sets = make_sets(min(N // 2, n), n, 10, bits=64)
    return planes, planes.server_load(sets.server), words, words.server_load(sets.server), sets


@pytest.mark.parametrize("N,bits,ell,mu,resident,passes", [
    (16384, [55] * 6 + [54] * 2, 128, 627, 607, 3),  # host pieces of 1 and 7 steps, 15 layers in the last tile
    (8192, [55, 55, 54, 54], 600, 70, 67, 2),        # long code: last stage of 2 steps
    (8192, [55, 54], 96, 333, 333, 2),               # 6 steps: a whole stage and a short one
    (4096, [36, 36, 37], 130, 200, 150, 2),          # 5 planes, 9 steps
    (8192, [58, 57], 144, 100, 85, 2),               # 8 planes
])
def test_plane_words_equal_regenerated_words(N, bits, ell, mu, resident, passes):
    torch = torch_cuda()
    planes, sp, words, sw, sets = _contexts(N, bits, ell, mu, resident)
    host, _ = planes.query(sets.client, 4)
    dev = to_dev(host)
    want, _ = words.eval_layers(sw, dev, 0, mu, want_e=False)
    for _ in range(passes):
        for req in (host, dev):
            assert np.array_equal(planes.eval_layers(sp, req, 0, mu, want_e=False)[0], want)
    for l0, nl in ((5, 30), (resident - 3, 3), (17, 1)):
        assert np.array_equal(planes.eval_layers(sp, dev, l0, nl, want_e=False)[0], want[l0:l0 + nl])
    del want
    # whole evaluations: one by one, and in batches that share the table's reads
    reqs = [dev] + [to_dev(planes.query(sets.client[::-1], 10 + i)[0]) for i in range(3)]
    one = [words.eval(sw, r) for r in reqs]
    assert np.array_equal(planes.eval(sp, host), one[0])
    planes.set_schedule(batch_requests=4)
    for q in (2, 3, 4):
        outs = [torch.zeros(one[0].size, dtype=torch.int64, device="cuda") for _ in range(q)]
        planes.eval_batch([sp] * q, reqs[:q], outs=outs)
        torch.cuda.synchronize()
        for i in range(q):
            assert np.array_equal(to_host(outs[i]).reshape(one[i].shape), one[i]), (q, i)
    assert planes.wait_probe(1) == 0  # no bounded wait expired
