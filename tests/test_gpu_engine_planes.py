"""Engine lanes, batches and captured evaluations over tables in byte planes,
wholly and partly resident (codes long enough for planes, N = 64): the oracle's
words with one to four requests in flight, as one request alone."""
import math
import os

import numpy as np
import pytest

from gpu_helpers import pair, to_dev, to_host, torch_cuda

pytestmark = pytest.mark.gpu

PAPER = [55, 55, 54, 54]
ALL = 0xFFFFFFFF
ELL, STEPS = 100, 7
LAYER = STEPS * 16 * 7 * len(PAPER) * 64  # bytes of a layer in byte planes


def _case(resident_layers, group=ALL):
    """A context whose set of 13 layers or more keeps `resident_layers` of them."""
    import oracle
    from paper_2310_14565_gb300.workload import make_sets

    torch_cuda()
    sets = make_sets(20, 120, 4, bits=32, seed_items=61, seed_plant=62)
    mu = max(13, oracle.simple_hash(0x5EED, 10, int(math.log2(64)), sets.server, 1000)[2])
    os.environ["PEPSI_CHUNK"] = "4"
    try:
        oc, gc, s, rlk = pair(64, PAPER, 4, 10, mu=mu, ell=ELL, rescale_group=group, response_primes=1,
                              resident_bytes=(resident_layers or mu) * LAYER)
    finally:
        os.environ.pop("PEPSI_CHUNK", None)
    sid = gc.server_load(sets.server)
    _, Ts, _ = oc.server_table(sets.server)
    reqs = [gc.query(sets.client[i::-1] if i else sets.client, 70 + i)[0] for i in range(6)]
    og = mu if group == ALL else 1
    want = [oc.mod_switch(oc.eval(rlk, r, Ts, mode=i & 1, mask_seed=i, group=og), 1) for i, r in enumerate(reqs)]
    return gc, sid, mu, reqs, want


@pytest.mark.parametrize("group", [0, ALL])
@pytest.mark.parametrize("resident", [0, 6])
def test_engine_lanes_over_planes(resident, group):
    import paper_2310_14565_gb300 as pepsi

    gc, sid, mu, reqs, want = _case(resident, group)
    for slots in (1, 2, 3, 4):
        for share in (1, 2, 4):
            gc.set_schedule(batch_requests=share)
            eng = pepsi.Engine([(gc, sid, slots)])
            tk = [eng.submit(0, r, mode=i & 1, mask_seed=i) for i, r in enumerate(reqs)]
            eng.run()
            for i, (t, out) in enumerate(tk):
                eng.wait(t)
                assert np.array_equal(out, want[i]), (slots, share, i)
            # a request's state: its formats, h' of a chunk, the layer sum and the run sum
            kN = gc.k * 64
            chunk = -(-mu // -(-mu // 4))
            words = chunk * 2 * kN + 3 * kN + STEPS * 32 * kN
            if resident:
                words += ELL * 3 * kN
            if group:
                words += 3 * (gc.k + gc.kb) * 64
            peak = eng.stats()["bytes_peak"]  # a finished request's state counts until its last step is seen done
            assert peak % (words * 8) == 0 and peak >= slots * words * 8
            eng.close()


@pytest.mark.parametrize("resident", [0, 6])
def test_engine_graph_over_planes(resident):
    import paper_2310_14565_gb300 as pepsi

    torch = torch_cuda()
    gc, sid, mu, reqs, want = _case(resident)
    gc.set_schedule(batch_requests=4)
    eng = pepsi.Engine([(gc, sid, 3)])
    dev = [to_dev(np.zeros_like(r)) for r in reqs]
    outs = [torch.zeros(2 * 64, dtype=torch.int64, device="cuda") for _ in reqs]
    for i in range(len(reqs)):
        eng.submit(0, dev[i], out=outs[i], mode=i & 1, mask_seed=i)
    graph = eng.capture()
    for _ in range(2):
        for d, r in zip(dev, reqs):
            d.copy_(to_dev(r))
        torch.cuda.synchronize()
        graph.launch()
        for i, o in enumerate(outs):
            assert np.array_equal(to_host(o).reshape(want[i].shape), want[i]), i
            o.zero_()
    graph.close()
    eng.close()


@pytest.mark.parametrize("resident", [0, 6])
def test_batches_and_captured_evaluation_over_planes(resident):
    torch = torch_cuda()
    gc, sid, mu, reqs, want = _case(resident)
    for n in (2, 3, 4, 6):
        gc.set_schedule(batch_requests=min(n, 4))
        outs = gc.eval_batch([sid] * n, reqs[:n], [i & 1 for i in range(n)], list(range(n)))
        for i in range(n):
            assert np.array_equal(outs[i], want[i]), (n, i)
    cts, out = to_dev(reqs[0]), torch.zeros(2 * 64, dtype=torch.int64, device="cuda")
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    gc.eval(sid, cts, out=out, stream=stream)  # creates the scratch
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
        gc.eval(sid, cts, out=out, stream=torch.cuda.current_stream())
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(to_host(out).reshape(want[0].shape), want[0])
