"""Two host threads update sketches of different shapes at once.  A kernel's largest dynamic shared memory is
state of the whole process: a call that set its own size could find it lowered by the other thread when it
launched, and was refused.  Every kernel whose launches differ in shared memory is taken: the multi-iteration
kernel (keys in device memory), chunk_update_kernel (keys in pinned memory) and the one-at-a-time window
kernel (its Slim)."""
import threading

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

CALLS, N = 1500, 64


@pytest.fixture(scope="module")
def sf():
    import paper_1701_04148_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("what,shapes", [
    ("multi", [(1009, 131_072), (1009, 1 << 20)]),
    ("pinned", [(1009, 131_072), (1009, 1 << 20)]),
    ("window", [(61, 1), (7001, 1)]),
])
def test_calls_of_two_shapes_from_two_threads(sf, what, shapes):
    import torch
    d, z, kb = 4, 4, 4
    r = np.random.RandomState(8)
    host = [torch.from_numpy(r.randint(0, 500, N).astype(np.int32)) for _ in shapes]
    keys = [h.pin_memory() if what == "pinned" else h.cuda() for h in host]
    streams = [torch.cuda.Stream() for _ in shapes]
    torch.cuda.synchronize()
    sk = [sf.Sketch(d, w, z, kb, 5, chunk, stream=s) for (w, chunk), s in zip(shapes, streams)]
    errors = []

    def client(i):
        try:
            torch.cuda.set_device(0)
            for _ in range(CALLS):
                sk[i].insert(keys[i])
                sk[i]._held.clear()
        except Exception as e:  # reported below, from the test's thread
            errors.append(e)

    th = [threading.Thread(target=client, args=(i,)) for i in range(len(shapes))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not errors, errors
    for i, (w, chunk) in enumerate(shapes):
        assert sk[i].sync_status() == sf.SF_OK
        o = oracle.Sketch(d, w, z, kb, 5)
        for _ in range(CALLS):
            o.update(host[i].numpy(), np.ones(N, np.int8), S=chunk if chunk > 1 else None)
        assert np.array_equal(sk[i].fat.cpu().numpy().view(np.uint32).reshape(o.B.shape), o.B)
        assert np.array_equal(sk[i].slim.cpu().numpy().view(np.uint32).reshape(o.A.shape), o.A)


def test_one_at_a_time_calls_on_two_streams(sf):
    """Cooperative launches of two sketches, of up to 128 blocks each, interleave on two streams."""
    import torch
    import workloads as wl
    n = 150_000
    streams = [torch.cuda.Stream() for _ in range(2)]
    st = [wl.mixed_stream(n, 7000, 1.0, f, 4, seed=60 + i)[0] for i, f in enumerate((0.0, 0.2))]
    keys, ops = [s.keys.cuda() for s in st], [s.ops.cuda() for s in st]
    torch.cuda.synchronize()
    sk = [sf.Sketch(4, 3000, 16, 4, 5, 1, stream=s) for s in streams]
    for part in (slice(0, 60_000), slice(60_000, n)):
        for i in range(2):
            sk[i].update(keys[i][part], ops[i][part])
    for i in range(2):
        o = oracle.Sketch(4, 3000, 16, 4, 5)
        o.update(st[i].keys.numpy(), st[i].ops.numpy())
        assert sk[i].sync_status() == sf.SF_OK
        assert np.array_equal(sk[i].fat.cpu().numpy().view(np.uint32).reshape(o.B.shape), o.B)
        assert np.array_equal(sk[i].slim.cpu().numpy().view(np.uint32).reshape(o.A.shape), o.A)
