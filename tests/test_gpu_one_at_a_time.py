"""The S = 1 path by sorts and scans against the oracle's sequential rule, at the sizes where it can go
wrong: one update past the window kernel's calls, block edges (1,024 entries), the step from every block
summing the digit counts itself to sharing the work (16 blocks), a piece's end (131,072 updates), one to
four radix passes, buckets of 1 to 64 counters, dense sketches that iterate from below, both deletion
rules, updates that do nothing, and sketches carried over from earlier calls.  Counters are whole
numbers: equality."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sf():
    import paper_1701_04148_gb300 as m
    m.load()
    return m


def _check(sf, d, w, z, kb, calls, rule="sff"):
    g = sf.Sketch(d, w, z, kb, 9, 1, delete_rule=rule)
    o = oracle.Sketch(d, w, z, kb, 9, delete_rule=rule)
    for keys, ops in calls:
        n = len(keys)
        if isinstance(ops, str):
            (g.insert if ops == "insert" else g.delete)(keys.cuda())
            o.update(keys.numpy(), (np.ones if ops == "insert" else lambda m, t: -np.ones(m, t))(n, np.int8))
        else:
            g.update(keys.cuda(), ops.cuda())
            o.update(keys.numpy(), ops.numpy())
        assert g.sync_status() == sf.SF_OK
        assert np.array_equal(g.fat.cpu().numpy().view(np.uint32).reshape(d, w, z), o.B)
        assert np.array_equal(g.slim.cpu().numpy().view(np.uint32).reshape(d, w), o.A)


@pytest.mark.parametrize("n", [65, 1023, 1024, 1025, 2049, 16_384, 16_385, 131_072, 131_073])
def test_lengths(sf, n):
    st, _ = wl.mixed_stream(n, max(8, n // 9), 1.0, 0.2, 4, seed=n)
    ins, _ = wl.insert_only_u32(n, max(8, n // 20), 0.8, seed=n + 1)
    _check(sf, 4, 1024, 16, 4, [(ins, "insert"), (st.keys, st.ops), (ins.flip(0).contiguous(), "delete")])


@pytest.mark.parametrize("d,w,z,kb,distinct,s,frac,rule", [
    (1, 1024, 1, 4, 3000, 1.0, 0.3, "sff"),
    (2, 1024, 1, 4, 20_000, 0.0, 0.0, "sff"),        # dense: tens of iterations from below
    (3, 1024, 2, 8, 20_000, 1.2, 0.25, "sff"),       # dense, with deletions
    (4, 1031, 64, 4, 500, 1.5, 0.4, "sff"),          # z = 64: two counters a lane
    (5, 40_000, 3, 4, 30_000, 0.99, 0.3, "sff"),
    (4, 1500, 7, 8, 2000, 1.0, 0.3, "sf4"),
    (6, 70_001, 33, 8, 9000, 0.5, 0.1, "sff"),       # three passes over the counters
    (8, 1024, 5, 4, 4000, 1.0, 0.2, "sf4"),
    (2, 1 << 21, 16, 4, 9000, 0.7, 0.2, "sff"),      # four passes
])
def test_shapes(sf, d, w, z, kb, distinct, s, frac, rule):
    n = 20_000
    a, _ = wl.mixed_stream(n, distinct, s, frac, kb, seed=d * 7 + z)
    b, _ = wl.mixed_stream(n // 2, distinct, s, frac, kb, seed=d * 7 + z)
    if frac == 0.0:
        _check(sf, d, w, z, kb, [(a.keys, "insert"), (b.keys, "insert")], rule)
        return
    _check(sf, d, w, z, kb, [(a.keys, a.ops), (b.keys, b.ops)], rule)


def test_updates_that_do_nothing(sf):
    """Operations of 0 between the others, some on keys in use."""
    import torch
    st, _ = wl.mixed_stream(9000, 300, 1.1, 0.2, 4, seed=5)
    gen = torch.Generator().manual_seed(1)
    at = torch.randint(0, 9000, (3000,), generator=gen).sort().values
    keys = torch.cat([st.keys, st.keys[at]])
    ops = torch.cat([st.ops, torch.zeros(3000, dtype=torch.int8)])
    order = torch.cat([torch.arange(9000) * 2, at * 2 + 1]).argsort(stable=True)
    for kb in (4, 13):
        k = keys[order] if kb == 4 else torch.cat([keys[order]] * 4, 1)[:, :13]
        _check(sf, 4, 1024, 4, kb, [(k.contiguous(), ops[order].contiguous())])


def test_captured_and_replayed(sf):
    """A captured call replays: the launch leaves the barrier words as it found them."""
    import torch
    st, _ = wl.mixed_stream(30_000, 2000, 1.0, 0.1, 4, seed=3)
    main = torch.cuda.Stream()
    keys, ops = st.keys.cuda(), st.ops.cuda()
    torch.cuda.synchronize()
    g = sf.Sketch(4, 2048, 16, 4, 9, 1, stream=main)
    o = oracle.Sketch(4, 2048, 16, 4, 9)
    g.update(keys, ops)
    o.update(st.keys.numpy(), st.ops.numpy())
    assert g.sync_status() == sf.SF_OK
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        g.update(keys, ops)
    for _ in range(2):
        with torch.cuda.stream(main):
            graph.replay()
        o.update(st.keys.numpy(), st.ops.numpy())
    assert g.sync_status() == sf.SF_OK
    assert np.array_equal(g.fat.cpu().numpy().view(np.uint32).reshape(4, 2048, 16), o.B)
    assert np.array_equal(g.slim.cpu().numpy().view(np.uint32).reshape(4, 2048), o.A)
