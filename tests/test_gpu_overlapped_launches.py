"""Slim export and queries, which are launched while the stream's previous kernel drains: they read what
that kernel wrote, at sizes around a vector, a block and the iterations of a thread, with destinations
off 16 bytes, inside a captured graph and behind another stream's event.  Whole numbers: equality."""
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


@pytest.mark.parametrize("d,w", [(1, 1), (1, 3), (3, 5), (1, 1023), (2, 513), (4, 4097), (8, 65_536)])
@pytest.mark.parametrize("shift", [0, 1])
def test_export_follows_the_update(sf, d, w, shift):
    import torch
    st, _ = wl.insert_only_u32(3000, 500, 0.8, seed=d * w)
    g = sf.Sketch(d, w, 2, 4, 3, 700)
    o = oracle.Sketch(d, w, 2, 4, 3)
    buf = torch.full((d * w + 8,), -1, dtype=torch.int32, device="cuda")
    keys = st.cuda()
    for _ in range(3):
        g.insert(keys)
        g.export_slim(buf[shift:shift + d * w])
        o.insert(st.numpy(), S=700)
    g.sync()
    got = buf.cpu().numpy()
    assert np.array_equal(got[shift:shift + d * w].view(np.uint32).reshape(d, w), o.A)
    assert (got[:shift] == -1).all() and (got[shift + d * w:] == -1).all()


@pytest.mark.parametrize("n", [1, 255, 256, 511, 512, 513, 70_001, 1_000_003])
def test_query_follows_the_export(sf, n):
    import torch
    st, _ = wl.insert_only_u32(4000, 900, 0.8, seed=n)
    g = sf.Sketch(4, 1000, 4, 4, 3, 1000)
    o = oracle.Sketch(4, 1000, 4, 4, 3)
    gen = torch.Generator().manual_seed(n)
    asked = torch.randint(0, 256, (n, 4), dtype=torch.uint8, generator=gen)
    asked[: min(n, 2000)] = st[: min(n, 2000)]
    g.insert(st.cuda())
    slim, hdr = g.export_slim()
    est = sf.query(slim, hdr, asked.cuda())
    g.sync()
    o.insert(st.numpy(), S=1000)
    assert np.array_equal(est.cpu().numpy().view(np.uint32), o.query(asked.numpy()))


def test_query_and_export_in_a_graph_and_behind_an_event(sf):
    import torch
    st, _ = wl.insert_only_u32(50_000, 5000, 0.9, seed=1)
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    keys = st.cuda()
    torch.cuda.synchronize()
    g = sf.Sketch(4, 4096, 4, 4, 3, 1000, stream=main)
    o = oracle.Sketch(4, 4096, 4, 4, 3)
    slim = torch.empty(4 * 4096, dtype=torch.int32, device="cuda")
    out = torch.empty(len(st), dtype=torch.int32, device="cuda")
    g.insert(keys)
    o.insert(st.numpy(), S=1000)
    _, hdr = g.export_slim(slim)
    # another stream queries behind an event, then the sketch's stream goes on behind that stream
    side.wait_event(main.record_event())
    sf.query(slim, hdr, keys, out, stream=side)
    main.wait_event(side.record_event())
    g.insert(keys)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint32), o.query(st.numpy()))
    o.insert(st.numpy(), S=1000)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        g.export_slim(slim)
        sf.query(slim, hdr, keys, out, stream=main)
    for _ in range(2):
        g.insert(keys)
        o.insert(st.numpy(), S=1000)
        with torch.cuda.stream(main):
            graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(slim.cpu().numpy().view(np.uint32).reshape(4, 4096), o.A)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), o.query(st.numpy()))
