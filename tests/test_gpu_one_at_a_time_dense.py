"""One-at-a-time updates of dense sketches (few counters a bucket, tens of updates each), whose raise targets
settle in the iterations from below: whole pieces of more than 16 blocks, a second piece behind the first,
warm sketches whose new keys meet counters of every height, hot keys whose runs cross blocks, and streams
with deletions, whose bounds between a key's updates take whole blocks at a time.  Counters equal the oracle's."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


def _run(sf, d, w, z, kb, calls, rule="sff"):
    g = sf.Sketch(d, w, z, kb, 9, 1, delete_rule=rule)
    o = oracle.Sketch(d, w, z, kb, 9, delete_rule=rule)
    for keys, ops in calls:
        if ops is None:
            g.insert(keys.cuda())
            o.update(keys.numpy(), np.ones(len(keys), np.int8))
        else:
            g.update(keys.cuda(), ops.cuda())
            o.update(keys.numpy(), ops.numpy())
        assert g.sync_status() == sf.SF_OK
        assert np.array_equal(g.fat.cpu().numpy().view(np.uint32).reshape(o.B.shape), o.B)
        assert np.array_equal(g.slim.cpu().numpy().view(np.uint32).reshape(o.A.shape), o.A)


@pytest.mark.parametrize("d,w,z,distinct,s", [
    (1, 1024, 1, 3000, 0.0), (1, 1024, 3, 3000, 1.0),
    (2, 1024, 1, 20_000, 0.0), (2, 1024, 1, 2000, 0.0), (2, 1024, 2, 9000, 1.0), (2, 16_384, 1, 2000, 0.0),
    (3, 1024, 1, 2000, 0.0), (4, 1024, 1, 20_000, 0.5), (4, 1100, 2, 5000, 1.3), (5, 1024, 1, 9000, 0.0),
    (6, 1024, 1, 3000, 1.0), (8, 1024, 1, 9000, 0.3),
])
def test_insertions(sf, d, w, z, distinct, s):
    calls = [(wl.mixed_stream(n, distinct, s, 0.0, 4, seed=100 * c + d)[0].keys, None)
             for c, n in enumerate([60_000, 140_001, 3000])]
    _run(sf, d, w, z, 4, calls)


@pytest.mark.parametrize("d,w,z,distinct,s,frac,rule", [
    (1, 1024, 2, 3000, 1.0, 0.3, "sff"), (2, 1024, 1, 9000, 0.0, 0.1, "sff"), (2, 1024, 1, 2000, 0.5, 0.45, "sff"),
    (3, 1024, 1, 9000, 1.2, 0.2, "sff"), (4, 1024, 1, 20_000, 0.0, 0.02, "sff"), (4, 1100, 2, 3000, 1.0, 0.3, "sf4"),
    (5, 1024, 1, 5000, 0.7, 0.2, "sff"), (8, 1024, 1, 5000, 0.0, 0.3, "sf4"),
])
def test_mixed(sf, d, w, z, distinct, s, frac, rule):
    calls = []
    for c, n in enumerate([50_000, 140_001]):
        st, _ = wl.mixed_stream(n, distinct, s, frac, 4, seed=100 * c + d)
        calls.append((st.keys, st.ops))
    _run(sf, d, w, z, 4, calls, rule)
