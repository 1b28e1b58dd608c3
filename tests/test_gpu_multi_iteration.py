"""chunk_multi_kernel (rounds above one update per lane, keys in device memory) and chunk_update_kernel's claim list
(the same rounds with keys in pinned memory) against the oracle's chunked semantics.  Chunks: one warp above the
lanes of the grid, 200,000, and 2^20, where thousands of keys meet another's fingerprint in their probe; few and
many rows, key widths 4, 8 and 13 bytes, insertions of mostly distinct keys (increments that return values, slacks,
skipped Fat reads), skewed ones (block merges), deletions under both rules, the smaller blocks, claim
lists in shared and in global memory, ragged last chunks."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


def _keys(st_keys, kb):
    import torch
    return st_keys if st_keys.shape[1] == kb else torch.cat([st_keys, st_keys.flip(1)], 1)[:, :kb].contiguous()


def _stream(n, distinct, s, frac, kb, seed):
    st, _ = wl.mixed_stream(n, distinct, s, frac, 4 if kb == 4 else 8, seed=seed)
    return _keys(st.keys, kb), st.ops


def _lanes():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count * 512


def _same(g, o):
    assert np.array_equal(g.fat.cpu().numpy().view(np.uint32).reshape(o.B.shape), o.B)
    assert np.array_equal(g.slim.cpu().numpy().view(np.uint32).reshape(o.A.shape), o.A)


@pytest.mark.parametrize("chunk", [0, 200_000, 1 << 20])   # 0: one warp above the lanes of the grid
@pytest.mark.parametrize("d,w,kb,distinct,s", [
    (1, 60_001, 8, 3_000_000, 0.0), (2, 30_011, 13, 200_000, 0.0), (3, 1 << 16, 4, 400_000, 0.6),
    (5, 50_021, 8, 1_000_000, 0.0), (4, 1 << 18, 13, 50_000, 1.1),
])
def test_insertions(sf, chunk, d, w, kb, distinct, s):
    chunk = chunk or _lanes() + 32
    n = 2 * chunk + chunk // 3 + 7
    keys, _ = _stream(n, distinct, s, 0.0, kb, seed=d * 31 + chunk % 97)
    g = sf.Sketch(d, w, 8, kb, 3, chunk)
    o = oracle.Sketch(d, w, 8, kb, 3)
    ones = np.ones(n, np.int8)
    for part in (slice(0, n), slice(0, n // 3)):  # the second call's first chunk meets a warm sketch
        g.insert(keys[part].cuda())
        o.update(keys[part].numpy(), ones[part], S=chunk)
    assert g.sync_status() == sf.SF_OK
    _same(g, o)


@pytest.mark.parametrize("d,w,z,kb,s,frac,rule,chunk", [
    (3, 20_011, 8, 8, 0.0, 0.3, "sff", 200_000), (5, 9001, 7, 13, 1.0, 0.2, "sf4", 200_000),
    (3, 70_001, 16, 4, 0.8, 0.1, "sf4", 0), (5, 33_001, 3, 8, 1.4, 0.4, "sff", 1 << 20), (1, 5003, 64, 8, 1.0, 0.2, "sff", 0),
])
def test_mixed(sf, d, w, z, kb, s, frac, rule, chunk):
    chunk = chunk or _lanes() + 32
    n = chunk + chunk // 2 + 5
    keys, ops = _stream(n, 150_000, s, frac, kb, seed=d + chunk % 89)
    g = sf.Sketch(d, w, z, kb, 3, chunk, delete_rule=rule)
    o = oracle.Sketch(d, w, z, kb, 3, delete_rule=rule)
    g.update(keys.cuda(), ops.cuda())
    o.update(keys.numpy(), ops.numpy(), S=chunk)
    assert g.sync_status() == sf.SF_OK
    _same(g, o)
    gone = keys[ops > 0][: n // 20].contiguous()  # inserted once more and taken back: a deletion-only call
    g.insert(gone.cuda())
    o.update(gone.numpy(), np.ones(len(gone), np.int8), S=chunk)
    g.delete(gone.cuda())
    o.update(gone.numpy(), -np.ones(len(gone), np.int8), S=chunk)
    assert g.sync_status() == sf.SF_OK
    _same(g, o)


@pytest.mark.parametrize("chunk", [100_000, 1 << 20])
@pytest.mark.parametrize("batch", [False, True])
def test_pinned_keys(sf, chunk, batch):
    """chunk_update_kernel's list: keys read over the host link, alone and in a batch with device keys beside."""
    n = chunk + chunk // 3 + 11
    keys, ops = _stream(n, 120_000, 0.9, 0.2, 8, seed=5)
    other, _ = _stream(n, 120_000, 0.0, 0.0, 8, seed=6)
    g, h = sf.Sketch(4, 30_011, 16, 8, 3, chunk), sf.Sketch(4, 40_009, 16, 8, 4, chunk)
    o, p = oracle.Sketch(4, 30_011, 16, 8, 3), oracle.Sketch(4, 40_009, 16, 8, 4)
    pk, po = keys.pin_memory(), ops.pin_memory()
    if batch:
        b = sf.Batch(2, max_round_slots=2 * (chunk + 32), group_bytes=0)
        b.update([(g, pk, po), (h, other.cuda(), None)])
        assert b.sync_status() == sf.SF_OK
        b.close()
    else:
        g.update(pk, po)
        h.insert(other.cuda())
        assert g.sync_status() == sf.SF_OK and h.sync_status() == sf.SF_OK
    o.update(keys.numpy(), ops.numpy(), S=chunk)
    p.update(other.numpy(), np.ones(n, np.int8), S=chunk)
    _same(g, o)
    _same(h, p)


@pytest.mark.parametrize("block", [128, 256, 512])
@pytest.mark.parametrize("per_lane,frac", [(2, 0.0), (2, 0.2), (15, 0.0), (15, 0.1)])
def test_blocks_and_lists(sf, block, per_lane, frac):
    """Insertions only and with deletions, at every block size, with claim lists in shared memory (two updates a
    lane) and in global memory (15: 7,680 claims a 512-thread block, above 112 KiB of 16 bytes)."""
    slots = _lanes() * per_lane
    chunks = [slots // 2, slots // 4 + 33, slots // 4 + 1]
    sk, orc, items = [], [], []
    for k, c in enumerate(chunks):
        n = c + c // 4 + 3
        keys, ops = _stream(n, [900_000, 50_000, 4000][k], [0.0, 0.5, 1.1][k], frac, 8, seed=40 + k)
        sk.append(sf.Sketch(4, 20_011 + k, 16, 8, k, c))
        orc.append(oracle.Sketch(4, 20_011 + k, 16, 8, k))
        items.append((sk[k], keys.cuda(), ops.cuda() if frac else None))
        orc[k].update(keys.numpy(), ops.numpy(), S=c)
    b = sf.Batch(3, max_round_slots=slots + 200, group_bytes=0, block_threads=block)
    b.update(items)
    assert b.sync_status() == sf.SF_OK
    b.close()
    for g, o in zip(sk, orc):
        _same(g, o)
