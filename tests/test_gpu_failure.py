"""Failure detection without a GPU fault: bounded device waits return an error status.

A cooperative launch in which one block never arrives at the grid barrier makes every other
block's wait run out after a short limit; the host reads SF_ERR_TIMEOUT and the context stays
usable (a normal launch and a sketch update succeed afterwards).  Host-side failures (bad
arguments, underflow, bad key ids) are covered in the parity and ABI tests."""
import pytest

pytestmark = pytest.mark.gpu


def test_barrier_wait_times_out_and_the_context_survives(sf):
    import torch
    L = sf.load_bench()
    scratch = torch.zeros(64, dtype=torch.int32, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    assert L.sf_bench_wait_timeout(scratch.data_ptr(), 0, 20_000_000, st) == sf.SF_OK
    assert L.sf_bench_wait_timeout(scratch.data_ptr(), 1, 20_000_000, st) == sf.SF_ERR_TIMEOUT
    assert L.sf_bench_wait_timeout(scratch.data_ptr(), 5, 20_000_000, st) == sf.SF_ERR_TIMEOUT
    # the context is still usable
    assert L.sf_bench_grid_barrier(scratch.data_ptr(), 10, st) == sf.SF_OK
    g = sf.Sketch(4, 1024, 16, 4, 1, 256)
    g.insert(torch.arange(1000, dtype=torch.int32, device="cuda"))
    assert g.sync_status() == sf.SF_OK
    assert int((g.fat.view(4, -1).to(torch.int64).sum(dim=1) == 1000).sum()) == 4


def test_wait_limit_is_bounded_by_the_api(sf):
    import torch
    L = sf.load_bench()
    scratch = torch.zeros(64, dtype=torch.int32, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    assert L.sf_bench_wait_timeout(scratch.data_ptr(), 1, 5_000_000_000, st) == sf.SF_ERR_INVALID


def test_timeout_status_rezeroes_shared_dictionaries_and_the_arena(sf):
    """A grid wait that gave up latches the timeout bit in the error word (the first control word
    of the scratch) and may leave dictionary entries claimed.  Here the host writes that bit and
    fills the dictionaries with stale claim words, standing in for such a launch (no kernel is made
    to time out): sf_sync returns SF_ERR_TIMEOUT and zeroes the scratch and the dictionary given by
    sf_set_dictionary, sf_batch_sync zeroes the batch's dictionary arena, and the next updates
    equal sketches that never saw the failure.  The stale words (0x11111111) carry no fingerprint a
    key can have, so a dictionary left dirty would show up as wrong counters or a full-dictionary
    error, never as a re-read of a key."""
    import torch
    import workloads as wl
    ins, dels, _ = wl.flows_with_deletes(60_000, 8_000, 1.0, 0.1, seed=91, device="cuda")
    need = sf.dictionary_bytes(4, 3001, 16, 13, 5, 4096)
    a = sf.Sketch(4, 3001, 16, 13, 5, 4096)
    b = sf.Sketch(4, 3001, 16, 13, 5, 4096, shared_dict=True)
    d = torch.empty(need, dtype=torch.uint8, device="cuda")
    b.set_dictionary(d)
    torch.cuda.synchronize()
    d.fill_(0x11)
    b.scratch[0] = 2
    torch.cuda.synchronize()
    assert b.sync_status() == sf.SF_ERR_TIMEOUT
    assert int(torch.count_nonzero(d)) == 0 and int(torch.count_nonzero(b.scratch[:64])) == 0
    assert b.sync_status() == sf.SF_OK
    for s in (a, b):
        s.insert(ins)
        s.delete(dels)
    assert a.sync_status() == sf.SF_OK and b.sync_status() == sf.SF_OK
    assert torch.equal(a.fat, b.fat) and torch.equal(a.slim, b.slim)

    c = sf.Sketch(4, 3001, 16, 13, 5, 4096, shared_dict=True)
    e = sf.Sketch(4, 3001, 16, 13, 5, 4096)
    bt = sf.Batch(2, dict_arena_bytes=need)
    torch.cuda.synchronize()
    bt.arena.fill_(0x11)
    bt.scratch[0] = 2
    torch.cuda.synchronize()
    assert bt.sync_status() == sf.SF_ERR_TIMEOUT
    assert int(torch.count_nonzero(bt.arena)) == 0
    bt.update([(c, ins, None)])
    e.insert(ins)
    assert bt.sync_status() == sf.SF_OK and e.sync_status() == sf.SF_OK
    assert torch.equal(c.fat, e.fat) and torch.equal(c.slim, e.slim)
    bt.close()


@pytest.mark.parametrize("stale", [1, 128, 1 << 40])
@pytest.mark.parametrize("kind", ["insert", "delete", "mixed"])
def test_one_at_a_time_launches_after_a_timeout_change_nothing(sf, kind, stale):
    """The host writes what a one-at-a-time launch that gave up leaves behind: the timeout bit, a barrier
    count that is not zero and a count of blocks that have left.  The pieces queued behind it (140,000
    updates: two) must leave every counter as it is; sf_sync reports the timeout and zeroes the words, and
    the same call then gives the oracle's counters."""
    import numpy as np
    import oracle
    import torch
    import workloads as wl
    n = 140_000
    st, _ = wl.mixed_stream(n, 9000, 1.0, 0.1, 4, seed=12)
    first, _ = wl.mixed_stream(n, 9000, 1.0, 0.0, 4, seed=12)
    keys, ops = first.keys.cuda(), None
    g = sf.Sketch(4, 2048, 16, 4, 9, 1)
    o = oracle.Sketch(4, 2048, 16, 4, 9)
    g.insert(keys)
    o.update(first.keys.numpy(), np.ones(n, np.int8))
    assert g.sync_status() == sf.SF_OK
    fat, slim = g.fat.clone(), g.slim.clone()
    words = g.scratch[:64]                            # the control words
    words[0] = 2                                      # the timeout bit
    words[2] = stale & 0x7FFFFFFF                     # the 64-bit barrier count
    words[3] = stale >> 32
    words[4] = 1                                      # blocks that have left
    torch.cuda.synchronize()
    if kind == "mixed":
        keys, ops = st.keys.cuda(), st.ops.cuda()
    call = {"insert": lambda: g.insert(keys), "delete": lambda: g.delete(keys), "mixed": lambda: g.update(keys, ops)}[kind]
    call()
    call()
    assert g.sync_status() == sf.SF_ERR_TIMEOUT
    assert torch.equal(g.fat, fat) and torch.equal(g.slim, slim)
    assert int(torch.count_nonzero(g.scratch[:64])) == 0
    call()
    op = {"insert": np.ones(n, np.int8), "delete": -np.ones(n, np.int8), "mixed": st.ops.numpy()}[kind]
    o.update((st.keys if kind == "mixed" else first.keys).numpy(), op)
    assert g.sync_status() == sf.SF_OK
    assert np.array_equal(g.fat.cpu().numpy().view(np.uint32).reshape(o.B.shape), o.B)
    assert np.array_equal(g.slim.cpu().numpy().view(np.uint32).reshape(o.A.shape), o.A)


@pytest.mark.parametrize("chunk", [4096, 100_000])
@pytest.mark.parametrize("kb", [4, 13])
def test_stale_claims_past_the_calls_end_are_not_followed(sf, chunk, kb):
    """A launch that timed out leaves claims of its chunk behind, and the calls made before sf_sync meet them
    (a batch's next launch runs to its end).  The host plants one in every key's home slot, with the key's
    fingerprint and a position past the call's last key: the key there is not read, the claim counts as
    another key's, and the counters equal the oracle's.  Chunks of 4,096 run the single-iteration kernel's
    dictionary (15-bit fingerprints, 16-bit positions), of 100,000 the multi-iteration one's (11 and 20)."""
    import numpy as np
    import oracle
    import torch
    U = np.uint64

    def fin(x):
        x = (x ^ (x >> U(30))) * U(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> U(27))) * U(0x94D049BB133111EB)
        return x ^ (x >> U(31))

    seed = 9
    r = np.random.RandomState(3)
    distinct = r.randint(0, 256, (200, kb)).astype(np.uint8)
    keys = distinct[r.randint(0, 200, 700)]
    full = np.zeros((200, 16), np.uint8)
    full[:, :kb] = distinct
    with np.errstate(over="ignore"):
        probe = fin(full.view("<u8")[:, 0] ^ fin(np.array([seed], U) + U(0x9E3779B97F4A7C15)))
        if kb > 8:
            probe = fin(probe ^ full.view("<u8")[:, 1])
    if chunk == 4096:
        entries = 16 * chunk
        claims = (U(0x8000) | probe >> U(49)) << U(16) | U(0xFFFF)
    else:
        entries = 1 << 20                              # the power of two from 8 * 100,000
        claims = U(0x80000000) | (probe >> U(53)) << U(20) | U(0xFFFFF)
    g = sf.Sketch(4, 3001, 16, kb, seed, chunk)
    slots = torch.from_numpy((probe & U(entries - 1)).astype(np.int64)).cuda()
    words = torch.from_numpy((claims & U(0xFFFFFFFF)).astype(np.uint32).view(np.int32)).cuda()
    g.scratch[64 + 2 * slots] = words
    planted = g.scratch[64 + 2 * slots]
    torch.cuda.synchronize()
    g.insert(torch.from_numpy(keys).cuda())
    assert g.sync_status() == sf.SF_OK
    o = oracle.Sketch(4, 3001, 16, kb, seed)
    o.update(keys, np.ones(700, np.int8), S=chunk)
    assert np.array_equal(g.fat.cpu().numpy().view(np.uint32).reshape(o.B.shape), o.B)
    assert np.array_equal(g.slim.cpu().numpy().view(np.uint32).reshape(o.A.shape), o.A)
    assert torch.equal(g.scratch[64 + 2 * slots], planted)  # nobody took or cleared them
