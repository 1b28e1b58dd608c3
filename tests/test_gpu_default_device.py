"""Calls under a default device of the user's program."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def test_query_of_pinned_keys_under_a_cuda_default_device(sf):
    """Keys in pinned memory are answered into pinned memory, whatever device tensors are made on by default."""
    import torch
    keys = torch.arange(500, dtype=torch.int32)
    g = sf.Sketch(4, 1000, 16, 4, 5, 64)
    g.insert(keys.cuda())
    slim, hdr = g.export_slim()
    g.sync()
    o = oracle.Sketch(4, 1000, 16, 4, 5)
    o.update(keys.numpy(), np.ones(500, np.int8), S=64)
    pinned = keys.pin_memory()
    with torch.device("cuda"):
        out = sf.query(slim, hdr, pinned)
    torch.cuda.synchronize()
    assert not out.is_cuda and out.is_pinned()
    assert np.array_equal(out.numpy().view(np.uint32), o.query(keys.numpy()))
