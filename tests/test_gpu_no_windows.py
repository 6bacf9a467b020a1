"""A library of reads shorter than k has no windows: the call stops after the validity bitmap."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [21, 31, 64])
def test_reads_shorter_than_k(have_gpu, k):
    import torch

    import paper_1305_1861_gb300 as pkg

    pkg.build()
    ctx = pkg.Context(0)
    for length, n in ((k - 1, 1), (k - 1, 3000), (5, 400), (k, 500)):
        bases = np.frombuffer(b"ACGT", np.uint8)[np.random.default_rng(n).integers(0, 4, length * n)]
        offs = np.arange(0, bases.size + 1, length, dtype=np.uint64)
        ok, oc, nw = oracle.count(bases, offs, k, 1)
        keys, counts, got = ctx.turtle_count_device(torch.from_numpy(bases).cuda(),
                                                    torch.from_numpy(offs.astype(np.int64)).cuda(), k, 1)
        assert got == nw and np.array_equal(keys.cpu().numpy().view(np.uint64).reshape(ok.shape), ok)
        assert np.array_equal(counts.cpu().numpy().astype(np.uint64), oc)
        assert (ctx.stats()["stage_launches"]["filter"] > 0) == (nw > 0)
    ctx.close()
