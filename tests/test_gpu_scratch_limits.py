"""Scratch at the allocator's limit (GPU): a batch bootstrap runs in the memory
that its own arrays take, the table of weights being a luxury."""
import time

import numpy as np
import pytest

from paper_1006_0252_gb300 import inputs, pa

pytestmark = pytest.mark.gpu


class LimitedAllocator:
    """PyTorch's caching allocator, refusing single requests above `limit` bytes."""

    def __init__(self, torch):
        self.limit = 1 << 60

        def _alloc(nbytes, stream, ctx):
            if nbytes > self.limit:
                return None
            return torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), int(stream or 0))

        def _free(ptr, nbytes, stream, ctx):
            torch.cuda.caching_allocator_delete(ptr)

        self._fa, self._ff = pa.ALLOC_FN(_alloc), pa.FREE_FN(_free)
        self.opts = pa.Opts()
        self.opts.alloc, self.opts.free = self._fa, self._ff


def test_batch_bootstrap_without_room_for_the_table():
    torch = pytest.importorskip("torch")
    a = LimitedAllocator(torch)
    M, count, B, groups = 25, 4, 16, 2
    betas = np.array([0.2, 0.5, 0.9])
    b = pa.Batch([inputs.RunSpec(3, 4, r // M, 40 + r, 300, betas, 1) for r in range(groups * M)], opts=a.opts)
    b.run(betas, thetas=1)
    assert not b.sync().any()
    want = b.bootstrap(M, count, B=B, seed=7)
    need = 8 * (3 * M + 2 * B + 2) * groups * count  # the documented scratch
    a.limit = (need + 255) // 256 * 256
    got = b.bootstrap(M, count, B=B, seed=7)
    for k, w in want.items():
        # sums of 25 terms in another order, values up to 50 in a spread of 1e-2
        assert np.allclose(got[k], w, rtol=1e-10, atol=1e-12), k
    a.limit = 256
    with pytest.raises(pa.PAError) as e:
        b.bootstrap(M, count, B=B, seed=7)
    assert e.value.code == pa.PA_ERR_OOM
    b.close()


# With the table a call takes no longer than without: groups of fewer runs than the
# threads that share a resample took up to 3.4 times as long.
@pytest.mark.parametrize("M", [1, 2, 4, 8])
def test_batch_bootstrap_table_costs_no_time(M):
    torch = pytest.importorskip("torch")
    a = LimitedAllocator(torch)
    count, B, groups = 40, 1000, 40
    betas = np.linspace(0.05, 1.0, count)
    b = pa.Batch([inputs.RunSpec(3, 4, r // M, 40 + r, 100, betas, 1) for r in range(groups * M)], opts=a.opts)
    b.run(betas, thetas=1)
    assert not b.sync().any()

    def seconds():
        best = float("inf")
        for _ in range(10):
            t = time.perf_counter()
            b.bootstrap(M, count, B=B, seed=7)
            best = min(best, time.perf_counter() - t)
        return best

    tabulated = seconds()
    a.limit = (8 * (3 * M + 2 * B + 2) * groups * count + 255) // 256 * 256
    assert tabulated <= 1.1 * seconds()
    b.close()
