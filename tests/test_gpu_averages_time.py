"""Times of the Sec. 3 averages on device arrays (GPU), against sizes at which the
library has always taken the same path."""
import ctypes
import time

import pytest

from paper_1006_0252_gb300 import pa

pytestmark = pytest.mark.gpu


# The rule's other side is a warp a group: from 609 groups on.  One group fewer must
# not take longer (a block a group took 1.2 to 2 times as long at these sizes).
@pytest.mark.parametrize("M", [33, 64, 100, 200])
@pytest.mark.parametrize("pairs", [False, True])
def test_many_short_groups_take_no_longer_by_block(M, pairs):
    torch = pytest.importorskip("torch")
    lib, stream = pa.load(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def us(G):
        a = [torch.rand(G * M, dtype=torch.float64, device="cuda") + 1.0 for _ in range(5)]
        out = [torch.zeros(G, dtype=torch.float64, device="cuda") for _ in range(2)]
        x1, x2, A, R1, R2, mean, fbar = (ctypes.c_void_p(t.data_ptr()) for t in a + out)
        best = float("inf")
        for _ in range(10):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(50):
                if pairs:
                    code = lib.pa_weighted_average_pairs_dev(G, M, x1, x2, A, R1, R2, mean, fbar, stream)
                else:
                    code = lib.pa_weighted_average_dev(G, M, x1, A, R1, mean, fbar, stream)
                assert code == pa.PA_OK
            torch.cuda.synchronize()
            best = min(best, (time.perf_counter() - t) / 50 * 1e6)
        return best

    assert us(608) <= 1.1 * us(609)
