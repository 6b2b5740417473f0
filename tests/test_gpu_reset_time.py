"""Time of a fresh population (GPU): a small one takes no longer than a large one."""
import time

import pytest

from paper_1006_0252_gb300 import inputs, pa

pytestmark = pytest.mark.gpu


# Blocks of a few slots read the couplings for a few replicas each: 300 replicas
# took 1.6 times as long as 17000.
@pytest.mark.parametrize("L", [8, 10])
def test_small_gauss_population_resets_as_fast_as_a_large_one(L):
    J = inputs.gaussian_couplings_3d(L, 2, 9)

    def us(R0):
        g = pa.Run(J, L, 3, R0, 3, gaussian=True)
        best = float("inf")
        for k in range(20):
            g.sync()
            t = time.perf_counter()
            for i in range(10):
                g.reset(k + i)
            g.sync()
            best = min(best, (time.perf_counter() - t) * 1e5)
        return best

    assert us(300) <= 1.2 * us(17000)
