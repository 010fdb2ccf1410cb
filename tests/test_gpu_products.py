"""The FP64 products of a window at the edges of their tiles (4 rows, 16
candidates, 128 inner indexes per chunk), against the oracle's chain: identical
decisions, vertex lists and times, N and sum sign G to 1e-10 (tests/
test_gpu_parity.py says why).  The order grows from 10 through 128 to about
160, so every remainder of the rows and both chunk counts occur."""
import pytest

from tests.test_gpu_parity import check, run_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_sub", [5, 17, 33, 64])
def test_candidate_products_at_the_edges_of_their_tiles(k_sub):
    check(run_pair(16, 1.0, 0.0, 6.0, 4.0, 3.0, 1024, k_sub=k_sub, sweeps=14, seed=k_sub, warmup=4, R=16))
