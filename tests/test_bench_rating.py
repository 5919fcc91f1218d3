"""bench.py rates a point against the tensor peak only where the library's dispatch sends it to the tensor cores."""
import pytest

import bench


@pytest.mark.parametrize("es,m,n,k,want", [
    (4, 32768, 16, 32768, 0), (4, 32768, 17, 32768, 6), (4, 32768, 64, 15, 0), (4, 100, 64, 16, 6),
    (4, 16384, 65, 32, 0), (4, 16384, 65, 33, 6),
    (8, 32768, 1, 32768, 0), (8, 32768, 2, 32768, 35), (8, 32768, 64, 32768, 28), (8, 32768, 64, 255, 0),
    (8, 2048, 16, 1024, 0), (8, 2441, 64, 256, 0), (8, 2442, 64, 256, 28), (8, 2442, 49, 256, 28), (8, 400, 64, (1 << 20) + 1, 0),
    (8, 16384, 16384, 3, 0), (8, 16384, 16384, 4, 36)])
def test_products_follow_the_dispatch(es, m, n, k, want):
    assert bench.tensor_products(es, m, n, k) == want
