"""The counting sort of the dispatch at the chunk counts where its ranking changes (296 chunks of 1024 slots: two per SM) and at the
expert counts that decide beside them."""
import pytest

from test_gpu_dispatch_index import test_dispatch_index_is_a_stable_sort as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,n,k", [(296 * 1024, 3, 1), (296 * 1024 + 1, 3, 1), (303105, 1, 1), (296 * 512 + 1, 2, 2), (101400, 220, 3),
                                   (151553, 2048, 2), (151553, 2049, 2), (60000, 1025, 6), (76000, 300, 4)])
def test_dispatch_index_of_many_chunks(T, n, k):
    check(T, n, k)
