"""The tcgen05 decode linears at 17 to 64 tokens where many CTAs share a row tile:
their sums are added several CTAs and 8 or 16 tokens at a time, so the numbers of CTAs
and tokens lie around those."""
import pytest

from tests.gpu_helpers import check_decode_linear, torch_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


@pytest.mark.parametrize("wq", [0, 2])
@pytest.mark.parametrize("m", [17, 24, 31, 33, 48, 49, 64])
@pytest.mark.parametrize("n,k,epi", [(6400, 4096, 0), (3328, 8192, 3), (2056, 13824, 1), (4104, 8192, 2)])
def test_shared_row_tiles(fp, wq, m, n, k, epi):
    check_decode_linear(fp, wq, m, n, k, epi)
