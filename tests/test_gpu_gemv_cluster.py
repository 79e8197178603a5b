"""The decode GEMV with a cluster of CTAs per row block: shares of uneven length,
clusters of three to eight, ragged rows and tokens, every epilogue and format, the
residual in place, and shapes on both sides of the rule."""
import pytest

from tests.gpu_helpers import check_decode_linear, torch_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


@pytest.mark.parametrize("wq", [0, 1, 2])
@pytest.mark.parametrize("m,n,k,epi", [
    (1, 128, 384, 0), (3, 130, 1152, 1), (8, 4104, 2176, 2), (9, 260, 640, 3), (16, 2056, 4224, 1), (16, 520, 1664, 2),
    (8, 12296, 1152, 0), (5, 6152, 3456, 3), (24, 1032, 1152, 1), (32, 776, 2176, 2),
    (12, 1032, 512, 0), (10, 8200, 640, 1), (40, 1160, 1664, 0)])
def test_cluster_shares(fp, wq, m, n, k, epi):
    check_decode_linear(fp, wq, m, n, k, epi)
