"""Vector-quantized forward at the edges of its product kernel: row blocks of 512, 256 and 128 rows and a partial last one,
codebooks narrower than, as wide as and wider than a stage of 256 columns (and not dividing it), a last stage of 64 columns,
fewer stages than multiprocessors and several row blocks per CTA, every token tile, both centroid dimensions."""
import pytest

from paper_2601_19675_b200 import lopro
from tests.test_gpu_vq import _check, _random_record

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 8, 9, 17, 32, 33])
@pytest.mark.parametrize("n,m,cr,cc,b,r,dim", [(320, 576, 512, 320, 64, 16, 4),      # 512-row blocks, the last of 64 rows; one wide codebook
                                              (1216, 1024, 512, 64, 64, 5, 4),      # four codebooks per stage, a last stage of 192 columns
                                              (1152, 640, 256, 192, 128, 16, 4),    # codebooks across stage boundaries
                                              (1024, 320, 128, 128, 256, 0, 4),     # 128-row blocks: four phases
                                              (2112, 1600, 512, 704, 64, 32, 4),    # 11 x 64 columns: two codebooks meet in a stage
                                              (832, 1088, 512, 64, 64, 16, 2), (1280, 512, 256, 256, 256, 7, 2),
                                              (256, 20480, 512, 256, 64, 16, 4)])   # one stage per row block
def test_vq_forward_at_the_edges_of_row_blocks_and_stages(T, n, m, cr, cc, b, r, dim):
    d = lopro.make_vq_desc(n, m, cr, cc, b, rank=r, dim=dim)
    _check(d, *_random_record(n, m, cr, cc, r, seed=n + T, dim=dim), T, seed=T)
