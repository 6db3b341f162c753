"""Stage-by-stage parity at the sizes where the choice of tile shape changes and where a staging unit of the GEMM
epilogues (32 rows x 64 columns) is only partly inside the output."""
import pytest

from paper_2608_00916_b200 import synth
from gpu_util import Run, oracle_run
from test_gpu_parity import check_all

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E,k,f,seed", [
    (640, 192, 8, 2, 320, 71),    # 160 rows per expert: row GEMMs on pairs, weight gradients not
    (1024, 128, 8, 2, 192, 72),   # 256: row GEMMs on one-CTA tiles
    (1532, 192, 8, 2, 64, 73),    # 383: the last size with one-CTA weight gradients
    (1540, 320, 8, 2, 192, 74),   # 385: weight gradients on pairs, output rows and columns beyond the last full tile
    (1750, 128, 8, 2, 320, 75),   # 437: row GEMMs on pairs again
    (3080, 192, 8, 2, 128, 76),   # 770: dgrad-down on pairs as well
])
def test_tile_shape_boundaries(T, d, E, k, f, seed):
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), seed, x_std=1.0)
    ofw, obw = oracle_run(inp, k, 0.05)
    check_all(Run(inp, k), ofw, obw, 0.05)
