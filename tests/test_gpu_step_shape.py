"""lbm_info reports the thread blocks of the step kernel that a box takes."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_09041_gb300 import lbm as L  # noqa: E402


@pytest.mark.parametrize("lattice,precision,shape,params,block", [
    ("d2q9", "fp64", (64, 64, 1), {}, (64, 1)),                        # two warps per 32 nodes
    ("d2q9", "fp64", (32, 448, 1), {}, (64, 1)),
    ("d2q9", "fp64", (32, 449, 1), {}, (32, 1)),                       # one
    ("d2q9", "fp64", (64, 64, 1), {"omega_bulk": 1.1}, (32, 1)),
    ("d2q9", "fp64", (64, 64, 1), {"index64": 1}, (32, 1)),
    ("d2q9", "fp64", (64, 64, 1), {"block_x": 128}, (128, 2)),
    ("d2q9", "fp16s", (192, 1600, 1), {}, (32, 4)),                    # pairs
    ("d2q9", "fp16s", (192, 1600, 1), {"omega_bulk": 1.1}, (64, 2)),   # one node per thread
    ("d2q9", "fp16s", (160, 1900, 1), {}, (64, 2)),
    ("d2q9", "fp32", (192, 1600, 1), {}, (64, 2)),
    ("d2q9", "fp32", (96, 100, 1), {}, (96, 2)),
    ("d3q27", "fp16s", (128, 256, 192), {}, (64, 1)),                  # pairs
    ("d3q27", "fp16s", (128, 256, 192), {"rows3d": 1}, (128, 1)),      # one node per thread
    ("d3q27", "fp32", (128, 256, 192), {}, (128, 1))])
def test_info_reports_the_blocks_of_the_step(lattice, precision, shape, params, block):
    lat = L.Lattice(lattice, *shape, Ra=1e4, precision=precision)
    for k, v in params.items():
        lat.set_param(k, v)
    info = lat.info()
    lat.close()
    assert (info.block_x, info.block_y) == block
