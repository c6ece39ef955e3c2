"""The rules by which a launch takes one kernel or another, at the sizes where the choice or a tile's edge matters."""
import numpy as np
import pytest
import torch

from paper_2305_09887_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def util():
    import gpu_util
    return gpu_util


def _workload(n, edges, dims, seed):
    w = inputs.tiny()
    w.graph = inputs.uniform_graph(n, edges, seed)
    w.dims = dims
    w.y = inputs.uniform_labels(n, dims[-1], seed + 1)
    w.X = inputs.normal_features(n, dims[0], seed + 2)
    w.params0 = inputs.xavier_params(dims, seed + 3)
    return w


# enough 128-row tiles for every SM and K >= 384: the products of the second layer go to pairs of blocks.  Parts of
# about 850 and 300 rows: the last 256-row tile of a part lies half, wholly or not at all past its end.
@pytest.mark.parametrize("n, M, dims, parts, gemm_dtype", [
    (19_600, 23, (70, 200, 200, 5), (0, 7, 22), 0),     # 224-column tiles over 200 columns
    (19_600, 23, (70, 200, 200, 5), (3,), 1),
    (19_000, 60, (20, 200, 136, 7), (0, 31, 59), 0),    # two or three 128-row tiles a part
    (19_600, 23, (40, 520, 520, 3), (5,), 0),           # three column tiles of 192
])
def test_products_on_pairs_of_blocks(util, n, M, dims, parts, gemm_dtype):
    w = _workload(n, 3 * n, dims, 11)
    util.check_one_step(w, M=M, gemm_dtype=gemm_dtype, only_parts=parts, gradients_against_plain=gemm_dtype == 0)
