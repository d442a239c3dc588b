"""Split searches at the edges of their count modes, word for word against the
oracle: four equal parts with and without a last word of fewer than 16 keys,
thresholds with and without four lanes per index, nodes staged in shared
memory and nodes read from global memory, one node in all (a whole CTA on it)
and more nodes than the grid has warps."""
import numpy as np
import pytest

from paper_1910_06416_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    (8, 32, 32), (8, 33, 33), (8, 100, 97), (8, 32, 170000),       # 32 = 4 x 8; 33 = 2 parts; 96 + 1
    (9, 36, 36), (9, 36, 20000), (10, 40, 39), (10, 40, 20000),    # 36 = 4 x 9, 40 = 4 x 10: a short last word
    (12, 240, 240), (12, 240, 7000),                               # 240 = 4 x 60
    (7, 21, 30000), (7, 63, 30000), (5, 15, 40000), (3, 6, 60000),  # three equal parts, two equal parts
    (6, 6, 50000), (4, 5, 150000), (2, 3, 20000),                  # few trials, few keys
    (16, 17, 2000), (16, 30, 2000), (16, 48, 1500),
    (8, 700, 20000), (5, 20000, 40000), (8, 20000, 20000),         # m above the staged keys of a CTA
]


@pytest.mark.parametrize("leaf,b,n", CASES)
def test_structures_equal_the_oracles(orc, leaf, b, n):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_1910_06416_gb300.recsplit as rs
    keys = inputs.u64_keys(n, 500 + leaf)
    got = rs.Structure.build_u64(torch.from_numpy(keys.view(np.int64)).cuda(), leaf, b).serialize()
    assert np.array_equal(got, orc.build_u64(keys, leaf, b, threads=16))
