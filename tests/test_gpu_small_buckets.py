"""Builds whose buckets are all smaller than the leaf size: there is no full leaf, and the kernels of
full leaves, which read the node table's entry of the leaf size, are not launched (the table ends at the
largest bucket)."""
import numpy as np
import pytest

from paper_1910_06416_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1910_06416_gb300 import build
    build.build()
    import paper_1910_06416_gb300.recsplit as rs
    rs.lib()
    return rs


def device_keys(keys):
    return torch.from_numpy(keys.view(np.int64)).cuda()


@pytest.mark.parametrize("leaf", [4, 8, 12, 16, 24])
@pytest.mark.parametrize("extra", [0, 2])
def test_structures_equal_the_oracles(rs, orc, leaf, extra):
    for n, b in ((1, 100), (2, 100), (min(leaf - 1, 14), 65535), (50, 1), (3000, 1), (40 * leaf, leaf // 4)):
        keys = inputs.u64_keys(n, 910 + leaf)
        got = rs.Structure.build_perfect_u64(device_keys(keys), leaf, b, extra).serialize()
        assert np.array_equal(got, orc.build_u64(keys, leaf, b, threads=16, extra=extra)), (n, b)


@pytest.mark.parametrize("leaf", [4, 8, 12, 16])
def test_leaf_launches(rs, leaf):
    """One bucket of n keys, n at most the leaf size: no leaf launch at n = 1, that of partial leaves
    from 2 keys, and that of full leaves at the leaf size."""
    def launches(n):
        before = rs.recsplit_launch_count()
        rs.Structure.build_u64(device_keys(inputs.u64_keys(n, 33)), leaf, 65535).free()
        return rs.recsplit_launch_count() - before

    one = launches(1)
    assert [launches(n) - one for n in (2, leaf - 1, leaf)] == [1, 1, 2]
