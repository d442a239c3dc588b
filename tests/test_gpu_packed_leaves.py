"""Full leaves of 4 to 10 keys, searched several to a warp: the structure is
the oracle's from one leaf in all (one leaf per warp, 32 lanes on it) to more
than four per warp of the grid (eight lanes each), at every number of indices
per lane, and repeated keys are still found."""
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


@pytest.mark.parametrize("leaf", range(4, 11))
def test_structures_equal_the_oracles(rs, orc, leaf):
    saved = rs.recsplit_get_tuning(leaf)
    # one leaf; a few; about two per warp of a 608-block grid; more than four
    for n, spl in ((leaf, 1), (23 * leaf + 3, 8), (12000 * leaf, 2), (23000 * leaf + 5, 4)):
        keys = inputs.u64_keys(n, 300 + leaf)
        ref = orc.build_u64(keys, leaf, 100, threads=16)
        try:
            rs.recsplit_set_tuning(leaf, dict(saved, leaf_two_phase=1, leaf_warps=1, leaf_seeds_per_lane=spl))
            got = rs.Structure.build_u64(device_keys(keys), leaf, 100).serialize()
        finally:
            rs.recsplit_set_tuning(leaf, saved)
        assert np.array_equal(got, ref), (leaf, n, spl)


@pytest.mark.parametrize("leaf,n", [(4, 900), (8, 900), (8, 200000), (10, 900)])
def test_repeated_key_in_a_leaf_is_reported(rs, leaf, n):
    keys = inputs.u64_keys(n, 9)
    keys[n // 2] = keys[0]
    with pytest.raises(rs.RecSplitError) as e:
        rs.Structure.build_u64(device_keys(keys), leaf, 100)
    assert e.value.code == rs.E_DUPLICATE
