"""Full leaves of 4 to 8 keys just above the number from which several share a warp (eight per SM): one, two and
four leaves per warp, at every number of indices per lane, word for word the oracle's structures."""
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


@pytest.mark.parametrize("leaf", range(4, 9))
@pytest.mark.parametrize("extra", [0, 1])
def test_structures_equal_the_oracles(rs, orc, leaf, extra):
    warps = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 4  # of the packed kernel's grid
    saved = rs.recsplit_get_tuning(leaf)
    # leaves (at most): the first number that is packed, fewer than two per warp, two to four, more
    for leaves, spl in ((warps // 4 + 1, 1), (warps // 4 + 7, 8), (warps, 4), (4 * warps, 2), (7 * warps + 3, 8)):
        keys = inputs.u64_keys(leaves * leaf, 820 + leaf)
        ref = orc.build_u64(keys, leaf, 100, threads=16, extra=extra)
        dev = torch.from_numpy(keys.view(np.int64)).cuda()
        try:
            rs.recsplit_set_tuning(leaf, dict(saved, leaf_two_phase=1, leaf_warps=1, leaf_seeds_per_lane=spl))
            got = rs.Structure.build_perfect_u64(dev, leaf, 100, extra).serialize()
        finally:
            rs.recsplit_set_tuning(leaf, saved)
        assert np.array_equal(got, ref), (leaves, spl)
