"""Builds whose number of buckets lies at the edges of the one-launch scans'
tiles (1024 buckets for the keys and codes, 2048 for the bit lengths) and beyond
one look-back window of 32 tiles, with a lane and with a warp per bucket for the
codes, alone and in a batch: word for word the oracle's structures."""
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


@pytest.mark.parametrize("buckets", [1, 2, 1023, 1024, 1025, 2047, 2048, 2049, 33 * 1024 + 5, 70001])
def test_structures_equal_the_oracles(rs, orc, buckets):
    for leaf, b, extra in ((2, 1, 0), (4, 3, 0), (3, 2, 1), (2, 40, 0)):
        if buckets * b > 300000:
            continue
        keys = inputs.u64_keys(buckets * b, 60 + leaf)
        got = rs.Structure.build_perfect_u64(device_keys(keys), leaf, b, extra).serialize()
        assert np.array_equal(got, orc.build_u64(keys, leaf, b, threads=16, extra=extra)), (leaf, b, extra)


def test_batch_of_lane_and_warp_buckets(rs, orc):
    shapes = [(2, 1, 1000), (8, 2000, 5000), (4, 3, 0), (5, 5, 5000), (3, 300, 1), (8, 100, 31), (2, 40, 70000)]
    keys = [inputs.u64_keys(n, 80 + i) for i, (_, _, n) in enumerate(shapes)]
    hs = rs.recsplit_build_batch([(device_keys(k), leaf, b) for k, (leaf, b, _) in zip(keys, shapes)])
    for h, k, (leaf, b, _) in zip(hs, keys, shapes):
        assert np.array_equal(rs.recsplit_serialize(h), orc.build_u64(k, leaf, b, threads=16)), (leaf, b)
        rs.recsplit_free(h)
