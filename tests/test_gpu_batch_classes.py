"""Batched builds of more parameter classes (pairs of leaf size and leaf range extra) than one pass of the
searches takes: every structure is the oracle's, and a failing set fails the call without a structure left."""
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


# 25 classes fill a pass, 26 need a second one, 58 a third; each class occurs twice
@pytest.mark.parametrize("classes", [25, 26, 58])
def test_structures_equal_the_oracles(rs, orc, classes):
    pairs = [(1 + i % 10, i // 10) for i in range(classes)]
    plan = [(leaf, extra, 7 + leaf, 300 + 11 * i) for i, (leaf, extra) in enumerate(pairs + pairs[::-1])]
    keys = [inputs.u64_keys(n, 400 + i) for i, (_, _, _, n) in enumerate(plan)]
    hs = rs.recsplit_build_batch([(device_keys(k), leaf, b, {"leaf_extra": extra})
                                  for k, (leaf, extra, b, _) in zip(keys, plan)])
    for h, k, (leaf, extra, b, _) in zip(hs, keys, plan):
        assert np.array_equal(rs.recsplit_serialize(h), orc.build_u64(k, leaf, b, threads=4, extra=extra)), (leaf, extra)
        rs.recsplit_free(h)


def test_failure_in_a_later_pass(rs):
    keys = [inputs.u64_keys(200, 700 + i) for i in range(30)]
    keys[28][5] = keys[28][9]  # a repeated key
    with pytest.raises(rs.RecSplitError) as e:
        rs.recsplit_build_batch([(device_keys(k), 2 + i % 10, 20, {"leaf_extra": i // 10})
                                 for i, k in enumerate(keys)])
    assert e.value.code == rs.E_DUPLICATE
