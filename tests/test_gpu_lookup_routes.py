"""Batches on either side of the sizes from which the buckets, and the codes, are
decoded first: values equal the oracle's, alone, as strings and batched."""
import numpy as np
import pytest

from paper_1910_06416_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LISTS, CODES = 1 << 18, 3 << 16  # queries from which the lists, and the codes, are decoded


@pytest.fixture(scope="module")
def rs():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1910_06416_gb300 import build
    build.build()
    import paper_1910_06416_gb300.recsplit as rs
    rs.lib()
    return rs


def gpu(a):
    return torch.from_numpy(a.view(np.int64)).cuda()


# buckets of less than two codes keep to the lists whatever the batch; l = 12, b = 2000
# has fixed parts and unary windows over several 64-bit words, 100 buckets are few
@pytest.mark.parametrize("leaf,b,n,extra", [(5, 5, 200001, 0), (12, 2000, 20000, 0), (8, 100, 400003, 0),
                                            (8, 100, 400003, 3), (2, 700, 30000, 0), (16, 100, 300, 0)])
def test_either_side_of_the_rules(rs, orc, leaf, b, n, extra):
    keys = inputs.u64_keys(n, 900 + leaf)
    blob = orc.build_u64(keys, leaf, b, threads=16, extra=extra)
    s = rs.Structure.deserialize(blob)
    st = s.stats()
    codes, nb = st["num_codes"], st["num_buckets"]
    pool = keys[inputs.query_indices(n, max(LISTS + nb // 2, CODES, 3 * codes // 2) + 2, 3)]
    pool[::8] = inputs.u64_keys(pool[::8].shape[0], 4)
    want = orc.lookup_u64(blob, pool)
    dev = gpu(pool)
    for at in (LISTS + nb // 2, max(CODES, (3 * codes + 1) // 2)):
        for q in (at - 1, at):
            out = torch.full((q,), -1, dtype=torch.int64, device="cuda")
            s.lookup_u64(dev[:q], out)
            assert np.array_equal(out.cpu().numpy().view(np.uint64), want[:q]), q


@pytest.mark.parametrize("q", [LISTS + 100, LISTS + 101])
def test_batched_lists(rs, orc, q):
    """200 buckets, too many codes for the batch to decode, and q one below and at the rule."""
    keys = [inputs.u64_keys(100000, 71), inputs.u64_keys(300000, 72)]
    blobs = [orc.build_u64(k, 2, 2000, threads=16, extra=e) for k, e in zip(keys, (0, 2))]
    hs = [rs.recsplit_deserialize(blob) for blob in blobs]
    ids = (np.arange(q) & 1).astype(np.uint32)
    qk = np.where(ids == 0, keys[0][inputs.query_indices(100000, q, 5)], keys[1][inputs.query_indices(300000, q, 6)])
    out = torch.empty(q, dtype=torch.int64, device="cuda")
    rs.recsplit_lookup_batch(hs, torch.from_numpy(ids.view(np.int32)).cuda(), gpu(qk), out)
    got = out.cpu().numpy().view(np.uint64)
    for i, blob in enumerate(blobs):
        assert np.array_equal(got[ids == i], orc.lookup_u64(blob, qk[ids == i])), i
    for h in hs:
        rs.recsplit_free(h)


@pytest.mark.parametrize("n", [76000000, 79000000])
def test_codes_beyond_the_cache(rs, n):
    """On either side of the size up to which the codes are decoded (2^24 places): the same
    values as batches too small to decode anything, and all different."""
    keys = inputs.device_splitmix64(11, n, device="cuda")
    s = rs.Structure.build_u64(keys, 8, 100)
    q = 3 * s.stats()["num_codes"] // 2 + 1
    out = torch.empty(q, dtype=torch.int64, device="cuda")
    s.lookup_u64(keys[:q], out)
    want = torch.empty_like(out)
    for a in range(0, q, 250000):
        s.lookup_u64(keys[a:min(q, a + 250000)], want[a:min(q, a + 250000)])
    assert torch.equal(out, want)
    assert int(out.min()) >= 0 and int(out.max()) < n
    seen = torch.zeros(n, dtype=torch.bool, device="cuda")
    seen[out] = True
    assert int(seen.sum()) == q
