"""Lookups of batches large enough to decode the codes first (and just below):
values equal the oracle's for members and for other keys, over buckets of a few
codes to buckets of tens of thousands, minimal and not, alone and batched."""
import numpy as np
import pytest

from paper_1910_06416_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [(8, 100, 30000, 0), (8, 100, 99, 0), (12, 2000, 9000, 0), (5, 700, 40000, 0), (3, 60000, 70000, 0),
         (8, 100, 20000, 2), (5, 2000, 9000, 3), (16, 300, 900, 0), (2, 9, 50000, 0)]


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


def queries(keys, q, seed):
    """Members with replacement, one in eight a random key."""
    out = keys[inputs.query_indices(keys.shape[0], q, seed)]
    out[::8] = inputs.u64_keys(out[::8].shape[0], seed + 1)
    return out


@pytest.mark.parametrize("leaf,b,n,extra", CASES)
def test_values_equal_the_oracles(rs, orc, leaf, b, n, extra):
    keys = inputs.u64_keys(n, 700 + leaf)
    blob = orc.build_u64(keys, leaf, b, threads=16, extra=extra)
    s = rs.Structure.deserialize(blob)
    codes = s.stats()["num_codes"]
    for q in (max(3 * codes, 1 << 18) - 1, max(3 * codes, 1 << 18)):
        qk = queries(keys, q, q)
        out = torch.full((q,), -1, dtype=torch.int64, device="cuda")
        s.lookup_u64(gpu(qk), out)
        assert np.array_equal(out.cpu().numpy().view(np.uint64), orc.lookup_u64(blob, qk)), q


def test_byte_strings(rs, orc):
    keys = inputs.byte_keys(20000, 5)
    blob = orc.build_bytes(keys.data, keys.offsets, 8, 100, threads=16)
    s = rs.Structure.deserialize(blob)
    qk = inputs.gather_byte_keys(keys, inputs.query_indices(20000, 300001, 9))
    out = torch.empty(300001, dtype=torch.int64, device="cuda")
    s.lookup_bytes(torch.from_numpy(qk.data).cuda(), gpu(qk.offsets), out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), orc.lookup_bytes(blob, qk.data, qk.offsets))


@pytest.mark.parametrize("extras", [(0,), (0, 2)])
def test_batched(rs, orc, extras):
    shapes = [(8, 100, 7000), (5, 2000, 9000), (8, 100, 0), (12, 700, 1500), (2, 5, 4000), (8, 100, 1)]
    blobs, sets, hs = [], [], []
    for i, (leaf, b, n) in enumerate(shapes):
        sets.append(inputs.u64_keys(n, 40 + i))
        blobs.append(orc.build_u64(sets[-1], leaf, b, threads=16, extra=extras[i % len(extras)]))
        hs.append(rs.recsplit_deserialize(blobs[-1]))
    q = 300007
    ids = (inputs.splitmix64(3, q) % np.uint64(len(hs) + 1)).astype(np.uint32)  # the last id is no structure
    keys = inputs.u64_keys(q, 4)
    for i, k in enumerate(sets):
        at = np.nonzero(ids == i)[0][::2]
        if k.shape[0]:
            keys[at] = k[inputs.query_indices(k.shape[0], at.shape[0], i)]
    out = torch.empty(q, dtype=torch.int64, device="cuda")
    rs.recsplit_lookup_batch(hs, torch.from_numpy(ids.view(np.int32)).cuda(), gpu(keys), out)
    got = out.cpu().numpy().view(np.uint64)
    assert (got[ids == len(hs)] == np.uint64(2**64 - 1)).all()
    for i, blob in enumerate(blobs):
        at = ids == i
        assert np.array_equal(got[at], orc.lookup_u64(blob, keys[at])), i
    for h in hs:
        rs.recsplit_free(h)
