"""Which batches decode the buckets, and the codes, of their structures first, seen from the number of kernels
that a call launches (two with a decode, one without), and the values on either side against the oracle's: many
structures with empty ones and ids of none among them, one query below each rule and at it, and strings over a
structure with a leaf range extra.

The rules: over several structures nothing is decoded below buckets / 2 + 2^18 queries; from there on the
codes are, if there are at least 1.5 queries per code and two codes per bucket, else the lists.  One structure
decodes its codes from 3 * 2^16 queries on under the same two conditions."""
import numpy as np
import pytest

from paper_1910_06416_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LISTS, CODES = 1 << 18, 3 << 16


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
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def counted(rs, call):
    before = rs.recsplit_launch_count()
    call()
    return rs.recsplit_launch_count() - before


# the same structures with few codes (one per six keys: the codes are decoded) and with many (the lists alone)
@pytest.mark.parametrize("leaf", [2, 8])
@pytest.mark.parametrize("extras", [(0,), (0, 3)])
def test_many_structures(rs, orc, leaf, extras):
    sizes = [0, 1] + [3000 + 311 * i for i in range(40)] + [0, 2, 17]
    sets = [inputs.u64_keys(n, 1000 + i) for i, n in enumerate(sizes)]
    blobs = [orc.build_u64(k, leaf, 200, threads=16, extra=extras[i % len(extras)]) for i, k in enumerate(sets)]
    hs = [rs.recsplit_deserialize(b) for b in blobs]
    stats = [rs.recsplit_stats(h) for h in hs]
    buckets, codes = (sum(s[k] for s in stats) for k in ("num_buckets", "num_codes"))
    rule = LISTS + buckets // 2
    assert (2 * rule >= 3 * codes) == (leaf == 8) and codes >= 2 * buckets
    ids = (inputs.splitmix64(5, rule) % np.uint64(len(hs) + 2)).astype(np.uint32)
    ids[ids == len(hs) + 1] = 0xFFFFFFFF  # the last two ids are no structure
    keys = inputs.u64_keys(rule, 6)
    want = np.full(rule, np.iinfo(np.uint64).max, dtype=np.uint64)
    for i, (k, blob) in enumerate(zip(sets, blobs)):
        at = np.nonzero(ids == i)[0]
        if k.shape[0]:
            keys[at[::2]] = k[inputs.query_indices(k.shape[0], at[::2].shape[0], i)]  # members, and other keys
        want[at] = orc.lookup_u64(blob, keys[at])
    dids, dkeys = torch.from_numpy(ids.view(np.int32)).cuda(), gpu(keys)
    for q, launches in ((rule - 1, 1), (rule, 2)):
        out = torch.empty(q, dtype=torch.int64, device="cuda")
        assert counted(rs, lambda: rs.recsplit_lookup_batch(hs, dids[:q], dkeys[:q], out)) == launches
        assert np.array_equal(out.cpu().numpy().view(np.uint64), want[:q]), q
    hout = np.zeros(rule, dtype=np.uint64)
    rs.recsplit_lookup_batch(hs, ids, keys, hout)
    assert np.array_equal(hout, want)
    for h in hs:
        rs.recsplit_free(h)


@pytest.mark.parametrize("extra", [0, 2])
def test_strings_with_decoded_codes(rs, orc, extra):
    keys = inputs.byte_keys(20000, 15)
    blob = orc.build_bytes(keys.data, keys.offsets, 8, 100, threads=16, extra=extra)
    s = rs.Structure.deserialize(blob)
    for q, launches in ((CODES - 1, 1), (CODES, 2), (300001, 2)):
        qk = inputs.gather_byte_keys(keys, inputs.query_indices(20000, q, 16))
        data, offsets = torch.from_numpy(qk.data).cuda(), gpu(qk.offsets)
        out = torch.empty(q, dtype=torch.int64, device="cuda")
        assert counted(rs, lambda: s.lookup_bytes(data, offsets, out)) == launches
        assert np.array_equal(out.cpu().numpy().view(np.uint64), orc.lookup_bytes(blob, qk.data, qk.offsets)), q
