"""Batches that one CTA takes whole: tables, statuses and counts equal the
oracle's at the edges of their range, with repeated and equal keys, full
tables, values and groups."""
import numpy as np
import pytest

from paper_2212_09005_gb300 import workloads as W
from gpu_util import dev_u64, zeros_u8, zeros_u64, host, first_diff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2212_09005_gb300 as gf

    gf.lib()
    return gf


def step(F, O, op, keys, status=True, **kw):
    st = zeros_u8(len(keys)) + 7
    if "values" in kw:
        import torch

        F.insert(dev_u64(keys), st, values=torch.from_numpy(kw["values"]).cuda())
        want = O.insert(keys, values=kw["values"])
    else:
        getattr(F, op)(dev_u64(keys), st if status else None)
        want = getattr(O, op)(keys)
    if status:
        assert np.array_equal(host(st), want), op
    d = first_diff(F.export(), O.export())
    assert d is None, (op, len(keys), d)


SIZES = [1, 2, 33, 1000, 2047, 2048, 2049]


@pytest.mark.parametrize("lg,f", [(6, 16), (11, 16), (13, 16), (20, 16), (7, 8), (13, 8)])
def test_tcf_equals_oracle(gf, oracle, lg, f):
    F, O = gf.TCF(lg, f, seed=lg, max_batch=4096), oracle.TCF(lg, f, seed=lg)
    keys = W.uniform_keys(lg, sum(SIZES))
    at = 0
    for n in SIZES:  # tables of 2^6 and 2^7 slots fill up: backing buckets, FULL
        batch = np.concatenate([keys[at:at + n - n // 4], keys[at:at + n // 4]])  # a quarter repeated
        at += n
        step(F, O, "insert", batch, status=n != 33)
        step(F, O, "remove", batch[::3])
    step(F, O, "insert", np.repeat(keys[:1], 2048))  # one hot block
    step(F, O, "remove", np.repeat(keys[:2], 900))


def test_tcf_values_equal_oracle(gf, oracle):
    F, O = gf.TCF(11, 16, seed=5, max_batch=2048, value_bits=4), oracle.TCF(11, 16, seed=5, value_bits=4)
    keys = W.uniform_keys(5, 1900)
    for part in (keys[:1100], keys[1000:]):
        step(F, O, "insert", part, values=(part & np.uint64(15)).astype(np.uint8))
    step(F, O, "remove", np.concatenate([keys[::2], keys[::2]]))


def test_tcf_group_equals_oracle(gf, oracle):
    import torch

    logs, seeds, sizes = [8, 12, 6, 10], [1, 2, 3, 4], [200, 900, 70, 0]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    keys = W.uniform_keys(9, int(off[-1]))
    G = gf.FilterGroup(gf.FILTER_TCF, logs, 16, seeds, max_total=len(keys))
    refs = [oracle.TCF(lg, 16, seed=s) for lg, s in zip(logs, seeds)]
    for op in ("insert", "insert", "remove"):
        st = zeros_u8(len(keys))
        getattr(G, op)(torch.from_numpy(off).cuda(), dev_u64(keys), st)
        want = [getattr(r, op)(keys[off[m]:off[m + 1]]) for m, r in enumerate(refs)]
        assert np.array_equal(host(st), np.concatenate(want)), op
        for m, r in enumerate(refs):
            assert first_diff(G.export(m), r.export()) is None, (op, m)


@pytest.mark.parametrize("q,r", [(6, 8), (12, 8), (17, 16), (20, 8)])
def test_gqf_equals_oracle(gf, oracle, q, r):
    F, O = gf.GQF(q, r, seed=q, max_batch=8192), oracle.GQF(q, r, seed=q)
    keys = W.uniform_keys(50 + q, 9000)
    at = 0
    for n in (1, 2, 31, 1000, 4095, 4096, 4097):
        k = min(n - n // 4, (1 << q) // 6 + 1)  # room for all of them
        batch = np.resize(keys[at:at + k], n)   # repeated in order
        at = (at + k) % 4500
        step(F, O, "insert", batch, status=n != 31)
        step(F, O, "remove", np.concatenate([batch[::2], keys[-7:]]))
    hot = np.repeat(keys[:1], 4096)
    step(F, O, "insert", hot)
    step(F, O, "insert", W.zipf_keys(3, 4000, 1.0, 1 << 12)[: 1 << min(q - 1, 12)])
    c = zeros_u64(1)
    F.count(dev_u64(keys[:1]), c)
    assert np.array_equal(host(c), O.count(keys[:1]))


def test_gqf_counts_ride_along(gf, oracle):
    import torch

    keys = W.uniform_keys(77, 4096)
    counts = (1 + (keys & np.uint64(3))).astype(np.uint32)
    for with_status in (False, True):
        F, O = gf.GQF(15, 8, seed=2, max_batch=4096), oracle.GQF(15, 8, seed=2)
        for lo, hi in ((0, 1000), (500, 4096)):
            st = zeros_u8(hi - lo) if with_status else None
            F.insert_counts(dev_u64(keys[lo:hi]), torch.from_numpy(counts[lo:hi].view(np.int32)).cuda(), st)
            O.insert_counts(keys[lo:hi], counts[lo:hi])
            assert first_diff(F.export(), O.export()) is None
