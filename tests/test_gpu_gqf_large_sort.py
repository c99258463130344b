"""The sort and reduction of large batches without statuses: tables equal the
oracle's at the sizes where the number of passes changes, with keys so hot
that their unit goes through the hash table or is squeezed first, with equal
keys only, and with fingerprints crowded into a sliver of their range."""
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


def check(gf, oracle, q, r, seed, steps):
    G = gf.GQF(q, r, seed=seed, max_batch=max(len(k) for _, k in steps))
    O = oracle.GQF(q, r, seed=seed)
    for op, keys in steps:
        getattr(G, op)(dev_u64(keys))
        getattr(O, op)(keys)
        d = first_diff(G.export(), O.export())
        assert d is None, (op, len(keys), d)
    assert G.stats()["status_word"] == 0
    return G, O


# one pass up to 2^20 keys (512 units of 2048), two above; 31 bits below the units' at most
@pytest.mark.parametrize("q,r,n", [(13, 8, 4097), (16, 8, 4 * 2048 + 1), (16, 16, 40_001), (21, 8, 1 << 20),
                                   (21, 8, (1 << 20) + 1), (22, 16, 1_500_007), (9, 8, 5000), (28, 16, 5000)])
def test_uniform_batches(gf, oracle, q, r, n):
    keys = W.uniform_keys(q + n, n)
    if q == 9:
        keys = np.resize(keys[:40], n)  # few values, many copies
    check(gf, oracle, q, r, 7, [("insert", keys[: n - 1]), ("remove", keys[::2]), ("insert", keys[::2])])


@pytest.mark.parametrize("copies", [4095, 4097, 16_384, 16_385, 300_000])
def test_hot_keys(gf, oracle, copies):
    base = W.uniform_keys(3, 20_000)
    keys = np.concatenate([base, np.repeat(base[5:8], [copies, 33, 2500]), base[:100]])
    rng = np.random.default_rng(copies)
    rng.shuffle(keys)
    G, O = check(gf, oracle, 16, 8, 11, [("insert", keys), ("remove", keys[::3]), ("insert", keys[::2])])
    c = zeros_u64(100)
    G.count(dev_u64(base[:100]), c)
    assert np.array_equal(host(c), O.count(base[:100]))


def test_equal_keys_only(gf, oracle):
    keys = np.full(50_000, 12345, np.uint64)
    check(gf, oracle, 12, 8, 1, [("insert", keys), ("insert", keys[:5000]), ("remove", keys[:20_000])])


def test_zipf_two_passes(gf, oracle):
    keys = W.zipf_keys(5, 3_000_001, 1.0, 1 << 24)
    check(gf, oracle, 22, 8, 3, [("insert", keys), ("remove", keys[::4])])


def test_fingerprints_of_one_sliver(gf, oracle):
    """Distinct fingerprints all in one unit: more than a chunk's table holds,
    so the chunks stay raw and the unit takes several ranges."""
    q, r, n = 20, 8, 20_000
    G = gf.GQF(q, r, seed=5, max_batch=2 * n)
    fps = np.arange(n, dtype=np.uint64) * np.uint64(419) + np.uint64(1 << 25)  # 2^23 of 2^28 values
    keys = zeros_u64(n)
    G.keys_of(dev_u64(fps), keys)
    keys = host(keys)
    O = oracle.GQF(q, r, seed=5)
    for op, batch in (("insert", keys), ("insert", np.concatenate([keys[::5], keys[::7]])), ("remove", keys[::2])):
        getattr(G, op)(dev_u64(batch))
        getattr(O, op)(batch)
        d = first_diff(G.export(), O.export())
        assert d is None, (op, d)


# (q, r, n): the batch index below the fingerprint, up to exactly 64 bits, and beside it above
@pytest.mark.parametrize("q,r,n", [(13, 8, 4097), (18, 16, 70001), (26, 16, 1 << 22), (26, 16, (1 << 22) + 1)])
def test_statuses_ride_with_the_sort(gf, oracle, q, r, n):
    base = W.uniform_keys(50 + q, n - n // 8)
    keys = np.concatenate([base, base[: n - len(base)]])  # some of them twice
    np.random.default_rng(n).shuffle(keys)
    O, G = oracle.GQF(q, r, seed=1), gf.GQF(q, r, seed=1, max_batch=n)
    gone = np.concatenate([keys[: n // 2], keys[: n // 4], W.uniform_keys(51, n - n // 2 - n // 4)])
    for op, ks in (("insert", keys), ("remove", gone)):
        st = zeros_u8(n)
        getattr(G, op)(dev_u64(ks), st)
        assert np.array_equal(host(st), getattr(O, op)(ks)), op
    assert first_diff(G.export(), O.export()) is None


@pytest.mark.parametrize("q,n", [(11, 9000), (12, 14_001), (13, 3 * 8192)])
def test_statuses_of_batches_that_do_not_fit(gf, oracle, q, n):
    """Inserts carry no indices until some group does not fit: the keys past the kept prefix are FULL."""
    keys = W.uniform_keys(70 + q, n)
    keys = np.concatenate([keys, keys[:500]])
    O, G = oracle.GQF(q, 16, seed=1), gf.GQF(q, 16, seed=1, max_batch=len(keys))
    for part in (keys[: n // 8], keys):
        st = zeros_u8(len(part))
        G.insert(dev_u64(part), st)
        want = O.insert(part)
        assert np.array_equal(host(st), want)
        assert first_diff(G.export(), O.export()) is None
    assert (want != 0).any()
