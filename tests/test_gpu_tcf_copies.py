"""TCF bulk calls with many copies of each key, far more than their blocks and
buckets hold: tables and statuses equal the oracle's on every path (the touched
blocks in one launch, over every block, by unit with buckets on either side of
what a thread takes), and the copies do not wait for one another."""
import numpy as np
import pytest

from paper_2212_09005_gb300 import workloads as W
from gpu_util import dev_u64, zeros_u8, host, first_diff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2212_09005_gb300 as gf

    gf.lib()
    return gf


def copies_of(seed, n, copies):
    keys = np.resize(np.repeat(W.uniform_keys(seed, (n + copies - 1) // copies), copies), n)
    np.random.default_rng(seed).shuffle(keys)
    return keys


# (log2 slots, tag bits, keys, copies of each, by unit)
@pytest.mark.parametrize("lg,f,n,copies,unit", [
    (18, 16, 5000, 7, False), (18, 16, 9000, 8, False), (18, 16, 9000, 9, False), (18, 8, 9000, 300, False),
    (18, 16, 12_000, 3000, False), (17, 16, 100_000, 100, False), (12, 16, 3000, 100, False), (12, 8, 3000, 40, False),
    (18, 16, 60_000, 100, True), (18, 16, 60_000, 511, True), (18, 16, 60_000, 513, True), (18, 8, 60_000, 100, True),
    (18, 16, 60_000, 6000, True), (22, 16, 200_000, 2, True),
])
def test_tables_equal_oracle(gf, oracle, lg, f, n, copies, unit):
    O, G = oracle.TCF(lg, f, seed=3), gf.TCF(lg, f, seed=3, max_batch=max(n, 1 << (lg - 1)))
    G.set_tuning(**({"tcf_path": gf.TCF_PATH_TILED} if unit else {}))
    base = W.uniform_keys(lg, 1 << (lg - 1))
    G.insert(dev_u64(base))
    O.insert(base)
    keys = copies_of(lg + n, n, copies)
    for op in ("insert", "remove", "insert", "remove"):
        st = zeros_u8(n)
        getattr(G, op)(dev_u64(keys), st)
        assert np.array_equal(host(st), getattr(O, op)(keys)), op
        assert first_diff(G.export(), O.export()) is None, op


@pytest.mark.parametrize("unit", [False, True])
def test_values_of_copies(gf, oracle, unit):
    import torch

    lg, n = 16, 20_000
    O, G = oracle.TCF(lg, 16, seed=4, value_bits=4), gf.TCF(lg, 16, seed=4, max_batch=n, value_bits=4)
    if unit:
        G.set_tuning(tcf_path=gf.TCF_PATH_TILED)
    keys = copies_of(5, n, 50)
    vals = np.random.default_rng(1).integers(0, 16, n).astype(np.uint8)
    st = zeros_u8(n)
    G.insert(dev_u64(keys), st, values=torch.from_numpy(vals).cuda())
    assert np.array_equal(host(st), O.insert(keys, values=vals))
    assert first_diff(G.export(), O.export()) is None
    st = zeros_u8(n)
    G.remove(dev_u64(keys), st)
    assert np.array_equal(host(st), O.remove(keys))
    assert first_diff(G.export(), O.export()) is None


@pytest.mark.parametrize("lg,n", [(24, 1 << 18), (26, 1 << 22)])
def test_time_of_a_hundred_copies(gf, lg, n):
    """Removes of a hundred copies of each key, by touched blocks and by unit: within
    twenty times the time of as many uniform keys; 21 and 37 times, where hot
    blocks fill the lanes of a few warps or wait for a CTA one after another."""
    import torch

    G = gf.TCF(lg, 16, seed=1, max_batch=n)
    best = {}
    for name, keys in (("uniform", W.uniform_keys(1, n)), ("copies", copies_of(2, n, 100))):
        k, t = dev_u64(keys), []
        for _ in range(4):
            G.insert(k)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            G.remove(k)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        best[name] = min(t)
    assert best["copies"] < 20 * best["uniform"], best
