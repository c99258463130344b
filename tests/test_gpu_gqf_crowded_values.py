"""GQF batches whose fingerprints are not spread: a stretch of a filter's
enumeration, inserted into and removed from another of its geometry. Tables
equal the oracle's on every way such a batch can take (in place with the
groups' number read or not, merged from one list or from units), and it takes
about the time of a batch of other keys."""
import numpy as np
import pytest

from paper_2212_09005_gb300 import workloads as W
from gpu_util import dev_u64, zeros_u64, host, first_diff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2212_09005_gb300 as gf

    gf.lib()
    return gf


def keys_of(G, fps):
    keys = zeros_u64(len(fps))
    G.keys_of(dev_u64(fps), keys)
    return host(keys)


# (q, r, stored keys, first and number of the stretch)
@pytest.mark.parametrize("q,r,stored,first,n", [
    (18, 8, 200_000, 90_000, 1 << 16),      # units, merged
    (18, 8, 200_000, 0, 12_001),            # one list, merged
    (22, 8, 1_000_000, 999_000 - 6000, 6000),  # the load is asked for
    (24, 8, 1_000_000, 400_000, 10_000),    # in place, unread
    (24, 8, 1_000_000, 400_000, 50_000),    # in place
    (24, 8, 4_000_000, 1_000_001, 300_000),  # units on a large table
])
def test_stretches_of_an_enumeration(gf, oracle, q, r, stored, first, n):
    O = oracle.GQF(q, r, seed=9)
    G = gf.GQF(q, r, seed=9, max_batch=stored)
    fps = np.unique(O.fingerprints(W.uniform_keys(q, stored)))
    keys = keys_of(G, fps[first:first + n])
    twice = np.concatenate([keys, keys[::16]])
    for op, batch in (("insert", keys), ("remove", twice), ("insert", twice), ("remove", keys[1::2])):
        getattr(G, op)(dev_u64(batch))
        getattr(O, op)(batch)
        d = first_diff(G.export(), O.export())
        assert d is None, (op, d)
    assert G.stats()["status_word"] == 0


def test_time_does_not_depend_on_the_values(gf, oracle):
    """2^16 distinct fingerprints of one of 32 units of 2^31 values: within ten
    times the time of as many uniform ones. A CTA that reads its unit once for
    every range of values that its table holds took 500 times as long."""
    import torch

    n = 1 << 16
    G = gf.GQF(28, 8, seed=3, max_batch=n)
    fps = np.arange(n, dtype=np.uint64) * np.uint64(1 << 15) + np.uint64(1 << 33)
    others = W.uniform_keys(1, n)
    crowded, uniform = dev_u64(keys_of(G, fps)), dev_u64(others)

    def best(op, back, keys):
        t = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            op(keys)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
            back(keys)
        return min(t)

    for op, back in ((G.insert, G.remove), (G.remove, G.insert)):
        if op == G.remove:
            G.insert(crowded)
            G.insert(uniform)
        t = {name: best(op, back, keys) for name, keys in (("crowded", crowded), ("uniform", uniform))}
        assert t["crowded"] < 10 * t["uniform"], (op.__name__, t)
    c = zeros_u64(n)
    G.count(crowded, c)
    assert np.array_equal(host(c), 1 + np.isin(fps, oracle.GQF(28, 8, seed=3).fingerprints(others)))
