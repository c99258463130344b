"""GQF batches of many copies of few keys on large tables: updated in place, as
their number of distinct fingerprints says, not merged as their number of keys
would have it; tables equal the oracle's."""
import numpy as np
import pytest

from paper_2212_09005_gb300 import workloads as W
from gpu_util import dev_u64, first_diff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2212_09005_gb300 as gf

    gf.lib()
    return gf


# (q, keys, distinct ones, bound set by the caller, in place): the sort leaves
# batches above four times the most that goes in place in units
@pytest.mark.parametrize("q,n,distinct,bound,in_place", [
    (24, (1 << 18) + 1, 1, 0, True),
    (24, 1 << 19, 1000, 0, True),
    (24, 1 << 23, 1 << 16, 0, True),             # as many as go in place
    (24, 1 << 23, (1 << 16) + 1, 0, False),
    (24, 1 << 24, 1000, 0, True),
    (16, 9000, 100, 8, True),                    # a small table, by the caller's bound
])
def test_copies_of_few_keys(gf, oracle, q, n, distinct, bound, in_place):
    O, G = oracle.GQF(q, 8, seed=2), gf.GQF(q, 8, seed=2, max_batch=n)
    if bound:
        G.set_tuning(gqf_region_groups=bound)
    keys = W.uniform_keys(q, 2 * distinct + 16)
    keys = keys[np.unique(O.fingerprints(keys), return_index=True)[1]][:distinct]
    batch = np.concatenate([keys, np.resize(keys, n - distinct)])
    np.random.default_rng(n).shuffle(batch)
    rest = W.uniform_keys(q + 1, min(n, (1 << q) // 3))
    G.insert(dev_u64(rest))
    O.insert(rest)
    for op, ks in (("insert", batch), ("remove", batch[:n - n // 16]), ("insert", batch)):
        ks_d = dev_u64(ks)
        gf.trace_reset()
        gf.trace_enable(True)
        try:
            getattr(G, op)(ks_d)
            names = set(gf.trace_summary())
        finally:
            gf.trace_enable(False)
        getattr(O, op)(ks)
        assert first_diff(G.export(), O.export()) is None, op
        if len(ks) == n:
            assert (f"gqf_{'insert' if op == 'insert' else 'delete'}_phase" in names) == in_place, (op, names)
    assert G.stats()["status_word"] == 0
