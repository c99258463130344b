"""In-place GQF updates, a warp or a thread per region: tables, statuses and
the counters' growth equal the oracle's at the sizes where the choice of
kernel or of region changes, at short and at long clusters."""
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


# (q, r, load, groups of the update): regions of one to many words, the whole
# table one region, the edges between the warp and the thread kernels
@pytest.mark.parametrize("q,r,load,m", [(6, 8, 0.5, 1), (8, 8, 0.9, 3), (12, 8, 0.85, 1), (14, 16, 0.95, 100),
                                        (16, 8, 0.93, 37), (18, 8, 0.85, 1000), (18, 16, 0.9, 2048),
                                        (19, 8, 0.4, 1 << 14), (20, 8, 0.8, (1 << 14) + 1),
                                        (23, 8, 0.5, (1 << 18) + 1)])
def test_updates_equal_oracle(gf, oracle, q, r, load, m):
    base = W.uniform_keys(100 + q, int(load * (1 << q)))
    fresh = W.uniform_keys(200 + q, m)
    again = np.concatenate([base[: m // 2 + 1], fresh[: m // 2]])  # counters grow by 1, then by 2
    O, G = oracle.GQF(q, r, seed=q), gf.GQF(q, r, seed=q, max_batch=max(len(base), 4 * m + 4))
    G.set_tuning(gqf_region_groups=8)  # in place wherever it can
    G.insert(dev_u64(base))
    O.insert(base)
    steps = [("insert", fresh), ("insert", again), ("insert", np.concatenate([again, again])),
             ("remove", np.concatenate([again, fresh])), ("remove", W.uniform_keys(300 + q, m)), ("remove", again)]
    for op, keys in steps:
        st = zeros_u8(len(keys))
        getattr(G, op)(dev_u64(keys), st)
        assert np.array_equal(host(st), getattr(O, op)(keys)), op
        d = first_diff(G.export(), O.export())
        assert d is None, (op, d, G.stats()["status_word"])


def test_removed_runs_and_counters_of_several_digits(gf, oracle):
    q, r = 10, 8
    base = W.uniform_keys(41, 600)
    hot = np.repeat(base[:4], [300, 70000, 2, 1])
    O, G = oracle.GQF(q, r, seed=3), gf.GQF(q, r, seed=3, max_batch=1 << 17)
    for op, keys in [("insert", base), ("insert", hot[:5]), ("insert", base[:1].repeat(260)), ("insert", hot),
                     ("remove", base[:2].repeat(3)), ("remove", base[:1].repeat(300)), ("remove", base[1:3]),
                     ("remove", base[::2])]:
        st = zeros_u8(len(keys))
        getattr(G, op)(dev_u64(keys), st)
        assert np.array_equal(host(st), getattr(O, op)(keys)), op
        d = first_diff(G.export(), O.export())
        assert d is None, (op, d, G.stats()["status_word"])
