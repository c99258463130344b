"""GQF inserts in place whose groups take several slots each (counters of one
to several digits): tables equal the oracle's, and few keys of many slots do not
wait for one another."""
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


def counts_of(c, m):
    import torch

    return torch.from_numpy(np.resize(np.asarray(c, np.int32), m)).cuda()


# counts: one slot each, one or three, three to six
@pytest.mark.parametrize("counts", [[1], [1, 2], [1, 2, 2], [2, 300, 70_000, 2_000_000]])
@pytest.mark.parametrize("q,r,load,m", [(9, 8, 0.3, 3), (14, 16, 0.5, 200), (16, 8, 0.4, 900), (16, 8, 0.85, 500)])
def test_tables_equal_oracle(gf, oracle, q, r, load, m, counts):
    base = W.uniform_keys(q, int(load * (1 << q)))
    keys = np.concatenate([W.uniform_keys(q + 7, m - m // 3), base[: m // 3]])
    O, G = oracle.GQF(q, r, seed=q), gf.GQF(q, r, seed=q, max_batch=max(len(base), 2 * m))
    G.set_tuning(gqf_region_groups=8)
    G.insert(dev_u64(base))
    O.insert(base)
    c = np.resize(np.asarray(counts, np.uint32), m)
    for _ in range(2):
        st = zeros_u8(m)
        G.insert_counts(dev_u64(keys), counts_of(counts, m), st)
        assert np.array_equal(host(st), O.insert_counts(keys, c))
        assert first_diff(G.export(), O.export()) is None
    both = np.concatenate([keys, keys])
    G.remove(dev_u64(both))
    O.remove(both)
    assert first_diff(G.export(), O.export()) is None


def test_time_of_counters_of_several_digits(gf):
    """1000 keys into 2^24 slots at 70 % load: counts of 70,000 (six slots a key) in
    less than 2.2 times the time of counts of 1; 2.8 times where regions are as
    large as the keys are apart, so that some of them take several keys in turn."""
    import torch

    base, keys = W.uniform_keys(1, int(0.7 * (1 << 24))), dev_u64(W.uniform_keys(2, 1000))
    G = gf.GQF(24, 8, seed=3, max_batch=len(base))
    G.insert(dev_u64(base))
    image, best = G.export(), {}
    for count in (1, 70_000):
        c, t = counts_of([count], 1000), []
        for _ in range(4):
            G.import_(image)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            G.insert_counts(keys, c)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        best[count] = min(t)
    assert best[70_000] < 2.2 * best[1], best
