"""The GQF merge by entries: tables and statuses equal the oracle's for tiles
of every density, runs that match, split and empty, counters of one to many
digits, tiles whose old slots or new groups exceed the stages, counts beyond
an entry's, and caller-owned images that are not 16-byte aligned."""
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


def dev_u32(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def step(G, O, op, keys):
    st = zeros_u8(len(keys))
    getattr(G, op)(dev_u64(keys), st)
    assert np.array_equal(host(st), getattr(O, op)(keys)), op
    d = first_diff(G.export(), O.export())
    assert d is None, (op, d, G.stats()["status_word"])


@pytest.mark.parametrize("r", [8, 16])
@pytest.mark.parametrize("q,load", [(6, 0.9), (10, 0.5), (11, 0.95), (12, 0.3), (13, 0.98), (17, 0.9)])
def test_merges_equal_oracle(gf, oracle, q, r, load):
    n = int(load * (1 << q))
    keys = W.uniform_keys(500 + q, n)
    half = keys[: n // 2]
    O, G = oracle.GQF(q, r, seed=q), gf.GQF(q, r, seed=q, max_batch=2 * n + 64)
    G.set_tuning(gqf_region_groups=1)
    step(G, O, "insert", half)
    step(G, O, "insert", keys[n // 2:])
    step(G, O, "remove", np.concatenate([keys[::3], W.uniform_keys(501, n // 3)]))
    if load < 0.9:  # matches: counters of 2, then of more
        step(G, O, "insert", half[: n // 4])
        step(G, O, "insert", np.concatenate([half[: n // 8]] * 3 + [keys[n // 2: n // 2 + n // 8]]))
    step(G, O, "remove", np.concatenate([half, half[::2]]))
    step(G, O, "remove", keys)


@pytest.mark.parametrize("r,copies", [(8, 300), (16, 300), (8, 70000)])
def test_tiles_beyond_the_stages(gf, oracle, r, copies):
    q = 12
    keys = W.uniform_keys(77, 1200)
    many = W.uniform_keys(78, 20000) >> np.uint64(40)  # (more groups than a tile stages, before they overflow)
    O, G = oracle.GQF(q, r, seed=5), gf.GQF(q, r, seed=5, max_batch=1 << 20)
    G.set_tuning(gqf_region_groups=1)
    reps = np.repeat(keys, 3) if copies > 1000 else np.repeat(keys, copies)
    step(G, O, "insert", reps)
    if copies > 1000:
        step(G, O, "insert", np.repeat(keys[:10], copies))
    step(G, O, "insert", many)
    step(G, O, "remove", np.concatenate([reps[::2], many[:500]]))


def test_counts_beyond_an_entry(gf, oracle):
    q = 6
    keys = W.uniform_keys(3, 3)
    O, G = oracle.GQF(q, 8, seed=2), gf.GQF(q, 8, seed=2, max_batch=64)
    G.set_tuning(gqf_region_groups=1)
    for k in range(36):  # the largest batch counts: 2^37 after 32 of them
        c = np.array([(1 << 32) - 10, 3, 1], dtype=np.uint32)
        st = zeros_u8(3)
        G.insert_counts(dev_u64(keys), dev_u32(c), st)
        assert np.array_equal(host(st), O.insert_counts(keys, c))
        assert first_diff(G.export(), O.export()) is None, k
    step(G, O, "remove", np.repeat(keys, 5))


@pytest.mark.parametrize("skip", [0, 8])
@pytest.mark.parametrize("r", [8, 16])
def test_images_off_sixteen_bytes(gf, r, skip):
    import torch

    q = 12
    keys = W.uniform_keys(90, 3000)
    G = gf.GQF(q, r, seed=4, max_batch=gf.NOALLOC_MAX_KEYS)
    size = G.export().size
    a, b = (torch.zeros(size + 16, dtype=torch.uint8, device="cuda")[skip:skip + size] for _ in range(2))
    for part in (keys[:1500], keys[1000:]):
        G.insert(dev_u64(part))
        gf.gqf_insert_noalloc(q, r, 4, a, b, dev_u64(part))
        assert np.array_equal(host(b), G.export())
        a, b = b, a
