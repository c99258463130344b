"""TCF group calls whose keys belong to a few members only: tables and statuses
equal the oracle's where the automatic choice leaves the unit path for them
(one and two partition passes, an insert and a remove, the first phase by
touched blocks and over every block), at even calls beside them, and such a
call takes about the time of the per-block path, whatever the members are."""
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


def make(gf, logs, sizes, f=16):
    import torch

    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    G = gf.FilterGroup(gf.FILTER_TCF, logs, f, [m + 1 for m in range(len(logs))], max_total=n)
    G.set_tuning()
    return G, off, torch.from_numpy(off).cuda(), W.uniform_keys(len(logs) + n, n)


# (log2 slots of the members, keys of each): the loaded members' units are
# above what the unit path takes of a group call
CASES = {
    # 2^12 blocks and 3 keys a block: removes go by unit, all keys in one unit
    "remove, one pass": ([14] + [10] * 48, [0] * 40 + [12_300] + [0] * 8, 16),
    "remove, even": ([14] + [10] * 48, [3072] + [192] * 48, 16),
    "remove, 8-bit tags": ([15] + [11] * 48, [0] * 3 + [6500, 6500] + [0] * 44, 8),
    # 2^22 blocks: inserts too
    "one pass": ([22] * 15 + [18] * 16, [0] * 20 + [90_000, 0, 120_000, 90_000, 0, 110_000, 0, 120_000] + [0] * 3, 16),
    "one pass, even": ([22] * 16, [34_000] * 16, 16),
    "two passes, every 32nd member": ([16] * 1024, [37_500 if m % 32 == 3 else 0 for m in range(1024)], 16),
    # 2^23 blocks, more than half a key a block: over every block
    "every block": ([24] * 8, [0, 0, (1 << 22) + 5] + [0] * 5, 16),
}


@pytest.mark.parametrize("case", list(CASES))
def test_tables_equal_oracle(gf, oracle, case):
    logs, sizes, f = CASES[case]
    G, off, off_d, keys = make(gf, logs, sizes, f)
    refs = {m: oracle.TCF(logs[m], f, seed=m + 1) for m in range(len(logs)) if sizes[m]}
    # fresh keys, stored ones again, and a remove of both
    for op, ks in (("insert", keys), ("remove", keys), ("insert", keys[::-1].copy()), ("remove", keys)):
        st = zeros_u8(len(keys))
        getattr(G, op)(off_d, dev_u64(ks), st)
        want = np.concatenate([getattr(r, op)(ks[off[m]:off[m + 1]]) for m, r in refs.items()])
        assert np.array_equal(host(st), want), op
        for m in list(refs)[:6]:
            assert first_diff(G.export(m), refs[m].export()) is None, (op, m)
    empty = [m for m in range(len(logs)) if not sizes[m]][:2]
    assert all(not G.export(m).any() for m in empty)


def test_hot_key_in_an_even_group(gf, oracle):
    """What the offsets do not tell: copies of a key stay with the unit path."""
    logs, sizes, f = CASES["remove, even"]
    G, off, off_d, keys = make(gf, logs, sizes, f)
    keys[:2000] = keys[0]
    refs = [oracle.TCF(lg, f, seed=m + 1) for m, lg in enumerate(logs)]
    for op in ("insert", "remove"):
        st = zeros_u8(len(keys))
        getattr(G, op)(off_d, dev_u64(keys), st)
        want = np.concatenate([getattr(r, op)(keys[off[m]:off[m + 1]]) for m, r in enumerate(refs)])
        assert np.array_equal(host(st), want), op
    assert all(first_diff(G.export(m), r.export()) is None for m, r in enumerate(refs))


def test_uneven_calls_take_the_per_block_time(gf):
    """900,000 keys of one member of 2^20 slots in a group of 2^26: eight units of
    512 hold them all. Within three times the per-block path's time; by unit
    such a call took several hundred times as long."""
    import torch

    G, off, off_d, keys = make(gf, [20] * 64, [0] * 17 + [900_000] + [0] * 46)
    k = dev_u64(keys)

    def best(op):
        t = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            getattr(G, op)(off_d, k)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
            getattr(G, "remove" if op == "insert" else "insert")(off_d, k)
        return min(t)

    times = {}
    for path in (gf.TCF_PATH_AUTO, gf.TCF_PATH_BLOCK):
        G.set_tuning(tcf_path=path)
        G.clear()
        times[path, "insert"] = best("insert")
        G.insert(off_d, k)
        times[path, "remove"] = best("remove")
    for op in ("insert", "remove"):
        assert times[gf.TCF_PATH_AUTO, op] < 3 * times[gf.TCF_PATH_BLOCK, op], (op, times)
