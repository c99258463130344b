"""The unit path of bulk TCF calls (tcf_path TILED): tables and statuses equal
the oracle's at the edges of one and two partition passes, with keys so hot
that their unit or their block exceeds what a CTA sorts, with full tables,
values and groups of uneven members."""
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


def check(G, O, steps, values=None):
    for k, (op, keys) in enumerate(steps):
        st = zeros_u8(len(keys))
        if values and op == "insert":
            import torch

            v = (keys & np.uint64(15)).astype(np.uint8)
            G.insert(dev_u64(keys), st, values=torch.from_numpy(v).cuda())
            want = O.insert(keys, values=v)
        else:
            getattr(G, op)(dev_u64(keys), st)
            want = getattr(O, op)(keys)
        assert np.array_equal(host(st), want), (op, k)
        d = first_diff(G.export(), O.export())
        assert d is None, (op, k, d)
    assert G.stats()["status_word"] in (0, 1 << 4)  # FULL at the most


# units of at most 2048 (or 128, 1024) candidates: 2^9 of them in one pass
@pytest.mark.parametrize("lg,f,n,target", [(12, 16, 2049, 0), (5, 16, 5000, 128), (16, 8, 30_001, 1024),
                                           (20, 16, 512 * 128, 128), (20, 16, 512 * 128 + 1, 128),
                                           (23, 16, 512 * 2048 + 1, 0), (24, 16, 60_001, 0), (22, 8, 700_003, 1024)])
def test_sizes(gf, oracle, lg, f, n, target):
    G, O = gf.TCF(lg, f, seed=lg, max_batch=n), oracle.TCF(lg, f, seed=lg)
    G.set_tuning(tcf_path=gf.TCF_PATH_TILED, tcf_tile_target=target)
    keys = W.uniform_keys(lg, 2 * n)
    check(G, O, [("insert", keys[:n]), ("insert", np.concatenate([keys[n:], keys[:n // 5]])[:n]),
                 ("remove", keys[n // 2: n // 2 + n]), ("remove", keys[: n])])


@pytest.mark.parametrize("f", [16, 8])
@pytest.mark.parametrize("copies", [64, 65, 2500, 3073, 9000])
def test_hot_blocks(gf, oracle, f, copies):
    base = W.uniform_keys(2, 30_000)
    hot = np.concatenate([base, np.repeat(base[7:10], [copies, 40, copies // 2])])
    np.random.default_rng(copies).shuffle(hot)
    G, O = gf.TCF(15, f, seed=4, max_batch=len(hot)), oracle.TCF(15, f, seed=4)
    G.set_tuning(tcf_path=gf.TCF_PATH_TILED)
    check(G, O, [("insert", base[:5000]), ("insert", hot), ("remove", hot[::-1]), ("remove", base[:3000])])


def test_values_and_hot_removes(gf, oracle):
    base = W.uniform_keys(6, 20_000)
    dup = np.concatenate([base, np.repeat(base[:2], 3000)])
    G, O = gf.TCF(15, 16, seed=4, max_batch=len(dup), value_bits=4), oracle.TCF(15, 16, seed=4, value_bits=4)
    G.set_tuning(tcf_path=gf.TCF_PATH_TILED)
    check(G, O, [("insert", base), ("insert", dup[::-1][:9000]), ("remove", dup), ("insert", base[:7000])], values=True)


def test_uneven_group(gf, oracle):
    import torch

    logs, seeds = [14, 6, 16, 9, 15], [1, 2, 3, 4, 5]
    sizes = [int(0.8 * (1 << lg)) for lg in logs]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    keys = W.uniform_keys(9, int(off[-1]))
    G = gf.FilterGroup(gf.FILTER_TCF, logs, 16, seeds, max_total=len(keys))
    G.set_tuning(tcf_path=gf.TCF_PATH_TILED, tcf_tile_target=512)
    refs = [oracle.TCF(lg, 16, seed=s) for lg, s in zip(logs, seeds)]
    for op in ("insert", "remove", "insert"):
        st = zeros_u8(len(keys))
        getattr(G, op)(torch.from_numpy(off).cuda(), dev_u64(keys), st)
        want = [getattr(r, op)(keys[off[m]:off[m + 1]]) for m, r in enumerate(refs)]
        assert np.array_equal(host(st), np.concatenate(want)), op
        for m, r in enumerate(refs):
            assert first_diff(G.export(m), r.export()) is None, (op, m)


@pytest.mark.parametrize("copies", [13, 20])  # rejects of the first phase: below, above a sixteenth of the keys
def test_later_phases_on_a_large_table(gf, oracle, copies):
    base = W.uniform_keys(11, 6000)
    keys = np.repeat(base, copies)
    G, O = gf.TCF(27, 16, seed=1, max_batch=len(keys)), oracle.TCF(27, 16, seed=1)
    for k, (op, ks) in enumerate([("insert", keys), ("remove", np.concatenate([keys[::2], keys[::3]]))]):
        st = zeros_u8(len(ks))
        getattr(G, op)(dev_u64(ks), st)
        assert np.array_equal(host(st), getattr(O, op)(ks)), (op, k)
    assert first_diff(G.export(), O.export()) is None


@pytest.mark.parametrize("lg,n", [(16, 4 * (1 << 12)), (16, 3 * (1 << 12)), (16, 3 * (1 << 12) - 1), (15, 8192)])
def test_auto_calls_leave_the_oracle_table(gf, oracle, lg, n):
    """Around the lines of the automatic choice, and of the one launch of the later phases."""
    keys = W.uniform_keys(lg, int(1.02 * (1 << lg)))
    G, O = gf.TCF(lg, 16, seed=2, max_batch=n), oracle.TCF(lg, 16, seed=2)
    G.set_tuning()
    check(G, O, [("insert", keys[i:i + n]) for i in range(0, len(keys), n)] + [("remove", keys[: n]), ("remove", keys[: n])])


@pytest.mark.parametrize("few", [255, 256, 257])
@pytest.mark.parametrize("f", [16, 8])
def test_few_keys_by_touched_blocks(gf, oracle, f, few):
    """Batches small against the table, every phase by touched blocks; the
    later phases on both sides of what one CTA takes."""
    base, hot = W.uniform_keys(21, 4000), W.uniform_keys(22, 3)
    cap = 3 * (32 if f == 8 else 16) // 4
    G, O = gf.TCF(18, f, seed=3, max_batch=8192), oracle.TCF(18, f, seed=3)
    G.set_tuning()
    # one block's shortcut leaves exactly `few` copies to the second phase
    one = np.concatenate([base, np.repeat(hot[:1], cap + few)])
    check(G, O, [("insert", one), ("insert", np.concatenate([base[:3000], np.repeat(hot, 300)])),
                 ("remove", one[::-1]), ("remove", np.concatenate([base, np.repeat(hot, 200)])), ("insert", base)])


@pytest.mark.parametrize("lg,n,path", [(18, 5000, 0), (18, 1 << 16, 1), (20, 1 << 17, 2)])
def test_calls_captured_in_a_graph(gf, oracle, lg, n, path):
    import torch

    keys = W.uniform_keys(lg, 2 * n)
    G, O = gf.TCF(lg, 16, seed=1, max_batch=n), oracle.TCF(lg, 16, seed=1)
    G.set_tuning(tcf_path=path)
    buf, st = dev_u64(keys[:n]), zeros_u8(n)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graphs = {}
    with torch.cuda.stream(s):
        G.insert(buf, st)  # (outside a capture first: what a call sets up once)
        G.remove(buf, st)
        for op in ("insert", "remove"):
            graphs[op] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graphs[op], stream=s):
                getattr(G, op)(buf, st)
    torch.cuda.synchronize()
    for op, ks in (("insert", keys[:n]), ("insert", keys[n:]), ("insert", keys[:n]), ("remove", keys[n:]), ("remove", keys[n:])):
        buf.copy_(dev_u64(ks))
        graphs[op].replay()
        torch.cuda.synchronize()
        assert np.array_equal(host(st), getattr(O, op)(ks)), op
        assert first_diff(G.export(), O.export()) is None, op
