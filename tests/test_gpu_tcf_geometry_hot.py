"""Packed block geometries with blocks that get more candidates than their
lanes stage (a hot key), just as many, and ragged numbers of queries."""
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


@pytest.mark.parametrize("f,B,staged", [(16, 8, 32), (12, 21, 32), (16, 32, 32), (8, 64, 64), (16, 64, 64),
                                        (16, 128, 128)])
def test_hot_blocks_equal_oracle(gf, oracle, f, B, staged):
    lb = (B - 1).bit_length()
    O = oracle.TCF(0, f, seed=3, block_slots=B, log2_blocks=12 - lb)
    G = gf.TCF(12, f, gf.MODE_BULK, seed=3, max_batch=8192, block_slots=B)
    keys = W.uniform_keys(17, 2500)
    hot = np.concatenate([np.repeat(keys[:1], staged), np.repeat(keys[1:2], staged + 1), keys[2:700]])
    for op, batch in [("insert", keys[:1500]), ("insert", hot[::-1]), ("remove", hot), ("insert", keys[1500:]),
                      ("remove", np.repeat(keys[1490:1510], 3)), ("remove", np.repeat(keys[:3], 400))]:
        st = zeros_u8(len(batch))
        getattr(G, op)(dev_u64(batch), st)
        assert np.array_equal(host(st), getattr(O, op)(batch)), op
        d = first_diff(G.export(), O.export())
        assert d is None, (op, d)
    for n in (1, 31, 33, 2499):
        probe = np.concatenate([keys[:n - n // 2], W.uniform_keys(18, n // 2)])
        found = zeros_u8(n)
        G.query(dev_u64(probe), found)
        assert np.array_equal(host(found), O.query(probe))
