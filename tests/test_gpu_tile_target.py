"""The unit path's target of candidates per unit: the default can be asked for
by its value, the library's bound is the header's, and tables are the same."""
import numpy as np
import pytest

from paper_2212_09005_gb300 import tuning, workloads as W
from gpu_util import dev_u64

pytestmark = pytest.mark.gpu


def test_up_to_the_default():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2212_09005_gb300 as gf

    keys = W.uniform_keys(4, 200_000)
    T = gf.TCF(18, 16, seed=1, max_batch=len(keys))
    images = []
    for target in (0, 128, 2048):
        T.set_tuning(tcf_path=gf.TCF_PATH_TILED, tcf_tile_target=target)
        T.clear()
        T.insert(dev_u64(keys))
        T.remove(dev_u64(keys[::3]))
        images.append(T.export())
    assert all(np.array_equal(images[0], x) for x in images[1:])
    for bad in (127, 2049):
        with pytest.raises(gf.FilterError):
            T.set_tuning(tcf_tile_target=bad)
    assert max(target for _, target in tuning.TCF_CANDIDATES) == 2048
