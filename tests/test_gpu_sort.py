"""The radix sort at the edges of its forms: one block up to 4096 pairs, tiles of 4096 with
look-back beyond, full and ragged last tiles; keys all different, all equal, few, and clustered
(equal high digits). Keys and order must equal a stable sort's exactly."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


def _points(kind, n):
    rng = np.random.default_rng(n)
    if kind == "equal":
        x = np.full((3, n), 0.3)
    elif kind == "few":
        x = rng.integers(0, 3, (3, n)) * 0.25
    elif kind == "clustered":
        x = 0.7 + 1e-4 * rng.random((3, n))
    else:
        x = rng.random((3, n))
    return np.minimum(x.astype(np.float32), workloads.ONE_BELOW)


@pytest.mark.parametrize("kind", ["uniform", "equal", "few", "clustered"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 256, 4095, 4096, 4097, 8192, 12289, 1 << 20])
def test_keys_and_order_are_the_stable_sorts(n, kind):
    import torch
    from paper_1902_08083_gb300 import trevr
    x = _points(kind, n)
    key = np.asarray(oracle.morton_keys(x, (0.0, 0.0, 0.0), 1.0)).astype(np.uint64)
    order = np.argsort(key, kind="stable")
    keys, perm = trevr.morton_sort_noalloc(torch.from_numpy(x).cuda())
    np.testing.assert_array_equal(keys.cpu().numpy().view(np.uint64), key[order])
    np.testing.assert_array_equal(perm.cpu().numpy(), order.astype(np.int32))
