"""The sources of a tree: in the order of the first particle of their leaf, as a stable sort of
those leaves gives it, and every cell's range of them. With as many sources as needs more of
the sort's scratch than the particles do (a smaller sort may have more tiles), which a scratch
sized by the particles alone refuses."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,s", [(5, 1), (600, 4096), (4097, 4097), (70000, 12289),
                                 ((1 << 18) + 1, 1 << 18), (20000, (1 << 18) + 1)])
def test_source_order_and_ranges(n, s):
    import torch
    from paper_1902_08083_gb300 import trevr
    P = workloads.uniform_box(n_gas=n, n_src=s, seed=n)
    # half of the sources in a small cube, so that leaves hold many
    P["src_xyz"][:, ::2] = (0.3 + 0.01 * P["src_xyz"][:, ::2]).astype(np.float32)
    t = {k: torch.from_numpy(P[k]).cuda() for k in ("gas_xyz", "alpha", "src_xyz", "src_lum")}
    E = trevr.build_tree(t["gas_xyz"], t["alpha"], t["src_xyz"], t["src_lum"]).export()
    E = {k: v.cpu().numpy() for k, v in E.items()}
    # the leaf of each source, down from the root by the cut planes on the integer grid
    g = np.minimum((P["src_xyz"] * np.float32(2097152.0)).astype(np.int64), 2097151)
    cell = np.ones(s, np.int64)
    child, lo = E["child"], E["glo"].reshape(-1, 3)
    while np.any(child[cell] >= 0):
        inner = child[cell] >= 0
        c = np.where(inner, child[cell], 0)
        ax = np.argmax(lo[c + 1] != lo[c], axis=1)
        up = g[ax, np.arange(s)] >= lo[c + 1, ax]
        cell = np.where(inner, c + up, cell)
    first = E["first"][cell]
    order = np.argsort(first, kind="stable")
    np.testing.assert_array_equal(E["src_order"], order)
    ids = np.arange(1, len(child))
    a = np.searchsorted(first[order], E["first"][ids])
    b = np.searchsorted(first[order], E["first"][ids] + E["count"][ids])
    np.testing.assert_array_equal(E["src_first"][ids], a)
    np.testing.assert_array_equal(E["src_count"][ids], b - a)
