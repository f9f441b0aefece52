"""The radix sort at the edges of its forms: one block up to 4096 pairs, tiles of 2048 with
look-back beyond, of 4096 from 2^18 on, full and ragged last tiles; keys all different, all
equal, few, and clustered (equal high digits). Keys and order must equal a stable sort's exactly. And the walk order of
a sink list: any order and repetition of the caller's indices gives each sink's own result."""
import numpy as np
import pytest

import oracle
import workloads
from _parity import gpu_tree

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
@pytest.mark.parametrize("n", [1, 2, 31, 33, 256, 4095, 4096, 4097, 8192, 12289, 1 << 18, (1 << 18) + 1, 1 << 20])
def test_keys_and_order_are_the_stable_sorts(n, kind):
    import torch
    from paper_1902_08083_gb300 import trevr
    x = _points(kind, n)
    key = np.asarray(oracle.morton_keys(x, (0.0, 0.0, 0.0), 1.0)).astype(np.uint64)
    order = np.argsort(key, kind="stable")
    keys, perm = trevr.morton_sort_noalloc(torch.from_numpy(x).cuda())
    np.testing.assert_array_equal(keys.cpu().numpy().view(np.uint64), key[order])
    np.testing.assert_array_equal(perm.cpu().numpy(), order.astype(np.int32))


@pytest.mark.parametrize("n_src", [1, 3, 40, 700])
@pytest.mark.parametrize("m", [1, 32, 33, 4096, 4097, 9001])
def test_sink_lists_in_any_order(m, n_src):
    import torch
    from paper_1902_08083_gb300 import trevr
    P = workloads.uniform_box(n_gas=6000, n_src=n_src, seed=m)
    rng = np.random.default_rng(m + 1)
    P["alpha"] = rng.lognormal(0.0, 1.0, 6000).astype(np.float32)
    G = gpu_tree(P)
    full, counts = trevr.compute_flux(G, 0.75, 0.1, counters=True)
    idx = torch.from_numpy(rng.integers(0, 6000, m)).cuda()
    f, c = trevr.compute_flux(G, 0.75, 0.1, sink_idx=idx, counters=True)
    # the same rays in the same order; its compensated parts may be dealt out differently
    np.testing.assert_allclose(f.cpu().numpy(), full[idx].cpu().numpy(), rtol=1e-6)
    assert torch.equal(c, counts[idx])
    g = torch.from_numpy(rng.standard_normal(m).astype(np.float32)).cuda()
    whole = torch.zeros(6000, device="cuda").index_add_(0, idx, g)
    want = trevr.compute_flux_backward(G, whole, 0.75, 0.1)
    got = trevr.compute_flux_backward(G, g, 0.75, 0.1, sink_idx=idx)
    for a, b in zip(got, want):  # g is summed in fp32 for a repeated sink
        scale = float(b.abs().max())
        np.testing.assert_allclose(a.cpu().numpy(), b.cpu().numpy(), rtol=2e-5, atol=2e-5 * scale)
    if m > 1:
        idx[m // 2] = 6000  # out of range: reported, and its sink gets zeros
        with pytest.raises(trevr.TrevrError):
            trevr.compute_flux(G, 0.75, 0.1, sink_idx=idx, stats=True)
        out = torch.full((m,), -1.0, device="cuda")
        trevr.compute_flux(G, 0.75, 0.1, sink_idx=idx, out=out)
        with pytest.raises(trevr.TrevrError):
            trevr.check(G)
        assert float(out[m // 2]) == 0.0
        keep = torch.arange(m, device="cuda") != m // 2
        np.testing.assert_allclose(out[keep].cpu().numpy(), full[idx[keep]].cpu().numpy(),
                                   rtol=1e-6)


def test_sources_that_need_more_tiles_than_the_particles():
    # 2^18 + 1 particles sort in 65 tiles, 2^18 sources in 128: the scratch holds either
    from paper_1902_08083_gb300 import trevr
    import torch
    rng = np.random.default_rng(4)
    n, s = (1 << 18) + 1, 1 << 18
    gas = torch.from_numpy(_points("uniform", n)).cuda()
    src = torch.from_numpy(_points("uniform", s)).cuda()
    lum = torch.from_numpy(rng.random(s).astype(np.float32)).cuda()
    tree = trevr.build_tree(gas, torch.ones(n, device="cuda"), src, lum)
    order = tree.export()["src_order"].long()
    assert torch.equal(order.sort().values, torch.arange(s, device="cuda"))
    first = tree.export()["src_first"].long(), tree.export()["src_count"].long()
    assert int(first[1][1]) == s  # the root holds them all
