"""The walk that cuts a ray's pieces from the common ancestor's clip, where the cuts can go
wrong: sinks and sources on the cells' planes and one ulp to either side of them, in domains
whose planes g * h are rounded (sides that are no power of two), rays that lie in a plane,
several sinks at one point, and one-leaf trees. The per-lane walk (variant 1) clips every
cell on its own: both must take the same decisions, and the oracle's.

The fluxes are held to the per-lane walk's. The oracle's are no measure here: where a ray
lies within an ulp of a plane, its FP64 lengths belong to a neighbouring cell's, and the
per-lane walk differs from it as well (by up to 27 %). The two walks add the same fp32
lengths in another order, both compensated, so an optical depth differs by a few ulp of
itself: tau 4 2^-24 < 2e-5 of a flux that fp32 holds (tau < 88)."""
import numpy as np
import pytest

import workloads
from _parity import gpu_tree, oracle_tree

pytestmark = pytest.mark.gpu


def _plane_points(rng, n, side, level):
    """Points on the planes of the level's grid in fp32, a third each one ulp below, on and
    one ulp above, inside [0, side)."""
    g = rng.integers(0, 1 << level, (3, n))
    x = (g * (np.float64(np.float32(side)) / (1 << level))).astype(np.float32)
    step = rng.integers(-1, 2, (3, n))
    x = np.where(step < 0, np.nextafter(x, np.float32(-1)), x)
    x = np.where(step > 0, np.nextafter(x, np.float32(2 * side)), x)
    top = np.nextafter(np.float32(side), np.float32(0))
    return np.clip(x, np.float32(0), top).astype(np.float32)


def _problem(side, level, n=3001, s=61, seed=5):
    rng = np.random.default_rng(seed)
    P = workloads.uniform_box(n_gas=n, n_src=s, seed=seed)
    P["gas_xyz"] = _plane_points(rng, n, side, level)
    P["src_xyz"] = _plane_points(rng, s, side, level)
    P["alpha"] = rng.lognormal(0.0, 1.5, n).astype(np.float32) / np.float32(side)
    P["side"] = float(np.float32(side))
    return P


@pytest.mark.parametrize("theta,tau_ref", [(0.75, 0.1), (0.0, 0.05), (0.9, 0.0)])
@pytest.mark.parametrize("side,level", [(1.0, 4), (0.7, 4), (0.7, 9), (0.3, 6), (3.0, 5)])
def test_points_on_the_planes(side, level, theta, tau_ref):
    from paper_1902_08083_gb300 import trevr
    P = _problem(side, level)
    G = gpu_tree(P)
    n = P["alpha"].shape[0]
    _, rc, _ = oracle_tree(P).flux(theta, tau_ref, with_counters=True)
    f1, c1 = trevr.compute_flux(G, theta, tau_ref, counters=True, walk_variant=1)
    for variant in (2, 3):
        f, c, st = trevr.compute_flux(G, theta, tau_ref, counters=True, stats=True,
                                      walk_variant=variant)
        plain = trevr.compute_flux(G, theta, tau_ref, walk_variant=variant)
        assert np.array_equal(f.cpu().numpy(), plain.cpu().numpy())
        np.testing.assert_allclose(f.cpu().numpy(), f1.cpu().numpy(), rtol=2e-5, atol=1e-30)
        for other in (c1.cpu().numpy(), rc):
            mism = np.count_nonzero(np.any(c.cpu().numpy() != other, axis=1))
            assert mism <= max(1, n // 1000), f"{mism} sinks with other decisions"


@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 33, 129])
def test_few_and_equal_points(n):
    from paper_1902_08083_gb300 import trevr
    P = _problem(0.7, 3, n=n, s=3, seed=n)
    P["gas_xyz"][:, : (n + 1) // 2] = P["gas_xyz"][:, :1]  # equal keys share a leaf
    G = gpu_tree(P)
    _, rc, _ = oracle_tree(P).flux(0.5, 0.01, with_counters=True)
    f1 = trevr.compute_flux(G, 0.5, 0.01, walk_variant=1)
    f, c = trevr.compute_flux(G, 0.5, 0.01, counters=True)
    np.testing.assert_allclose(f.cpu().numpy(), f1.cpu().numpy(), rtol=2e-5, atol=1e-30)
    np.testing.assert_array_equal(c.cpu().numpy(), rc.astype(np.int32))


@pytest.mark.parametrize("n_src", [1, 31, 32, 33, 64, 65, 100])
@pytest.mark.parametrize("n_gas", [5, 600])
def test_many_sources_in_a_leaf(n_gas, n_src):
    # every other source dark, all within one leaf's cell
    from paper_1902_08083_gb300 import trevr
    rng = np.random.default_rng(n_src)
    P = workloads.uniform_box(n_gas=n_gas, n_src=n_src, seed=n_src)
    P["src_xyz"] = (0.3 + 0.004 * rng.random((3, n_src))).astype(np.float32)
    P["src_lum"][1::2] = 0.0
    P["alpha"] = rng.lognormal(0.0, 1.0, n_gas).astype(np.float32)
    G = gpu_tree(P)
    ref, rc, _ = oracle_tree(P).flux(0.3, 0.1, with_counters=True)
    f, c = trevr.compute_flux(G, 0.3, 0.1, counters=True)
    np.testing.assert_array_equal(c.cpu().numpy(), rc.astype(np.int32))
    np.testing.assert_allclose(f.cpu().numpy(), ref, rtol=1e-3)  # the parity tests' bound


def test_stack_limit_counts_dark_cells():
    # sources in one corner: a stack of two entries has no room below the root's children,
    # whether or not their siblings hold light
    from paper_1902_08083_gb300 import trevr
    P = workloads.uniform_box(n_gas=4096, n_src=40, seed=3)
    P["src_xyz"] = (P["src_xyz"] * np.float32(0.1)).astype(np.float32)
    G = gpu_tree(P)
    with pytest.raises(trevr.TrevrError) as ei:
        trevr.compute_flux(G, 0.1, 0.1, stats=True, stack_depth=2)
    assert ei.value.code == 3
    trevr.compute_flux(G, 0.1, 0.1, stats=True)


def test_gradient_of_rays_with_more_segments_than_are_kept():
    # buckets of one and full refinement: rays across the box have some 80 segments, more
    # than the 64 that are kept for the replay, and are traced a second time; the per-lane
    # walk traces every ray twice. Both sum fp32 terms in FP64 and other orders: d(tau)/dq
    # is a sum of ~100 terms of both signs, 100 * 2^-24 = 6e-6 of its largest.
    import torch
    from paper_1902_08083_gb300 import trevr
    P = workloads.uniform_box(n_gas=60000, n_src=8, seed=17, bucket=1)
    P["alpha"] = np.random.default_rng(18).lognormal(0.0, 1.0, 60000).astype(np.float32)
    G = gpu_tree(P)
    sinks = torch.arange(0, 60000, 29, device="cuda")
    g = torch.from_numpy(np.random.default_rng(19).standard_normal(sinks.shape[0])
                         .astype(np.float32)).cuda()
    _, c = trevr.compute_flux(G, 0.75, 0.0, sink_idx=sinks, counters=True)
    assert int((c[:, 1] / c[:, 0].clamp(min=1)).max()) > 64
    want = trevr.compute_flux_backward(G, g, 0.75, 0.0, sink_idx=sinks, walk_variant=1)
    got = trevr.compute_flux_backward(G, g, 0.75, 0.0, sink_idx=sinks)
    for a, b in zip(got, want):
        assert float((a - b).norm() / b.norm()) < 2e-5
        assert float((a - b).abs().max() / b.abs().max()) < 2e-5
