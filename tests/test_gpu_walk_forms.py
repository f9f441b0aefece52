"""The forms that one walk takes: with and without counters, in groups of 32 sinks that one,
two, four or eight warps share (from the most sinks to the fewest), and over sinks in other
company. A sink's results are its own in every form, bit for bit."""
import numpy as np
import pytest

import workloads
from _parity import gpu_tree, oracle_tree
from test_gpu_termination import _check

pytestmark = pytest.mark.gpu


def _problem(n, s, seed=7):
    P = workloads.uniform_box(n_gas=n, n_src=s, seed=seed)
    rng = np.random.default_rng(seed + 1)
    P["alpha"] = workloads.lognormal_alpha(rng, P["gas_xyz"], 6.0, 1.5, 0.08, n_modes=64)
    return P


@pytest.mark.parametrize("bg_radius", [0.0, 0.45])
@pytest.mark.parametrize("n", [33, 4097, 60000, 120000, 330000])
def test_tau_stop_is_one_walk_with_and_without_counters(n, bg_radius):
    from paper_1902_08083_gb300 import trevr
    if bg_radius:
        P = workloads.background_shell(n_gas=n, n_bg=700, radius=0.45, alpha=8.0)
    else:
        P = _problem(n, 100)
    G = gpu_tree(P)
    kw = dict(bg_radius=bg_radius, tau_stop=2.0)
    f = trevr.compute_flux(G, 0.6, 0.1, **kw)
    fc, c = trevr.compute_flux(G, 0.6, 0.1, counters=True, **kw)
    fs, st = trevr.compute_flux(G, 0.6, 0.1, stats=True, **kw)
    assert np.array_equal(f.cpu().numpy(), fc.cpu().numpy())
    assert np.array_equal(f.cpu().numpy(), fs.cpu().numpy())
    # the walk without a threshold: the same rays, a cut one adds fewer segments
    _, whole, wst = trevr.compute_flux(G, 0.6, 0.1, counters=True, stats=True,
                                       bg_radius=bg_radius)
    c, whole = c.cpu().numpy(), whole.cpu().numpy()
    np.testing.assert_array_equal(c[:, [0, 2]], whole[:, [0, 2]])
    assert np.all(c[:, [1, 3]] <= whole[:, [1, 3]])
    assert st["interactions"] == wst["interactions"] and st["segments"] == int(c[:, 1].sum())
    assert st["refine_expansions"] == int(c[:, 3].sum())
    # a threshold that no ray passes: every number is the complete walk's
    _, c, st = trevr.compute_flux(G, 0.6, 0.1, counters=True, stats=True, bg_radius=bg_radius,
                                  tau_stop=1e30)
    np.testing.assert_array_equal(c.cpu().numpy(), whole)
    assert {k: v for k, v in st.items() if not k.endswith("_ms")} == \
        {k: v for k, v in wst.items() if not k.endswith("_ms")}


@pytest.mark.parametrize("n", [33, 4097, 60000])
def test_tau_stop_without_counters_against_the_oracle(n):
    from paper_1902_08083_gb300 import trevr
    P = _problem(n, 100)
    sinks = np.arange(n) if n < 5000 else workloads.sink_sample(n, 2048, seed=42)
    f = trevr.compute_flux(gpu_tree(P), 0.6, 0.1, tau_stop=2.0).cpu().numpy()[sinks]
    of = oracle_tree(P).flux_terminated(0.6, 0.1, 2.0, sinks=sinks)
    f0 = oracle_tree(dict(P, alpha=np.zeros_like(P["alpha"]))).flux(0.6, 0.1, sinks=sinks)
    _check(f, of, f0, 2.0, f"n={n}")
