"""The gradients as vectors against the FP64 adjoint: in norm, where the elementwise bound of
1e-3 is wide. Per ray there are some 35 boundaries and segments. A segment's length in fp32 is
the difference of two numbers near one, good to 35 * 2^-24 = 2e-6 of itself, and a contribution
f carries some ten roundings; the cells' sums are FP64: 1e-5 bounds the absorption's gradient.
The luminosities' has d(tau)/dq, a sum of terms of both signs at the boundaries: 35 * 3 * 2^-24
= 6e-6 of the sum of their sizes, up to some eight times their sum: 5e-5."""
import numpy as np
import pytest

import workloads
from _parity import gpu_tree, oracle_tree

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [1, 3])
@pytest.mark.parametrize("n,s,theta,tau_ref,sigma", [(6000, 80, 0.75, 0.1, 1.0),
                                                    (20000, 300, 0.6, 0.01, 2.0),
                                                    (3000, 20, 0.45, 0.05, 1.5)])
def test_gradients_in_norm(n, s, theta, tau_ref, sigma, variant):
    import torch
    from paper_1902_08083_gb300 import trevr
    P = workloads.uniform_box(n_gas=n, n_src=s, seed=n)
    P["alpha"] = workloads.lognormal_alpha(np.random.default_rng(s), P["gas_xyz"], 1.0, sigma,
                                           0.1, n_modes=64)
    T = oracle_tree(P)
    g = np.random.default_rng(3).standard_normal(n) / T.flux(theta, tau_ref)
    g = g.astype(np.float32)
    want = T.adjoint(theta, tau_ref, g.astype(np.float64))
    got = trevr.compute_flux_backward(gpu_tree(P), torch.from_numpy(g).cuda(), theta, tau_ref,
                                      walk_variant=variant)
    for a, b, bound in zip(got, want, (5e-5, 1e-5)):
        a = a.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(a - b) / np.linalg.norm(b) < bound
