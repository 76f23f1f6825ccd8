"""The 16- and 24-wide tiles of the setup's products, and the Gram contraction's chunks.

V^{-1/2} and [K]^L come from products of N_aux rows; a small N_aux takes the narrow tiles,
whose edges lie between the sizes here.  V is well conditioned, so that the Newton-Schulz
root is within 1e-11 of the eigen-decomposition's largest element in either arithmetic
(fp64 ~1e-15 and double-float ~1e-13 per product, some tens of products), the bar the
parity tests put on it at larger sizes.
"""
import numpy as np
import pytest

import oracle as O
from paper_2005_12338_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("na", [3, 15, 16, 17, 24, 25, 47, 48, 49, 73, 97])
@pytest.mark.parametrize("dd", [0, 1], ids=["fp64", "df64"])
def test_metric_root_at_tile_edges(na, dd):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding as B, build
    build.build()
    s = synth.make_system(12, 5, na, 2, input_seed=na)
    w = O.metric_inv_sqrt(s.metric)
    kl, _ = O.large_factor(O.screen(s.eri3, 0.02)[0], w, 0.0)
    h = B.Handle(0)
    h.setup(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
              (s.eri3, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)],
            n_occ=s.n_occ, mu=s.mu, beta=s.beta, opts=B.Handle.options(0.02, 0.0, 2, 1, dd_arith=dd))
    assert np.abs(h.export("W").reshape(na, na) - w).max() <= 1e-11 * np.abs(w).max()
    got = h.export("K_L").reshape(12, 12, na)
    assert np.abs(got - kl.reshape(12, 12, na)).max() <= 1e-11 * np.abs(kl).max()
    h.close()
