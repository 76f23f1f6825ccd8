"""Products of more rows than a grid of narrow tiles holds.

[K]^L is one product with a row per kept pair, up to n^2 of them, and a launch has at most
65,535 rows of tiles: 1,048,560 product rows of 16-wide tiles.  n = 1025 with nothing screened
out has 1,050,625.  N_aux = 2 keeps the problem small, and eps = 0.9 the kept pairs few.

Each element of [K]^L is a sum of two products of a metric root that agrees with the
eigen-decomposition's to 1e-11 of its largest element (the bar of the metric tests), so they
agree to a few times that of the largest; elements within that of the cut may fall on either
side of it."""
import numpy as np
import pytest

import oracle as O
from paper_2005_12338_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dd", [0, 1, 2], ids=["fp64", "df64", "sliced"])
def test_more_rows_than_a_grid_of_narrow_tiles(dd):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding as B, build
    build.build()
    n, na, eps = 1025, 2, 0.9
    s = synth.make_system(n, 500, na, 1, input_seed=5)
    kl = s.eri3.reshape(n * n, na) @ O.metric_inv_sqrt(s.metric)
    top = np.abs(kl).max()
    h = B.Handle(0)
    o = B.Handle.options(0.0, eps, 2, 1, dd_arith=dd)
    h.setup(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
              (s.eri3, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)],
            n_occ=s.n_occ, mu=s.mu, beta=s.beta, opts=o)
    got = h.export("K_L").reshape(n * n, na)
    h.close()
    tol = 1e-10 * top
    assert np.abs(got - kl)[np.abs(got) > 0].max() <= tol
    assert np.abs(kl)[got == 0].max() <= eps * top + tol
