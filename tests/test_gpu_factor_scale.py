"""Stochastic factors far from 1, made up for by G.

The double-float chain takes factors and G of magnitudes in [2^-40, 2^40].  With integrals times
2^k and a chemical potential that multiplies G(tau) by 2^-k and G(beta - tau) by 2^k, every
intermediate of the general products stays in fp32's range at k = +-33 (X G Y ~ 2^k, F ~ 2^3k);
the chain on the orbitals, which forms products of four factors before G's magnitude comes in,
must match it as it does at k = 0: 1e-11 relative, as in the other tests of the two forms."""
import numpy as np
import pytest

import oracle as O
from paper_2005_12338_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = 1e-11


@pytest.mark.parametrize("k", [0, 33, -33])
@pytest.mark.parametrize("n,n_occ", [(24, 9), (41, 25)])
def test_forms_agree_on_scaled_factors(n, n_occ, k):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding as B, build
    build.build()
    s = synth.make_system(n, n_occ, 60, 1, input_seed=n)
    mu = s.mu - k * np.log(2.0) / s.tau[0]
    g, gb = O.green(s.orb_e, s.orb_c, n_occ, mu, s.tau[0])
    o = B.Handle.options(0.02, 0.1, 6, 3, precision=B.RSSRI_PREC_DF64)
    h = B.Handle(0)
    h.setup(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
              (s.eri3 * 2.0 ** k, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)],
            n_occ=n_occ, mu=mu, beta=s.beta, opts=o)
    out = []
    for gg in ((None, None), [torch.from_numpy(np.array(x)[None].copy()).cuda() for x in (g, gb)]):
        sig = torch.empty((1, n, n), dtype=torch.float64, device="cuda")
        ep = torch.empty(6, dtype=torch.float64, device="cuda")
        h.sigma(o, sig, ep, g=gg[0], gb=gg[1])
        torch.cuda.synchronize()
        out.append((sig.cpu().numpy()[0], ep.cpu().numpy()))
    h.close()
    (a, ea), (b, eb) = out
    assert np.linalg.norm(a - b) <= TOL * np.linalg.norm(b)
    assert np.abs(ea - eb).max() <= TOL * np.abs(eb).max()
