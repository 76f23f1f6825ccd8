"""The sliced Gram block over many row tiles and over chunks of tau points.

n = 300, 513 and 900 take 3, 5 and 8 tiles of 128 rows (6, 15 and 36 tiles on and above the
diagonal); at n = 300 the digits of 5 of the 8 tau points fit their buffer, which leaves a
shorter last chunk of 3, and at n = 900 those of one.  One occupied orbital keeps the
contraction short, nothing is cut (P = n^2 pairs, far too many for the contraction over
pairs, so that both arithmetics take the Gram matrix, which the flops booked for each
say too).  The reference is the fp64 Gram matrix, other kernels throughout; the bound on the
left-out digit products, sqrt(K) 2^-46 of the largest element, is taken 8 times."""
import numpy as np
import pytest

from paper_2005_12338_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,n_tau", [(300, 8), (513, 3), (900, 2)])
def test_sliced_gram_over_many_tiles(n, n_tau):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding as B, build
    build.build()
    s = synth.make_system(n, 1, 24, n_tau, input_seed=n)
    arrays = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
              (s.eri3, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)]
    sig = torch.empty((n_tau, n, n), dtype=torch.float64, device="cuda")
    K = (n - 1) ** 2
    spmm = B.PROF_CLASSES.index("dd_spmm")
    out = {}
    for dd, gflop in ((0, 0.0), (2, 1e-9 * n * n * K * n_tau)):
        h = B.Handle(0)
        o = B.Handle.options(0.0, 0.0, 2, 1, dd_arith=dd)
        h.setup(*arrays, n_occ=1, mu=s.mu, beta=s.beta, opts=o)
        _, _, st = h.sigma(o, sig)
        assert st["prof_gflop"][spmm] == pytest.approx(gflop, rel=1e-12)
        out[dd] = h.export("SIGMA_DD").reshape(n_tau, n, n)
        h.close()
    for x, y in zip(out[2], out[0]):
        assert np.abs(x - y).max() <= 8.0 * (n - 1) * 2.0 ** -46 * np.abs(y).max()
