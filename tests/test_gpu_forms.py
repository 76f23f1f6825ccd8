"""Which form the comparisons of forms compare.

test_gpu_orbitals.py holds the chain and the block on the orbitals against the general
products at its sizes; that says something only while the rules of the forms take the orbitals
there.  The flops that the library books tell: the block on the orbitals books no exchange
over the kept pairs (sliced, from n = 33 on: n^2 K per tau point for the Gram matrices), and
the chain on the orbitals books 8 n^2 n_v for the transforms of the two factors and 2 n^3 per
tau point, pair and kind, plus 4 n^3 per tau point for the sum's way back."""
import numpy as np
import pytest

from paper_2005_12338_gb300 import synth
from test_gpu_orbitals import BLOCKS, SIZES

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def gflops(s, n_s, eps_prime, eps, dd=0):
    """Booked GFLOP per class of one setup and sampling call."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding as B, build
    build.build()
    h = B.Handle(0)
    o = B.Handle.options(eps_prime, eps, n_s, 6, dd_arith=dd)
    h.setup(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
              (s.eri3, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)],
            n_occ=s.n_occ, mu=s.mu, beta=s.beta, opts=o)
    st = h.sigma(o, torch.empty((s.n_tau, s.n, s.n), dtype=torch.float64, device="cuda"))[2]
    h.close()
    return dict(zip(B.PROF_CLASSES, st["prof_gflop"]))


# (double-float: the rule of fp64, and some of these inputs are out of its range)
@pytest.mark.parametrize("n,n_occ,n_aux", BLOCKS)
@pytest.mark.parametrize("dd", [0, 2], ids=["fp64", "sliced"])
def test_block_on_the_orbitals(n, n_occ, n_aux, dd):
    s = synth.make_system(n, n_occ, n_aux, 8, input_seed=n + 1)
    want = 1e-9 * n * n * n_occ * (n - n_occ) ** 2 * 8 if dd == 2 and n > 32 else 0.0
    assert gflops(s, 4, 0.0, 0.0, dd)["dd_spmm"] == pytest.approx(want, rel=1e-12)


@pytest.mark.parametrize("n,n_occ,n_aux,n_tau", SIZES)
def test_chain_on_the_orbitals(n, n_occ, n_aux, n_tau):
    s = synth.make_system(n, n_occ, n_aux, n_tau, input_seed=n)
    pairs_kinds = 7 * 2
    want = pairs_kinds * (8.0 * n * n * (n - n_occ) + 2.0 * n ** 3 * n_tau) + 4.0 * n ** 3 * n_tau
    assert gflops(s, 7, 0.02, 1e-2)["chain_gemm"] == pytest.approx(1e-9 * want, rel=1e-12)
