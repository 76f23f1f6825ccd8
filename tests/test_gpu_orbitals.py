"""The orbital-basis chain against the general one.

rssri_sigma evaluates S8 on the orbitals of the setup's G; rssri_sigma_from_g
given that same G evaluates it with the general products.  Both sum the same
terms in fp64 (or in double-float, ~1e-13 per product), in other orders, so
they agree to rounding: 1e-12 relative per tau point in fp64 (contractions of
at most a few hundred terms, three in a row, ~1e-15 each), 1e-11 in
double-float.  Sizes sit at the edges of the kernels' tiles (24, 32, 40, 48,
64, 100) and at extreme numbers of occupied orbitals.
"""
import numpy as np
import pytest

import oracle as O
from paper_2005_12338_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding, build
    build.build()
    return binding


def both(B, s, opts):
    """(Sigma, pair energies, E_corr) from the orbitals and from the same G given explicitly."""
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
           for a in (s.eri3, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)]
    gs, gbs = zip(*(O.green(s.orb_e, s.orb_c, s.n_occ, s.mu, t) for t in s.tau))
    h = B.Handle(0)
    h.setup(*dev, n_occ=s.n_occ, mu=s.mu, beta=s.beta, opts=opts)
    out = []
    for g in ((None, None), (torch.from_numpy(np.array(gs)).cuda(),
                             torch.from_numpy(np.array(gbs)).cuda())):
        sig = torch.empty((s.n_tau, s.n, s.n), dtype=torch.float64, device="cuda")
        ep = torch.empty(opts.n_s, dtype=torch.float64, device="cuda")
        e, _, _ = h.sigma(opts, sig, ep, g=g[0], gb=g[1])
        torch.cuda.synchronize()
        out.append((sig.cpu().numpy(), ep.cpu().numpy(), e))
    h.close()
    return out


def close(a, b, tol):
    for x, y in zip(a[0], b[0]):
        assert np.linalg.norm(x - y) <= tol * np.linalg.norm(y)
    assert np.abs(a[1] - b[1]).max() <= tol * np.abs(b[1]).max()
    assert abs(a[2] - b[2]) <= tol * abs(b[2])


def out_of_range(s):
    """Whether some G(tau) or G(beta - tau) leaves the range the double-float forms take (a lone
    occupied orbital far below mu does)."""
    m = [np.abs(x).max() for t in s.tau for x in O.green(s.orb_e, s.orb_c, s.n_occ, s.mu, t)]
    return min(m) < 2.0 ** -40 or max(m) > 2.0 ** 40


SIZES = [(2, 1, 3, 2), (24, 12, 30, 5), (25, 24, 31, 4), (33, 1, 40, 3), (40, 13, 50, 4),
         (49, 30, 60, 3), (65, 32, 70, 2), (101, 47, 110, 2)]


@pytest.mark.parametrize("n,n_occ,n_aux,n_tau", SIZES)
@pytest.mark.parametrize("prec", [0, 3], ids=["fp64", "df64"])
def test_orbital_and_general_form_agree(B, n, n_occ, n_aux, n_tau, prec):
    s = synth.make_system(n, n_occ, n_aux, n_tau, input_seed=n)
    refused = prec and out_of_range(s)
    for kw in (dict(), dict(estimator=B.RSSRI_EST_SRI), dict(pair_batch=3)):
        o = B.Handle.options(0.02, 1e-2, 7, 5, precision=prec, dd_arith=1 if prec else 0, **kw)
        if refused:
            with pytest.raises(B.RssriError) as err:
                both(B, s, o)
            assert err.value.code == -9
            continue
        a, b = both(B, s, o)
        close(a, b, 1e-11 if prec else 1e-12)


# The deterministic block as a Gram matrix over (virtual, virtual, occupied)
# triples against the contraction over the kept pairs: nothing cut (eps = eps' =
# 0, P = n^2) and n_tau = 8, so that the orbital form is the cheaper one; numbers of
# virtual orbitals around the packing tiles' 32, one occupied orbital, one virtual, and
# n just above the tensor cores' 128-row tile (a last column tile of 16).  n = 32 and 33: the sliced
# form takes fp64 up to 32.
BLOCKS = [(20, 4, 24), (21, 20, 24), (40, 7, 42), (70, 38, 40), (66, 1, 40), (45, 13, 60),
          (130, 62, 33), (129, 100, 48), (32, 15, 64), (33, 16, 66)]


@pytest.mark.parametrize("n,n_occ,n_aux", BLOCKS)
@pytest.mark.parametrize("dd", [0, 1, 2], ids=["fp64", "df64", "sliced"])
def test_gram_block_equals_the_pair_contraction(B, n, n_occ, n_aux, dd):
    s = synth.make_system(n, n_occ, n_aux, 8, input_seed=n + 1)
    o = B.Handle.options(0.0, 0.0, 4, 6, dd_arith=dd)
    if dd == 1 and out_of_range(s):
        with pytest.raises(B.RssriError) as err:
            both(B, s, o)
        assert err.value.code == -9
        return
    a, b = both(B, s, o)
    # the sliced products: the library's fp64-accuracy bar
    close(a, b, (1e-12, 1e-11, 1e-10)[dd])


def test_orbitals_that_are_not_orthonormal_keep_the_general_form(B):
    """G = -C_v g C_v^T is formed from whatever C is given; an estimate that
    used C^T C = I would be off by the deviation, 1e-6 here."""
    s = synth.make_system(40, 13, 50, 4, input_seed=3)
    rng = np.random.default_rng(4)
    s.orb_c = s.orb_c + 1e-6 * rng.standard_normal(s.orb_c.shape)
    o = B.Handle.options(0.02, 1e-2, 7, 5)
    a, b = both(B, s, o)
    close(a, b, 1e-12)


# Blocks of 16 columns that are small at a tau point have only their leading digits
# multiplied on the tensor cores: at large tau most triples are, so that all levels occur,
# in runs of whatever length, with n below and above one 128-row tile.  A digit product
# that is left out (p + q >= 6) is at most 2^-46 of the product of its rows' maxima, of
# either sign, a handful per term: over the K = n_occ n_virt^2 terms they add up like
# sqrt(K) 2^-46 of the largest element, taken 8 times.
@pytest.mark.parametrize("n,n_occ", [(37, 11), (130, 40)])
def test_gram_levels(B, n, n_occ):
    s = synth.make_system(n, n_occ, 3 * n, 24, input_seed=n)
    tol = 8.0 * n_occ ** 0.5 * (n - n_occ) * 2.0 ** -46
    sig = {}
    for dd in (0, 2):
        h = B.Handle(0)
        o = B.Handle.options(0.0, 0.0, 2, 1, dd_arith=dd)
        h.setup(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
                  (s.eri3, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)],
                n_occ=s.n_occ, mu=s.mu, beta=s.beta, opts=o)
        h.sigma(o, torch.empty((s.n_tau, n, n), dtype=torch.float64, device="cuda"))
        sig[dd] = h.export("SIGMA_DD").reshape(s.n_tau, n, n)
        h.close()
    for x, y in zip(sig[2], sig[0]):
        assert np.abs(x - y).max() <= tol * np.abs(y).max()
