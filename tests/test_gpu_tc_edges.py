"""The reduced-precision chains at the edges of the dC / C^L kernel's tiles:
128-row and 128-column tiles, column steps of 32 (bf16) and 16 (tf32), one
more and one less, odd sizes whose fp32 rows are not 16-byte aligned, an odd
number of pairs, and more tau points than one chunk of 12 holds.

The reference is the same chain with the same operand roundings, products in
fp64 rounded to fp32.  The library's fp32 sums differ from that by ~1e-6
relative, so an operand rounds the other way with probability ~1e-6 / u (u =
2^-8, 2^-11) and is then off by u: over the three roundings on the path that
is below 3 u sqrt(1e-6 / u), 2e-4 (bf16) and 7e-5 (tf32) of the summed terms'
norms; a few elements at the small sizes can do worse than that average.  The
tests allow u / 4 of those norms; a misplaced tile, row or step is of order one.
"""
import numpy as np
import pytest

import oracle as O
from paper_2005_12338_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = {1: 2.0 ** -8, 2: 2.0 ** -11}


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding, build
    build.build()
    return binding


def rounded(x, prec):
    """fp32 and then bf16 (nearest even) or tf32 (nearest, ties away), as float64."""
    bits = np.asarray(x, dtype=np.float32).view(np.uint32).astype(np.uint64)
    if prec == 1:
        bits = (bits + 0x7FFF + ((bits >> 16) & 1)) & 0xFFFF0000
    else:
        bits = (bits + 0x1000) & 0xFFFFE000
    return bits.astype(np.uint32).view(np.float32).astype(np.float64)


def f32(x):
    return x.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,n_occ,n_aux,n_tau,n_s", [
    (16, 7, 20, 13, 2), (33, 12, 40, 2, 3), (48, 20, 50, 1, 5), (127, 60, 90, 1, 2),
    (128, 64, 90, 1, 3), (129, 50, 90, 1, 2), (161, 80, 100, 1, 2)])
@pytest.mark.parametrize("prec", [1, 2], ids=["bf16", "tf32"])
def test_chain_at_tile_edges(B, n, n_occ, n_aux, n_tau, n_s, prec):
    s = synth.make_system(n, n_occ, n_aux, n_tau, input_seed=n)
    opts = B.Handle.options(0.02, 0.1, n_s, 17, precision=prec)
    dev = [torch.from_numpy(a).cuda() for a in (s.eri3, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)]
    h = B.Handle(0)
    h.setup(*dev, n_occ=s.n_occ, mu=s.mu, beta=s.beta, opts=opts)
    sig = torch.empty((n_tau, n, n), dtype=torch.float64, device="cuda")
    h.sigma(opts, sig)
    raw = h.export("SIGMA_RAW").reshape(n_tau, n, n)
    sdd = h.export("SIGMA_DD").reshape(n_tau, n, n)
    r = h.export("R").reshape(2, n_s, n, n)
    rl = h.export("R_L").reshape(2, n_s, n, n)
    h.close()
    q = lambda x: rounded(x, prec)
    for t in range(n_tau):
        g, gb = (q(x) for x in O.green(s.orb_e, s.orb_c, s.n_occ, s.mu, s.tau[t]))
        ref, scale = np.zeros((n, n)), 0.0
        for x in range(n_s):
            ps, pl = q(f32(q(r[0, x] - rl[0, x]) @ g)), q(f32(q(rl[0, x]) @ g))
            dc = f32(ps @ q(r[1, x]) + pl @ q(r[1, x] - rl[1, x]))
            cl = f32(pl @ q(rl[1, x]))
            xm, ym = f32(q(dc) @ gb), f32(q(cl) @ gb)
            a = q(f32(2 * np.trace(xm) * np.eye(n)) - xm)
            b = q(f32(2 * np.trace(ym) * np.eye(n)) - ym)
            c, d = q(f32(cl + dc)), q(dc)
            ref += (a @ c + b @ d) / n_s
            scale += (np.linalg.norm(a) * np.linalg.norm(c) +
                      np.linalg.norm(b) * np.linalg.norm(d)) / n_s
        assert np.linalg.norm(raw[t] - sdd[t] - ref) < 0.25 * U[prec] * scale, t
