"""Orbitals that are far from orthonormal in scale.

G = -C_v exp(-(e_v - mu) tau) C_v^T is all that the deterministic block needs of the orbitals,
so C times 2^70 with the exponentials times 2^-140 (by shifted energies, one tau point) is the
same problem.  It must give the same block in every arithmetic: pairs of floats, which
C^2 ~ 2^140 would overflow, are formed from quantities in their range only.

The exponentials of shifted energies, x + 97, are off by ~97 2^-53 = 1e-14, far below the bar
of 1e-10 of the fp64-accurate forms."""
import numpy as np
import pytest

from paper_2005_12338_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,n_occ", [(24, 9), (40, 13)])
@pytest.mark.parametrize("dd", [0, 1, 2], ids=["fp64", "df64", "sliced"])
def test_block_depends_on_the_orbitals_through_g_alone(n, n_occ, dd):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding as B, build
    build.build()
    s = synth.make_system(n, n_occ, 60, 1, input_seed=3)
    o = B.Handle.options(0.02, 1e-2, 2, 3, dd_arith=dd)
    out = []
    for k in (0, 70):
        e = s.orb_e.copy()
        e[n_occ:] += 2 * k * np.log(2.0) / s.tau[0]
        e[:n_occ] -= 2 * k * np.log(2.0) / s.tau[0]
        h = B.Handle(0)
        h.setup(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
                  (s.eri3, s.metric, e, s.orb_c * 2.0 ** k, s.tau, s.tau_w)],
                n_occ=n_occ, mu=s.mu, beta=s.beta, opts=o)
        out.append(h.export("SIGMA_DD"))
        h.close()
    assert np.abs(out[0]).max() > 0
    assert np.abs(out[1] - out[0]).max() <= 1e-10 * np.abs(out[0]).max()
