"""What a product's first call costs.

The fp64 products choose their tile on the first call of a shape by timing six candidates.  A
large product must not be run six times more for that: the candidates take a part of it that
keeps the chip busy.  R = U^T (ij|A) at n = 300 with 512 pairs has 92 million results, five
times that part, so a first call takes about 1 + 6 / 5 times as long as the next one and seven
times if every candidate runs the whole; 4 lies between.  The part leaves nothing behind:
both calls give the same bits.  The shape occurs nowhere else in the suite."""
import numpy as np
import pytest

from paper_2005_12338_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_first_call_of_a_large_product():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding as B, build
    build.build()
    n, ns = 300, 512
    s = synth.make_system(n, 140, 101, 1, input_seed=1)
    o = B.Handle.options(0.02, 0.5, ns, 1, profile=1)
    h = B.Handle(0)
    h.setup(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
              (s.eri3, s.metric, s.orb_e, s.orb_c, s.tau, s.tau_w)],
            n_occ=s.n_occ, mu=s.mu, beta=s.beta, opts=o)
    sig = torch.empty((1, n, n), dtype=torch.float64, device="cuda")
    cls = B.PROF_CLASSES.index("factor_gemm")
    ms, r = [], []
    for _ in range(2):
        ms.append(h.sigma(o, sig)[2]["prof_ms"][cls])
        r.append(h.export("R"))
    h.close()
    assert ms[0] < 4.0 * ms[1], ms
    assert np.array_equal(r[0], r[1])
