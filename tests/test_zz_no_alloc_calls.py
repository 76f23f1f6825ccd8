"""rssri_energy_static over changing sizes, and after calls that overlapped.

Its blocks count themselves in static device memory; a call must leave those counters as it
found them, whatever the size of the calls before it, and also when calls overlapped on the
GPU, which the interface forbids and which may spoil those calls alone.  Runs last (file
name), with the other test of the entry point.

The reference is torch's fp64 sum of the same n^2 n_tau products in another order: either sum
is within n^2 n_tau 2^-53 of the products' magnitudes, 3e-11 of them at the largest size here;
random signs leave far less, and the bound taken is 1e-12.
"""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2005_12338_gb300 import binding, build
    build.build()
    return binding.lib()


class Call:
    def __init__(self, n, n_tau, seed):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        kw = dict(dtype=torch.float64, device="cuda", generator=gen)
        self.n, self.n_tau = n, n_tau
        self.x, self.y = torch.randn((n_tau, n, n), **kw), torch.randn((n_tau, n, n), **kw)
        self.w = torch.rand(n_tau, **kw)
        self.e = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
        prod = self.x * self.y.transpose(1, 2)
        self.want = -float((self.w * prod.sum((1, 2))).sum()) / 6.0
        self.tol = 1e-12 * float((self.w * prod.abs().sum((1, 2))).sum()) / 6.0

    def run(self, lib, stream):
        assert lib.rssri_energy_static(self.x.data_ptr(), self.y.data_ptr(), self.w.data_ptr(),
                                       self.n, self.n_tau, 3, self.e.data_ptr(),
                                       C.c_void_p(stream.cuda_stream)) == 0

    def check(self, lib, stream):
        with torch.cuda.stream(stream):
            self.e.fill_(float("nan"))
        self.run(lib, stream)
        stream.synchronize()
        assert abs(float(self.e.item()) - self.want) <= self.tol, (self.n, self.n_tau)


# one block, one per tau point, several per tau point (2 x 2 up to 13 x 13 tiles of 32), the most
# tau points
SIZES = [(1, 1), (31, 7), (33, 2), (65, 45), (400, 8), (40, 32), (3, 4096), (400, 1)]


def test_changing_sizes(lib):
    calls = [Call(n, t, 10 + k) for k, (n, t) in enumerate(SIZES)]
    torch.cuda.synchronize()
    s = torch.cuda.current_stream()
    for c in calls + calls[::-1] + calls[::3]:
        c.check(lib, s)


def test_calls_after_overlapping_ones(lib):
    a, b, c = Call(400, 8, 1), Call(400, 8, 2), Call(300, 11, 3)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    for _ in range(200):
        for call, s in zip((a, b, c), streams):
            call.run(lib, s)
    torch.cuda.synchronize()
    for call in (a, b, c, a, c):
        call.check(lib, streams[0])
