"""The advection at every line length around the edges of the register kernels' length classes and
beyond them, in all three dimensions at once, with short and long stencils, positive and negative
shifts, against the oracle.

Tolerances as everywhere in these tests: 1e-12 relative L2 in double precision; in the
FP32-mixed form 1e-6: three passes with about ten FP32 operations per value each (sqrt(30) 2^-24 =
3e-7), smooth data whose spline coefficients stay within a factor of two of it."""
import numpy as np
import pytest

import synth
from oracle import chasm_oracle as O

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LO, HI, LK, NK = (-3.0, -2.5, -2.0), (2.5, 3.0, 2.8), 3.0, 8


@pytest.fixture(scope="module")
def ch():
    import paper_2205_02380_gb300 as pkg
    pkg.chasm.lib()
    assert torch.cuda.is_available()
    return pkg


def _data(nx, seed):
    rng = np.random.default_rng(seed)
    pk = [synth.packet(rng.uniform(-1, 1, 3), rng.uniform(-1, 1, 3)) for _ in range(2)]
    f = synth.gaussian_packets(nx, NK, LO, HI, LK, pk)
    return f + 1e-3 * f.max() * rng.standard_normal(f.shape)


@pytest.mark.parametrize("name,tol", [("fp64", 1e-12), ("fp32", 1e-6)])
@pytest.mark.parametrize("nx,n_nb,tau", [
    ((4, 5, 7), 20, 0.05), ((8, 9, 15), 5, -0.04), ((16, 17, 6), 30, 0.02), ((23, 4, 25), 20, -0.05),
    ((31, 4, 33), 20, 0.05), ((4, 39, 5), 5, 0.03), ((5, 40, 4), 20, -0.05), ((41, 4, 5), 30, 0.04),
    ((4, 5, 47), 20, 0.05), ((4, 49, 5), 5, -0.03), ((55, 5, 4), 20, 0.05), ((5, 4, 56), 20, -0.04),
    ((4, 57, 4), 20, 0.05), ((63, 4, 4), 5, 0.04), ((4, 4, 65), 20, 0.05)])
def test_advection_matches_the_oracle_at_every_length(ch, name, tol, nx, n_nb, tau):
    f = _data(nx, sum(nx))
    dtype = torch.float64 if name == "fp64" else torch.float32
    d = torch.from_numpy(f).to("cuda", dtype)
    prob = O.Problem(nx=nx, nk=NK, x_lo=LO, x_hi=HI, lk=LK, kappa=1.0, n_nb=n_nb)
    want = O.advect(d.double().cpu().numpy(), prob, tau)
    with ch.Solver(nx, NK, LO, HI, LK, kappa=1.0, n_nb=n_nb,
                   precision=ch.FP64 if name == "fp64" else ch.FP32_MIXED) as s:
        s.advect(d, tau)
        s.sync()
    assert O.rel_l2(d.double().cpu().numpy(), want) <= tol


@pytest.mark.parametrize("nx", [(16, 4, 4), (9, 4, 5)])
def test_fp32_data_at_an_odd_address(ch, nx):
    """f may start at any float: the kernels with 8-byte accesses are not taken then."""
    f = torch.from_numpy(_data(nx, 3)).to("cuda", torch.float32)
    buf = torch.zeros(f.numel() + 1, device="cuda", dtype=torch.float32)
    odd = buf[1:].view(f.shape)
    odd.copy_(f)
    with ch.Solver(nx, NK, LO, HI, LK, kappa=1.0) as s:
        s.advect(f, 0.03)
        s.advect(odd, 0.03)
        s.sync()
    assert O.rel_l2(odd.double().cpu().numpy(), f.double().cpu().numpy()) <= 1e-6
    assert float(buf[0]) == 0.0
