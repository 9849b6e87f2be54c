"""A(tau) in single precision with N_k = 8 and line lengths 4, 8, 12 and 16, whose three passes run in one
launch: against the oracle on mixed lengths, up to the largest grid and just beyond it, with shifts that
differ within a pair of adjacent k.

Tolerance: each pass rounds a value a few times in FP32 (solve and four taps, every factor below 2 in the
norm), 2^-24 each: under 3 x 8 x 2^-24 = 1.4e-6, as for the passes one by one."""
import numpy as np
import pytest

from oracle import chasm_oracle as O

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = 1.5e-6
LO, HI, LK = (-2.0, -1.5, -2.5), (2.5, 1.0, 2.0), 4.0


@pytest.fixture(scope="module")
def ch():
    import paper_2205_02380_gb300 as pkg
    pkg.chasm.lib()
    assert torch.cuda.is_available()
    return pkg


@pytest.mark.parametrize("shift", [0.4, 1.3])
@pytest.mark.parametrize("nx,launches", [((4, 4, 4), 1), ((8, 12, 4), 1), ((4, 8, 16), 1), ((16, 12, 4), 1),
                                         ((12, 8, 8), 1), ((8, 8, 16), 3), ((8, 6, 8), 3), ((20, 4, 8), 3)])
def test_three_passes_in_one_launch(ch, nx, launches, shift):
    """shift: the largest k's foot in cells of the coarsest dimension's spacing (1.3: the integer
    shifts run over -2..1 along it, and change within a pair)"""
    h = [(b - a) / (n - 1) for a, b, n in zip(LO, HI, nx)]
    tau = shift * max(h) / LK if shift < 1 else shift * min(h) / LK
    f = np.random.default_rng(sum(nx)).standard_normal(tuple(nx) + (8,) * 3).astype(np.float32)
    prob = O.Problem(nx=nx, nk=8, x_lo=LO, x_hi=HI, lk=LK, nuclei=[])
    with ch.Solver(nx, 8, LO, HI, LK, precision=ch.FP32_MIXED) as s:
        d = torch.from_numpy(f).cuda()
        c0 = s.launch_count()
        s.advect(d, tau)
        s.sync()
        if shift == 1.3:
            assert s.launch_count() - c0 == launches
        got = d.cpu().numpy()
        want = O.advect(f.astype(np.float64), prob, tau)
        assert O.rel_l2(got, want) <= TOL
        if launches == 1:   # an address of four bytes' alignment goes pass by pass
            buf = torch.empty(f.size + 1, device="cuda")
            e = buf[1:].view(f.shape)
            e.copy_(torch.from_numpy(f))
            c0 = s.launch_count()
            s.advect(e, tau)
            s.sync()
            assert s.launch_count() - c0 == 3
            assert O.rel_l2(e.cpu().numpy(), want) <= TOL
