"""Single-precision table form with N_k = 16 (its own kernel, two CTAs per SM): every call that reaches
it, on fewer and on more x points than CTAs run at once.

Every x point goes through the same operations whichever CTA does it, so a lattice of 360 x points
(more than two CTAs on each of 152 SMs) gives the bits of its two halves (180); spacing and origin are
dyadic, so the halves' x points have the same coordinates.  Against the oracle: 1e-5 relative L2 as for
every FP32-mixed call of these tests."""
import numpy as np
import pytest

import synth
from oracle import chasm_oracle as O

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

NK, H, LO = 16, 0.25, (-1.0, -0.75, -1.25)
NUC = [((0.3, -0.2, 0.1), 1.0), ((-0.4, 0.35, 0.6), 0.5)]


@pytest.fixture(scope="module")
def ch():
    import paper_2205_02380_gb300 as pkg
    pkg.chasm.lib()
    assert torch.cuda.is_available()
    return pkg


def _solver(ch, nx, lo, **kw):
    hi = tuple(a + H * (n - 1) for a, n in zip(lo, nx))
    return ch.Solver(nx, NK, lo, hi, 4.0, nuclei=NUC, precision=ch.FP32_MIXED, theta_form=ch.THETA_TABLE, **kw)


@pytest.mark.parametrize("call", ["theta", "pflow", "tkm_convolve"])
def test_more_x_points_than_ctas_give_the_same_bits(ch, call):
    nx, half = (10, 4, 9), (5, 4, 9)
    u = np.random.default_rng(7).standard_normal(nx + (NK,) * 3).astype(np.float32)

    def run(part, lo):
        d = torch.from_numpy(np.ascontiguousarray(part)).cuda()
        out = d if call == "pflow" else torch.empty_like(d)
        with _solver(ch, part.shape[:3], lo) as s:
            if call == "pflow":
                s.pflow(d, 0.02)
            else:
                getattr(s, call)(d, out)
            s.sync()
        return out.cpu().numpy()

    got = run(u, LO)
    assert np.array_equal(got[:5], run(u[:5], LO))
    assert np.array_equal(got[5:], run(u[5:], (LO[0] + 5 * H,) + LO[1:]))
    assert half == u[:5].shape[:3]


@pytest.mark.parametrize("nx", [(4, 5, 4), (8, 5, 9)])
def test_lpc1_step_matches_the_oracle(ch, nx):
    hi = tuple(a + H * (n - 1) for a, n in zip(LO, nx))
    prob = O.Problem(nx=nx, nk=NK, x_lo=LO, x_hi=hi, lk=4.0, nuclei=NUC)
    rng = np.random.default_rng(8)
    f = synth.gaussian_packets(nx, NK, LO, hi, 4.0, [synth.packet((0.2, -0.1, 0.0), (0.3, 0.0, -0.2))])
    f = (f + 1e-3 * f.max() * rng.standard_normal(f.shape)).astype(np.float32)
    d = torch.from_numpy(f).cuda()
    with _solver(ch, nx, LO, integrator=ch.LPC1) as s:
        s.step(d, 0.005, 1)
        s.sync()
    want = O.lpc1_step(f.astype(np.float64), prob, 0.005)
    assert O.rel_l2(d.cpu().numpy(), want) <= 1e-5
