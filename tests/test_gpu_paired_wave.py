"""Single-precision P(dt) and Theta with N_k = 32 where the x points left for the last wave are worked on
by pairs of CTAs: the same bits as one CTA per x point.

Every line and slab goes through the same operations in the same order whichever CTA holds it, so the
outputs are equal bit by bit; spacing and origin are dyadic, so the x points of the grids below
have the same coordinates.  (4, 4, 4) is one partial wave of pairs, (5, 4, 8) and (6, 4, 9) are a full wave
of 152 and 8 or 64 x points by pairs, (4, 4, 9) one partial wave without pairs (144 x points)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

NK, H, LO = 32, 0.25, (-1.0, -0.75, -1.25)
NUC = [((0.3, -0.2, 0.1), 1.0), ((-0.4, 0.35, 0.6), 0.5)]
WHOLE = (6, 4, 9)


@pytest.fixture(scope="module")
def ch():
    import paper_2205_02380_gb300 as pkg
    pkg.chasm.lib()
    assert torch.cuda.is_available()
    return pkg


@pytest.fixture(scope="module")
def data():
    return np.random.default_rng(11).standard_normal(WHOLE + (NK,) * 3).astype(np.float32)


def _run(ch, data, nx, call, first=0):
    """call's outputs at the x points first.. of the whole lattice's first axis, nx of them"""
    lo = (LO[0] + H * first,) + LO[1:]
    hi = tuple(a + H * (n - 1) for a, n in zip(lo, nx))
    with ch.Solver(nx, NK, lo, hi, 4.0, nuclei=NUC, precision=ch.FP32_MIXED, theta_form=ch.THETA_TABLE) as s:
        d = torch.from_numpy(np.ascontiguousarray(data[first:first + nx[0], :nx[1], :nx[2]])).cuda()
        if call == "theta":
            out = torch.empty_like(d)
            s.theta(d, out)
        else:
            out = d
            s.pflow(d, 0.02)
        s.sync()
        return out.cpu().numpy()


@pytest.mark.parametrize("call", ["theta", "pflow"])
@pytest.mark.parametrize("nx", [(4, 4, 4), (5, 4, 8), (6, 4, 9)])
def test_pairs_give_the_same_bits(ch, data, call, nx):
    got = _run(ch, data, nx, call)
    for first in range(0, nx[0], 4):
        n0 = min(4, nx[0] - first)
        ref = _run(ch, data, (4, 4, 9), call, min(first, WHOLE[0] - 4))
        skip = first - min(first, WHOLE[0] - 4)
        assert np.array_equal(got[first:first + n0], ref[skip:skip + n0, :, :nx[2]])
