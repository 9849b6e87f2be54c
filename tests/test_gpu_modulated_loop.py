"""Modulated form in single precision with N_k = 32 on more x points than CTAs: 320 x points go through
the persistent loop of one CTA per SM two or three times, and give the bits of the same x points in
lattices of 128, one per CTA.  Spacing and origin are dyadic, so the parts have the same coordinates;
two nuclei, so that the spectrum scratch is reused within an x point too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

NK, H, LO = 32, 0.25, (-1.0, -0.75, -1.25)
NUC = [((0.3, -0.2, 0.1), 1.0), ((-0.4, 0.35, 0.6), 0.5)]
WHOLE = (10, 4, 8)


@pytest.fixture(scope="module")
def ch():
    import paper_2205_02380_gb300 as pkg
    pkg.chasm.lib()
    assert torch.cuda.is_available()
    return pkg


def _run(ch, part, first, call):
    lo = (LO[0] + H * first,) + LO[1:]
    hi = tuple(a + H * (n - 1) for a, n in zip(lo, part.shape[:3]))
    d = torch.from_numpy(np.ascontiguousarray(part)).cuda()
    out = d if call == "pflow" else torch.empty_like(d)
    with ch.Solver(part.shape[:3], NK, lo, hi, 4.0, nuclei=NUC, precision=ch.FP32_MIXED,
                   theta_form=ch.THETA_MODULATED) as s:
        if call == "pflow":
            s.pflow(d, 0.02)
        else:
            s.theta(d, out)
        s.sync()
    return out.cpu().numpy()


@pytest.mark.parametrize("call", ["theta", "pflow"])
def test_more_x_points_than_ctas_give_the_same_bits(ch, call):
    assert torch.cuda.get_device_properties(0).multi_processor_count < int(np.prod(WHOLE))
    u = np.random.default_rng(9).standard_normal(WHOLE + (NK,) * 3).astype(np.float32)
    got = _run(ch, u, 0, call)
    for first in (0, 4, 6):
        assert np.array_equal(got[first:first + 4], _run(ch, u[first:first + 4], first, call))
