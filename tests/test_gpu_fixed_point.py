"""Theta and P(dt) in double precision, Coulomb and quadratic, whose transforms run in block fixed
point: against the oracle at every N_k, exact under scaling by powers of two, with zero, tiny and
non-finite data.

Tolerance against the oracle: a transform's entries carry 57 bits below the vector's largest
entry and leave it about 3 units of the last one off, i.e. 2^-55; a padded vector's largest entry
is at most 2^2.5 times its root mean square for the seeded data here; three forward and three
inverse passes and the symbol product add up to under 8 2^-52.5 = 1.3e-15, and the oracle's own
FFTs are off by about as much: 1e-14.  The quadratic passes transform each line twice per dimension:
6 2^-54 and the oracle's part stay below it as well."""
import numpy as np
import pytest

from oracle import chasm_oracle as O

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = 1e-14
LO, HI, LK = (-2.0, -1.5, -2.5), (2.5, 1.0, 2.0), 4.0
NUC = [((0.3, -0.2, 0.1), 1.0), ((-0.4, 0.35, 0.6), 0.5)]
GRIDS = [(8, (5, 4, 6)), (16, (4, 5, 4)), (32, (4, 4, 5))]


@pytest.fixture(scope="module")
def ch():
    import paper_2205_02380_gb300 as pkg
    pkg.chasm.lib()
    assert torch.cuda.is_available()
    return pkg


def _solver(ch, nx, nk):
    return ch.Solver(nx, nk, LO, HI, LK, nuclei=NUC, precision=ch.FP64, theta_form=ch.THETA_TABLE)


def _theta(s, u):
    out = torch.empty_like(u)
    s.theta(u, out)
    s.sync()
    return out


def _data(nx, nk, seed):
    return np.random.default_rng(seed).standard_normal(tuple(nx) + (nk,) * 3)


@pytest.mark.parametrize("nk,nx", GRIDS)
def test_theta_and_pflow_match_the_oracle(ch, nk, nx):
    u = _data(nx, nk, nk)
    prob = O.Problem(nx=nx, nk=nk, x_lo=LO, x_hi=HI, lk=LK, nuclei=NUC)
    with _solver(ch, nx, nk) as s:
        d = torch.from_numpy(u).cuda()
        assert O.rel_l2(_theta(s, d).cpu().numpy(), O.theta(u, prob)) <= TOL
        s.pflow(d, 0.02)
        s.sync()
        assert O.rel_l2(d.cpu().numpy(), O.pflow(u, prob, 0.02)) <= TOL


@pytest.mark.parametrize("nk,nx", GRIDS)
@pytest.mark.parametrize("power", [-900, -40, 900])
def test_theta_scales_exactly_with_powers_of_two(ch, nk, nx, power):
    u = torch.from_numpy(_data(nx, nk, 1)).cuda()
    with _solver(ch, nx, nk) as s:
        want = _theta(s, u)
        got = _theta(s, torch.ldexp(u, torch.tensor(power // 2)).ldexp(torch.tensor(power - power // 2)))
        assert torch.equal(got, want.ldexp(torch.tensor(power // 2)).ldexp(torch.tensor(power - power // 2)))


@pytest.mark.parametrize("nk,nx", GRIDS)
def test_zero_lines_and_mixed_magnitudes(ch, nk, nx):
    """Zero data gives zero; an x point whose lines differ by 2^200 is as exact as its largest."""
    u = _data(nx, nk, 2)
    u[0] = 0.0
    u[1, 0, 0, 0] *= 2.0 ** -200
    u[1, 0, 0, 1:] = 0.0
    prob = O.Problem(nx=nx, nk=nk, x_lo=LO, x_hi=HI, lk=LK, nuclei=NUC)
    want = O.theta(u, prob)
    with _solver(ch, nx, nk) as s:
        got = _theta(s, torch.from_numpy(u).cuda()).cpu().numpy()
    assert np.all(got[0] == 0.0)
    for x in ((1, 0, 0), (1, 1, 1)):
        assert O.rel_l2(got[x], want[x]) <= TOL


@pytest.mark.parametrize("nk,nx", GRIDS)
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_a_non_finite_entry_makes_its_x_point_nan_and_no_other(ch, nk, nx, value):
    u = _data(nx, nk, 3)
    with _solver(ch, nx, nk) as s:
        want = _theta(s, torch.from_numpy(u).cuda())
        u[1, 2, 1, 3, 0, 5] = value
        got = _theta(s, torch.from_numpy(u).cuda())
    assert bool(torch.isnan(got[1, 2, 1]).all())
    got[1, 2, 1] = want[1, 2, 1]
    assert torch.equal(got, want)


def _quadratic(ch, nx, nk):
    return ch.Solver(nx, nk, LO, HI, LK, kappa=0.7, precision=ch.FP64)


@pytest.mark.parametrize("nk,nx", GRIDS + [(32, (4, 4, 4)), (8, (7, 4, 9))])
def test_quadratic_shift_and_derivative_match_the_oracle(ch, nk, nx):
    u = _data(nx, nk, nk + 1)
    prob = O.Problem(nx=nx, nk=nk, x_lo=LO, x_hi=HI, lk=LK, kappa=0.7)
    with _quadratic(ch, nx, nk) as s:
        d = torch.from_numpy(u).cuda()
        assert O.rel_l2(_theta(s, d).cpu().numpy(), O.theta(u, prob)) <= TOL
        s.pflow(d, 0.3)
        s.sync()
        assert O.rel_l2(d.cpu().numpy(), O.pflow(u, prob, 0.3)) <= TOL


@pytest.mark.parametrize("nk,nx", GRIDS)
def test_quadratic_lines_keep_their_own_scale(ch, nk, nx):
    """Lines of neighbouring k3 are transformed together in the k1 and k2 passes: every second one
    scaled by 2^300 comes out scaled (compared at the potential's centre in x_3, where k3 is not
    shifted); scaling everything by a power of two is exact."""
    u = torch.from_numpy(_data(nx, nk, 4)).cuda()
    small = u * 2.0 ** -900
    big = u.clone()
    big[..., 1::2] *= 2.0 ** 300
    c3 = (0.0, 0.0, LO[2])   # the first x_3 is the centre
    with ch.Solver(nx, nk, LO, HI, LK, kappa=0.7, center=c3, precision=ch.FP64) as s:
        for f in (u, small, big):
            s.pflow(f, 0.3)
    assert torch.equal(small, u * 2.0 ** -900)
    got, want = big[:, :, 0], u[:, :, 0]
    assert torch.allclose(got[..., 1::2] * 2.0 ** -300, want[..., 1::2], rtol=0, atol=1e-14)


@pytest.mark.parametrize("nk,nx", GRIDS)
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_a_non_finite_entry_of_the_quadratic_passes_stays_in_its_x_point(ch, nk, nx, value):
    u = _data(nx, nk, 5)
    with _quadratic(ch, nx, nk) as s:
        want = torch.from_numpy(u).cuda()
        s.pflow(want, 0.3)
        u[1, 2, 1, 3, 0, 5] = value
        got = torch.from_numpy(u).cuda()
        s.pflow(got, 0.3)
    assert not bool(torch.isfinite(got[1, 2, 1]).any())
    got[1, 2, 1] = want[1, 2, 1]
    assert torch.equal(got, want)
