"""LPC1 without a potential: Theta is zero, so a step is the advection by dt, bit by bit (the
predictor and corrector add products with zero), in both precisions and at every N_k."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ch():
    import paper_2205_02380_gb300 as pkg
    pkg.chasm.lib()
    assert torch.cuda.is_available()
    return pkg


@pytest.mark.parametrize("name", ["fp64", "fp32"])
@pytest.mark.parametrize("nk,nx", [(8, (5, 9, 4)), (16, (4, 5, 4)), (32, (4, 4, 5))])
@pytest.mark.parametrize("graphs", [True, False])
def test_a_free_step_is_the_advection(ch, name, nk, nx, graphs):
    rng = np.random.default_rng(nk)
    f = torch.from_numpy(rng.standard_normal(nx + (nk,) * 3)).to(
        "cuda", torch.float64 if name == "fp64" else torch.float32)
    want = f.clone()
    with ch.Solver(nx, nk, -2.0, 2.0, 3.0, integrator=ch.LPC1, use_graphs=graphs,
                   precision=ch.FP64 if name == "fp64" else ch.FP32_MIXED) as s:
        s.step(f, 0.05, 2)
        s.advect(want, 0.05)
        s.advect(want, 0.05)
        s.sync()
    assert torch.equal(f, want)
